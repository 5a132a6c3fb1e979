// The 5D-local block descriptor and its derived constants: plain host C++ (no
// CUDA), shared by the kernels, their launchers and the host tests.
#pragma once

#include <cmath>

#define EOFA_MAX_LS 64

// 5D-local operator on each (4D site, component) column over s, per chirality
// h = 0 (P_+, components 0..5) and h = 1 (P_-, components 6..11):
//   u   = B1^{-1} x                   (if inv[h]; else u = x)
//   out = B2 u + sigma[h] w[h] (v[h] . u)   (B2 if fwd[h]; else identity)
//   out = a_out * out + b_in * y      (optional axpy with a second field y)
// with Bk = p I + q L_dir and L_dir the down-shift (dir 0, L_+ shape) or the
// up-shift (dir 1, L_- shape), both with corner -mass.
struct Op5 {
    int inv[2], fwd[2];
    double p1[2], q1[2], p2[2], q2[2];
    int dir1[2], dir2[2];
    double mass;
    double sigma[2];
    const double* w[2];  // device, Ls each
    const double* v[2];
    double a_out, b_in;  // out = a_out * op(x) + b_in * y
    // derived constants of the inverse (filled by op_finalize on the host):
    // mr = -q1/p1, invp = 1/p1, invN = 1/(p1 (1 + mass mr^Ls))
    double mr[2], invp[2], invN[2];
    // the same block without its leading factor (col_lead, dslash_impl.cuh): lead = p2 / p1 (1 / p1
    // without a matrix), ratio = q2 / p2, nrm = 1 / (1 + mass mr^Ls), sigl = sigma / p2; lead 0:
    // no inverse, p2 = 0 or two directions
    double lead[2], ratio[2], nrm[2], sigl[2];
};

// The derived constants of op at Ls slices.  They are formed anew on every call
// (two powers, a few divisions): a block edited after an earlier call never
// keeps the constants of its old coefficients.
inline Op5 op_finalize(Op5 op, int Ls) {
    for (int h = 0; h < 2; h++) {
        if (op.inv[h]) {
            op.mr[h] = -op.q1[h] / op.p1[h];
            op.invp[h] = 1.0 / op.p1[h];
            const double corner = 1.0 + op.mass * std::pow(op.mr[h], Ls);
            op.nrm[h] = 1.0 / corner;
            op.invN[h] = 1.0 / (op.p1[h] * corner);
        } else {
            op.mr[h] = op.invp[h] = op.invN[h] = op.nrm[h] = 0.0;
        }
        op.lead[h] = op.ratio[h] = op.sigl[h] = 0.0;
        if (op.inv[h] && (!op.fwd[h] || (op.p2[h] != 0.0 && op.dir2[h] == op.dir1[h]))) {
            op.lead[h] = (op.fwd[h] ? op.p2[h] : 1.0) * op.invp[h];
            op.ratio[h] = op.fwd[h] ? op.q2[h] / op.p2[h] : 0.0;
            op.sigl[h] = op.fwd[h] ? op.sigma[h] / op.p2[h] : op.sigma[h];
        }
    }
    return op;
}
