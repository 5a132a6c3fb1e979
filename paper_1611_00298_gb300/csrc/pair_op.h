// The 5D-local block as the two-slice kernels apply it (dslash_pair.cuh): plain
// host C++ (no CUDA), shared with the host tests.
#pragma once
#include "op5.h"

namespace dsl {

// B in the form v_s = x_s + mr v_{s-1}, out = c1 v_s + c2 v_{s-1} + w (sig vv . v),
// mirrored in s for the chirality whose shift runs the other way.  On a pair
// (x_0 first in its direction, k the carry):
//   out_0 = c1 x_0 + k0 k,  out_1 = c1 x_1 + k0 x_0 + k1 k.
struct PairOp {
    float mr[2], m2[2], c1[2], k0[2], k1[2], cor[2], sig[2];
    float pw[2][EOFA_MAX_LS / 2];  // mr^(2 i)
};

// factor B as pair_op (dslash_pair.cuh) applies it; false for forms that it does not take: no inverse,
// two directions on one chirality, and a rank-one term on both chiralities (their partial sums share
// one region of shared memory).
// up: direction of the upper chirality that the kernel is built for.
inline bool pair_op_of(const Op5& op, int Ls, bool up, double factor, PairOp& o) {
    if (op.sigma[0] != 0.0 && op.sigma[1] != 0.0) return false;
    for (int h = 0; h < 2; h++) {
        if (!op.inv[h] || (op.fwd[h] && op.dir2[h] != op.dir1[h]) || (op.dir1[h] == 0) != (h == 0 ? up : !up)) return false;
        const double mr = op.mr[h], f = factor * op.invp[h];
        const double c1 = f * (op.fwd[h] ? op.p2[h] : 1.0), c2 = f * (op.fwd[h] ? op.q2[h] : 0.0);
        o.mr[h] = (float)mr;
        o.m2[h] = (float)(mr * mr);
        o.c1[h] = (float)c1;
        o.k0[h] = (float)(c1 * mr + c2);
        o.k1[h] = (float)((c1 * mr + c2) * mr);
        o.cor[h] = (float)(-op.mass * op.nrm[h]);
        o.sig[h] = (float)(op.sigma[h] * f);
        double p = 1.0;
        for (int i = 0; i < Ls / 2; i++, p *= mr * mr) o.pw[h][i] = (float)p;
    }
    return true;
}

}  // namespace dsl
