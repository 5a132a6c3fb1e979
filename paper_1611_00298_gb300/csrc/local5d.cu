// 5D-local operators (the s-structure of Eq. (3)): bidiagonal-plus-corner
// matrices p + q L and their inverses, applied per 4D site and spin-colour
// component in O(Ls), plus an optional rank-one term and axpy.
//
// L_+ = down-shift with corner -m_f, L_- = L_+^T.  The inverse of
// B = p + q L_+ follows from L_+^Ls = -m_f: with r = q / p,
//   u_0 = [x_0 - m_f sum_{j>=1} (-r)^(Ls-j) x_j] / (p (1 + m_f (-r)^Ls)),
//   u_s = (x_s - q u_{s-1}) / p                 (s = 1 .. Ls-1),
// and the mirror image for L_-.  The Cayley factorisation of Eq. (3) makes
// every block used here (D-tilde, the even-odd diagonal block
// M = (4 - M5) D-tilde + 1 - L, G = M D-tilde^{-1}, G^{-1} = D-tilde M^{-1},
// their transposes, and the EOFA rank-one corrections by Sherman-Morrison)
// a product of at most one such inverse and one such matrix.
//
// Blocks without an inverse (D-tilde, M) are a two-point stencil in s: one
// thread per (site, s) reads its slice and, through L1, the neighbouring one
// of each chirality.  All others, and a stencil that writes its own input (the
// D-tilde^T passes of D_DWF^+), run as the launch of the CG's residual update
// without its update (local5_kernel, dslash_impl.cuh): whole 4D sites staged in
// shared memory, one thread per (site, component) column.
//
// What bounds them: the generic column loops that both kinds ran as before
// reached 0.62 TB/s in FP64 (serial shared-memory steps).  The stencil takes
// 48 to 72 FP64 instructions a site and slice, the columns 3 per real number.
// D_DWF and D_DWF^+ on a 16^3 x 32 x 12 field (8 such passes and 4 hops):
// 9.05 -> 6.74 ms with the hop's own share (4 x 1.61 -> 4 x 1.25 ms).
#include "field.cuh"
#include "fused.h"

namespace {

struct Fwd5 {
    double p[2], q[2];  // out = p x_s + q x_n, n the neighbour of the chirality's direction
    int dir[2];
    double mass, b;
};

__global__ void __launch_bounds__(256) fwd5_kernel(Geom g, Fwd5 o, const double2* __restrict__ x, const double2* y,
                                                   double2* out) {
    const long long n5 = (long long)g.Vh * g.Ls;
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= n5) return;
    const int Ls = g.Ls;
    const long long j = t / Ls;
    const int s = (int)(t - j * Ls);
    const double2* xs = x + j * 12 * Ls;
    double2* os = out + j * 12 * Ls;
#pragma unroll
    for (int h = 0; h < 2; h++) {
        int n;
        double q = o.q[h];
        if (o.dir[h] == 0) {
            n = s - 1;
            if (n < 0) { n = Ls - 1; q *= -o.mass; }
        } else {
            n = s + 1;
            if (n == Ls) { n = 0; q *= -o.mass; }
        }
        double2 a[6], b[6], c[6];
#pragma unroll
        for (int k = 0; k < 6; k++) {
            a[k] = __ldg(xs + (6 * h + k) * Ls + s);
            b[k] = __ldg(xs + (6 * h + k) * Ls + n);
            if (y) c[k] = __ldcs(y + (j * 12 + 6 * h + k) * Ls + s);
        }
#pragma unroll
        for (int k = 0; k < 6; k++) {
            double re = fma(o.p[h], a[k].x, q * b[k].x), im = fma(o.p[h], a[k].y, q * b[k].y);
            if (y) {
                re = fma(o.b, c[k].x, re);
                im = fma(o.b, c[k].y, im);
            }
            os[(6 * h + k) * Ls + s] = make_double2(re, im);
        }
    }
}

}  // namespace

void launch_op5(const eofa_ctx* ctx, int prec, const Op5& op, const void* x, const void* y, void* out,
                cudaStream_t st) {
    const void* yy = op.b_in != 0.0 ? y : nullptr;
    const bool stencil = !op.inv[0] && !op.inv[1] && op.sigma[0] == 0.0 && op.sigma[1] == 0.0;
    // (out = x in place goes through shared memory: the stencil's threads read each other's slices)
    if (prec != P64 || !stencil || x == out) {
        fused_local5(ctx, prec, op, x, nullptr, 0.0, nullptr, 0, 0, nullptr, out, op.a_out, nullptr, 0, st, yy, op.b_in);
        return;
    }
    Fwd5 o;
    for (int h = 0; h < 2; h++) {
        o.p[h] = op.a_out * (op.fwd[h] ? op.p2[h] : 1.0);
        o.q[h] = op.a_out * (op.fwd[h] ? op.q2[h] : 0.0);
        o.dir[h] = op.dir2[h];
    }
    o.mass = op.mass;
    o.b = op.b_in;
    const Geom g = ctx_geom(ctx);
    const long long n5 = (long long)g.Vh * g.Ls;
    prof_begin(ctx, 3 + P64, st, (double)n5 * 192.0 * (yy ? 3.0 : 2.0));
    fwd5_kernel<<<(unsigned)((n5 + 255) / 256), 256, 0, st>>>(g, o, (const double2*)x, (const double2*)yy, (double2*)out);
    EOFA_LAUNCHED();
    prof_end(ctx, st);
}
