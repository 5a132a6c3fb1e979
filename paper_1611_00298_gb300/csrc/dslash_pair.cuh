// Even-odd dslash with two s-slices per thread (FP32 arithmetic, FP32 or FP16
// storage, even Ls): out = a (-1/2) B[hop] + b y and the CG epilogues of
// dslash_impl.cuh (the same MODEs and the same Epi).
//
// What bounds the hop: a lane's loads return through the SM's 128 byte / clock
// L1 data path, and the neighbours come from L2 at 12-14 TB/s, of the 20 that a
// resident buffer of this size reads at.  With one slice per thread a
// direction returns 96 bytes of spinor and 72 of link per (site, slice), 43% of
// it the same link sent to all slices of the site again.  Two slices per thread
// send each link once for both (132 bytes instead of 168), and the two slices
// are the two lanes of the f32x2 multiply-adds: the link elements are splatted
// once per direction and 36 f32x2 instructions do the work of 72 per slice,
// with no swaps (74 against 137 million warp instructions, issue 26% of the
// time against 46%).  The spinors of two neighbouring slices are one 32-byte
// load per row of chunks, and those of the next direction are on their way
// while the products of the present one are formed (168 registers, 12 warps an
// SM: as many bytes in flight as 24 warps with one slice each; 128 registers
// and 15 warps measured 5% slower).
//
// B: with mr = -q1 / p1 the inverse's recurrence is v_s = x_s + mr v_{s-1}
// (u = v / p1) and the cyclic corner is v_{-1} = -mass v_{Ls-1}; a thread's
// two slices need only the carry v_{2i-1}.  The threads write the end values
// of their pairs (for zero carry) to shared memory, one thread per (site,
// component) column scans the Ls / 2 of them, closes the corner and leaves
// the carries, and each thread finishes its pair from its registers: half of
// the shared-memory bytes and half of the serial steps of passing the whole
// column through (dslash_impl.cuh).
//
// One slice per thread -> two, one GB300: 24^3 x 64 x 24 FP32 hop 0.660 ->
// 0.585 ms, with G^-1 0.862 -> 0.725 ms, CG iteration 4.95 -> 4.46 ms; FP16
// 0.664 -> 0.588, 0.881 -> 0.673, 4.94 -> 3.98 ms; 16^4 x 16 iteration FP32
// 0.311 -> 0.282, FP16 0.304 -> 0.252 ms; 8^4 x 8 iteration FP32 55.5 -> 50.0
// us.  So every even Ls takes it.
//
// Tried and dropped (24^3 x 64 x 24, FP32 hop): links staged in shared memory
// and splatted there 0.81 ms, or copied one tile ahead with cp.async 0.61-0.65;
// the next tile's neighbour entries and first spinors loaded ahead 0.65-0.69;
// tiles dealt so that each half of the SMs sweeps its own half of t 0.68.  The
// epilogue's first field loaded before the block's barriers spills: with G^-1
// at 24^3 x 32 x 24 0.456 ms instead of 0.366.
#pragma once
#include "dslash_impl.cuh"
#include "mrhs.h"
#include "pair_op.h"

#include <algorithm>
#include <climits>
#include <cmath>

// 96 / (Ls / 2) whole sites a block: all threads at work for Ls 2, 4, 6, 8, 12, 16, 24,
// 32, 48 and 64, at worst 75 of 96 (Ls 50)
#define PAIR_THREADS 96
namespace dsl {
namespace {

__device__ __forceinline__ f2p add2(f2p a, f2p b) {
    f2p r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2p neg1add2(f2p a, f2p b) { return fma2(b, 0xBF800000BF800000ull, a); }  // a - b
__device__ __forceinline__ f2p pack2(float a, float b) {
    f2p r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float lo2(f2p a) { return __uint_as_float((unsigned)a); }
__device__ __forceinline__ float hi2(f2p a) { return __uint_as_float((unsigned)(a >> 32)); }

// ---------------------------------------------------------------- two slices of a field

// 32 bytes: the same 16-byte chunk row of slices 2 sp and 2 sp + 1.  HOP: the
// neighbour spinors of the hop (read by other threads at other times, never
// again by this SM soon: kept out of L1, which then holds the links); else
// streamed fields, some of them updated in place.
template <bool HOP>
__device__ __forceinline__ void ld32(const void* p, unsigned* w) {
    if (HOP)
        asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                     : "l"(p));
    else
        asm volatile("ld.global.L1::no_allocate.L2::evict_first.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                     : "l"(p)
                     : "memory");
}
__device__ __forceinline__ void st32(void* p, const unsigned* w) {
    asm volatile("st.global.L1::no_allocate.L2::evict_first.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p),
                 "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
}

template <int P>
struct Pair;

template <>
struct Pair<P32> {
    static constexpr int NCH = 6;  // chunk rows of a site
    template <bool HOP>
    static __device__ __forceinline__ void load_raw(const void* base, int j, int sp, int Ls, unsigned (*w)[8]) {
        const char* b = (const char*)base + ((long long)j * NCH * Ls + 2 * sp) * 16;
#pragma unroll
        for (int k = 0; k < NCH; k++) ld32<HOP>(b + (long long)k * Ls * 16, w[k]);
    }
    static __device__ __forceinline__ void unpack(const unsigned (*w)[8], cpx<float> (*v)[12]) {
#pragma unroll
        for (int k = 0; k < NCH; k++)
#pragma unroll
            for (int t = 0; t < 2; t++) {
                v[t][2 * k] = mk(__uint_as_float(w[k][4 * t]), __uint_as_float(w[k][4 * t + 1]));
                v[t][2 * k + 1] = mk(__uint_as_float(w[k][4 * t + 2]), __uint_as_float(w[k][4 * t + 3]));
            }
    }
    static __device__ __forceinline__ void load(const void* base, int j, int sp, int Ls, long long, cpx<float> (*v)[12]) {
        unsigned w[NCH][8];
        load_raw<false>(base, j, sp, Ls, w);
        unpack(w, v);
    }
    static __device__ __forceinline__ void store(void* base, int j, int sp, int Ls, long long,
                                                 const cpx<float> (*v)[12]) {
        char* b = (char*)base + ((long long)j * NCH * Ls + 2 * sp) * 16;
#pragma unroll
        for (int k = 0; k < NCH; k++) {
            unsigned w[8];
#pragma unroll
            for (int t = 0; t < 2; t++) {
                w[4 * t] = __float_as_uint(v[t][2 * k].re);
                w[4 * t + 1] = __float_as_uint(v[t][2 * k].im);
                w[4 * t + 2] = __float_as_uint(v[t][2 * k + 1].re);
                w[4 * t + 3] = __float_as_uint(v[t][2 * k + 1].im);
            }
            st32(b + (long long)k * Ls * 16, w);
        }
    }
};

template <>
struct Pair<P16> {
    static constexpr int NCH = 3;
    template <bool HOP>
    static __device__ __forceinline__ void load_raw(const void* base, int j, int sp, int Ls, unsigned (*w)[8]) {
        const char* b = (const char*)base + ((long long)j * NCH * Ls + 2 * sp) * 16;
#pragma unroll
        for (int k = 0; k < NCH; k++) ld32<HOP>(b + (long long)k * Ls * 16, w[k]);
    }
    // the stored (unit-scale) values
    static __device__ __forceinline__ void unpack(const unsigned (*w)[8], cpx<float> (*v)[12]) {
#pragma unroll
        for (int k = 0; k < NCH; k++)
#pragma unroll
            for (int t = 0; t < 2; t++)
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    unsigned u = w[k][4 * t + e];
                    const float2 f = __half22float2(*reinterpret_cast<__half2*>(&u));
                    v[t][4 * k + e] = mk(f.x, f.y);
                }
    }
    static __device__ __forceinline__ const float2* scales(const void* base, int j, int sp, int Ls, long long n5) {
        return reinterpret_cast<const float2*>((const char*)base + n5 * 48 + ((long long)j * Ls + 2 * sp) * 4);
    }
    static __device__ __forceinline__ void load(const void* base, int j, int sp, int Ls, long long n5,
                                                cpx<float> (*v)[12]) {
        unsigned w[NCH][8];
        load_raw<false>(base, j, sp, Ls, w);
        const float2 sc = *scales(base, j, sp, Ls, n5);
        unpack(w, v);
#pragma unroll
        for (int c = 0; c < 12; c++) {
            v[0][c] = sc.x * v[0][c];
            v[1][c] = sc.y * v[1][c];
        }
    }
    static __device__ __forceinline__ void store(void* base, int j, int sp, int Ls, long long n5,
                                                 const cpx<float> (*v)[12]) {
        float m[2], inv[2];
#pragma unroll
        for (int t = 0; t < 2; t++) {
            m[t] = 0.f;
#pragma unroll
            for (int c = 0; c < 12; c++) m[t] = fmaxf(m[t], fmaxf(fabsf(v[t][c].re), fabsf(v[t][c].im)));
            inv[t] = m[t] > 0.f ? 1.f / m[t] : 0.f;
        }
        char* b = (char*)base + ((long long)j * NCH * Ls + 2 * sp) * 16;
#pragma unroll
        for (int k = 0; k < NCH; k++) {
            unsigned w[8];
#pragma unroll
            for (int t = 0; t < 2; t++)
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    __half2 h = __floats2half2_rn(v[t][4 * k + e].re * inv[t], v[t][4 * k + e].im * inv[t]);
                    w[4 * t + e] = *reinterpret_cast<unsigned*>(&h);
                }
            st32(b + (long long)k * Ls * 16, w);
        }
        *const_cast<float2*>(scales(base, j, sp, Ls, n5)) = make_float2(m[0], m[1]);
    }
};

// ---------------------------------------------------------------- hop

// half spinors of both slices, (slice 0, slice 1) in the lanes: real parts hr, imaginary parts hm
template <int MU, int SG>
__device__ __forceinline__ void project_pair(const cpx<float> (*psi)[12], f2p* hr, f2p* hm) {
    cpx<float> a[6], b[6];
    project<MU, SG>(psi[0], a);
    project<MU, SG>(psi[1], b);
#pragma unroll
    for (int c = 0; c < 6; c++) {
        hr[c] = pack2(a[c].re, b[c].re);
        hm[c] = pack2(a[c].im, b[c].im);
    }
}

// mac_row (dslash_impl.cuh) on both slices: row a of V h to the upper spins and through A^+ to the lower
template <int MU, int SG>
__device__ __forceinline__ void mac_row_pair(const cpx<float>* u, int a, const f2p* hr, const f2p* hm, f2p* ar, f2p* ai) {
    f2p wr[2], wi[2];
    f2p ur[3], ui[3], nu[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        ur[k] = splat2(u[k].re);
        ui[k] = splat2(u[k].im);
        nu[k] = splat2(-u[k].im);
    }
#pragma unroll
    for (int q = 0; q < 2; q++) {
        const f2p *x = hr + 3 * q, *y = hm + 3 * q;
        f2p r = mul2(ur[0], x[0]), i = mul2(ur[0], y[0]);
        r = fma2(nu[0], y[0], r);
        i = fma2(ui[0], x[0], i);
#pragma unroll
        for (int k = 1; k < 3; k++) {
            r = fma2(ur[k], x[k], r);
            i = fma2(ur[k], y[k], i);
            r = fma2(nu[k], y[k], r);
            i = fma2(ui[k], x[k], i);
        }
        wr[q] = r;
        wi[q] = i;
    }
    ar[a] = add2(ar[a], wr[0]);
    ai[a] = add2(ai[a], wi[0]);
    ar[3 + a] = add2(ar[3 + a], wr[1]);
    ai[3 + a] = add2(ai[3 + a], wi[1]);
    // lower spins: SG A^+ (w0, w1); (source spin, swap with i, sign) per mu as in mac_row
    constexpr bool sw = MU == 0 || MU == 1;  // lower spin 0 takes w1
    constexpr bool im = MU == 0 || MU == 2;  // times +-i
    const f2p x0r = sw ? wr[1] : wr[0], x0i = sw ? wi[1] : wi[0];
    const f2p x1r = sw ? wr[0] : wr[1], x1i = sw ? wi[0] : wi[1];
    constexpr bool s0 = SG > 0, s1 = (SG > 0) == (MU == 0 || MU == 3);
    if (im) {  // + i x = (-xi, xr)
        ar[6 + a] = s0 ? neg1add2(ar[6 + a], x0i) : add2(ar[6 + a], x0i);
        ai[6 + a] = s0 ? add2(ai[6 + a], x0r) : neg1add2(ai[6 + a], x0r);
        ar[9 + a] = s1 ? neg1add2(ar[9 + a], x1i) : add2(ar[9 + a], x1i);
        ai[9 + a] = s1 ? add2(ai[9 + a], x1r) : neg1add2(ai[9 + a], x1r);
    } else {
        ar[6 + a] = s0 ? add2(ar[6 + a], x0r) : neg1add2(ar[6 + a], x0r);
        ai[6 + a] = s0 ? add2(ai[6 + a], x0i) : neg1add2(ai[6 + a], x0i);
        ar[9 + a] = s1 ? add2(ar[9 + a], x1r) : neg1add2(ar[9 + a], x1r);
        ai[9 + a] = s1 ? add2(ai[9 + a], x1i) : neg1add2(ai[9 + a], x1i);
    }
}

// Direction D (2 mu: forward, 2 mu + 1: backward) from the raw spinors w; the
// loads of direction D + 1 go out between the projection and the products.
template <int P, int DAG, int D>
__device__ __forceinline__ void hop_pair(const Geom& g, int par, int j, const int* ent, int sp, int Ls, long long n5,
                                         const void* in, const void* gauge, unsigned (*w)[8], float2& sc, f2p* ar,
                                         f2p* ai) {
    constexpr int MU = D / 2;
    constexpr int SG = (D % 2 == 0) == (DAG == 1) ? 1 : -1;
    f2p hr[6], hm[6];
    {
        cpx<float> psi[2][12];
        Pair<P>::unpack(w, psi);
        project_pair<MU, SG>(psi, hr, hm);
    }
    if constexpr (P == P16) {
        const f2p s2 = pack2(sc.x, sc.y);
#pragma unroll
        for (int c = 0; c < 6; c++) {
            hr[c] = mul2(s2, hr[c]);
            hm[c] = mul2(s2, hm[c]);
        }
    }
    const int jn = ent[D];
    if constexpr (D < 7) {
        Pair<P>::template load_raw<true>(in, ent[D + 1], sp, Ls, w);
        if constexpr (P == P16) sc = __ldg(Pair<P16>::scales(in, ent[D + 1], sp, Ls, n5));
    }
    const long long lidx =
        D % 2 == 0 ? (long long)((par * 4 + MU) * g.Vh + j) : (long long)(((1 - par) * 4 + MU) * g.Vh + jn);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        cpx<float> u[3];
        link_row<float>(gauge, lidx, a, D % 2 == 1, u);
        mac_row_pair<MU, SG>(u, a, hr, hm, ar, ai);
    }
}

// ---------------------------------------------------------------- 5D-local block on pairs

struct ColumnPlan {
    int lhp;              // stride of a column's carries (odd: conflict-free)
    int carry, dot, sum;  // offsets in 8-byte units: carries, rank-one partial sums (one chirality's: pair_op_of), rank-one sums
    int bytes;
};
inline __host__ __device__ ColumnPlan column_plan(int NS, int Ls) {
    ColumnPlan p;
    p.lhp = (Ls / 2) | 1;
    p.carry = 0;
    p.dot = NS * 12 * p.lhp;
    p.sum = p.dot + NS * 6 * p.lhp;
    p.bytes = (p.sum + NS * 12) * 8;
    return p;
}

__device__ __forceinline__ cpx<float> fma_c(float a, cpx<float> x, cpx<float> y) {
    return mk(fmaf(a, x.re, y.re), fmaf(a, x.im, y.im));
}

// The column pass: carries of one (site, component) column from its pairs' end values.
// UP: s ascending (shift from s - 1).
template <int LH, bool UP, int H>
__device__ __forceinline__ void scan_column(const PairOp& o, int lh, cpx<float>* e, const cpx<float>* dp, const float* vv,
                                            cpx<float>* sum) {
    const int n = LH > 0 ? LH : lh;
    const float m2 = o.m2[H], mr = o.mr[H];
    const bool r1 = o.sig[H] != 0.f;
    cpx<float> P = mk(0.f, 0.f), d = mk(0.f, 0.f);
    // P_{i+1} = e_i + m2 P_i; P_i is the carry into pair i for an open start
    if constexpr (LH > 0) {
        cpx<float> c[LH];
#pragma unroll
        for (int i = 0; i < LH; i++) c[i] = lds(e + (UP ? i : LH - 1 - i));
#pragma unroll
        for (int i = 0; i < LH; i++) {
            const cpx<float> x = c[i];
            c[i] = P;
            P = fma_c(m2, P, x);
        }
        const cpx<float> t = o.cor[H] * P;  // v_{-1} of the cyclic corner
#pragma unroll
        for (int i = 0; i < LH; i++) {
            c[i] = fma_c(o.pw[H][i], t, c[i]);
            sts(e + (UP ? i : LH - 1 - i), c[i]);
        }
        if (r1) {
#pragma unroll
            for (int i = 0; i < LH; i++) {
                const int q = UP ? i : LH - 1 - i;
                d = fma_c(fmaf(vv[UP ? 2 * q + 1 : 2 * q], m2, vv[UP ? 2 * q : 2 * q + 1] * mr), c[i], d + lds(dp + q));
            }
        }
    } else {
        for (int i = 0; i < n; i++) {
            const int q = UP ? i : n - 1 - i;
            const cpx<float> x = lds(e + q);
            sts(e + q, P);
            P = fma_c(m2, P, x);
        }
        cpx<float> t = o.cor[H] * P;
        for (int i = 0; i < n; i++) {
            const int q = UP ? i : n - 1 - i;
            const cpx<float> c = lds(e + q) + t;
            sts(e + q, c);
            t = m2 * t;
            if (r1)
                d = fma_c(fmaf(vv[UP ? 2 * q + 1 : 2 * q], m2, vv[UP ? 2 * q : 2 * q + 1] * mr), c, d + lds(dp + q));
        }
    }
    if (r1) sts(sum, o.sig[H] * d);
}

// the pairs' end values of one chirality (and its rank-one partial sums) to shared memory
template <bool UP, int H>
__device__ __forceinline__ void pair_ends(const PairOp& o, const ColumnPlan& pl, int Ls, int ls, int sp, cpx<float>* sm,
                                          const float* wv, const cpx<float> (*v)[12]) {
    const float mr = o.mr[H];
#pragma unroll
    for (int c = 6 * H; c < 6 * H + 6; c++)
        sts(sm + pl.carry + (ls * 12 + c) * pl.lhp + sp, fma_c(mr, v[UP ? 0 : 1][c], v[UP ? 1 : 0][c]));
    if (o.sig[H] != 0.f) {
        const float* vv = wv + (2 * H + 1) * Ls;
        const float vf = vv[UP ? 2 * sp : 2 * sp + 1], vs = vv[UP ? 2 * sp + 1 : 2 * sp];
        const float vfm = fmaf(vs, mr, vf);  // vf x_0 + vs (x_1 + mr x_0)
#pragma unroll
        for (int c = 0; c < 6; c++)
            sts(sm + pl.dot + (ls * 6 + c) * pl.lhp + sp, fma_c(vfm, v[UP ? 0 : 1][6 * H + c], vs * v[UP ? 1 : 0][6 * H + c]));
    }
}

template <bool UP, int H>
__device__ __forceinline__ void pair_finish(const PairOp& o, const ColumnPlan& pl, int Ls, int ls, int sp,
                                            const cpx<float>* sm, const float* wv, cpx<float> (*v)[12]) {
    const float c1 = o.c1[H], k0 = o.k0[H], k1 = o.k1[H];
    const bool r1 = o.sig[H] != 0.f;
    const float w0 = r1 ? wv[2 * H * Ls + 2 * sp] : 0.f, w1 = r1 ? wv[2 * H * Ls + 2 * sp + 1] : 0.f;
#pragma unroll
    for (int c = 6 * H; c < 6 * H + 6; c++) {
        const cpx<float> k = lds(sm + pl.carry + (ls * 12 + c) * pl.lhp + sp);
        const cpx<float> x0 = v[UP ? 0 : 1][c], x1 = v[UP ? 1 : 0][c];
        v[UP ? 0 : 1][c] = fma_c(k0, k, c1 * x0);
        v[UP ? 1 : 0][c] = fma_c(k1, k, fma_c(k0, x0, c1 * x1));
        if (r1) {
            const cpx<float> d = lds(sm + pl.sum + ls * 12 + c);
            v[0][c] = fma_c(w0, d, v[0][c]);
            v[1][c] = fma_c(w1, d, v[1][c]);
        }
    }
}

// out = B x on the pairs of a tile; x, out in v (both slices of the thread's site ls, pair sp).
// UP: direction of the upper chirality, the lower one runs the other way.
// wv: the rank-one vectors [h][w, vv][s] (stage_wv).  Every thread of the block calls it.
template <int LH, bool UP>
__device__ __forceinline__ void pair_op(const PairOp& o, int NS, int nsites, int ls, int sp, int lh, bool ok,
                                        unsigned char* smraw, const float* wv, cpx<float> (*v)[12]) {
    const int LHn = LH > 0 ? LH : lh, Ls = 2 * LHn;
    const ColumnPlan pl = column_plan(NS, Ls);
    cpx<float>* sm = reinterpret_cast<cpx<float>*>(smraw);
    if (ok) {
        pair_ends<UP, 0>(o, pl, Ls, ls, sp, sm, wv, v);
        pair_ends<!UP, 1>(o, pl, Ls, ls, sp, sm, wv, v);
    }
    __syncthreads();
    // half of the threads take the columns of each chirality
    const int half = blockDim.x / 2, hh = threadIdx.x >= half;
    for (int idx = threadIdx.x - hh * half; idx < nsites * 6; idx += half) {
        const int site = idx / 6, c = idx - site * 6;
        cpx<float>* e = sm + pl.carry + (site * 12 + 6 * hh + c) * pl.lhp;
        const cpx<float>* dp = sm + pl.dot + idx * pl.lhp;
        cpx<float>* sum = sm + pl.sum + site * 12 + 6 * hh + c;
        if (hh) scan_column<LH, !UP, 1>(o, lh, e, dp, wv + 3 * Ls, sum);
        else scan_column<LH, UP, 0>(o, lh, e, dp, wv + Ls, sum);
    }
    __syncthreads();
    if (ok) {
        pair_finish<UP, 0>(o, pl, Ls, ls, sp, sm, wv, v);
        pair_finish<!UP, 1>(o, pl, Ls, ls, sp, sm, wv, v);
    }
}

// ---------------------------------------------------------------- kernel

// the outputs beside the first, as in Epi
struct EpiPair {
    void* out2;
    const void* aux;
    void* out3;
    const void* aux2;
    int it, slot2;
};

// Sweep order: z in n blocks, each swept along t before the next (tiles: the
// tiles of one block's slab of a time slice).
struct ZBlocks {
    int n, tiles;
};

// One launch of one system.  r1, r2: the blocks whose rank-one vectors go with op, op2.
template <int P, int DAG, int LS, bool HASOP, int MODE>
__device__ __forceinline__ void pair_body(const Geom& g, int par, const void* __restrict__ in, void* out,
                                          const void* __restrict__ gauge, const PairOp& op, const Op5& r1,
                                          const PairOp& op2, const Op5& r2, const void* y, float a_out, float b_in,
                                          double* red, int slot, int NS, const ZBlocks& zb, const EpiPair& ep) {
    extern __shared__ __align__(128) unsigned char smraw[];
    constexpr int LH = LS / 2;
    const int Ls = LS > 0 ? LS : g.Ls, lh = Ls / 2;
    __shared__ float wv_s[HASOP ? 4 * EOFA_MAX_LS : 1];
    __shared__ float wv2_s[MODE == 1 ? 4 * EOFA_MAX_LS : 1];
    if (HASOP) stage_wv<float>(r1, Ls, wv_s);
    if (MODE == 1) stage_wv<float>(r2, Ls, wv2_s);
    if (HASOP || MODE == 1) __syncthreads();
    const float cz = MODE == 2 ? (float)(-cg_alpha(red, ep.it)) : 0.f;
    const float ax = MODE == 3 ? (float)cg_alpha(red, ep.it) : 0.f;
    const long long n5 = (long long)g.Vh * Ls;
    const int ls = threadIdx.x / lh, sp = threadIdx.x - ls * lh;
    const int ntiles = (g.Vh + NS - 1) / NS;
    const int* nb = par ? g.nbr[1] : g.nbr[0];
    double nacc = 0.0, nacc2 = 0.0;
    for (int it = blockIdx.x; it < ntiles; it += gridDim.x) {
        int tile = it;
        if (zb.n > 1) {  // block of z, then t, then the tiles of the block's slab
            const int b = it / (zb.tiles * g.T), r = it - b * (zb.tiles * g.T), t = r / zb.tiles;
            tile = (t * zb.n + b) * zb.tiles + (r - t * zb.tiles);
        }
        const int j = tile * NS + ls;
        const bool ok = ls < NS && j < g.Vh;
        cpx<float> v[2][12];
        if (ok) {
            f2p ar[12], ai[12];
#pragma unroll
            for (int c = 0; c < 12; c++) ar[c] = ai[c] = 0ull;
            int ent[8];
#pragma unroll
            for (int d = 0; d < 8; d++) ent[d] = __ldg(nb + d * g.Vh + j);
            unsigned w[Pair<P>::NCH][8];
            float2 sc = make_float2(1.f, 1.f);
            Pair<P>::template load_raw<true>(in, ent[0], sp, Ls, w);
            if constexpr (P == P16) sc = __ldg(Pair<P16>::scales(in, ent[0], sp, Ls, n5));
            hop_pair<P, DAG, 0>(g, par, j, ent, sp, Ls, n5, in, gauge, w, sc, ar, ai);
            hop_pair<P, DAG, 1>(g, par, j, ent, sp, Ls, n5, in, gauge, w, sc, ar, ai);
            hop_pair<P, DAG, 2>(g, par, j, ent, sp, Ls, n5, in, gauge, w, sc, ar, ai);
            hop_pair<P, DAG, 3>(g, par, j, ent, sp, Ls, n5, in, gauge, w, sc, ar, ai);
            hop_pair<P, DAG, 4>(g, par, j, ent, sp, Ls, n5, in, gauge, w, sc, ar, ai);
            hop_pair<P, DAG, 5>(g, par, j, ent, sp, Ls, n5, in, gauge, w, sc, ar, ai);
            hop_pair<P, DAG, 6>(g, par, j, ent, sp, Ls, n5, in, gauge, w, sc, ar, ai);
            hop_pair<P, DAG, 7>(g, par, j, ent, sp, Ls, n5, in, gauge, w, sc, ar, ai);
#pragma unroll
            for (int c = 0; c < 12; c++) {
                v[0][c] = mk(lo2(ar[c]), lo2(ai[c]));
                v[1][c] = mk(hi2(ar[c]), hi2(ai[c]));
            }
        }
        const int nsites = min(NS, g.Vh - tile * NS);
        if (HASOP) pair_op<LH, DAG == 0>(op, NS, nsites, ls, sp, lh, ok, smraw, wv_s, v);
        if (ok) {
            if (!HASOP) {  // (a block's constants carry the factor)
                const float scale = -0.5f * a_out;
#pragma unroll
                for (int t = 0; t < 2; t++)
#pragma unroll
                    for (int c = 0; c < 12; c++) v[t][c] = scale * v[t][c];
            }
            if (y != nullptr) {
                cpx<float> yv[2][12];
                Pair<P>::load(y, j, sp, Ls, n5, yv);
#pragma unroll
                for (int t = 0; t < 2; t++)
#pragma unroll
                    for (int c = 0; c < 12; c++) v[t][c] = v[t][c] + b_in * yv[t][c];
                if (MODE == 2 && ep.out2 != nullptr) {
                    cpx<float> rv[2][12];
                    Pair<P>::load(ep.out2, j, sp, Ls, n5, rv);
#pragma unroll
                    for (int t = 0; t < 2; t++) {
#pragma unroll
                        for (int c = 0; c < 12; c++) rv[t][c] = rv[t][c] + cz * yv[t][c];
                        nacc2 += site_norm2<float>(rv[t]);
                    }
                    Pair<P>::store(ep.out2, j, sp, Ls, n5, rv);
                }
            }
            if (MODE == 2) {
                cpx<float> zv[2][12];
                Pair<P>::load(out, j, sp, Ls, n5, zv);
#pragma unroll
                for (int t = 0; t < 2; t++)
#pragma unroll
                    for (int c = 0; c < 12; c++) v[t][c] = zv[t][c] + cz * v[t][c];
            }
            Pair<P>::store(out, j, sp, Ls, n5, v);
            if (red && slot >= 0) nacc += site_norm2<float>(v[0]) + site_norm2<float>(v[1]);
            if (MODE == 3) {
                cpx<float> pv[2][12], xv[2][12];
                Pair<P>::load(ep.aux, j, sp, Ls, n5, pv);
                Pair<P32>::load(ep.out2, j, sp, Ls, n5, xv);
#pragma unroll
                for (int t = 0; t < 2; t++)
#pragma unroll
                    for (int c = 0; c < 12; c++) xv[t][c] = xv[t][c] + ax * pv[t][c];
                Pair<P32>::store(ep.out2, j, sp, Ls, n5, xv);
                if (ep.out3 != nullptr) {
                    Pair<P>::load(ep.aux2, j, sp, Ls, n5, pv);
                    Pair<P>::load(ep.out3, j, sp, Ls, n5, xv);
#pragma unroll
                    for (int t = 0; t < 2; t++) {
#pragma unroll
                        for (int c = 0; c < 12; c++) xv[t][c] = xv[t][c] - ax * pv[t][c];
                        nacc2 += site_norm2<float>(xv[t]);
                    }
                    Pair<P>::store(ep.out3, j, sp, Ls, n5, xv);
                }
            }
        }
        if (MODE == 1) {
            __syncthreads();  // the first block's carries are still being read
            pair_op<LH, DAG != 0>(op2, NS, nsites, ls, sp, lh, ok, smraw, wv2_s, v);
            if (ok) Pair<P>::store(ep.out2, j, sp, Ls, n5, v);
        }
        if (HASOP) __syncthreads();
    }
    if (MODE == 3) {
        if (ep.out3 != nullptr) grid_sum(nacc2, red, ep.slot2);
    } else if (red && slot >= 0) {
        if (MODE == 2 && ep.out2 != nullptr) grid_sum2(nacc, nacc2, red, slot, ep.slot2);
        else grid_sum(nacc, red, slot);
    }
}

template <int P, int DAG, int LS, bool HASOP, int MODE>
__global__ void __launch_bounds__(PAIR_THREADS, 4)
    dslash_pair_kernel(Geom g, int par, const void* __restrict__ in, void* out, const void* __restrict__ gauge, PairOp op,
                       Op5 r1, PairOp op2, Op5 r2, const void* y, float a_out, float b_in, double* red, int slot, int NS,
                       ZBlocks zb, EpiPair ep) {
    chain_wait();
    pair_body<P, DAG, LS, HASOP, MODE>(g, par, in, out, gauge, op, r1, op2, r2, y, a_out, b_in, red, slot, NS, zb,
                                              ep);
}

// The same launch for several systems on one lattice: system blockIdx.y, its
// fields and scratch in a, its blocks in ops, ops2 (and r1, r2).
template <int P, int DAG, int LS, bool HASOP, int MODE>
__global__ void __launch_bounds__(PAIR_THREADS, 4)
    mr_pair_kernel(Geom g, int par, MRPtrs a, const void* __restrict__ gauge, const PairOp* __restrict__ ops,
                   const Op5* __restrict__ r1, const PairOp* __restrict__ ops2, const Op5* __restrict__ r2, float a_out,
                   float b_in, int slot, int NS, ZBlocks zb, int it, int slot2) {
    const int r = blockIdx.y;
    __shared__ PairOp op_s, op2_s;
    if (HASOP) {
        for (int i = threadIdx.x; i < (int)(sizeof(PairOp) / 4); i += blockDim.x) {
            reinterpret_cast<unsigned*>(&op_s)[i] = reinterpret_cast<const unsigned*>(ops + r)[i];
            if (MODE == 1) reinterpret_cast<unsigned*>(&op2_s)[i] = reinterpret_cast<const unsigned*>(ops2 + r)[i];
        }
        __syncthreads();
    }
    EpiPair ep = {a.out2[r], nullptr, nullptr, nullptr, it, slot2};
    pair_body<P, DAG, LS, HASOP, MODE>(g, par, a.in[r], a.out[r], gauge, op_s, r1[r], op2_s, r2[r], a.y[r], a_out, b_in,
                                       a.red[r], slot, NS, zb, ep);
}

// ---------------------------------------------------------------- launch

// A neighbour slab is fetched for t + 1 and used again for t and t - 1: three
// slabs and the output have to stay in the L2 of a die (half of 126 MB, both
// dies read most lines).  Slabs of up to 10 MB do; larger time slices are swept
// in blocks of z.  24^3 x 64 x 24, hop: FP32, 15.9 MB a slice, 0.594 ms
// unblocked, 0.574 in two blocks, 0.579 in three, 0.594 in six; FP16, 8.6 MB,
// 0.588 ms unblocked, 0.599 in two.  A block's slab has to hold whole tiles:
// where no count of blocks divides it so (32^3 x Ls 16: tiles of 12 sites, slabs
// of 16384; most Ls that are no divisor of 192) the sweep stays unblocked.
inline ZBlocks z_blocks(const Geom& g, int NS, int spinor) {
    const long long slice = (long long)(g.X / 2) * g.Y * g.Z;
    ZBlocks z = {1, 0};
    for (int n = 1; n <= g.Z / 2; n++) {
        if (g.Z % n || (slice / n) % NS) continue;
        z.n = n;
        z.tiles = (int)(slice / n / NS);
        if (slice / n * g.Ls * spinor <= (10LL << 20)) return z;
    }
    return ZBlocks{1, 0};
}

// block shape of a launch: sites, threads, dynamic shared memory
struct PairShape {
    int NS, threads;
    size_t smem;
};
inline PairShape pair_shape(int Ls, bool hasop) {
    PairShape p;
    p.threads = PAIR_THREADS;
    p.NS = PAIR_THREADS / (Ls / 2);
    p.smem = hasop ? column_plan(p.NS, Ls).bytes : 0;
    return p;
}

template <int P, int DAG, int LS, bool HASOP, int MODE>
void launch_pair(const eofa_ctx* ctx, int par, const PairArgs& a, const PairOp& o, const PairOp& o2, const EpiPair& e,
                 cudaStream_t st) {
    Geom g = ctx_geom(ctx);
    const PairShape s = pair_shape(g.Ls, HASOP);
    auto k = dslash_pair_kernel<P, DAG, LS, HASOP, MODE>;
    const int ntiles = (g.Vh + s.NS - 1) / s.NS;
    const unsigned grid = grid_size(k, s.threads, s.smem, ntiles, ctx->sms);
    launch_chained(chain_pays(CHAIN_PAIR, grid, (int)grid == ntiles, ctx->sms), k, grid, s.threads, s.smem, st, g, par, a.in,
                   a.out, (const void*)ctx->gauge[P32], o, a.op ? *a.op : Op5(), o2, a.op2 ? *a.op2 : Op5(), a.y,
                   (float)a.a_out, (float)a.b_in, a.red, a.slot, s.NS, z_blocks(g, s.NS, P == P16 ? 52 : 96), e);
    EOFA_LAUNCHED();
}

template <int P, int LS>
void launch_pair_ls(const eofa_ctx* ctx, int par, int dag, const PairArgs& a, const PairOp& o, const PairOp& o2,
                    const EpiPair& e, cudaStream_t st) {
    if (a.mode == 1) launch_pair<P, 0, LS, true, 1>(ctx, par, a, o, o2, e, st);
    else if (a.mode == 2) launch_pair<P, 1, LS, false, 2>(ctx, par, a, o, o2, e, st);
    else if (a.mode == 3) launch_pair<P, 1, LS, true, 3>(ctx, par, a, o, o2, e, st);
    else if (a.op && dag) launch_pair<P, 1, LS, true, 0>(ctx, par, a, o, o2, e, st);
    else if (a.op) launch_pair<P, 0, LS, true, 0>(ctx, par, a, o, o2, e, st);
    else if (dag) launch_pair<P, 1, LS, false, 0>(ctx, par, a, o, o2, e, st);
    else launch_pair<P, 0, LS, false, 0>(ctx, par, a, o, o2, e, st);
}

template <int P>
bool pair_dslash(const eofa_ctx* ctx, int par, int dag, const PairArgs& a, cudaStream_t st) {
    const int Ls = ctx->Ls;
    if ((Ls & 1) || ctx->forced_cfg) return false;
    // the CG uses MODE 1 with the operator and MODE 2, 3 with its adjoint only
    if ((a.mode == 1 && dag) || (a.mode >= 2 && !dag)) return false;
    for (const void* q : {a.in, (const void*)a.out, a.y, (const void*)a.out2, a.aux, (const void*)a.out3, a.aux2})
        if ((uintptr_t)q & 31) return false;
    PairOp o = {}, o2 = {};
    if (a.op && !pair_op_of(*a.op, Ls, dag == 0, -0.5 * a.a_out, o)) return false;
    if (a.op2 && !pair_op_of(*a.op2, Ls, dag != 0, 1.0, o2)) return false;
    const EpiPair e = {a.out2, a.aux, a.out3, a.aux2, a.it, a.slot2};
    switch (Ls) {
        case 8: launch_pair_ls<P, 8>(ctx, par, dag, a, o, o2, e, st); break;
        case 12: launch_pair_ls<P, 12>(ctx, par, dag, a, o, o2, e, st); break;
        case 16: launch_pair_ls<P, 16>(ctx, par, dag, a, o, o2, e, st); break;
        case 24: launch_pair_ls<P, 24>(ctx, par, dag, a, o, o2, e, st); break;
        default: launch_pair_ls<P, 0>(ctx, par, dag, a, o, o2, e, st); break;
    }
    return true;
}

// ---------------------------------------------------------------- several systems

template <int P, int DAG, int LS, bool HASOP, int MODE>
void launch_mr_pair(const eofa_ctx* ctx, int par, const MRPtrs& a, const PairOp* ops, const Op5* r1, const PairOp* ops2,
                    const Op5* r2, int nr, double a_out, double b_in, int slot, int it, int slot2, cudaStream_t st) {
    Geom g = ctx_geom(ctx);
    const PairShape s = pair_shape(g.Ls, HASOP);
    const int ntiles = (g.Vh + s.NS - 1) / s.NS;
    auto k = mr_pair_kernel<P, DAG, LS, HASOP, MODE>;
    const int all = (int)grid_size(k, s.threads, s.smem, INT_MAX, ctx->sms);  // resident blocks, over the systems
    const int gx = std::max(1, std::min(ntiles, (all + nr - 1) / nr));
    k<<<dim3(gx, nr), s.threads, s.smem, st>>>(g, par, a, ctx->gauge[P32], ops, r1, ops2, r2, (float)a_out, (float)b_in, slot,
                                              s.NS, z_blocks(g, s.NS, P == P16 ? 52 : 96), it, slot2);
    EOFA_LAUNCHED();
}

// The launches of the lock-step iteration (batch.cu): blocks by kind, MR_MAX systems each
// (0: G'^-1 of te = G'^-1 D p, 1: of q = p - G'^-1 D te, 2: G'^-T of te = G'^-T D^+ to, 3: of to = G'^-T q).
template <int P, int LS>
void mr_pair_ls(const eofa_ctx* ctx, int par, int dag, int mode, const MRPtrs& a, const PairOp* po, const Op5* ops,
                const Op5* ops2, int nr, double a_out, double b_in, int slot, int it, int slot2, cudaStream_t st) {
    if (mode == 1)
        launch_mr_pair<P, 0, LS, true, 1>(ctx, par, a, po + MR_MAX, ops, po + 3 * MR_MAX, ops2, nr, a_out, b_in, slot, it,
                                          slot2, st);
    else if (mode == 2)
        launch_mr_pair<P, 1, LS, false, 2>(ctx, par, a, po, ops, po, ops2, nr, a_out, b_in, slot, it, slot2, st);
    else if (dag)
        launch_mr_pair<P, 1, LS, true, 0>(ctx, par, a, po + 2 * MR_MAX, ops, po, ops2, nr, a_out, b_in, slot, it, slot2, st);
    else
        launch_mr_pair<P, 0, LS, true, 0>(ctx, par, a, po, ops, po, ops2, nr, a_out, b_in, slot, it, slot2, st);
}

// (unrolled builds as for one system; eight systems on 8^4 x 24: 103 -> 97 ms in FP32, 100 -> 97 in FP16)
template <int P>
void mr_pair(const eofa_ctx* ctx, int par, int dag, int mode, const MRPtrs& a, const void* pops, const Op5* ops,
             const Op5* ops2, int nr, double a_out, double b_in, int slot, int it, int slot2, cudaStream_t st) {
    const PairOp* po = (const PairOp*)pops;
    switch (ctx->Ls) {
        case 8: mr_pair_ls<P, 8>(ctx, par, dag, mode, a, po, ops, ops2, nr, a_out, b_in, slot, it, slot2, st); break;
        case 12: mr_pair_ls<P, 12>(ctx, par, dag, mode, a, po, ops, ops2, nr, a_out, b_in, slot, it, slot2, st); break;
        case 16: mr_pair_ls<P, 16>(ctx, par, dag, mode, a, po, ops, ops2, nr, a_out, b_in, slot, it, slot2, st); break;
        case 24: mr_pair_ls<P, 24>(ctx, par, dag, mode, a, po, ops, ops2, nr, a_out, b_in, slot, it, slot2, st); break;
        default: mr_pair_ls<P, 0>(ctx, par, dag, mode, a, po, ops, ops2, nr, a_out, b_in, slot, it, slot2, st); break;
    }
}

}  // namespace
}  // namespace dsl
