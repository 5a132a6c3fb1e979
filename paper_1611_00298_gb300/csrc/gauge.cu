// Wilson plaquette gauge action and its force on the canonical links
// (U[i][mu][a][b], i = x + X (y + Y (z + Z t)), periodic), the gauge part of
// the HMC Hamiltonian that the paper's EOFA runs integrate beside the
// fermion force (Sec. 5):
//   S_g = (beta / 3) sum_{x, mu < nu} Re tr (1 - U_mu(x) U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+),
//   F_mu(x) = sum_a T^a dS_g / dw^a  (U_mu(x) -> exp(i w T^a) U_mu(x))
//           = -i (beta / 12) [(X - X^+) - tr (X - X^+) / 3],  X = U_mu(x) A_mu(x),
// with A_mu(x) the sum of the six staples around U_mu(x).  FP64 throughout;
// one thread per site (action) or per link (force); the action's sum is a
// fixed-order two-pass reduction (bitwise reproducible).
#include "api_util.h"

namespace {

struct M3 {
    double2 e[9];
};

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

__device__ __forceinline__ M3 ld(const double2* U, long long i, int mu) {
    M3 m;
    const double2* p = U + (i * 4 + mu) * 9;
#pragma unroll
    for (int k = 0; k < 9; k++) m.e[k] = __ldg(p + k);
    return m;
}

// c + (a or a*) (b or b*) as multiply-adds (first: c is zero)
template <bool CA, bool CB>
__device__ __forceinline__ double2 cma(double2 a, double2 b, double2 c, bool first) {
    const double ai = CA ? -a.y : a.y, bi = CB ? -b.y : b.y;
    double re = first ? a.x * b.x : fma(a.x, b.x, c.x), im = first ? a.x * bi : fma(a.x, bi, c.y);
    re = fma(-ai, bi, re);
    im = fma(ai, b.x, im);
    return make_double2(re, im);
}
// products of 3x3 matrices, each 108 multiply-adds: a b, a b^+ and a^+ b, added to c (ADD) or alone
template <bool CA, bool CB, bool ADD>
__device__ __forceinline__ void mm(const M3& a, const M3& b, M3& c) {
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            double2 s = c.e[3 * i + j];
#pragma unroll
            for (int k = 0; k < 3; k++)
                s = cma<CA, CB>(a.e[CA ? 3 * k + i : 3 * i + k], b.e[CB ? 3 * j + k : 3 * k + j], s, !ADD && k == 0);
            c.e[3 * i + j] = s;
        }
}
__device__ __forceinline__ M3 mul(const M3& a, const M3& b) {
    M3 c;
    mm<false, false, false>(a, b, c);
    return c;
}
__device__ __forceinline__ M3 mul_nd(const M3& a, const M3& b) {
    M3 c;
    mm<false, true, false>(a, b, c);
    return c;
}

struct Lat {
    int d[4];
    long long V;
};

// index offsets of the eight neighbours of site i (periodic)
struct Steps {
    int up[4], dn[4];
};
__device__ __forceinline__ Steps steps(const Lat& L, int i) {
    Steps s;
    int rest = i, stride = 1;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int n = L.d[k], c = rest % n;
        rest /= n;
        s.up[k] = c + 1 == n ? -(n - 1) * stride : stride;
        s.dn[k] = c == 0 ? (n - 1) * stride : -stride;
        stride *= n;
    }
    return s;
}

// per block: sum over its sites of sum_{mu<nu} (3 - Re tr U_mu,nu(x))
__global__ void __launch_bounds__(256) plaquette_kernel(Lat L, const double2* __restrict__ U, double* part) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    double v = 0.0;
    if (i < L.V) {
        const Steps st = steps(L, (int)i);
#pragma unroll
        for (int mu = 0; mu < 4; mu++) {
            const M3 Um = ld(U, i, mu);
#pragma unroll
            for (int nu = mu + 1; nu < 4; nu++) {
                const M3 A = mul(Um, ld(U, i + st.up[mu], nu));               // U_mu(x) U_nu(x+mu)
                const M3 B = mul(ld(U, i, nu), ld(U, i + st.up[nu], mu));     // U_nu(x) U_mu(x+nu)
                double tr = 0.0;                                              // Re tr (A B^+)
#pragma unroll
                for (int k = 0; k < 9; k++) tr += A.e[k].x * B.e[k].x + A.e[k].y * B.e[k].y;
                v += 3.0 - tr;
            }
        }
    }
    __shared__ double ws[8];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += ws[w];
        part[blockIdx.x] = t;
    }
}

// fixed-order sum of n partials into out[0], scaled
__global__ void __launch_bounds__(256) sum_kernel(const double* part, int n, double scale, double* out) {
    __shared__ double ws[8];
    double v = 0.0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) v += part[k];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += ws[w];
        out[0] = scale * t;
    }
}

// sum of the six staples around U_MU(x)
template <int MU>
__device__ __forceinline__ M3 staples(const double2* U, long long i, const Steps& st) {
    M3 A;
#pragma unroll
    for (int k = 0; k < 9; k++) A.e[k] = make_double2(0.0, 0.0);
#pragma unroll
    for (int nu = 0; nu < 4; nu++) {
        if (nu == MU) continue;
        // U_nu(x+mu) U_mu(x+nu)^+ U_nu(x)^+
        mm<false, true, true>(mul_nd(ld(U, i + st.up[MU], nu), ld(U, i + st.up[nu], MU)), ld(U, i, nu), A);
        // U_nu(x+mu-nu)^+ U_mu(x-nu)^+ U_nu(x-nu) = (U_mu(x-nu) U_nu(x+mu-nu))^+ U_nu(x-nu)
        const long long y = i + st.dn[nu];
        mm<true, false, true>(mul(ld(U, y, MU), ld(U, y + st.up[MU], nu)), ld(U, y, nu), A);
    }
    return A;
}

// F_mu(x) (= or +=) the gauge force, one thread per link, one direction per
// block (the blocks of the four directions of a run of sites are neighbours in
// the grid and share their links in L2).  FP64-bound: 13 products of 108
// multiply-adds a link, against 144 instructions with separate products and
// sums.  16^3 x 32: 2.49 -> 1.26 ms.  The longer chains cost part of a last bit:
// momenta of a four-step trajectory on 8^4 1.26e-15 off 64-bit torch instead of
// 1.17e-15 (its links 1.11e-15 instead of 1.14e-15).
__global__ void __launch_bounds__(128) gauge_force_kernel(Lat L, const double2* __restrict__ U, double beta,
                                                          int accumulate, double2* F) {
    const int mu = blockIdx.x & 3;
    const long long i = (blockIdx.x >> 2) * (long long)blockDim.x + threadIdx.x;
    if (i >= L.V) return;
    const Steps st = steps(L, (int)i);
    const M3 A = mu == 0 ? staples<0>(U, i, st) : mu == 1 ? staples<1>(U, i, st) : mu == 2 ? staples<2>(U, i, st)
                                                                                       : staples<3>(U, i, st);
    const long long l = i * 4 + mu;
    const M3 X = mul(ld(U, i, mu), A);
    // M = X - X^+ (anti-Hermitian); F = -i (beta / 12) (M - tr M / 3)
    double2 Mv[9];
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const double2 x = X.e[3 * a + b], y = X.e[3 * b + a];
            Mv[3 * a + b] = make_double2(x.x - y.x, x.y + y.y);
        }
    const double trim = (Mv[0].y + Mv[4].y + Mv[8].y) / 3.0;  // tr M is imaginary
    const double c = beta / 12.0;
    double2* out = F + l * 9;
#pragma unroll
    for (int k = 0; k < 9; k++) {
        double2 m = Mv[k];
        if (k == 0 || k == 4 || k == 8) m.y -= trim;
        const double2 f = make_double2(c * m.y, -c * m.x);  // -i c m
        out[k] = accumulate ? cadd(out[k], f) : f;
    }
}

inline unsigned nblk(long long n, int b) { return (unsigned)((n + b - 1) / b); }

Lat lat_of(const eofa_ctx* ctx) {
    Lat L;
    for (int k = 0; k < 4; k++) L.d[k] = ctx->dims[k];
    L.V = ctx->V;
    return L;
}

}  // namespace

double gauge_action_now(eofa_ctx* ctx, const double* U, double beta, cudaStream_t st) {
    const Lat L = lat_of(ctx);
    const unsigned nb = nblk(L.V, 256);
    double* part = (double*)ctx_buffer(ctx, "gauge_part", (size_t)(nb + 1) * sizeof(double));
    plaquette_kernel<<<nb, 256, 0, st>>>(L, (const double2*)U, part);
    EOFA_LAUNCHED();
    sum_kernel<<<1, 256, 0, st>>>(part, (int)nb, beta / 3.0, part + nb);
    EOFA_LAUNCHED();
    EOFA_CUDA(cudaMemcpyAsync(ctx->red_host, part + nb, sizeof(double), cudaMemcpyDeviceToHost, st));
    EOFA_CUDA(cudaStreamSynchronize(st));
    return ctx->red_host[0];
}

void gauge_force_launch(eofa_ctx* ctx, const double* U, double beta, int accumulate, double* F, cudaStream_t st) {
    const Lat L = lat_of(ctx);
    gauge_force_kernel<<<4 * nblk(L.V, 128), 128, 0, st>>>(L, (const double2*)U, beta, accumulate, (double2*)F);
    EOFA_LAUNCHED();
}

extern "C" {

int eofa_gauge_action_dev(eofa_ctx* ctx, double beta, const double* U_dev, double* S, void* stream) {
    if (!ctx || !S) return fail(ctx, EOFA_EINVAL, "null argument");
    try {
        const double* U = U_dev;
        if (!U) {
            require_gauge(ctx);
            U = (const double*)ctx_buffer(ctx, "U", 0);
        }
        *S = gauge_action_now(ctx, U, beta, (cudaStream_t)stream);
    } catch (const eofa_error& e) {
        return fail(ctx, e.code, e.msg);
    }
    return EOFA_OK;
}

int eofa_gauge_force_dev(eofa_ctx* ctx, double beta, const double* U_dev, double* F_dev, int accumulate,
                         void* stream) {
    if (!ctx || !F_dev) return fail(ctx, EOFA_EINVAL, "null argument");
    try {
        const double* U = U_dev;
        if (!U) {
            require_gauge(ctx);
            U = (const double*)ctx_buffer(ctx, "U", 0);
        }
        gauge_force_launch(ctx, U, beta, accumulate ? 1 : 0, F_dev, (cudaStream_t)stream);
    } catch (const eofa_error& e) {
        return fail(ctx, e.code, e.msg);
    }
    return EOFA_OK;
}

}  // extern "C"
