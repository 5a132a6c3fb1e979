// Two-slices-per-thread dslash kernels, FP32 storage (dslash_pair.cuh).
#include "dslash_pair.cuh"

bool pair_dslash_p32(const eofa_ctx* ctx, int par, int dag, const PairArgs& a, cudaStream_t st) {
    return dsl::pair_dslash<P32>(ctx, par, dag, a, st);
}
