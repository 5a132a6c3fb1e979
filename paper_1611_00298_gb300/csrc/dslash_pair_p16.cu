// Two-slices-per-thread dslash kernels, FP16 storage (dslash_pair.cuh).
#include "dslash_pair.cuh"

bool pair_dslash_p16(const eofa_ctx* ctx, int par, int dag, const PairArgs& a, cudaStream_t st) {
    return dsl::pair_dslash<P16>(ctx, par, dag, a, st);
}
