// Two-slices-per-thread dslash kernels, FP16 storage (dslash_pair.cuh).
#include "dslash_pair.cuh"

bool pair_dslash_p16(const eofa_ctx* ctx, int par, int dag, const PairArgs& a, cudaStream_t st) {
    return dsl::pair_dslash<P16>(ctx, par, dag, a, st);
}

void mr_pair_p16(const eofa_ctx* ctx, int par, int dag, int mode, const MRPtrs& a, const void* pops, const Op5* ops,
                 const Op5* ops2, int nr, double a_out, double b_in, int slot, int it, int slot2, cudaStream_t st) {
    dsl::mr_pair<P16>(ctx, par, dag, mode, a, pops, ops, ops2, nr, a_out, b_in, slot, it, slot2, st);
}
