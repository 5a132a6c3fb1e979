// Two-slices-per-thread dslash kernels, FP32 storage (dslash_pair.cuh).
#include "dslash_pair.cuh"

bool pair_dslash_p32(const eofa_ctx* ctx, int par, int dag, const PairArgs& a, cudaStream_t st) {
    return dsl::pair_dslash<P32>(ctx, par, dag, a, st);
}

void mr_pair_p32(const eofa_ctx* ctx, int par, int dag, int mode, const MRPtrs& a, const void* pops, const Op5* ops,
                 const Op5* ops2, int nr, double a_out, double b_in, int slot, int it, int slot2, cudaStream_t st) {
    dsl::mr_pair<P32>(ctx, par, dag, mode, a, pops, ops, ops2, nr, a_out, b_in, slot, it, slot2, st);
}

size_t mr_pair_ops_bytes() { return 4 * MR_MAX * sizeof(dsl::PairOp); }

bool mr_pair_ops_fill(const Op5* Gi, const Op5* GiT, int n, int Ls, void* host) {
    if (Ls & 1) return false;
    dsl::PairOp* o = (dsl::PairOp*)host;
    for (int a = 0; a < n; a++) {
        if (!dsl::pair_op_of(Gi[a], Ls, true, -0.5, o[a]) || !dsl::pair_op_of(Gi[a], Ls, true, 0.5, o[MR_MAX + a]) ||
            !dsl::pair_op_of(GiT[a], Ls, false, -0.5, o[2 * MR_MAX + a]) ||
            !dsl::pair_op_of(GiT[a], Ls, false, 1.0, o[3 * MR_MAX + a]))
            return false;
    }
    return true;
}
