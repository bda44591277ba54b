// The variants of the low-rank passes for any shape (conef_lrgen.cuh): one translation unit per codec.
#pragma once
#include "conef_lrgen.cuh"

namespace conef {

template <int CK, bool HALF, bool PARTIAL, int R>
static cudaError_t gen_pass_launch(int pass, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, size_t smem2)
{
    const dim3 grid(tiles, V.n_workers);
    if (pass == 1)
        return launch(k_gen_pass<1, CK, HALF, PARTIAL, R>, grid, kGenThreads, kGenP1Smem, s, V, pfx);
    if (pass == 2)
        return launch(k_gen_pass<2, CK, HALF, PARTIAL, R>, grid, kGenThreads, smem2, s, V, pfx);
    return launch(k_gen_pass<3, CK, HALF, PARTIAL, R>, grid, kGenThreads, kGenP3Smem, s, V, pfx);
}

template <int CK>
cudaError_t gen_launch_codec(int pass, int rank, bool exact, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, size_t smem2)
{
    auto by_rank = [&](auto half, auto partial) {
        constexpr bool H = decltype(half)::value != 0, P = decltype(partial)::value != 0;
        // (rank 8 on int8: gen_tile, BOTH)
        switch (exact || (rank == 8 && CK == CONEF_C_INT8) ? gen_rank(rank) : -gen_rank(rank)) {
        case 1: return gen_pass_launch<CK, H, P, 1>(pass, V, pfx, tiles, s, smem2);
        case 2: return gen_pass_launch<CK, H, P, 2>(pass, V, pfx, tiles, s, smem2);
        case 4: return gen_pass_launch<CK, H, P, 4>(pass, V, pfx, tiles, s, smem2);
        case 8: return gen_pass_launch<CK, H, P, 8>(pass, V, pfx, tiles, s, smem2);
        case -2: return gen_pass_launch<CK, H, P, -2>(pass, V, pfx, tiles, s, smem2);
        case -4: return gen_pass_launch<CK, H, P, -4>(pass, V, pfx, tiles, s, smem2);
        default: return gen_pass_launch<CK, H, P, -8>(pass, V, pfx, tiles, s, smem2);
        }
    };
    if (V.beta != 0.f)
        return V.scale_half ? by_rank(IntC<1>(), IntC<1>()) : by_rank(IntC<0>(), IntC<1>());
    return V.scale_half ? by_rank(IntC<1>(), IntC<0>()) : by_rank(IntC<0>(), IntC<0>());
}

}  // namespace conef
