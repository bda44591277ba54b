// Launcher of the low-rank passes for any shape (conef_lrgen.cuh): one translation unit for their variants.
#include "conef_lrgen.cuh"

namespace conef {

template <int CK, int R>
static void launch(int pass, int unit, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s)
{
    const dim3 grid(tiles, V.n_workers);
    if (pass == 1)
        k_gen_pass<1, CK, R, 1><<<grid, kGenThreads, 0, s>>>(V, pfx);
    else if (pass == 2)
        k_gen_pass<2, CK, R, 1><<<grid, kGenThreads, 0, s>>>(V, pfx);
    else if (unit == 256)
        k_gen_pass<3, CK, R, 8><<<grid, kGenThreads, 0, s>>>(V, pfx);
    else if (unit == 128)
        k_gen_pass<3, CK, R, 4><<<grid, kGenThreads, 0, s>>>(V, pfx);
    else if (CK == CONEF_C_INT4 || unit == 64)   // (int4 blocks are 64 or more)
        k_gen_pass<3, CK, R, 2><<<grid, kGenThreads, 0, s>>>(V, pfx);
    else if constexpr (CK == CONEF_C_INT8)
        k_gen_pass<3, CK, R, 1><<<grid, kGenThreads, 0, s>>>(V, pfx);
}

cudaError_t gen_launch(int pass, int ckind, int rank, int unit, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s)
{
    if (tiles <= 0)
        return cudaSuccess;
#define CONEF_GEN_CK(CKV)                                                                  \
    if (ckind == CKV) {                                                                    \
        switch (rank) {                                                                    \
        case 1: launch<CKV, 1>(pass, unit, V, pfx, tiles, s); return cudaSuccess;          \
        case 2: launch<CKV, 2>(pass, unit, V, pfx, tiles, s); return cudaSuccess;          \
        case 4: launch<CKV, 4>(pass, unit, V, pfx, tiles, s); return cudaSuccess;          \
        case 8: launch<CKV, 8>(pass, unit, V, pfx, tiles, s); return cudaSuccess;          \
        default: launch<CKV, 0>(pass, unit, V, pfx, tiles, s); return cudaSuccess;         \
        }                                                                                  \
    }
    CONEF_GEN_CK(CONEF_C_INT8)
    CONEF_GEN_CK(CONEF_C_INT4)
#undef CONEF_GEN_CK
    return cudaErrorNotSupported;
}

}  // namespace conef
