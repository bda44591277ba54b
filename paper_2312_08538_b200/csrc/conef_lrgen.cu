// Launcher of the low-rank passes for any shape (conef_lrgen.cuh): one translation unit for their variants.
#include "conef_lrgen.cuh"

namespace conef {

template <int CK, int R>
static cudaError_t pass_launch(int pass, int unit, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, bool coop)
{
    const dim3 grid(tiles, V.n_workers);
    if (pass == 1)
        return launch(k_gen_pass<1, CK, R, 1>, grid, kGenThreads, 0, s, V, pfx);
    if (pass == 2)
        return launch(k_gen_pass<2, CK, R, 1>, grid, kGenThreads, coop ? kGenCoopSmem : 0, s, V, pfx);
    if (unit == 256)
        return launch(k_gen_pass<3, CK, R, 8>, grid, kGenThreads, 0, s, V, pfx);
    if (unit == 128)
        return launch(k_gen_pass<3, CK, R, 4>, grid, kGenThreads, 0, s, V, pfx);
    if (CK == CONEF_C_INT4 || unit == 64)   // (int4 blocks are 64 or more)
        return launch(k_gen_pass<3, CK, R, 2>, grid, kGenThreads, 0, s, V, pfx);
    else if constexpr (CK == CONEF_C_INT8)
        return launch(k_gen_pass<3, CK, R, 1>, grid, kGenThreads, 0, s, V, pfx);
    return cudaErrorNotSupported;
}

cudaError_t gen_launch(int pass, int ckind, int rank, int unit, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, bool coop)
{
    if (tiles <= 0)
        return cudaSuccess;
#define CONEF_GEN_CK(CKV)                                                                  \
    if (ckind == CKV) {                                                                    \
        switch (rank) {                                                                    \
        case 1: return pass_launch<CKV, 1>(pass, unit, V, pfx, tiles, s, coop); \
        case 2: return pass_launch<CKV, 2>(pass, unit, V, pfx, tiles, s, coop); \
        case 4: return pass_launch<CKV, 4>(pass, unit, V, pfx, tiles, s, coop); \
        case 8: return pass_launch<CKV, 8>(pass, unit, V, pfx, tiles, s, coop); \
        default: return pass_launch<CKV, 0>(pass, unit, V, pfx, tiles, s, coop); \
        }                                                                                  \
    }
    CONEF_GEN_CK(CONEF_C_INT8)
    CONEF_GEN_CK(CONEF_C_INT4)
#undef CONEF_GEN_CK
    return cudaErrorNotSupported;
}

}  // namespace conef
