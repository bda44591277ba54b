// Launcher of the low-rank passes for any shape (conef_lrgen.cuh).
#include "conef_lrgen.cuh"

namespace conef {

cudaError_t gen_launch(int pass, int ckind, int rank, bool exact, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, size_t smem2)
{
    if (tiles <= 0)
        return cudaSuccess;
    if (ckind == CONEF_C_INT8)
        return gen_launch_codec<CONEF_C_INT8>(pass, rank, exact, V, pfx, tiles, s, smem2);
    if (ckind == CONEF_C_INT4)
        return gen_launch_codec<CONEF_C_INT4>(pass, rank, exact, V, pfx, tiles, s, smem2);
    return cudaErrorNotSupported;
}

}  // namespace conef
