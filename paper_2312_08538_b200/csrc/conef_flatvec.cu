// Launcher of the tuned fused step (conef_flatvec.cuh): one translation unit for its many variants.
#include "conef_flatvec.cuh"

namespace conef {

// bytes of the copy ring (below the 48 KB that need no opt-in)
static size_t fv_smem_bytes(int ckind)
{
    const int cw = ckind == CONEF_C_INT4 ? 1 : 2;
    return (size_t)kFvRing * kFvThreads * (32 + 4 * (cw + 2) + 8);
}

cudaError_t flatvec_launch(int qkind, int ckind, int half, const DevView &V, const int32_t *pfx, int tiles,
                           cudaStream_t s)
{
    if (tiles <= 0)
        return cudaSuccess;
    dim3 grid(tiles, V.n_workers);
#define CONEF_FV_CASE(QV, CKV, HV)                                                           \
    if (qkind == QV && ckind == CKV && (half != 0) == HV) {                                  \
        k_flat_vec2<QV, CKV, HV><<<grid, kFvThreads, fv_smem_bytes(CKV), s>>>(V, pfx);       \
        return cudaSuccess;                                                                  \
    }
#define CONEF_FV_Q(QV)                       \
    CONEF_FV_CASE(QV, CONEF_C_INT8, false)   \
    CONEF_FV_CASE(QV, CONEF_C_INT8, true)    \
    CONEF_FV_CASE(QV, CONEF_C_INT4, false)   \
    CONEF_FV_CASE(QV, CONEF_C_INT4, true)
    CONEF_FV_Q(CONEF_Q_RANDK)
    CONEF_FV_Q(CONEF_Q_RANDBLOCK)
#undef CONEF_FV_Q
#undef CONEF_FV_CASE
    return cudaErrorNotSupported;
}

}  // namespace conef
