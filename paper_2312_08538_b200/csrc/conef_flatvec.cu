// Launcher of the tuned fused step (conef_flatvec.cuh): one translation unit for its many variants.
#include "conef_flatvec.cuh"

namespace conef {

// bytes of the copy ring (below the 48 KB that need no opt-in)
inline size_t fv_smem_bytes(int ckind, int ico)
{
    const int cw = ckind == CONEF_C_INT4 ? 1 : 2;
    return (size_t)kFvRing * kFvThreads * (32 + 4 * (cw + 2) + (ico == 1 ? 4 * (cw + 1) : ico == 2 ? 8 : 0));
}

cudaError_t flatvec_launch(int qkind, int ckind, int half, const DevView &V, const int32_t *pfx, int tiles,
                                  cudaStream_t s)
{
    if (tiles <= 0)
        return cudaSuccess;
    dim3 grid(tiles, V.n_workers);
    const int ico = V.iconef;
    if (V.iconef) {   // iConEF-v1: the variants with a second state; -v2: with e~ as the values of a second draw
#define CONEF_FV_ICO(QV, CKV, HV)                                               \
    if (qkind == QV && ckind == CKV && (half != 0) == HV) {                     \
        if (V.iconef == 1)                                                      \
            k_flat_vec<QV, CKV, HV, 1><<<grid, kFvThreads, fv_smem_bytes(CKV, ico), s>>>(V, pfx);     \
        else if (QV != CONEF_Q_IDENTITY)                                        \
            k_flat_vec<QV == CONEF_Q_IDENTITY ? CONEF_Q_RANDK : QV, CKV, HV, 2><<<grid, kFvThreads, fv_smem_bytes(CKV, ico), s>>>(V, pfx); \
        else                                                                    \
            return cudaErrorNotSupported;                                       \
        return cudaSuccess;                                                     \
    }
#define CONEF_FV_ICO_Q(QV)                  \
    CONEF_FV_ICO(QV, CONEF_C_INT8, false)   \
    CONEF_FV_ICO(QV, CONEF_C_INT8, true)    \
    CONEF_FV_ICO(QV, CONEF_C_INT4, false)   \
    CONEF_FV_ICO(QV, CONEF_C_INT4, true)
        CONEF_FV_ICO_Q(CONEF_Q_IDENTITY)
        CONEF_FV_ICO_Q(CONEF_Q_RANDK)
        CONEF_FV_ICO_Q(CONEF_Q_RANDBLOCK)
#undef CONEF_FV_ICO_Q
#undef CONEF_FV_ICO
        return cudaErrorNotSupported;
    }
#define CONEF_FV_CASE(QV, CKV, HV)                                              \
    if (qkind == QV && ckind == CKV && (half != 0) == HV) {                     \
        k_flat_vec<QV, CKV, HV><<<grid, kFvThreads, fv_smem_bytes(CKV, ico), s>>>(V, pfx);            \
        return cudaSuccess;                                                     \
    }
#define CONEF_FV_Q(QV)                       \
    CONEF_FV_CASE(QV, CONEF_C_INT8, false)   \
    CONEF_FV_CASE(QV, CONEF_C_INT8, true)    \
    CONEF_FV_CASE(QV, CONEF_C_INT4, false)   \
    CONEF_FV_CASE(QV, CONEF_C_INT4, true)    \
    CONEF_FV_CASE(QV, CONEF_C_STOCHQUANT, false)
    CONEF_FV_Q(CONEF_Q_IDENTITY)
    CONEF_FV_Q(CONEF_Q_RANDK)
    CONEF_FV_Q(CONEF_Q_RANDBLOCK)
#undef CONEF_FV_Q
#undef CONEF_FV_CASE
    return cudaErrorNotSupported;
}

}  // namespace conef
