// Launcher of the tuned fused step (conef_flat16.cuh): one translation unit for its many variants.
#include "conef_flat16.cuh"

namespace conef {

template <int QK, int CK, bool HALF, int ICO>
static cudaError_t flat16(const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s)
{
    constexpr size_t smem = (size_t)(kF16Threads / 32) * f16_ring(ICO) * sizeof(F16Stage<CK, ICO>);
    static int done[64];
    const cudaError_t e = opt_in_smem(k_flat16<QK, CK, HALF, ICO>, smem, done);
    if (e != cudaSuccess)
        return e;
    return launch(k_flat16<QK, CK, HALF, ICO>, dim3(tiles, V.n_workers), kF16Threads, smem, s, V, pfx);
}

cudaError_t flat16_launch(int qkind, int ckind, int half, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s)
{
    if (tiles <= 0)
        return cudaSuccess;
#define CONEF_F16_CASE(QV, CKV, HV, IV)                                                     \
    if (qkind == QV && ckind == CKV && (half != 0) == HV && (V.iconef == 1) == (IV == 1))   \
        return flat16<QV, CKV, HV, IV>(V, pfx, tiles, s);
#define CONEF_F16_Q(QV)                          \
    CONEF_F16_CASE(QV, CONEF_C_INT8, false, 0)   \
    CONEF_F16_CASE(QV, CONEF_C_INT8, true, 0)    \
    CONEF_F16_CASE(QV, CONEF_C_INT4, false, 0)   \
    CONEF_F16_CASE(QV, CONEF_C_INT4, true, 0)    \
    CONEF_F16_CASE(QV, CONEF_C_INT8, false, 1)   \
    CONEF_F16_CASE(QV, CONEF_C_INT8, true, 1)    \
    CONEF_F16_CASE(QV, CONEF_C_INT4, false, 1)   \
    CONEF_F16_CASE(QV, CONEF_C_INT4, true, 1)    \
    CONEF_F16_CASE(QV, CONEF_C_STOCHQUANT, false, 0)
    CONEF_F16_Q(CONEF_Q_IDENTITY)
    CONEF_F16_Q(CONEF_Q_RANDK)
    CONEF_F16_Q(CONEF_Q_RANDBLOCK)
#undef CONEF_F16_Q
#undef CONEF_F16_CASE
    return cudaErrorNotSupported;
}

}  // namespace conef
