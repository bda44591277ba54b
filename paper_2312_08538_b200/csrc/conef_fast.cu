// Launchers of the tuned low-rank passes (conef_fast.cuh): one translation unit for their many variants.
#include "conef_fast.cuh"

namespace conef {

template <int PASS, int CK, int R, bool HALF, bool NARROW = false, bool PARTIAL = false>
inline cudaError_t fast_launch_pass23(const DevView &V, const int32_t *pfx, int tiles, int threads, cudaStream_t s,
                                      size_t stage)
{
    const size_t smem = (size_t)ring_depth(PASS, R) * threads * (32 + (CK == CONEF_C_INT4 ? 4 : 8)) + stage;
    static int done[64];
    const cudaError_t e = opt_in_smem(k_fast_pass<PASS, CK, R, HALF, NARROW, PARTIAL>, smem, done);
    if (e != cudaSuccess)
        return e;
    return launch(k_fast_pass<PASS, CK, R, HALF, NARROW, PARTIAL>, dim3(tiles, V.n_workers), threads, smem, s, V, pfx);
}

cudaError_t fast_launch(int pass, int ckind, int rank, int half, const DevView &V, const int32_t *pfx,
                               int tiles, int threads, cudaStream_t s, bool narrow, size_t stage)
{
    if (tiles <= 0)
        return cudaSuccess;
#define CONEF_FAST_CASE_P(CKV, RV, HV, PV)                                                                \
    if (ckind == CKV && rank == RV && (half != 0) == HV && (V.beta != 0.f) == PV) {                       \
        if (pass == 1 && narrow) return fast_launch_pass23<1, CKV, RV, HV, true, PV>(V, pfx, tiles, threads, s, stage); \
        if (pass == 1) return fast_launch_pass23<1, CKV, RV, HV, false, PV>(V, pfx, tiles, threads, s, stage);          \
        if (pass == 2) return fast_launch_pass23<2, CKV, RV, HV, false, PV>(V, pfx, tiles, threads, s, stage);          \
        return fast_launch_pass23<3, CKV, RV, HV, false, PV>(V, pfx, tiles, threads, s, stage);           \
    }
#define CONEF_FAST_CASE(CKV, RV, HV) CONEF_FAST_CASE_P(CKV, RV, HV, false) CONEF_FAST_CASE_P(CKV, RV, HV, true)
    CONEF_FAST_CASE(CONEF_C_INT4, 4, true)
    CONEF_FAST_CASE(CONEF_C_INT4, 8, true)
    CONEF_FAST_CASE(CONEF_C_INT8, 4, true)
    CONEF_FAST_CASE(CONEF_C_INT8, 8, true)
    CONEF_FAST_CASE(CONEF_C_INT4, 4, false)
    CONEF_FAST_CASE(CONEF_C_INT4, 8, false)
    CONEF_FAST_CASE(CONEF_C_INT8, 4, false)
    CONEF_FAST_CASE(CONEF_C_INT8, 8, false)
#undef CONEF_FAST_CASE
#undef CONEF_FAST_CASE_P
    return cudaErrorNotSupported;
}

cudaError_t fast_launch_p1_combine(int rank, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s)
{
    if (tiles <= 0)
        return cudaSuccess;
    return launch(rank == 4 ? k_fast_p1_combine<4> : k_fast_p1_combine<8>, dim3(tiles, V.n_workers), 256, 0, s, V, pfx);
}

}  // namespace conef
