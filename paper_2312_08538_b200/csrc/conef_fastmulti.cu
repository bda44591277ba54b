// The passes over all tensors in one launch (conef_fastmulti.cuh): one translation unit for their variants.
#include "conef_fastmulti.cuh"

namespace conef {

template <int PASS, int CK, int R, bool HALF, bool PARTIAL>
__global__ void __launch_bounds__(kMultiThreads, multi_ctas(PASS, R))
k_fast_multi(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
    extern __shared__ __align__(128) uint8_t smem_raw[];
    grid_release();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const uint32_t tile = blockIdx.x - pfx[li];
    if (L.fast == 1) {
        const int bd = L.f_threads, sub = threadIdx.x / (unsigned)bd, nsub = L.f_nsub;
        const uint32_t local = tile * (uint32_t)nsub + sub;
        const uint32_t n = (uint32_t)(PASS == 1 ? L.f_rt1 : PASS == 2 ? L.f_rt2 : L.f_rt3) * (uint32_t)L.f_ncg;
        if (sub >= nsub || local >= n)   // (all threads of a tile together)
            return;
        const int it = PASS == 1 ? L.f_it1 : PASS == 2 ? L.f_it2 : L.f_it3;
        uint8_t *mine = smem_raw + sub * multi_tile_bytes(PASS, R, CK == CONEF_C_INT4 ? 1 : 2, HALF ? 2 : 4, it, L.f_subs, bd, L.unit);
        const int tid = threadIdx.x - sub * bd;
        if (PASS == 1 && L.cols < 256)
            fast_tile<PASS, CK, R, HALF, PASS == 1, PARTIAL, true>(V, &L, local, tid, bd, mine, sub + 1);
        else
            fast_tile<PASS, CK, R, HALF, false, PARTIAL, true>(V, &L, local, tid, bd, mine, sub + 1);
        return;
    }
    grid_wait();
    if (L.fast == 3) {
        gen_tile<PASS, CK, HALF, PARTIAL, -R>(V, L, tile, (float *)smem_raw);
    } else if (PASS == 1 && !L.compressed) {
        pass_tile(V, L, tile);
    }
}

template <int PASS, int CK, int R, bool HALF, bool PARTIAL>
static cudaError_t multi(const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, size_t smem)
{
    static int done[64];
    const cudaError_t e = opt_in_smem(k_fast_multi<PASS, CK, R, HALF, PARTIAL>, smem, done);
    if (e != cudaSuccess)
        return e;
    return launch(k_fast_multi<PASS, CK, R, HALF, PARTIAL>, dim3(tiles, V.n_workers), kMultiThreads, smem, s, V, pfx);
}

cudaError_t multi_launch(int pass, int ckind, int rank, int half, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s,
                         size_t smem)
{
    if (tiles <= 0)
        return cudaSuccess;
#define CONEF_MULTI_CASE_P(CKV, RV, HV, PV)                                                 \
    if (ckind == CKV && rank == RV && (half != 0) == HV && (V.beta != 0.f) == PV)           \
        return pass == 1   ? multi<1, CKV, RV, HV, PV>(V, pfx, tiles, s, smem)     \
               : pass == 2 ? multi<2, CKV, RV, HV, PV>(V, pfx, tiles, s, smem)     \
                           : multi<3, CKV, RV, HV, PV>(V, pfx, tiles, s, smem);
#define CONEF_MULTI_CASE(CKV, RV, HV) CONEF_MULTI_CASE_P(CKV, RV, HV, false) CONEF_MULTI_CASE_P(CKV, RV, HV, true)
    CONEF_MULTI_CASE(CONEF_C_INT4, 4, true)
    CONEF_MULTI_CASE(CONEF_C_INT4, 8, true)
    CONEF_MULTI_CASE(CONEF_C_INT8, 4, true)
    CONEF_MULTI_CASE(CONEF_C_INT8, 8, true)
    CONEF_MULTI_CASE(CONEF_C_INT4, 4, false)
    CONEF_MULTI_CASE(CONEF_C_INT4, 8, false)
    CONEF_MULTI_CASE(CONEF_C_INT8, 4, false)
    CONEF_MULTI_CASE(CONEF_C_INT8, 8, false)
#undef CONEF_MULTI_CASE
#undef CONEF_MULTI_CASE_P
    return cudaErrorNotSupported;
}

}  // namespace conef
