// Fused step on a dense fp32 error (C = identity: Alg. 1, EFSGD, and Alg. 4 with beta) for Q in {identity,
// random-k, random-block-k}: p = eta g + e, message, e <- p - Delta.  HBM-bound, 12 bytes per element:
// four 16-byte loads of each stream in flight per thread; gradients off a 16-byte boundary are
// read four bytes at a time, a warp 128 contiguous bytes, with the same number in flight.
// ResNet-50 list, random-block-k, four workers: one element at a time in each thread took 415 us
// (3.0 TB/s), this takes 194 us (6.3 TB/s).
#pragma once
#include "conef_decode.cuh"

namespace conef {

template <int QK, int VEC>
__device__ __forceinline__ void dense_tile(const DevView &V, const LayerDesc &L, int li, uint32_t j0, uint32_t n)
{
    constexpr int B = 16 / VEC;   // vectors per thread: kDecTile elements per CTA
    const int worker = blockIdx.y;
    const uint32_t d = (uint32_t)L.d, kept = (uint32_t)L.k;
    const float *__restrict__ g = V.grads[worker] + L.g_off + j0;
    float *__restrict__ e = (float *)(V.state + worker * V.state_stride + L.a_off) + j0;
    float *__restrict__ msg = V.msgv + worker * V.msgv_stride + L.msgv_off;
    uint32_t *__restrict__ idx = V.idx + L.idx_off;
    const float lr = V.lr, omb = V.omb, beta = V.beta;
    uint32_t blk_start = 0;
    if (QK == CONEF_Q_RANDBLOCK)
        blk_start = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)V.step), d, kept);
    // (a tile holds all or none of the block in most cases)
    const bool near_block = QK == CONEF_Q_RANDBLOCK && j0 < blk_start + kept && j0 + n > blk_start;
    float gv[B][VEC], ev[B][VEC];
    uint32_t word[B];
#pragma unroll
    for (int u = 0; u < B; ++u) {
        const uint32_t q = (u * kDecThreads + threadIdx.x) * VEC;
        word[u] = 0;
        if (VEC == 4) {
            const float4 a = __ldcs((const float4 *)(g + q)), b = *(const float4 *)(e + q);
            gv[u][0] = a.x; gv[u][1 % VEC] = a.y; gv[u][2 % VEC] = a.z; gv[u][3 % VEC] = a.w;
            ev[u][0] = b.x; ev[u][1 % VEC] = b.y; ev[u][2 % VEC] = b.z; ev[u][3 % VEC] = b.w;
        } else {
            gv[u][0] = q < n ? __ldcs(g + q) : 0.f;
            ev[u][0] = q < n ? e[q] : 0.f;
        }
        if (QK == CONEF_Q_RANDK && (VEC == 4 || q < n))
            word[u] = V.selbits[L.selbits_off + ((j0 + q) >> 5)];
    }
#pragma unroll
    for (int u = 0; u < B; ++u) {
        const uint32_t q = (u * kDecThreads + threadIdx.x) * VEC, j = j0 + q;
        float r[VEC];
        uint32_t slot = 0;
        if (QK == CONEF_Q_RANDK && ((word[u] >> (j & 31u)) & ((1u << VEC) - 1u)))
            slot = draw_slot(L, V.wordoff, V.tileoff, word[u], j);
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            const float p = __fmaf_rn(lr, gv[u][v], __fmul_rn(omb, ev[u][v]));   // Alg. 2 line 5, Alg. 4 line 5
            r[v] = p;
            if (QK == CONEF_Q_IDENTITY) {
                gv[u][v] = p;
                r[v] = 0.f;
            } else if (QK == CONEF_Q_RANDK) {
                if ((word[u] >> ((j + v) & 31u)) & 1u) {
                    msg[slot] = p;
                    if (worker == 0)
                        idx[slot] = j + v;
                    ++slot;
                    r[v] = 0.f;
                }
            } else if (near_block) {
                const uint32_t sl = j + v - blk_start;   // wraps to a large value below the block
                if (sl < kept && (VEC == 4 || q < n)) {
                    msg[sl] = p;
                    if (worker == 0)
                        idx[sl] = j + v;
                    r[v] = 0.f;
                }
            }
            if (beta != 0.f)
                r[v] = __fmaf_rn(beta, ev[u][v], r[v]);   // Alg. 4 line 9
        }
        if (VEC == 4) {
            *(float4 *)(e + q) = make_float4(r[0], r[1 % VEC], r[2 % VEC], r[3 % VEC]);
        } else if (q < n) {
            e[q] = r[0];
        }
        if (QK == CONEF_Q_IDENTITY) {
#pragma unroll
            for (int v = 0; v < VEC; ++v)
                if (VEC == 4 || q < n)
                    msg[j + v] = gv[u][v];
        }
    }
}

template <int QK>
__global__ void __launch_bounds__(kDecThreads) k_flat_dense(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
    grid_release();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    if (!L.compressed) {   // (a 1-D tensor: its message in the same launch)
        grid_wait();
        pass_tile(V, L, blockIdx.x - pfx[li]);
        return;
    }
    const uint32_t j0 = (blockIdx.x - pfx[li]) * (uint32_t)kDecTile, n = min((uint32_t)L.d - j0, (uint32_t)kDecTile);
    grid_wait();
    if (n == (uint32_t)kDecTile && ((uintptr_t)(V.grads[blockIdx.y] + L.g_off) & 15) == 0)
        dense_tile<QK, 4>(V, L, li, j0, n);
    else
        dense_tile<QK, 1>(V, L, li, j0, n);
}

}  // namespace conef
