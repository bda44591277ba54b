// The stored error expanded to fp32 (Alg. 2 line 5's decode alone) for the quantised states: int8, int4,
// stochastic levels in one byte, and the sum of the two states of iConEF-v1.
//
// HBM-bound: the codes in, 4 bytes per element out.  A thread takes four consecutive elements (one
// 2- or 4-byte load of codes, one scale, one 16-byte store; a warp's stores are 512 contiguous bytes)
// and has four of them in flight (small models: one, in four times the CTAs).  Where the output is not 16-byte aligned, and at the end of a
// tensor, a thread takes single elements, a warp 32 consecutive ones.  Transformer-big list, int4 / 128 /
// fp16: one element at a time in each thread took 564 us per worker (1.7 TB/s), this takes 159 us (6.0 TB/s).
#pragma once
#include "conef_common.cuh"

namespace conef {

constexpr int kDecThreads = 256;
constexpr int kDecBatch = 4;
__host__ __device__ constexpr int dec_tile(int batch) { return kDecThreads * 4 * batch; }   // elements per CTA
constexpr int kDecTile = dec_tile(kDecBatch);
// Below about four CTAs of the large kind per SM a launch takes the time of its slowest CTA, not of its bytes:
// one worker, int8, one vector and four vectors per thread, captured calls: 32 k elements 1.56, 1.85 us; 0.5 M
// 1.93, 2.30; 1 M 2.38, 2.38; 2 M 3.03, 3.36 (int4 the same within 0.2).
inline int dec_batch(int64_t elements) { return elements < (int64_t)dec_tile(kDecBatch) * kPlanSMs * 4 ? 1 : kDecBatch; }

// four codes, element 0 in the low bits, times the scale; each product is rounded once
template <bool INT4>
__device__ __forceinline__ float4 decode4(uint32_t w, float s)
{
    constexpr float off = INT4 ? 8388616.f : 8388736.f;   // 2^23 + the bias that makes codes non-negative
    w ^= INT4 ? 0x8888u : 0x80808080u;
    float v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t u = INT4 ? (w >> (4 * q)) & 0xFu : (w >> (8 * q)) & 0xFFu;
        v[q] = __fmul_rn(__fsub_rn(__uint_as_float(0x4B000000u | u), off), s);
    }
    return make_float4(v[0], v[1], v[2], v[3]);
}

template <bool INT4, bool SECOND, int BATCH>
__global__ void __launch_bounds__(kDecThreads) k_decode(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx,
                                                        int worker, float *__restrict__ out)
{
    constexpr int kTile = dec_tile(BATCH);
    grid_release();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const uint8_t *__restrict__ st = V.state + worker * V.state_stride;
    const uint8_t *__restrict__ codes[2] = {st + L.a_off, st + L.a2_off};
    const uint8_t *__restrict__ scales[2] = {st + L.b_off, st + L.b2_off};
    const bool half = V.scale_half && V.ckind != CONEF_C_STOCHQUANT;
    const int shift = 31 - __clz(L.unit);
    const uint32_t d = (uint32_t)L.d, j0 = (blockIdx.x - pfx[li]) * (uint32_t)kTile;
    float *__restrict__ o = out + L.e_off;
    const uint32_t n = min(d - j0, (uint32_t)kTile);
    grid_wait();
    if (n == (uint32_t)kTile && ((uintptr_t)(o + j0) & 15) == 0) {
        uint32_t w[2][BATCH];
        float s[2][BATCH];
#pragma unroll
        for (int x = 0; x < (SECOND ? 2 : 1); ++x)
#pragma unroll
            for (int u = 0; u < BATCH; ++u) {
                const uint32_t j = j0 + (u * kDecThreads + threadIdx.x) * 4;
                w[x][u] = INT4 ? (uint32_t)__ldcs((const unsigned short *)(codes[x] + j / 2)) : __ldcs((const uint32_t *)(codes[x] + j));
                s[x][u] = load_scale(scales[x], j >> shift, half);
            }
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
            float4 e = decode4<INT4>(w[0][u], s[0][u]);
            if (SECOND) {   // e~ + q
                const float4 q = decode4<INT4>(w[1][u], s[1][u]);
                e = make_float4(__fadd_rn(e.x, q.x), __fadd_rn(e.y, q.y), __fadd_rn(e.z, q.z), __fadd_rn(e.w, q.w));
            }
            __stcs((float4 *)(o + j0) + u * kDecThreads + threadIdx.x, e);
        }
        return;
    }
    auto one = [&](int x, uint32_t j) {
        const uint32_t w = INT4 ? codes[x][j >> 1] >> (4 * (j & 1u)) : codes[x][j];
        return decode4<INT4>(INT4 ? w & 0xFu : w, load_scale(scales[x], j >> shift, half)).x;
    };
    if (((uintptr_t)(o + j0) & 15) == 0) {   // a tensor's last tile
        for (uint32_t q = threadIdx.x * 4; q + 4 <= n; q += kDecThreads * 4) {
            const uint32_t j = j0 + q;
            float4 e[2];
#pragma unroll
            for (int x = 0; x < (SECOND ? 2 : 1); ++x)
                e[x] = decode4<INT4>(INT4 ? (uint32_t)__ldcs((const unsigned short *)(codes[x] + j / 2)) : __ldcs((const uint32_t *)(codes[x] + j)),
                                     load_scale(scales[x], j >> shift, half));
            if (SECOND)
                e[0] = make_float4(__fadd_rn(e[0].x, e[1].x), __fadd_rn(e[0].y, e[1].y), __fadd_rn(e[0].z, e[1].z), __fadd_rn(e[0].w, e[1].w));
            __stcs((float4 *)(o + j), e[0]);
        }
        const uint32_t q = (n & ~3u) + threadIdx.x;
        if (q < n) {
            float e = one(0, j0 + q);
            if (SECOND)
                e = __fadd_rn(e, one(1, j0 + q));
            o[j0 + q] = e;
        }
        return;
    }
#pragma unroll 8
    for (uint32_t q = threadIdx.x; q < n; q += kDecThreads) {
        float e = one(0, j0 + q);
        if (SECOND)
            e = __fadd_rn(e, one(1, j0 + q));
        o[j0 + q] = e;
    }
}

template <int BATCH>
inline void decode_launch_batch(bool int4, bool second, const DevView &V, const int32_t *pfx, int tiles, int worker, float *out,
                                cudaStream_t s)
{
    auto *k = int4 ? (second ? k_decode<true, true, BATCH> : k_decode<true, false, BATCH>)
                   : (second ? k_decode<false, true, BATCH> : k_decode<false, false, BATCH>);
    launch(k, dim3(tiles), kDecThreads, 0, s, V, pfx, worker, out);
}
inline void decode_launch(int batch, bool int4, bool second, const DevView &V, const int32_t *pfx, int tiles, int worker, float *out,
                          cudaStream_t s)
{
    if (batch == 1)
        decode_launch_batch<1>(int4, second, V, pfx, tiles, worker, out, s);
    else
        decode_launch_batch<kDecBatch>(int4, second, V, pfx, tiles, worker, out, s);
}

}  // namespace conef
