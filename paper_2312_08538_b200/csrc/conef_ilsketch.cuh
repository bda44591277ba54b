// Fused step for the count sketch hashed over whole tensors (Alg. 2 lines 5, 6, 9 with C = count sketch,
// Sec. 4.2.2) and Q in {identity, random-k, random-block-k}.
//
// Every element reads v buckets of the old sketch and adds to the same v buckets of the new one, at
// random places of arrays that do not fit an SM.  The buckets depend on the element only, not on the
// worker.  What bounds the step is the number of requests that cross from the SMs to L2 (83 % of the
// peak rate with one worker at a time, L2 tag lookups 76 %, DRAM 3 %), so the workers of a context are
// handled together: their sketches are interleaved, workers innermost, and one request of up to 32
// bytes reads, and one adds to, the bucket of up to eight workers.  An element is one lane's for up to
// four workers and a pair of lanes' for eight (the two 16-byte accesses of a pair make one request).
//
// The state stays one contiguous sketch per worker: a group of tensors is interleaved into a scratch
// (k_sketch_swap, which also clears the new sketch), stepped, and written back.  Groups are as many
// tensors as keep the scratch inside L2, or one larger tensor.
//
// Transformer-big list (210 M elements), 5 x d/10 buckets, eight workers: 90 ms per step one worker at a
// time, 25.3 ms now, of which interleaving takes 3.3; the requests still bound it, ten per element.
// Three CTAs per SM (80 registers); with four (spills) 24.8 ms instead of 23.0 for k_sketch_il.
#pragma once
#include "conef_common.cuh"

namespace conef {

constexpr int kIlThreads = 256;
constexpr int kIlTile = 1024;          // elements per CTA
constexpr int kIlEntries = 1024;       // sketch entries (of every worker) per CTA of the interleaving kernels
// Old (and as many new) bytes per group of tensors: both stay in L2.  (20, 40, 64 MB: 27.6, 26.7, 26.9 ms.)
constexpr int64_t kIlGroupBytes = 40ll << 20;

// A group whose records are larger than this (one tensor that does not fit L2) has the old and the new
// values of an entry side by side, so that the addition finds in L2 what the read brought; in a group
// that fits they are apart, since an addition next to a read of the same sector waits for it.  Eight
// workers, Transformer-big: 25.0 ms with this line, 26.8 always side by side, 28.0 always apart; four
// workers, 16 M elements in L2: 476 us apart, 728 side by side.
constexpr int64_t kIlTogether = 100ll << 20;
// Below this many elements over all workers the two kernels that interleave cost more than they save.
constexpr int64_t kIlDirect = 1ll << 20;
// workers per bucket record: 1, 2, 4 or a multiple of 8
__host__ __device__ inline int il_width(int n_workers)
{
    return n_workers <= 1 ? 1 : n_workers <= 2 ? 2 : n_workers <= 4 ? 4 : (n_workers + 7) / 8 * 8;
}

template <int W>
struct IlVec {
    float v[W];
};
template <int W>
__device__ __forceinline__ IlVec<W> il_load(const float *p)
{
    IlVec<W> r;
    if constexpr (W == 4) {
        const float4 t = *(const float4 *)p;
        r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
    } else if constexpr (W == 2) {
        const float2 t = *(const float2 *)p;
        r.v[0] = t.x; r.v[1] = t.y;
    } else {
        r.v[0] = *p;
    }
    return r;
}
template <int W>
__device__ __forceinline__ void il_add(float *p, const IlVec<W> &a)
{
    if constexpr (W == 4)
        asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};"
                     ::"l"(p), "f"(a.v[0]), "f"(a.v[1]), "f"(a.v[2]), "f"(a.v[3]) : "memory");
    else if constexpr (W == 2)
        asm volatile("red.relaxed.gpu.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a.v[0]), "f"(a.v[1]) : "memory");
    else
        asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(a.v[0]) : "memory");
}

// The old values of a sketch entry are `stride` floats apart from entry to entry, groups of GW = W * LP
// workers (blockIdx.y) follow one another within an entry; the new values lie newoff floats after the old.
//
// VR sketch rows (0: V.cs_rows, up to 7); W workers per lane, LP lanes per element.  GW = 1: no records,
// the states themselves.
template <int QK, int VR, int W, int LP>
__global__ void __launch_bounds__(kIlThreads, W == 4 ? 3 : 4)
k_sketch_il(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx, int first, float *records, uint32_t stride, int64_t newoff)
{
    constexpr int VM = VR ? VR : 7, GW = W * LP;
    const int v = VR ? VR : V.cs_rows;
    const int tile = first + (int)blockIdx.x;
    const int li = find_layer(pfx, V.n_layers, tile);
    const LayerDesc &L = V.layers[li];
    const uint32_t d = (uint32_t)L.d, w = (uint32_t)L.w;
    const uint32_t j0 = (uint32_t)(tile - pfx[li]) * (uint32_t)kIlTile;
    const uint32_t left = min(d - j0, (uint32_t)kIlTile);   // elements of this tile
    const int sub = threadIdx.x & (LP - 1);
    const int w0 = blockIdx.y * GW + sub * W;               // this lane's first worker
    if (GW == 1)
        stride = 1u;
    const float *So;
    float *Sn;
    if (GW == 1) {
        So = (const float *)(V.state + w0 * V.state_stride + L.a_off);
        Sn = (float *)(V.state_new + w0 * V.state_stride + L.a_off);
    } else {
        So = records + L.sk_off * stride + blockIdx.y * (stride / gridDim.y) + sub * W;
        Sn = records + L.sk_off * stride + blockIdx.y * (stride / gridDim.y) + sub * W + newoff;
    }
    __shared__ uint64_t keys[7];
    if (threadIdx.x < 7)
        keys[threadIdx.x] = stream_key(V.seed_c, (uint64_t)li, (uint64_t)threadIdx.x);
    __syncthreads();
    uint32_t blk_start = 0;
    if (QK == CONEF_Q_RANDBLOCK)
        blk_start = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)V.step), d, (uint32_t)L.k);
    const uint32_t *__restrict__ bits = V.selbits + L.selbits_off;
    const uint32_t kept = (uint32_t)L.k;
    const int64_t goff = L.g_off, moff = L.msgv_off;
    const float lr = V.lr, omb = V.omb, beta = V.beta;
    for (uint32_t q = threadIdx.x / LP; q < left; q += kIlThreads / LP) {
        const uint32_t j = j0 + q;
        uint32_t bk[VM];    // bucket
        uint32_t sign = 0;  // bit i: negative sign in row i
        IlVec<W> rec[VM];
#pragma unroll
        for (int i = 0; i < VM; ++i) {
            bk[i] = 0;
            if (VR || i < v) {
                const uint64_t u = h64(keys[i], j);
                bk[i] = (uint32_t)(((u >> 32) * (uint64_t)w) >> 32);
                sign |= (uint32_t)(u & 1) << i;
                rec[i] = il_load<W>(So + ((uint64_t)i * w + bk[i]) * stride);
            }
        }
        float gv[W];
#pragma unroll
        for (int x = 0; x < W; ++x)
            gv[x] = w0 + x < V.n_workers ? __ldcs(V.grads[w0 + x] + goff + j) : 0.f;
        bool sel = QK == CONEF_Q_IDENTITY;
        uint32_t slot = j;
        if (QK == CONEF_Q_RANDK) {
            const uint32_t word = bits[j >> 5];
            sel = (word >> (j & 31u)) & 1u;
            if (sel)
                slot = draw_slot(L, V.wordoff, V.tileoff, word, j);
        } else if (QK == CONEF_Q_RANDBLOCK) {
            slot = j - blk_start;   // wraps to a large value below the block
            sel = slot < kept;
        }
        IlVec<W> val;
#pragma unroll
        for (int x = 0; x < W; ++x) {
            float est[VM];
#pragma unroll
            for (int i = 0; i < VM; ++i)
                est[i] = (VR || i < v) ? __uint_as_float(__float_as_uint(rec[i].v[x]) ^ (((sign >> i) & 1u) << 31)) : 0.f;
            const float e = median_small(est, v);
            const float p = __fmaf_rn(lr, gv[x], __fmul_rn(omb, e));   // Alg. 2 line 5 (Alg. 4 line 5 with beta)
            if (sel && w0 + x < V.n_workers)
                V.msgv[(w0 + x) * V.msgv_stride + moff + slot] = p;
            // r = p - Delta (zero on a transmitted coordinate); Alg. 4 line 9 keeps beta e as well
            val.v[x] = sel ? 0.f : p;
            if (beta != 0.f)
                val.v[x] = __fmaf_rn(beta, e, val.v[x]);
        }
        if (QK != CONEF_Q_IDENTITY && sel && w0 == 0)
            V.idx[L.idx_off + slot] = j;
        bool any = false;
#pragma unroll
        for (int x = 0; x < W; ++x)
            any |= val.v[x] != 0.f;
        if (any) {
#pragma unroll
            for (int i = 0; i < VM; ++i)
                if (VR || i < v) {
                    IlVec<W> a;
#pragma unroll
                    for (int x = 0; x < W; ++x)
                        a.v[x] = __uint_as_float(__float_as_uint(val.v[x]) ^ (((sign >> i) & 1u) << 31));
                    il_add<W>(Sn + ((uint64_t)i * w + bk[i]) * stride, a);
                }
        }
    }
}

// IN: states -> old values of the records, new ones cleared; else: new values -> states.  A thread has one
// entry of all GW workers (coalesced over the entries of a worker); the records, exchanged through
// shared memory, are accessed 16 bytes per lane over contiguous memory.
template <int GW, bool IN>
__global__ void __launch_bounds__(kIlThreads) k_sketch_swap(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx,
                                                            int first, float *__restrict__ records, uint32_t stride, int64_t newoff)
{
    constexpr int PW = GW == 2 ? 2 : 4, H = GW / PW;   // floats per piece, pieces of a record's old (or new) values
    constexpr int PITCH = GW == 8 ? 9 : GW;            // (entries of a warp in different banks)
    using Piece = typename std::conditional<PW == 2, float2, float4>::type;
    __shared__ float buf[kIlThreads * PITCH];
    const int tile = first + (int)blockIdx.x;
    const int li = find_layer(pfx, V.n_layers, tile);
    const LayerDesc &L = V.layers[li];
    const int64_t n = (int64_t)V.cs_rows * L.w;
    const int64_t e0 = (int64_t)(tile - pfx[li]) * kIlEntries;
    const int w0 = blockIdx.y * GW, t = threadIdx.x;
    uint8_t *base = IN ? V.state : V.state_new;
    for (int q = 0; q < kIlEntries / kIlThreads; ++q) {
        const int64_t b = e0 + q * kIlThreads, e = b + t;
        if (b >= n)
            return;   // (uniform over the CTA)
        const int have = (int)min((int64_t)kIlThreads, n - b);
        float *rec = records + (L.sk_off + b) * stride + blockIdx.y * (stride / gridDim.y);
        float r[GW];
        if (IN) {
#pragma unroll
            for (int x = 0; x < GW; ++x)
                r[x] = t < have && w0 + x < V.n_workers ? __ldcs((const float *)(base + (int64_t)(w0 + x) * V.state_stride + L.a_off) + e) : 0.f;
        }
        if (q)
            __syncthreads();
        if (IN) {
#pragma unroll
            for (int x = 0; x < GW; ++x)
                buf[t * PITCH + x] = r[x];
            __syncthreads();
        }
#pragma unroll
        for (int k = 0; k < H; ++k) {
            const int f = k * kIlThreads + t, en = f / H, part = f % H;
            if (en < have) {
                float *at = rec + (int64_t)en * stride + part * PW, *p = buf + en * PITCH + part * PW;
                Piece z;
                float *zf = (float *)&z;
                if (IN) {
#pragma unroll
                    for (int x = 0; x < PW; ++x)
                        zf[x] = p[x];
                    *(Piece *)at = z;
#pragma unroll
                    for (int x = 0; x < PW; ++x)
                        zf[x] = 0.f;
                    *(Piece *)(at + newoff) = z;
                } else {
                    z = *(const Piece *)(at + newoff);
#pragma unroll
                    for (int x = 0; x < PW; ++x)
                        p[x] = zf[x];
                }
            }
        }
        if (!IN) {
            __syncthreads();
            if (t < have) {
#pragma unroll
                for (int x = 0; x < GW; ++x)
                    if (w0 + x < V.n_workers)
                        __stcs((float *)(base + (int64_t)(w0 + x) * V.state_stride + L.a_off) + e, buf[t * PITCH + x]);
            }
        }
    }
}

template <int QK, int W, int LP>
inline void il_step(const DevView &V, const int32_t *pfx, int first, int tiles, int groups, float *records, uint32_t stride, int64_t newoff, cudaStream_t s)
{
    const dim3 grid(tiles, groups);
    if (V.cs_rows == 5)
        k_sketch_il<QK, 5, W, LP><<<grid, kIlThreads, 0, s>>>(V, pfx, first, records, stride, newoff);
    else if (V.cs_rows == 3)
        k_sketch_il<QK, 3, W, LP><<<grid, kIlThreads, 0, s>>>(V, pfx, first, records, stride, newoff);
    else
        k_sketch_il<QK, 0, W, LP><<<grid, kIlThreads, 0, s>>>(V, pfx, first, records, stride, newoff);
}
// the step on the states themselves, one worker per blockIdx.y, all tensors
template <int QK>
inline void il_launch_direct(const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s)
{
    il_step<QK, 1, 1>(V, pfx, 0, tiles, V.n_workers, nullptr, 1, 0, s);
}
// the step of a group of tensors: tiles [first, first + tiles) of elements, [efirst, efirst + etiles) of
// sketch entries.  Returns the number of kernels launched.
template <int QK>
inline int il_launch(const DevView &V, const int32_t *pfx, int first, int tiles, const int32_t *epfx, int efirst, int etiles,
                     int64_t n_records, float *records, cudaStream_t s)
{
    const int NW = il_width(V.n_workers);
    const bool together = n_records * 8 * NW > kIlTogether;
    const uint32_t stride = (uint32_t)(together ? 2 * NW : NW);
    const int64_t newoff = together ? std::min(NW, 8) : n_records * NW;
#define CONEF_IL_CASE(W, LP)                                                                                        \
    {                                                                                                               \
        const int groups = NW / (W * LP);                                                                           \
        k_sketch_swap<W * LP, true><<<dim3(etiles, groups), kIlThreads, 0, s>>>(V, epfx, efirst, records, stride, newoff);          \
        il_step<QK, W, LP>(V, pfx, first, tiles, groups, records, stride, newoff, s);                                               \
        k_sketch_swap<W * LP, false><<<dim3(etiles, groups), kIlThreads, 0, s>>>(V, epfx, efirst, records, stride, newoff);         \
        return 3;                                                                                                   \
    }
    if (NW == 2)
        CONEF_IL_CASE(2, 1)
    if (NW == 4)
        CONEF_IL_CASE(4, 1)
    CONEF_IL_CASE(4, 2)
#undef CONEF_IL_CASE
}

}  // namespace conef
