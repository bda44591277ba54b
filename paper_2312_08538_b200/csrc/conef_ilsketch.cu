// Launchers of the count-sketch step over whole tensors (conef_ilsketch.cuh): one translation unit for its
// many variants.
#include "conef_ilsketch.cuh"

namespace conef {

// SPLIT's last step: `records`, one sketch after the other (n_records floats apart), -> states, whose padding
// (to 64 floats) is cleared again.  blockIdx.y: worker of the batch.
static __global__ void __launch_bounds__(kIlThreads) k_sketch_back(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx,
                                                                   int first, int worker0, const float *records,
                                                                   int64_t n_records)
{
    grid_release();
    const int tile = first + (int)blockIdx.x;
    const int li = find_layer(pfx, V.n_layers, tile);
    const LayerDesc &L = V.layers[li];
    grid_wait();
    const int64_t n = (int64_t)V.cs_rows * L.w, room = (n + 63) / 64 * 64;
    const int64_t e0 = (int64_t)(tile - pfx[li]) * kIlEntries + threadIdx.x;
    const float *src = records + blockIdx.y * n_records + L.sk_off;
    float *__restrict__ dst = (float *)(V.state + (worker0 + (int)blockIdx.y) * V.state_stride + L.a_off);
#pragma unroll
    for (int q = 0; q < kIlEntries / kIlThreads; ++q) {
        const int64_t e = e0 + q * kIlThreads;
        if (e < room)
            dst[e] = e < n ? __ldcs(src + e) : 0.f;
    }
}

// FOLD, one tensor, whose first tile of entries is `first`.  `half` entries are in the scratch.
//   0  states -> scratch: the old values of entry e and, in the new one's slot, of entry half + e
//   1  the latter -> their records among the states; all new values cleared
//   2  the new values among the states -> the old slots of the scratch
//   3  scratch -> states, whose padding is cleared again
template <int GW, int PART>
static __global__ void __launch_bounds__(kIlThreads) k_sketch_fold(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx,
                                                                   int first, int worker0, float *records)
{
    constexpr int F = 2 * GW, PITCH = F + 1, PW = GW < 4 ? GW : 4;   // floats per record and per piece
    using Piece = typename std::conditional<PW == 2, float2, float4>::type;
    __shared__ float buf[PART == 0 || PART == 3 ? kIlThreads * PITCH : 1];
    grid_release();
    const LayerDesc &L = V.layers[find_layer(pfx, V.n_layers, first)];
    grid_wait();
    const uint32_t n = (uint32_t)(V.cs_rows * L.w), half = (n + 1u) / 2u, t = threadIdx.x;
    float *const states = (float *)(V.state + worker0 * V.state_stride + L.a_off);
    const int64_t pitch = V.state_stride / 4;
    const IlSlices slices(n, F, V.state_stride);
    if constexpr (PART == 1 || PART == 2) {
        constexpr uint32_t H = GW / PW;   // a thread has one piece of a record's old (or new) values
        const uint64_t f0 = (uint64_t)blockIdx.x * (kIlEntries * H) + t;
#pragma unroll
        for (uint32_t q = 0; q < kIlEntries * H / kIlThreads; ++q) {
            const uint32_t e = (uint32_t)((f0 + q * kIlThreads) / H), part = (uint32_t)((f0 + q * kIlThreads) % H);
            if (e < half) {
                Piece *const mine = (Piece *)(records + (uint64_t)e * F + part * PW);
                Piece *const other = (Piece *)(states + slices.at(e, F) + part * PW);
                const Piece zero = {};
                if (PART == 1) {
                    if (half + e < n) {
                        *other = mine[H];
                        other[H] = zero;
                    }
                    mine[H] = zero;
                } else if (half + e < n) {
                    *mine = other[H];
                }
            }
        }
    } else {
        for (int q = 0; q < kIlEntries / kIlThreads; ++q) {
            const uint32_t b = blockIdx.x * kIlEntries + q * kIlThreads, e = b + t;
            if (b >= half)
                break;   // (uniform over the CTA)
            const uint32_t have = min((uint32_t)kIlThreads, half - b);
            float *const rec = records + (uint64_t)b * F;
            if (q)
                __syncthreads();
            if (PART == 0) {
#pragma unroll
                for (int x = 0; x < GW; ++x) {
                    buf[t * PITCH + x] = t < have ? __ldcs(states + x * pitch + e) : 0.f;
                    buf[t * PITCH + GW + x] = t < have && half + e < n ? __ldcs(states + x * pitch + half + e) : 0.f;
                }
                __syncthreads();
            }
#pragma unroll
            for (int k = 0; k < F / PW; ++k) {
                const uint32_t f = k * kIlThreads + t, en = f / (F / PW), part = f % (F / PW);
                if (en < have) {
                    float *const at = rec + (uint64_t)en * F + part * PW, *const p = buf + en * PITCH + part * PW;
                    Piece z;
                    float *const zf = (float *)&z;
                    if (PART == 3)
                        z = *(const Piece *)at;
#pragma unroll
                    for (int x = 0; x < PW; ++x)
                        (PART == 0 ? zf[x] : p[x]) = PART == 0 ? p[x] : zf[x];
                    if (PART == 0)
                        *(Piece *)at = z;
                }
            }
            if (PART == 3) {
                __syncthreads();
                if (t < have) {
#pragma unroll
                    for (int x = 0; x < GW; ++x) {
                        __stcs(states + x * pitch + e, buf[t * PITCH + GW + x]);
                        if (half + e < n)
                            __stcs(states + x * pitch + half + e, buf[t * PITCH + x]);
                    }
                }
            }
        }
        if (PART == 3 && blockIdx.x == 0 && t < 64 && n + t < (n + 63u) / 64u * 64u) {
#pragma unroll
            for (int x = 0; x < GW; ++x)
                states[x * pitch + n + t] = 0.f;
        }
    }
}

template <int QK, int W, int LP, int FORM, int WALK = 0>
static void step(const DevView &V, const int32_t *pfx, int first, int tiles, int worker0, int groups, float *records, uint32_t stride,
                 int64_t newoff, cudaStream_t s, float *resid = nullptr)
{
    const dim3 grid(tiles, groups);
    if (V.cs_rows == 5)
        launch(k_sketch_il<QK, 5, W, LP, FORM, WALK>, dim3(grid), kIlThreads, 0, s, V, pfx, first, worker0, records, stride, newoff, resid);
    else if (V.cs_rows == 3)
        launch(k_sketch_il<QK, 3, W, LP, FORM, WALK>, dim3(grid), kIlThreads, 0, s, V, pfx, first, worker0, records, stride, newoff, resid);
    else
        launch(k_sketch_il<QK, 0, W, LP, FORM, WALK>, dim3(grid), kIlThreads, 0, s, V, pfx, first, worker0, records, stride, newoff, resid);
}

// a group of tensors
struct Group {
    const DevView &V;
    const int32_t *pfx;
    int first, tiles;
    const int32_t *epfx;
    int efirst, etiles;
    int64_t n_records;
    float *records;
    bool second;
    cudaStream_t s;
};

// `batches` batches of W * LP workers from worker0 on
template <int QK, int W, int LP>
static int together(const Group &G, int worker0, int batches, int64_t bytes)
{
    constexpr int GW = W * LP;
    const int NW = GW * batches;
    const bool two = il_two_walks(G.n_records, G.tiles, NW, GW, G.V.cs_rows, bytes), near = !two && G.n_records * 8 * NW > kIlTogether;
    const uint32_t stride = (uint32_t)(near ? 2 * NW : NW);
    const int64_t newoff = near ? GW : G.n_records * NW;
    const dim3 egrid(G.etiles, batches);
    launch(k_sketch_swap<GW, true, false>, dim3(egrid), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records, stride, newoff);
    if (two) {
        float *const resid = G.records + G.n_records * 2 * NW;
        step<QK, W, LP, IL_SCRATCH, 1>(G.V, G.pfx, G.first, G.tiles, worker0, batches, G.records, stride, newoff, G.s, resid);
        step<QK, W, LP, IL_SCRATCH, 2>(G.V, G.pfx, G.first, G.tiles, worker0, batches, G.records, stride, newoff, G.s, resid);
    } else {
        step<QK, W, LP, IL_SCRATCH>(G.V, G.pfx, G.first, G.tiles, worker0, batches, G.records, stride, newoff, G.s);
    }
    launch(k_sketch_swap<GW, false, false>, dim3(egrid), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records, stride, newoff);
    return two ? 4 : 3;
}
template <int QK, int W, int LP>
static int split(const Group &G, int worker0)
{
    constexpr int GW = W * LP;
    if constexpr (GW > 1) {
        if (G.n_records * 8 * GW > kIlTogether) {   // (one tensor: a group of several is at most 2 kIlGroupBytes)
            const int tiles = (int)(((G.n_records + 1) / 2 + kIlEntries - 1) / kIlEntries);
            launch(k_sketch_fold<GW, 0>, dim3(tiles), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records);
            launch(k_sketch_fold<GW, 1>, dim3(tiles), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records);
            step<QK, W, LP, IL_FOLD>(G.V, G.pfx, G.first, G.tiles, worker0, 1, G.records, GW, 0, G.s);
            launch(k_sketch_fold<GW, 2>, dim3(tiles), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records);
            launch(k_sketch_fold<GW, 3>, dim3(tiles), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records);
            return 5;
        }
    }
    launch(k_sketch_swap<GW, true, true>, dim3(G.etiles), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records, GW, 0);
    step<QK, W, LP, IL_SPLIT>(G.V, G.pfx, G.first, G.tiles, worker0, 1, G.records, GW, 0, G.s);
    if (GW == 1)   // (its one slice is the state)
        return 2;
    launch(k_sketch_swap<GW, false, true>, dim3(G.etiles), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records, GW, G.second ? -1 : G.n_records);
    if (G.second)
        return 3;
    launch(k_sketch_back, dim3(dim3(G.etiles, GW)), kIlThreads, 0, G.s, G.V, G.epfx, G.efirst, worker0, G.records, G.n_records);
    return 4;
}

template <int QK>
static int group(const Group &G, int64_t bytes)
{
    const int n = G.V.n_workers, batch = il_batch(n), all = il_width(n) / batch;
    const int at_once = il_at_once(n, G.n_records, bytes);
    int launched = 0;
    for (int b = 0; at_once > 0 && b < all; b += at_once) {
        const int now = std::min(at_once, all - b);
        launched += batch == 2 ? together<QK, 2, 1>(G, 0, now, bytes) : batch == 4 ? together<QK, 4, 1>(G, 0, now, bytes) : together<QK, 4, 2>(G, 8 * b, now, bytes);
    }
    for (int w = 0; at_once == 0 && w < n;) {
        const int left = n - w, now = left >= 8 ? 8 : left >= 4 ? 4 : left >= 2 ? 2 : 1;
        launched += now == 8 ? split<QK, 4, 2>(G, w) : now == 4 ? split<QK, 4, 1>(G, w) : now == 2 ? split<QK, 2, 1>(G, w) : split<QK, 1, 1>(G, w);
        w += now;
    }
    return launched;
}

int il_launch_direct(int qkind, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s)
{
    if (qkind == CONEF_Q_IDENTITY)
        step<CONEF_Q_IDENTITY, 1, 1, IL_SCRATCH>(V, pfx, 0, tiles, 0, V.n_workers, nullptr, 1, 0, s);
    else if (qkind == CONEF_Q_RANDK)
        step<CONEF_Q_RANDK, 1, 1, IL_SCRATCH>(V, pfx, 0, tiles, 0, V.n_workers, nullptr, 1, 0, s);
    else
        step<CONEF_Q_RANDBLOCK, 1, 1, IL_SCRATCH>(V, pfx, 0, tiles, 0, V.n_workers, nullptr, 1, 0, s);
    return 1;
}

int il_launch(int qkind, const DevView &V, const int32_t *pfx, int first, int tiles, const int32_t *epfx, int efirst, int etiles,
              int64_t n_records, float *records, int64_t bytes, bool second, cudaStream_t s)
{
    const Group G{V, pfx, first, tiles, epfx, efirst, etiles, n_records, records, second, s};
    if (qkind == CONEF_Q_IDENTITY)
        return group<CONEF_Q_IDENTITY>(G, bytes);
    return qkind == CONEF_Q_RANDK ? group<CONEF_Q_RANDK>(G, bytes) : group<CONEF_Q_RANDBLOCK>(G, bytes);
}

}  // namespace conef
