// Fused step for the count sketch hashed over whole tensors (Alg. 2 lines 5, 6, 9 with C = count sketch,
// Sec. 4.2.2) and Q in {identity, random-k, random-block-k}.
//
// Every element reads v buckets of the old sketch and adds to the same v buckets of the new one, at
// random places of arrays that do not fit an SM.  The buckets depend on the element only, not on the
// worker.  What bounds the step is the number of random requests, ten per element: to L2 where a group of
// tensors fits it, to DRAM beyond (about 64 bytes each).  Their rate hardly depends on their width, so
// the workers of a context are handled together: their sketches are interleaved, workers innermost, and
// one request of up to 32 bytes reads, and one adds to, the bucket of up to eight workers.  An element is
// one lane's for up to four workers and a pair of lanes' for eight (the two 16-byte accesses of a pair
// make one request).
//
// The state stays one contiguous sketch per worker: a group of tensors is interleaved into a scratch
// (k_sketch_swap, which also clears the new sketch), stepped, and written back to where it was.  Groups
// are as many tensors as keep the scratch inside L2, or one larger tensor.  The scratch is the memory of
// the second sketch, which one worker at a time needs and this does not.  Where the old and the new
// records of a group do not fit it together (a group with more than half of a model), the workers go in
// batches of eight where that is enough; else the states themselves lend the other half (IlForm), at
// the price of one or two more passes over the sketch.
//
// Transformer-big list (210 M elements), 5 x d/10 buckets, eight workers: 90 ms per step one worker at a
// time, 23.2 ms now, of which interleaving takes 3.1; the requests still bound it, ten per element.
// Three CTAs per SM (80 registers); with four (spills) 24.8 ms instead of 23.0 for k_sketch_il.
#pragma once
#include <algorithm>
#include <type_traits>

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
// workers, Transformer-big, in one walk: 25.0 ms with this line, 26.8 always side by side, 28.0 always apart; four
// workers, 16 M elements in L2: 476 us apart, 728 side by side.
constexpr int64_t kIlTogether = 100ll << 20;
// ... unless the old values alone, and then the new ones, mostly stay in L2, and the scratch has room for r: then the sketch is read in one
// walk over the elements and added to in a second, for a write and a read of r and a second hash of the elements.  Steps of models
// of five or six such tensors, 5 x d/10 buckets, one walk and two: eight workers, 4 M elements (64 MB of old values) 2728 and 2345 us,
// 4.8 M (77 MB) 3702 and 3031, 5.9 M (94 MB) 5319 and 4533; four workers, 8 M (64 MB) 5307 and 3102, 12 M (96 MB) 9322 and 6211; two
// workers, 16 M (64 MB) 8853 and 4358.  Above L2: eight workers, 6.9 M (110 MB) 5720 and 5155, 9 M (144 MB) 8505 and 8475; two workers,
// 30 M (120 MB) 20.5 and 13.6 ms.  Transformer-big list, eight workers 24.6 and 23.2 ms.
constexpr int64_t kIlOneSide = 150ll << 20;
// What is saved are requests (two per sketch row), what it costs are 8 bytes of r per element and worker: with batches of eight workers, whose
// requests are a sector each, it does not pay beyond half of L2 but at five rows, nor for the general number of rows.  Eight workers, one walk and
// two, old values in MB: three rows 1.8 M elements, d/5 (58) 986 and 908 us, 6 M, d/10 (58) 2558 and 2240, 2 M, d/2 (96) 1065 and 1088, 6 M, d/5 (115)
// 2650 and 2709, 13 M, d/10 (125) 8068 and 8395; seven rows 5 M, d/20 (56) 9292 and 9077, 2 M, d/5 (90) 2919 and 3112, 5 M, d/10 (112) 9835 and
// 11325; one row 7 M, d/2 (112) 1981 and 2357; five rows 3 M, d/5 (96) 1963 and 1756, 7 M, d/10 (112) 6713 and 6128, 7 M, d/20 (56) 4380 and
// 3382.  Sixteen: three rows 3 M, d/5 (115) 2804 and 2722, 6 M, d/10 (115) 7342 and 7203, seven rows 2 M, d/10 (90) 8073 and 8260.  Two and
// four workers at one, three, five and seven rows, d/2 to d/20, 60 to 130 MB: 0 to 48 % less time.
constexpr int64_t kIlOneSide8 = 70ll << 20;
// n_records of n workers, in batches of gw
inline bool il_two_walks(int64_t n_records, int64_t tiles, int n, int gw, int cs_rows, int64_t bytes)
{
    const int64_t most = gw < 8 || cs_rows == 5 || (cs_rows == 3 && n > 8) ? kIlOneSide : kIlOneSide8;
    return n_records * 8 * n > kIlTogether && n_records * 4 * n <= most && (n_records * 8 + tiles * kIlTile * 4) * n <= bytes;
}
// Below this many elements over all workers the two kernels that interleave cost more than they save: 5 x d/10
// buckets, steps on the states and on records, two, four and eight workers: 256 k elements 29.7, 27.7, 27.7 and
// 32.8, 30.8, 36.5 us; 512 k 45.4, 42.0, 40.0 and 40.9, 32.8, 38.7; 1 M 66.0, 63.5, 60.6 and 53.4, 42.3, 41.0.
constexpr int64_t kIlDirect = 3ll << 17;
// workers of a batch, and of a whole bucket record: 1, 2, 4 or a multiple of 8
inline int il_batch(int n_workers) { return n_workers <= 1 ? 1 : n_workers <= 2 ? 2 : n_workers <= 4 ? 4 : 8; }
inline int il_width(int n_workers) { return (n_workers + il_batch(n_workers) - 1) / il_batch(n_workers) * il_batch(n_workers); }
// Batches stepped together in a scratch of `bytes`; 0: one batch of 8, 4, 2 or 1 workers at a time, with
// records in the states too.
inline int il_at_once(int n_workers, int64_t n_records, int64_t bytes)
{
    return (int)std::min<int64_t>(il_width(n_workers) / il_batch(n_workers), bytes / (n_records * 8 * il_batch(n_workers)));
}

// Whether a group that is the whole model ends in the second sketch (SPLIT, all workers in one batch)
inline bool il_second(int n_workers, int64_t n_records, int64_t bytes)
{
    return il_at_once(n_workers, n_records, bytes) == 0 && (n_workers == 2 || n_workers == 4 || n_workers == 8) &&
           n_records * 8 * n_workers <= kIlTogether;
}
// Where the records are:
//   SCRATCH  all in the scratch, next to one another or apart (kIlTogether)
//   SPLIT    old ones in the scratch, new ones in the place of the states; for groups inside L2
//   FOLD     a tensor beyond L2, old next to new: the first half of the entries in the scratch, the second in
//            the place of the states.  On the way in and out a record of the scratch carries the entry of
//            the second half in the slot that is not in use, which frees the states.
// 5 x d/10 buckets of one 8192 x 8192 matrix: two, four, eight workers 16.2, 17.5, 17.6 ms with room for all
// records, 19.4, 23.1, 27.0 under SPLIT, 16.9, 18.4, 18.0 under FOLD.  Three and five workers go as 2 + 1 and
// 4 + 1 (30.5 and 32.0 ms) where records of four and eight fit and take 17.4 with room for them: no
// form holds more records than two sketches per worker have room for.
enum IlForm { IL_SCRATCH, IL_SPLIT, IL_FOLD };

// Where record e (of F floats) of a batch lies among its states: in slice e / (c / F) of the c floats (a
// multiple of 64) of each, counted from the first
struct IlSlices {
    uint32_t per, magic;   // records per slice
    int64_t stride;        // floats from state to state
    __device__ __forceinline__ IlSlices(uint32_t n, uint32_t F, int64_t state_stride)
    {
        per = (n + 63u) / 64u * (64u / F);
        magic = 0xFFFFFFFFu / per;
        stride = state_stride / 4;
    }
    __device__ __forceinline__ int64_t at(uint32_t e, uint32_t F) const
    {
        uint32_t q = __umulhi(e, magic), r = e - q * per;   // e / per or one less
        if (r >= per) {
            r -= per;
            ++q;
        }
        return q * stride + (int64_t)r * F;
    }
};

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
// r of an element, between the two walks
template <int W>
__device__ __forceinline__ IlVec<W> il_load_once(const float *p)
{
    IlVec<W> r;
    if constexpr (W == 4) {
        const float4 t = __ldcs((const float4 *)p);
        r.v[0] = t.x; r.v[1] = t.y; r.v[2] = t.z; r.v[3] = t.w;
    } else if constexpr (W == 2) {
        const float2 t = __ldcs((const float2 *)p);
        r.v[0] = t.x; r.v[1] = t.y;
    } else {
        r.v[0] = __ldcs(p);
    }
    return r;
}
template <int W>
__device__ __forceinline__ void il_store_once(float *p, const IlVec<W> &a)
{
    if constexpr (W == 4)
        __stcs((float4 *)p, make_float4(a.v[0], a.v[1], a.v[2], a.v[3]));
    else if constexpr (W == 2)
        __stcs((float2 *)p, make_float2(a.v[0], a.v[1]));
    else
        __stcs(p, a.v[0]);
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
// VR sketch rows (0: V.cs_rows, up to 7); W workers per lane, LP lanes per element, the first of them
// worker0.  GW = 1 in SCRATCH form: no records, the states themselves.
//
// WALK 0: the whole step; 1: without the additions, r to `resid` (GW floats per element, elements by tile); 2: the additions.
template <int QK, int VR, int W, int LP, int FORM, int WALK>
__global__ void __launch_bounds__(kIlThreads, W == 4 ? 3 : 4)
k_sketch_il(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx, int first, int worker0, float *records, uint32_t stride,
            int64_t newoff, float *resid)
{
    constexpr int VM = VR ? VR : 7, GW = W * LP;
    const int v = VR ? VR : V.cs_rows;
    grid_release();
    const int tile = first + (int)blockIdx.x;
    const int li = find_layer(pfx, V.n_layers, tile);
    const LayerDesc &L = V.layers[li];
    const uint32_t d = (uint32_t)L.d, w = (uint32_t)L.w;
    const uint32_t j0 = (uint32_t)(tile - pfx[li]) * (uint32_t)kIlTile;
    const uint32_t left = min(d - j0, (uint32_t)kIlTile);   // elements of this tile
    const int sub = threadIdx.x & (LP - 1);
    const int w0 = worker0 + blockIdx.y * GW + sub * W;     // this lane's first worker
    if (GW == 1)
        stride = 1u;
    const float *So;
    float *Sn;
    const IlSlices slices((uint32_t)(FORM != IL_SCRATCH ? v * w : 1u), FORM == IL_FOLD ? 2 * GW : GW, V.state_stride);
    const uint32_t half = ((uint32_t)v * w + 1u) / 2u;   // FOLD: entries in the scratch
    if (FORM != IL_SCRATCH) {
        So = records + L.sk_off * stride + sub * W;
        Sn = (float *)(V.state + worker0 * V.state_stride + L.a_off) + sub * W;
    } else if (GW == 1) {
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
    grid_wait();
    uint32_t blk_start = 0;
    if (QK == CONEF_Q_RANDBLOCK)
        blk_start = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)V.step), d, (uint32_t)L.k);
    const uint32_t *__restrict__ bits = V.selbits + L.selbits_off;
    const uint32_t kept = (uint32_t)L.k;
    const int64_t goff = L.g_off, moff = L.msgv_off;
    const float lr = V.lr, omb = V.omb, beta = V.beta;
    if (WALK != 0)
        resid += ((uint64_t)blockIdx.y * gridDim.x + blockIdx.x) * (kIlTile * GW) + sub * W;
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
                const uint32_t e = (uint32_t)i * w + bk[i];
                if (WALK == 2)
                    continue;
                if (FORM == IL_FOLD)
                    rec[i] = il_load<W>(e < half ? So + (uint64_t)e * (2 * GW) : Sn + slices.at(e - half, 2 * GW));
                else
                    rec[i] = il_load<W>(So + ((uint64_t)i * w + bk[i]) * stride);
            }
        }
        IlVec<W> val;
        if (WALK == 2) {
            val = il_load_once<W>(resid + q * GW);
        } else {
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
            if (WALK == 1) {
                il_store_once<W>(resid + q * GW, val);
                continue;
            }
        }
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
                    const uint32_t e = (uint32_t)i * w + bk[i];
                    if (FORM == IL_FOLD)
                        il_add<W>((e < half ? records + sub * W + (uint64_t)e * (2 * GW) : Sn + slices.at(e - half, 2 * GW)) + GW, a);
                    else if (FORM == IL_SPLIT && GW > 1)
                        il_add<W>(Sn + slices.at(e, GW), a);
                    else
                        il_add<W>(Sn + ((uint64_t)i * w + bk[i]) * stride, a);
                }
        }
    }
}

// IN: states -> old values of the records, and the new ones cleared (SPLIT: the states, whose place they
// take); else: new values -> states (SPLIT: from their slices to one sketch after the other in `records`, or
// to the second sketch, padding included, with newoff < 0).  A thread has one entry of all GW workers (coalesced over the entries of a worker); the records,
// exchanged through shared memory, are accessed 16 bytes per lane over contiguous memory.
template <int GW, bool IN, bool SPLIT>
__global__ void __launch_bounds__(kIlThreads) k_sketch_swap(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx,
                                                            int first, int worker0, float *records, uint32_t stride,
                                                            int64_t newoff)
{
    constexpr int PW = GW < 4 ? GW : 4, H = GW / PW;   // floats per piece, pieces of a record's old (or new) values
    constexpr int PITCH = GW == 8 ? 9 : GW;            // (entries of a warp in different banks)
    using Piece = typename std::conditional<PW == 1, float, typename std::conditional<PW == 2, float2, float4>::type>::type;
    __shared__ float buf[kIlThreads * PITCH];
    grid_release();
    const int tile = first + (int)blockIdx.x;
    const int li = find_layer(pfx, V.n_layers, tile);
    const LayerDesc &L = V.layers[li];
    grid_wait();
    const int64_t n = (int64_t)V.cs_rows * L.w;
    const int64_t e0 = (int64_t)(tile - pfx[li]) * kIlEntries;
    const int w0 = worker0 + blockIdx.y * GW, t = threadIdx.x;
    float *const states = (float *)(V.state + w0 * V.state_stride + L.a_off);
    const int64_t pitch = V.state_stride / 4;
    const IlSlices slices((uint32_t)(SPLIT ? n : 1), GW, V.state_stride);
    for (int q = 0; q < kIlEntries / kIlThreads; ++q) {
        const int64_t b = e0 + q * kIlThreads, e = b + t;
        if (b >= n)
            return;   // (uniform over the CTA)
        const int have = (int)min((int64_t)kIlThreads, n - b);
        float *rec = records + (L.sk_off + b) * stride + blockIdx.y * (stride / gridDim.y);
        float r[GW];
        if (IN) {
#pragma unroll
            for (int x = 0; x < GW; ++x) {
                const bool in = t < have && w0 + x < V.n_workers;
                r[x] = in ? __ldcs(states + x * pitch + e) : 0.f;
                if (SPLIT && in)
                    states[x * pitch + e] = 0.f;
            }
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
                    if (!SPLIT) {
#pragma unroll
                        for (int x = 0; x < PW; ++x)
                            zf[x] = 0.f;
                        *(Piece *)(at + newoff) = z;
                    }
                } else {
                    z = *(const Piece *)(SPLIT ? states + slices.at((uint32_t)(b + en), GW) + part * PW : at + newoff);
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
                    if (SPLIT && newoff < 0)
                        ((float *)(V.state_new + (w0 + x) * V.state_stride + L.a_off))[e] = buf[t * PITCH + x];
                    else if (SPLIT)
                        records[x * newoff + L.sk_off + e] = buf[t * PITCH + x];
                    else if (w0 + x < V.n_workers)
                        __stcs(states + x * pitch + e, buf[t * PITCH + x]);
            } else if (SPLIT && newoff < 0 && e < (n + 63) / 64 * 64) {
#pragma unroll
                for (int x = 0; x < GW; ++x)
                    ((float *)(V.state_new + (w0 + x) * V.state_stride + L.a_off))[e] = 0.f;
            }
        }
    }
}

// launchers (conef_ilsketch.cu), each of which returns the number of kernels launched: the step on the states themselves,
// one worker per blockIdx.y, all tensors; and the step of a group of n_records records: tiles [first, first + tiles) of
// elements, [efirst, efirst + etiles) of sketch entries, in a scratch of `bytes`; second: the result of a group that
// il_second accepts is left in V.state_new.
int il_launch_direct(int qkind, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s);
int il_launch(int qkind, const DevView &V, const int32_t *pfx, int first, int tiles, const int32_t *epfx, int efirst, int etiles,
              int64_t n_records, float *records, int64_t bytes, bool second, cudaStream_t s);

}  // namespace conef
