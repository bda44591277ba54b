// Device helpers shared by the kernel headers: tile -> tensor search, warp reductions, decoding of a
// stored error element (Alg. 2 line 5), membership in a stored draw of Q.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <float.h>

#include "conef_internal.h"
#include "conef_hash.cuh"

namespace conef {

// Last tensor l with pfx[l] <= bid (prefix tables have n + 1 entries), by a whole warp: 32 entries per
// round, so two dependent loads for up to 1024 tensors.  A binary search was eight to ten of them, each a
// trip to L2 at the start of a kernel.
__device__ __forceinline__ int find_layer(const int32_t *__restrict__ pfx, int n, int bid)
{
    const int lane = threadIdx.x & 31;
    int lo = 0;   // pfx[lo] <= bid, and the tensor is one of the n from lo on
    while (n > 1) {
        const int step = (n + 31) >> 5, at = lane * step;
        const bool le = at < n && __ldg(pfx + lo + at) <= bid;
        const int skip = (__popc(__ballot_sync(0xffffffffu, le)) - 1) * step;
        lo += skip;
        n = min(step, n - skip);
    }
    return lo;
}

// For kernels launched by launch() (conef_internal.h).  The kernel ahead in the stream is done and what it
// wrote is visible:
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// ... and a pointer to what it wrote, so that no load through it (loads of constant memory, as __ldg is taken
// for, may pass a memory clobber) comes before the wait:
template <class T>
__device__ __forceinline__ T *fresh(T *p)
{
    asm volatile("" : "+l"(p));
    return p;
}
// ... or, of a kernel whose registers do not allow that, the tensor, before anything is computed from it:
__device__ __forceinline__ void grid_wait(int &li) { asm volatile("griddepcontrol.wait;" : "+r"(li) : : "memory"); }
// The kernel behind may come onto the SMs before this one's CTAs leave them.  For grids that leave room on the SMs
// only: CTAs that wait hold registers and shared memory.  Released always, the count sketch over whole tensors
// took 36 ms instead of 24; never, the index sets of 54 convolutions 499 us instead of 408 (one CTA per SM; with two or
// eight 430).
__device__ __forceinline__ void grid_release()
{
    if (gridDim.x * gridDim.y <= (unsigned)kPlanSMs)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Loads of what the kernel itself does not write: as free to be moved and batched as __ldg (they depend on the address
// alone, which has to come from behind grid_wait(), by fresh() or through the tensor), but not by the non-coherent path, which
// is for memory that nobody writes while the grid lives: a chained kernel's CTAs live while the one ahead writes its results.
__device__ __forceinline__ float load_global(const float *p)
{
    float v;
    asm("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float2 load_global(const float2 *p)
{
    float2 v;
    asm("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 load_global(const float4 *p)
{
    float4 v;
    asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t load_global(const uint32_t *p)
{
    uint32_t v;
    asm("ld.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ uint2 load_global(const uint2 *p)
{
    uint2 v;
    asm("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ uint32_t load_global(const uint8_t *p)
{
    uint32_t v;
    asm("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ unsigned short load_global(const unsigned short *p)
{
    unsigned short v;
    asm("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// ... OFF bytes behind p
template <int OFF>
__device__ __forceinline__ float load_global_at(const float *p)
{
    float v;
    asm("ld.global.f32 %0, [%1+%2];" : "=f"(v) : "l"(p), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ float2 load_global_at(const float2 *p)
{
    float2 v;
    asm("ld.global.v2.f32 {%0, %1}, [%2+%3];" : "=f"(v.x), "=f"(v.y) : "l"(p), "n"(OFF));
    return v;
}
template <int OFF>
__device__ __forceinline__ float4 load_global_at(const float4 *p)
{
    float4 v;
    asm("ld.global.v4.f32 {%0, %1, %2, %3}, [%4+%5];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "n"(OFF));
    return v;
}

template <int OFF>   // ... of what is not read again
__device__ __forceinline__ float load_stream_at(const float *p)
{
    float v;
    asm("ld.global.cs.f32 %0, [%1+%2];" : "=f"(v) : "l"(p), "n"(OFF));
    return v;
}

template <int OFF>   // ... where `in` says so, without a branch; v stays what it is elsewhere
__device__ __forceinline__ void load_stream_if(float &v, const float *p, uint32_t in)
{
    asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t@q ld.global.cs.f32 %0, [%1+%2];\n\t}" : "+f"(v) : "l"(p), "n"(OFF), "r"(in));
}

// Loads of what other CTAs of the same launch wrote before a ticket or a flag: past L1, and volatile with
// a memory clobber, so that the compiler may not move them ahead of it (it may move __ldcg, whose
// result depends on its address alone).
__device__ __forceinline__ uint32_t load_cg(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.global.cg.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint2 load_cg(const uint2 *p)
{
    uint2 v;
    asm volatile("ld.global.cg.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float4 load_cg(const float4 *p)
{
    float4 v;
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void load_cg(const uint32_t *p, uint32_t (&v)[8])   // 32 bytes, 16-byte aligned
{
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "l"(p) : "memory");
    asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]) : "l"(p + 4) : "memory");
}

// one tile of a 1-D tensor that passes through, by 256 threads: message eta g
__device__ __forceinline__ void pass_tile(const DevView &V, const LayerDesc &L, int tile)
{
    constexpr int PER = kPassTile / 256;
    const int worker = blockIdx.y;
    const int64_t j0 = (int64_t)tile * kPassTile;
    const float *__restrict__ g = V.grads[worker] + L.g_off + j0;
    float *__restrict__ out = V.msg1d + worker * V.msg1d_stride + L.msg1d_off + j0;
    const int n = (int)min((int64_t)kPassTile, L.d - j0);
    float v[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int q = u * 256 + threadIdx.x;
        v[u] = q < n ? __ldcs(g + q) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int q = u * 256 + threadIdx.x;
        if (q < n)
            out[q] = __fmul_rn(V.lr, v[u]);
    }
}

__device__ __forceinline__ float warp_max(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// ------------------------------------------------------------------ decode (S1)
__device__ __forceinline__ float load_scale(const uint8_t *__restrict__ b, int64_t blk, int half)
{
    if (half)
        return __half2float(__ushort_as_half(((const unsigned short *)b)[blk]));
    return ((const float *)b)[blk];
}

__device__ __forceinline__ float median_small(float *x, int v)
{
    if (v == 1)
        return x[0];
    if (v == 3)
        return fmaxf(fminf(x[0], x[1]), fminf(fmaxf(x[0], x[1]), x[2]));
    if (v == 5) {
        // median of five by a fixed exchange network
        float a = fminf(x[0], x[1]), b = fmaxf(x[0], x[1]);
        float c = fminf(x[2], x[3]), d = fmaxf(x[2], x[3]);
        float lo = fmaxf(a, c);   // the smaller of the two minima cannot be the median
        float hi = fminf(b, d);   // nor the larger of the two maxima
        float e = x[4];
        // median of {lo, hi, e} together with the leftover middle pair
        float m1 = fminf(lo, hi), m2 = fmaxf(lo, hi);
        return fmaxf(m1, fminf(m2, e));
    }
    // v == 7: insertion sort
    for (int a = 1; a < v; ++a) {
        float val = x[a];
        int b = a - 1;
        while (b >= 0 && x[b] > val) {
            x[b + 1] = x[b];
            --b;
        }
        x[b + 1] = val;
    }
    return x[v / 2];
}

struct SketchKeys {
    uint64_t st[7];
};
__device__ __forceinline__ SketchKeys sketch_keys(uint64_t seed, int tensor, int v)
{
    SketchKeys k;
#pragma unroll
    for (int i = 0; i < 7; ++i)
        k.st[i] = i < v ? stream_key(seed, (uint64_t)tensor, (uint64_t)i) : 0;
    return k;
}

// Count sketch applied run by run (cs_chunk > 0): the window [lo, lo + width) of every sketch row
// that the run of element j owns.  Runs are cs_chunk consecutive elements, the last one also takes
// the remainder; windows are cut in proportion to the elements.  One run: the whole row.
__device__ __forceinline__ void sketch_window_of_run(uint32_t c, uint32_t nc, uint32_t chunk, uint32_t d, uint32_t w,
                                                     uint32_t &lo, uint32_t &width)
{
    const uint64_t b0 = c == 0 ? 0ull : (uint64_t)w * ((uint64_t)c * chunk) / d;          // w c E <= w d < 2^64
    const uint64_t b1 = c == nc - 1 ? (uint64_t)w : (uint64_t)w * ((uint64_t)(c + 1) * chunk) / d;
    lo = (uint32_t)b0;
    width = (uint32_t)(b1 - b0);
}
__device__ __forceinline__ void sketch_window(const DevView &V, const LayerDesc &L, uint32_t j, uint32_t &lo,
                                              uint32_t &width)
{
    lo = 0;
    width = (uint32_t)L.w;
    if (V.cs_chunk > 0) {
        const uint32_t chunk = (uint32_t)V.cs_chunk, d = (uint32_t)L.d;
        uint32_t nc = d / chunk;
        nc = nc < 1 ? 1 : nc;
        uint32_t c = j / chunk;
        c = c > nc - 1 ? nc - 1 : c;
        if (nc > 1)
            sketch_window_of_run(c, nc, chunk, d, (uint32_t)L.w, lo, width);
    }
}

// Alg. 2 line 5, p = eta g + e; with partial error feedback (Alg. 4 line 5) p = eta g + (1-beta) e,
// the product rounded first.  V.omb is 1 for beta = 0, and 1 * e is e.
__device__ __forceinline__ float form_p(const DevView &V, float g, float e)
{
    return __fmaf_rn(V.lr, g, __fmul_rn(V.omb, e));
}
// whether this codec keeps the second state of iConEF-v1 (Alg. 3)
template <int CK>
__device__ __forceinline__ bool has_second(const DevView &V)
{
    return (CK == CONEF_C_IDENTITY || CK == CONEF_C_INT8 || CK == CONEF_C_INT4) && V.iconef == 1;
}

// iConEF-v2: the second application of Q in a step draws from the stream of step t + 2^62
constexpr int64_t kSecondDraw = 1ll << 62;
// Message slot of member j of a random-k draw whose bitmap word is `word` (conef_select.cuh)
__device__ __forceinline__ uint32_t draw_slot(const LayerDesc &L, const uint16_t *__restrict__ wordoff,
                                              const uint32_t *__restrict__ tileoff, uint32_t word, uint32_t j)
{
    return tileoff[L.tileoff_off + j / kHistTile] + wordoff[L.wordoff_off + (j >> 5)] + __popc(word & ((1u << (j & 31u)) - 1u));
}
// Whether element j belongs to a stored draw of Q (the bitmap and offsets the selection leaves, or
// the block of random-block-k), and its slot among the k values.
template <int QK>
__device__ __forceinline__ bool draw_member(const LayerDesc &L, const uint32_t *__restrict__ selbits,
                                            const uint16_t *__restrict__ wordoff,
                                            const uint32_t *__restrict__ tileoff, uint32_t blk_start, uint32_t j,
                                            uint32_t &slot)
{
    if (QK == CONEF_Q_RANDBLOCK) {
        slot = j - blk_start;   // wraps to a large value below the block
        return slot < (uint32_t)L.k;
    }
    const uint32_t word = selbits[L.selbits_off + (j >> 5)];
    if (!((word >> (j & 31u)) & 1u))
        return false;
    slot = draw_slot(L, wordoff, tileoff, word, j);
    return true;
}

// e_j of one element from a worker's stored state (Alg. 2 line 5, decode).
// Row-sketch entries are fp32 or, with a binary16 sketch, halves (stored saturated to the finite
// half range, rounded to nearest even).  idx counts entries.
__device__ __forceinline__ float rs_load1(const void *T, size_t idx, bool half)
{
    return half ? __half2float(((const __half *)T)[idx]) : ((const float *)T)[idx];
}
__device__ __forceinline__ void rs_load4(const void *T, size_t idx, bool half, float (&out)[4])
{
    if (half) {
        const uint2 raw = *(const uint2 *)((const __half *)T + idx);
        const float2 a = __half22float2(*(const __half2 *)&raw.x), b = __half22float2(*(const __half2 *)&raw.y);
        out[0] = a.x; out[1] = a.y; out[2] = b.x; out[3] = b.y;
    } else {
        const float4 t = *(const float4 *)((const float *)T + idx);
        out[0] = t.x; out[1] = t.y; out[2] = t.z; out[3] = t.w;
    }
}
__device__ __forceinline__ unsigned short rs_to_half(float f)
{
    f = f > 65504.0f ? 65504.0f : f;
    f = f < -65504.0f ? -65504.0f : f;
    return __half_as_ushort(__float2half_rn(f));
}
__device__ __forceinline__ void rs_store1(void *T, size_t idx, bool half, float f)
{
    if (half)
        ((unsigned short *)T)[idx] = rs_to_half(f);
    else
        ((float *)T)[idx] = f;
}
__device__ __forceinline__ void rs_store4(void *T, size_t idx, bool half, float a, float b, float c, float d)
{
    if (half) {
        uint2 raw;
        raw.x = (uint32_t)rs_to_half(a) | ((uint32_t)rs_to_half(b) << 16);
        raw.y = (uint32_t)rs_to_half(c) | ((uint32_t)rs_to_half(d) << 16);
        *(uint2 *)((unsigned short *)T + idx) = raw;
    } else {
        *(float4 *)((float *)T + idx) = make_float4(a, b, c, d);
    }
}

// second: the state q of iConEF (Alg. 3) instead of the first one.
template <int CK>
__device__ __forceinline__ float decode_elem(const DevView &V, const LayerDesc &L,
                                             const uint8_t *__restrict__ st, uint32_t j,
                                             const SketchKeys &keys, bool second = false)
{
    const int64_t aoff = second ? L.a2_off : L.a_off, boff = second ? L.b2_off : L.b_off;
    if (CK == CONEF_C_IDENTITY)
        return ((const float *)(st + aoff))[j];
    if (CK == CONEF_C_INT8) {
        int c = ((const signed char *)(st + aoff))[j];
        return __fmul_rn((float)c, load_scale(st + boff, j / (uint32_t)L.unit, V.scale_half));
    }
    if (CK == CONEF_C_INT4) {
        unsigned byte = (st + aoff)[j >> 1];
        int nib = (j & 1) ? (byte >> 4) : (byte & 0xF);
        int c = (nib ^ 8) - 8;
        return __fmul_rn((float)c, load_scale(st + boff, j / (uint32_t)L.unit, V.scale_half));
    }
    if (CK == CONEF_C_STOCHQUANT) {
        const int c = V.sq_wide ? (int)((const short *)(st + L.a_off))[j] : (int)((const signed char *)(st + L.a_off))[j];
        return __fmul_rn((float)c, ((const float *)(st + L.b_off))[j / (uint32_t)L.unit]);
    }
    if (CK == CONEF_C_ROWSKETCH) {
        // row sketch: median over sketch rows of s_i(a) * T_i[h_i(a)][b]; buckets and signs of
        // the matrix rows come from the table built when the context was created
        const void *T = st + L.a_off;
        const bool th = V.scale_half != 0;
        const uint32_t m = (uint32_t)L.cols, a = j / m, b = j - a * m;
        const uint32_t *info = V.rs + L.rs_info_off;
        float est[7];
#pragma unroll
        for (int i = 0; i < 7; ++i) {
            if (i < V.cs_rows) {
                const uint32_t in = info[(int64_t)i * L.rows + a];
                const float t = rs_load1(T, (size_t)(((int64_t)i * L.w + (in & 0x7FFFFFFFu)) * m + b), th);
                est[i] = (in >> 31) ? -t : t;
            } else
                est[i] = 0.f;
        }
        return median_small(est, V.cs_rows);
    }
    // count sketch: median over rows of s_i(j) * S[i][h_i(j)]
    const float *S = (const float *)(st + L.a_off);
    float est[7];
    uint32_t lo, width;
    sketch_window(V, L, j, lo, width);
#pragma unroll
    for (int i = 0; i < 7; ++i) {
        if (i < V.cs_rows) {
            uint64_t u = h64(keys.st[i], j);
            uint64_t b = lo + (((u >> 32) * (uint64_t)width) >> 32);
            float s = S[(int64_t)i * L.w + (int64_t)b];
            est[i] = (u & 1) ? -s : s;
        } else
            est[i] = 0.f;
    }
    return median_small(est, V.cs_rows);
}

}  // namespace conef
