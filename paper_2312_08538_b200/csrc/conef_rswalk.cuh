// The low-rank passes on a row-sketch state with one sketch row (conef_rowsketch.cuh) where 16-byte loads line up.
//
// A CTA owns kRsBuckets buckets and 512 columns, four per thread, and walks the rows of its buckets in the order of
// the bucket lists, as one sequence.  The entries (row, sign) of all its buckets, which are contiguous in the tables, and their
// rows of P_hat are in shared memory before the walk starts.  The gradient comes by asynchronous copies, a batch of rows ahead, each
// thread's own, so that it takes no registers and no barrier; the old sketch entry of the next bucket is loaded at the start of the one before.
// The rank is a constant (2, 4) where it is the configured one; arrays have room for the configured one elsewhere.
//
// GPT-2-small list, rank 4, binary16 sketch, one worker: with the gradient in registers, the old entries in shared memory and
// the body for any rank beside it (94 registers, five CTAs per SM) the passes took 169 / 148 / 177 us, issue slots 40 to 50 % busy;
// now 131 / 114 / 125 us (72 registers, seven CTAs; step and update 698 -> 579 us), 60 to 72 % busy.  Rank 2, 33 M elements of two
// workers, fp32 sketch: 120 / 98 / 130 -> 64 / 59 / 69 us (eight CTAs).  The single-phase compressors stay with rs_body (3 % slower here).
#pragma once
#include "conef_fast.cuh"
#include "conef_kernels.cuh"

namespace conef {

constexpr int kRwBatch = 4;      // rows of a batch
// Rows of the gradient under way per thread, in shared memory.  Sixteen leave room for six CTAs per SM: passes 147 / 134 / 145 us instead
// of 131 / 117 / 127 on the list above.
constexpr int kRwRing = 8;
constexpr int kRwEntries = 128;  // entries staged at a time (eight buckets of ten rows expect 80)
constexpr int kRwCols = kRsThreads * 4;

struct alignas(16) RwShared {
    float4 ring[kRwRing][kRsThreads];                  // each thread's own
    float ph[kRwEntries + kRwBatch][CONEF_MAX_RANK];   // rows of P_hat of the staged entries; a constant rank: packed
    uint32_t ent[kRwEntries + kRwBatch];               // row | sign << 31
    uint32_t start[kRsBuckets + 1];
};

// PASS 1, 2, 3: the low-rank passes; 3 writes the new sketch.  EXACT: rank RK (2, 4) and rows of the factors on their vector's
// boundaries; else any rank up to RK.
template <int PASS, int RK, bool EXACT>
__device__ __forceinline__ void rs_walk(const DevView &V, const LayerDesc &L, const uint32_t local, RwShared &S)
{
    constexpr bool NEED_PH = PASS != 1;
    static_assert(!EXACT || RK == 2 || RK == 4, "vectors of a row");
    const int worker = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t m = (uint32_t)L.cols, w = (uint32_t)L.w, slabs = (m + kRwCols - 1) / kRwCols;
    const uint32_t grp = local / slabs, slab = local - grp * slabs, h0 = grp * kRsBuckets, nb = min((uint32_t)kRsBuckets, w - h0);
    const uint32_t b = slab * kRwCols + tid * 4;   // this thread's first column
    const bool colok = b < m;                      // (four divides cols: all or none of them exist)
    const bool live = b - lane * 4u < m;           // some of the warp's do; a warp without any helps to stage and no more
    const bool th = V.scale_half != 0;
    const int r = EXACT ? RK : L.rank;
    if (!colok) {
#pragma unroll
        for (int u = 0; u < kRwRing; ++u)
            S.ring[u][tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if ((uint32_t)tid <= nb)
        S.start[tid] = V.rs[L.rs_ptr_off + h0 + tid];
    __syncthreads();
    const uint32_t *__restrict__ brow = V.rs + L.rs_row_off;
    const uint32_t first = S.start[0], last = S.start[nb];
    grid_wait();   // (the tables do not change)
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off) + (colok ? b : 0u);
    const float *__restrict__ phat = fresh(V.phat + L.msgp_off);
    // the old entries of the next bucket, as stored (binary16: half of them)
    const uint8_t *told_at = fresh(V.state + worker * V.state_stride + L.a_off) + ((size_t)h0 * m + (colok ? b : 0u)) * (th ? 2 : 4);
    const size_t told_step = (size_t)m * (th ? 2 : 4);
    uint4 told = make_uint4(0u, 0u, 0u, 0u);
    auto fetch_told = [&] {
        if (!colok) {
        } else if (th) {
            const uint2 t = load_global((const uint2 *)told_at);
            told.x = t.x; told.y = t.y;
        } else {
            const float4 t = load_global((const float4 *)told_at);
            told = make_uint4(__float_as_uint(t.x), __float_as_uint(t.y), __float_as_uint(t.z), __float_as_uint(t.w));
        }
        told_at += told_step;
    };
    fetch_told();

    float q[4][RK];   // PASS 1: Q_{t-1}[b .. b + 3][:], 2: accumulators of Q_i[b .. b + 3][:], 3: Q_i[...]
    {
        const float *__restrict__ qp = fresh((PASS == 1 ? V.qprev : V.msgq + worker * V.msgq_stride) + L.msgq_off) + (size_t)(colok ? b : 0u) * r;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            if (PASS == 2) {
#pragma unroll
                for (int c = 0; c < RK; ++c)
                    q[x][c] = 0.f;
            } else if (EXACT && RK == 4) {
                const float4 t = load_global((const float4 *)qp + x);
                q[x][0] = t.x; q[x][1] = t.y; q[x][2 % RK] = t.z; q[x][3 % RK] = t.w;
            } else if (EXACT && RK == 2) {
                const float2 t = load_global((const float2 *)qp + x);
                q[x][0] = t.x; q[x][1] = t.y;
            } else {
#pragma unroll
                for (int c = 0; c < RK; ++c)
                    q[x][c] = c < r ? load_global(qp + x * r + c) : 0.f;
            }
            if (PASS == 1 && !colok) {   // (columns that do not exist add nothing to a row's sum)
#pragma unroll
                for (int c = 0; c < RK; ++c)
                    q[x][c] = 0.f;
            }
        }
    }
    // PASS 1: which of a warp's totals of kRwBatch rows ends up in this lane
    constexpr int NV = kRwBatch * RK;
    int p1_idx = 0, p1_plain = 32;
    float *__restrict__ ppart = nullptr;
    if (PASS == 1) {
        int hh = NV;
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1)
            if (hh > 1) {
                hh >>= 1;
                if (lane & o)
                    p1_idx += hh;
                p1_plain = o;
            }
        ppart = V.ppart + worker * V.ppart_stride + L.pp_off + (size_t)(slab * (kRsThreads / 32) + warp) * (uint32_t)L.rows * r;
    }
    void *Tnew = V.state_new + worker * V.state_stride + L.a_off;
    const float lr = V.lr, omb = V.omb, beta = V.beta;

    double acc[4];
    float eb[4];              // (1 - beta) e, but for the row's sign
    uint32_t bucket = 0, next = first;   // the bucket that ends before entry `next`, one past the current one
    auto open = [&]() {       // the first row of a bucket
        float t[4];
        if (th) {
            const float2 u = __half22float2(*(const __half2 *)&told.x), v = __half22float2(*(const __half2 *)&told.y);
            t[0] = u.x; t[1] = u.y; t[2] = v.x; t[3] = v.y;
        } else {
            t[0] = __uint_as_float(told.x); t[1] = __uint_as_float(told.y); t[2] = __uint_as_float(told.z); t[3] = __uint_as_float(told.w);
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            eb[x] = __fmul_rn(omb, t[x]);   // (the sign commutes with the rounding)
            if (PASS == 3)
                acc[x] = (double)__fmul_rn(beta, t[x]);
        }
        ++bucket;
        next = S.start[bucket];
        if (bucket < nb)
            fetch_told();
    };
    auto close = [&]() {      // ... and its last
        if (PASS == 3 && colok)
            rs_store4(Tnew, (size_t)(h0 + bucket - 1) * m + b, th, (float)acc[0], (float)acc[1], (float)acc[2], (float)acc[3]);
    };

    for (uint32_t c0 = first; c0 < last || c0 == first; c0 += kRwEntries) {
        const uint32_t n = min((uint32_t)kRwEntries, last - c0);   // entries of this chunk
        if (c0 != first)
            __syncthreads();   // (the previous chunk is done)
        for (uint32_t x = tid; x < n; x += kRsThreads)
            S.ent[x] = brow[c0 + x];
        __syncthreads();
        if (NEED_PH) {
            for (uint32_t x = tid; x < n; x += kRsThreads) {
                const float *src = phat + (size_t)(S.ent[x] & 0x7FFFFFFFu) * r;
                float *const dst = EXACT ? &S.ph[0][0] + x * RK : S.ph[x];
                if (EXACT && RK == 4) {
                    cp_async16(dst, src);
                } else if (EXACT && RK == 2) {
                    cp_async_small<8>(dst, src);
                } else {
                    for (int c = 0; c < r; ++c)
                        cp_async_small<4>(dst + c, src + c);
                }
            }
        }
        cp_async_commit();
        // a batch of rows is one group of copies; one batch of the ring is read while the others are under way
        auto issue = [&](uint32_t x0) {
#pragma unroll
            for (int u = 0; u < kRwBatch; ++u)
                if (x0 + u < n && colok)
                    cp_async16(&S.ring[(x0 + u) % kRwRing][tid], g + (size_t)(S.ent[x0 + u] & 0x7FFFFFFFu) * m);
            cp_async_commit();
        };
#pragma unroll
        for (int u = 0; u < kRwRing - kRwBatch; u += kRwBatch)
            issue(u);
        if (NEED_PH) {
            cp_async_wait<kRwRing / kRwBatch - 1>();
            __syncthreads();
        }
        if (PASS == 1 && !live)   // (their partial sums are added like all others)
            for (uint32_t x = lane; x < n * r; x += 32)
                ppart[(size_t)(S.ent[x / r] & 0x7FFFFFFFu) * r + x % r] = 0.f;
        for (uint32_t x0 = 0; live && x0 < n; x0 += kRwBatch) {
            issue(x0 + kRwRing - kRwBatch);
            cp_async_wait<kRwRing / kRwBatch - 1>();
            float pr[PASS == 1 ? kRwBatch : 1][RK];
#pragma unroll
            for (int u = 0; u < kRwBatch; ++u) {
                const uint32_t x = x0 + u;
                if (PASS == 1) {
#pragma unroll
                    for (int c = 0; c < RK; ++c)
                        pr[PASS == 1 ? u : 0][c] = 0.f;
                }
                if (x >= n)
                    continue;   // (uniform)
                while (c0 + x == next) {   // (uniform; buckets without rows open and close at once)
                    if (bucket)
                        close();
                    open();
                }
                const uint32_t sgn = S.ent[x] & 0x80000000u;
                const float4 gv = S.ring[x % kRwRing][tid];
                const float gq[4] = {gv.x, gv.y, gv.z, gv.w};
                float p[4];
#pragma unroll
                for (int y = 0; y < 4; ++y)   // Alg. 2 (4) line 5
                    p[y] = __fmaf_rn(lr, gq[y], __uint_as_float(__float_as_uint(eb[y]) ^ sgn));
                if constexpr (PASS == 1) {
#pragma unroll
                    for (int c = 0; c < RK; ++c)
#pragma unroll
                        for (int y = 0; y < 4; ++y)
                            pr[u][c] = __fmaf_rn(p[y], q[y][c], pr[u][c]);
                } else {
                    float ph[RK];
                    if constexpr (EXACT && RK == 4) {
                        const float4 t = ((const float4 *)S.ph)[x];
                        ph[0] = t.x; ph[1] = t.y; ph[2] = t.z; ph[3] = t.w;
                    } else if constexpr (EXACT && RK == 2) {
                        const float2 t = ((const float2 *)S.ph)[x];
                        ph[0] = t.x; ph[1] = t.y;
                    } else {
#pragma unroll
                        for (int c = 0; c < RK; ++c)
                            ph[c] = c < r ? S.ph[x][c] : 0.f;
                    }
                    if constexpr (PASS == 2) {
#pragma unroll
                        for (int y = 0; y < 4; ++y)
#pragma unroll
                            for (int c = 0; c < RK; ++c)
                                q[y][c] = __fmaf_rn(p[y], ph[c], q[y][c]);
                    } else {
                        float res[4];
#pragma unroll
                        for (int y = 0; y < 4; ++y) {
                            res[y] = p[y];
#pragma unroll
                            for (int c = 0; c < RK; ++c)
                                if (EXACT || c < r)
                                    res[y] = __fmaf_rn(-ph[c], q[y][c], res[y]);   // r = p - P_hat Q_i^T
                        }
#pragma unroll
                        for (int y = 0; y < 4; ++y)
                            acc[y] += (double)__uint_as_float(__float_as_uint(res[y]) ^ sgn);   // s_i(a) r, exact
                    }
                }
            }
            if constexpr (PASS == 1) {
                float t[NV];
#pragma unroll
                for (int u = 0; u < kRwBatch; ++u)
#pragma unroll
                    for (int c = 0; c < RK; ++c)
                        t[u * RK + c] = pr[u][c];
                warp_reduce_many<NV>(t, lane);   // (the tree over the lanes does not depend on how many values share it)
                const uint32_t u = (uint32_t)p1_idx / RK, c = (uint32_t)p1_idx % RK, x = x0 + u;
                if ((lane & (p1_plain - 1)) == 0 && x < n && (EXACT || c < (uint32_t)r))
                    ppart[(size_t)(S.ent[x] & 0x7FFFFFFFu) * r + c] = t[0];
            }
        }
        cp_async_wait<0>();
    }
    if (PASS == 3 && live) {
        while (true) {   // the last bucket with rows, and those without after it
            if (bucket)
                close();
            if (bucket == nb)
                break;
            open();
        }
    }
    if (PASS == 2 && colok) {
        float *__restrict__ part = V.part + worker * V.part_stride + L.part_off + ((size_t)grp * m + b) * r;
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
            for (int c = 0; c < RK; ++c)
                if (EXACT || c < r)
                    part[(size_t)y * r + c] = q[y][c];
    }
}

// Whether a tensor takes the walk with its rank as a constant
__host__ __device__ __forceinline__ bool rs_exact(const LayerDesc &L, int rank)
{
    return (rank == 2 || rank == 4) && L.rank == rank && ((L.msgp_off | L.msgq_off) & (rank - 1)) == 0;
}

}  // namespace conef
