// The low-rank passes on a row-sketch state with one sketch row (conef_rowsketch.cuh) where 16-byte loads line up.
//
// A CTA owns kRsBuckets buckets and 512 columns, four per thread, and walks the rows of its buckets in the order of
// the bucket lists, as one sequence.  What a row needs besides the gradient is in shared memory before the walk
// starts: the entries (row, sign) of all its buckets, which are contiguous in the tables, their rows of P_hat, and
// the old sketch entries, each thread's own.  The walk has no load but the gradient's, a batch of rows ahead in
// registers, and only a bucket's first and last row touch the sketch.
//
// Before, every thread loaded entries, rows of P_hat and sketch entries when they were due, two rows at a time: a chain of
// trips to L2.  GPT-2-small list, rank 4, binary16 sketch, one worker: passes 204 / 183 / 239 us, now 169 / 148 / 177 us
// (4.4 B per element: 3.1 - 3.7 TB/s).  Bound by latency: 17 warps per SM (94 registers), issue slots 35 to 44 % busy.  With single loads
// four rows ahead instead of batches the waits ran to the youngest load: 266 / 246 / 259 us.  The single-phase compressors
// have no such chain in their step and stay with rs_body (3 % slower here).
#pragma once
#include "conef_fast.cuh"
#include "conef_kernels.cuh"

namespace conef {

constexpr int kRwDepth = 4;      // rows of a batch
constexpr int kRwEntries = 128;  // entries staged at a time (eight buckets of ten rows expect 80)
constexpr int kRwCols = kRsThreads * 4;

struct alignas(16) RwShared {
    uint32_t ent[kRwEntries + kRwDepth];               // row | sign << 31
    float ph[kRwEntries + kRwDepth][CONEF_MAX_RANK];   // their rows of P_hat; rank 4: [..][4], packed
    uint32_t start[kRsBuckets + 1];
    uint4 told[kRsBuckets][kRsThreads];                // the old entries of a thread's columns (binary16: half of each)
};

// PASS 1, 2, 3: the low-rank passes; 3 writes the new sketch.  RK: 4 for rows of P_hat of exactly four floats on 16-byte
// boundaries, else 8 (any rank).
template <int PASS, int RK>
__device__ __forceinline__ void rs_walk(const DevView &V, const LayerDesc &L, const uint32_t local, RwShared &S)
{
    constexpr bool NEED_PH = PASS != 1;
    const int worker = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t m = (uint32_t)L.cols, w = (uint32_t)L.w, slabs = (m + kRwCols - 1) / kRwCols;
    const uint32_t grp = local / slabs, slab = local - grp * slabs, h0 = grp * kRsBuckets, nb = min((uint32_t)kRsBuckets, w - h0);
    const uint32_t b = slab * kRwCols + tid * 4;   // this thread's first column
    const bool colok = b < m;                      // (four divides cols: all or none of them exist)
    const bool th = V.scale_half != 0;
    const int r = RK == 4 ? 4 : L.rank;
    if ((uint32_t)tid <= nb)
        S.start[tid] = V.rs[L.rs_ptr_off + h0 + tid];
    __syncthreads();
    const uint32_t *__restrict__ brow = V.rs + L.rs_row_off;
    const uint32_t first = S.start[0], last = S.start[nb];
    grid_wait();   // (the tables do not change)
    const uint8_t *__restrict__ Told = fresh(V.state + worker * V.state_stride + L.a_off);
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off) + b;
    const float *__restrict__ phat = fresh(V.phat + L.msgp_off);
    if (colok) {
        for (uint32_t x = 0; x < nb; ++x) {
            const size_t at = (size_t)(h0 + x) * m + b;
            if (th)
                cp_async_small<8>(&S.told[x][tid], Told + at * 2);
            else
                cp_async16(&S.told[x][tid], Told + at * 4);
        }
    }
    cp_async_commit();

    float q[4][RK];   // PASS 1: Q_{t-1}[b .. b + 3][:], 2: accumulators of Q_i[b .. b + 3][:], 3: Q_i[...]
    {
        const float *__restrict__ qp = fresh((PASS == 1 ? V.qprev : V.msgq + worker * V.msgq_stride) + L.msgq_off);
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int c = 0; c < RK; ++c)
                q[x][c] = PASS != 2 && colok && c < r ? qp[(size_t)(b + x) * r + c] : 0.f;
    }
    // PASS 1: which of a warp's totals of kRwDepth rows ends up in this lane
    constexpr int NV = kRwDepth * RK;
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
        float t[4] = {0.f, 0.f, 0.f, 0.f};
        if (!colok) {
        } else if (th) {
            const uint2 raw = *(const uint2 *)&S.told[bucket][tid];
            const float2 u = __half22float2(*(const __half2 *)&raw.x), v = __half22float2(*(const __half2 *)&raw.y);
            t[0] = u.x; t[1] = u.y; t[2] = v.x; t[3] = v.y;
        } else {
            const float4 u = *(const float4 *)&S.told[bucket][tid];
            t[0] = u.x; t[1] = u.y; t[2] = u.z; t[3] = u.w;
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            eb[x] = __fmul_rn(omb, t[x]);   // (the sign commutes with the rounding)
            if (PASS == 3)
                acc[x] = (double)__fmul_rn(beta, t[x]);
        }
        ++bucket;
        next = S.start[bucket];
    };
    auto close = [&]() {      // ... and its last
        if (PASS == 3 && colok)
            rs_store4(Tnew, (size_t)(h0 + bucket - 1) * m + b, th, (float)acc[0], (float)acc[1], (float)acc[2], (float)acc[3]);
    };

    for (uint32_t c0 = first; c0 < last || c0 == first; c0 += kRwEntries) {
        const uint32_t n = min((uint32_t)kRwEntries, last - c0);   // entries of this chunk
        if (c0 != first)
            __syncthreads();   // (the previous chunk is done)
        for (uint32_t x = tid; x < n + kRwDepth; x += kRsThreads)
            S.ent[x] = x < n ? brow[c0 + x] : 0u;   // (rows past the last one: loaded, not used)
        __syncthreads();
        float4 gv[2][kRwDepth];
        // the loads of a batch are issued together, and the next batch's before the first is used: a wait for one of several
        // loads in flight ends only when the youngest of them is there
        auto fetch = [&](auto buf, uint32_t x0) {
            constexpr int B = decltype(buf)::value;
#pragma unroll
            for (int u = 0; u < kRwDepth; ++u) {
                const uint32_t a = S.ent[x0 + u] & 0x7FFFFFFFu;
                if (colok)
                    gv[B][u] = __ldcs((const float4 *)(g + (size_t)a * m));
            }
        };
#pragma unroll
        for (int u = 0; u < kRwDepth; ++u)
            gv[0][u] = gv[1][u] = make_float4(0.f, 0.f, 0.f, 0.f);
        fetch(IntC<0>(), 0);
        if (NEED_PH) {   // (while those are under way)
            for (uint32_t x = tid; x < n; x += kRsThreads) {
                const float *src = phat + (size_t)(S.ent[x] & 0x7FFFFFFFu) * r;
                if (RK == 4) {
                    cp_async16(&((float4 *)S.ph)[x], src);
                } else {
                    for (int c = 0; c < r; ++c)
                        cp_async_small<4>(&S.ph[x][c], src + c);
                }
            }
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        auto batch = [&](auto buf, uint32_t x0) {
            constexpr int B = decltype(buf)::value;
            if (x0 + kRwDepth < n)
                fetch(IntC<1 - B>(), x0 + kRwDepth);
            float pr[PASS == 1 ? kRwDepth : 1][RK];
#pragma unroll
            for (int u = 0; u < kRwDepth; ++u) {
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
                const float gq[4] = {gv[B][u].x, gv[B][u].y, gv[B][u].z, gv[B][u].w};
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
                    if (NEED_PH) {
                        if (RK == 4) {
                            const float4 t = ((const float4 *)S.ph)[x];
                            ph[0] = t.x; ph[1] = t.y; ph[2] = t.z; ph[3] = t.w;
                        } else {
#pragma unroll
                            for (int c = 0; c < RK; ++c)
                                ph[c] = c < r ? S.ph[x][c] : 0.f;
                        }
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
                                if (RK == 4 || c < r)
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
                for (int u = 0; u < kRwDepth; ++u)
#pragma unroll
                    for (int c = 0; c < RK; ++c)
                        t[u * RK + c] = pr[u][c];
                warp_reduce_many<NV>(t, lane);   // (the tree over the lanes does not depend on how many values share it)
                const uint32_t u = (uint32_t)p1_idx / RK, c = (uint32_t)p1_idx % RK, x = x0 + u;
                if ((lane & (p1_plain - 1)) == 0 && x < n && (RK == 4 || c < (uint32_t)r))
                    ppart[(size_t)(S.ent[x] & 0x7FFFFFFFu) * r + c] = t[0];
            }
        };
        for (uint32_t x0 = 0; x0 < n; x0 += 2 * kRwDepth) {
            batch(IntC<0>(), x0);
            if (x0 + kRwDepth < n)
                batch(IntC<1>(), x0 + kRwDepth);
        }
    }
    if (PASS == 3) {
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
                if (RK == 4 || c < r)
                    part[(size_t)y * r + c] = q[y][c];
    }
}

}  // namespace conef
