// Error state kept as a count sketch over matrix rows (Sec. 4.2.2, the tensor
// trick; the form the experiments of Sec. 5.4 run) with partial error feedback
// (Alg. 4).  One fused kernel per step does, for one worker:
//
//   e = decode(T)                       median over sketch rows of s_i(a) T_i[h_i(a)][b]
//   p = eta g + (1 - beta) e            Alg. 4 line 5 (beta = 0: Alg. 2 line 5)
//   Delta = Q(p), message               identity / shared random-k / rank-r residual
//   T' = beta T + sketch(p - Delta)     Alg. 4 line 9 in its linear form: no re-decode
//
// A scatter (one atomic per element and sketch row) is turned into a gather:
// the buckets of the matrix rows do not depend on the step, so the rows of
// every bucket are listed once when the context is created, and a CTA owns
// whole buckets: thread = one column, loop over the bucket's rows in ascending
// order, accumulate in a register (fp64, the old term first, rounded once), one
// store.  All loads of the gradient are row-contiguous and coalesced, every
// sketch entry is read and written once, and the result does not depend on
// scheduling.  HBM-bound: 4 B of gradient per element plus 8 v w / rows bytes
// of sketch.
#pragma once
#include "conef_kernels.cuh"
#include "conef_fast.cuh"
#include "conef_rswalk.cuh"

namespace conef {

#ifndef CONEF_RS_ROWS
#define CONEF_RS_ROWS 2
#endif
// Rows of a bucket whose loads are issued together.  Measured with a low-rank Q and one sketch row, which rs_walk takes now
// where 16-byte loads line up, on the two-block GPT-2-XL list: 2 rows 1.05 ms, 4 rows 1.16 ms, 8 rows 1.24 ms (registers
// against occupancy).
constexpr int kRsRows = CONEF_RS_ROWS;

// The single-phase compressors, and the low-rank residual with several sketch rows or where 16-byte loads do not line up.
// VEC columns per thread (4: 16-byte loads; needs cols % 4 == 0 and 16-byte aligned gradients; 1: any shape).  The CTA covers kRsThreads * VEC columns of kRsBuckets
// buckets of one sketch row.
// A low-rank Q has room for any rank: a body for rank 4 with one 16-byte load per row of P_hat takes as long (two matrices of
// 4 M elements, two workers, rank 4, three sketch rows: 399 us in binary16 with both, 394 and 403 us in fp32 without and with it).
template <int QK, int VEC, bool V1>
__device__ __forceinline__ void rs_body(const DevView &V, const LayerDesc &L, const int li, uint32_t local)
{
    const int worker = blockIdx.y;
    const uint32_t m = (uint32_t)L.cols, n = (uint32_t)L.rows, w = (uint32_t)L.w, d = (uint32_t)L.d;
    const int v = V.cs_rows;
    constexpr uint32_t CW = kRsThreads * VEC;               // columns per CTA
    const uint32_t slabs = (m + CW - 1) / CW;
    const uint32_t groups = (w + kRsBuckets - 1) / kRsBuckets;
    const uint32_t slab = local % slabs;
    local /= slabs;
    const uint32_t grp = local % groups;
    const uint32_t i = local / groups;                      // sketch row this CTA builds
    const uint32_t b = slab * CW + threadIdx.x * VEC;       // this thread's first column
    const bool colok = b < m;                               // VEC divides cols: all or none of the thread's columns exist

    const uint32_t *__restrict__ info = V.rs + L.rs_info_off;
    const uint32_t *__restrict__ bptr = V.rs + L.rs_ptr_off + (size_t)i * (w + 1);
    const uint32_t *__restrict__ brow = V.rs + L.rs_row_off + (size_t)i * n;
    const void *__restrict__ Told = V.state + worker * V.state_stride + L.a_off;
    void *__restrict__ Tnew = V.state_new + worker * V.state_stride + L.a_off;
    const bool th = V.scale_half != 0;   // the sketch is stored in binary16
    const float *__restrict__ g = V.grads[worker] + L.g_off;
    float *__restrict__ msg = V.msgv + worker * V.msgv_stride + L.msgv_off;

    const uint32_t *__restrict__ selbits = V.selbits + L.selbits_off;
    uint32_t blk_start = 0;
    if (QK == CONEF_Q_RANDBLOCK)
        blk_start = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)V.step), d, (uint32_t)L.k);
    const int r = L.rank;
    constexpr int RK = QK == CONEF_Q_LOWRANK ? CONEF_MAX_RANK : 1;
    float qreg[VEC][RK];   // Q_i[b..b+VEC-1][:], fixed for the thread
    const float *__restrict__ phat = fresh(V.phat + L.msgp_off);
    if (QK == CONEF_Q_LOWRANK) {
        const float *qi = V.msgq + worker * V.msgq_stride + L.msgq_off;
#pragma unroll
        for (int x = 0; x < VEC; ++x)
#pragma unroll
            for (int c = 0; c < RK; ++c)
                qreg[x][c] = (c < r && colok) ? qi[(size_t)(b + x) * r + c] : 0.f;
    }

    auto load_vec = [&](const float *p, float (&out)[VEC]) {
        if (VEC == 4) {
            const float4 t = *(const float4 *)p;
            out[0] = t.x; out[1 % VEC] = t.y; out[2 % VEC] = t.z; out[3 % VEC] = t.w;
        } else {
            out[0] = *p;
        }
    };
    auto load_t = [&](size_t idx, float (&out)[VEC]) {   // VEC entries of the old sketch
        if (VEC == 4) {
            float t4[4];
            rs_load4(Told, idx, th, t4);
            out[0] = t4[0]; out[1 % VEC] = t4[1]; out[2 % VEC] = t4[2]; out[3 % VEC] = t4[3];
        } else {
            out[0] = rs_load1(Told, idx, th);
        }
    };

    const uint32_t h_end = min(w, (grp + 1) * kRsBuckets);
    for (uint32_t h = grp * kRsBuckets; h < h_end; ++h) {
        const uint32_t lo = bptr[h], hi = bptr[h + 1];
        float told[VEC];
#pragma unroll
        for (int x = 0; x < VEC; ++x)
            told[x] = 0.f;
        if (colok)
            load_t(((size_t)i * w + h) * m + b, told);
        double acc[VEC];
#pragma unroll
        for (int x = 0; x < VEC; ++x)
            acc[x] = (double)__fmul_rn(V.beta, told[x]);
        for (uint32_t k0 = lo; k0 < hi; k0 += kRsRows) {
            uint32_t ent[kRsRows];
            float gv[kRsRows][VEC];
#pragma unroll
            for (int u = 0; u < kRsRows; ++u) {   // the loads of several rows are in flight together
                ent[u] = k0 + u < hi ? brow[k0 + u] : 0u;
#pragma unroll
                for (int x = 0; x < VEC; ++x)
                    gv[u][x] = 0.f;
                if (k0 + u < hi && colok)
                    load_vec(g + ((ent[u] & 0x7FFFFFFFu) * m + b), gv[u]);
            }
#pragma unroll
            for (int u = 0; u < kRsRows; ++u) {
                if (k0 + u >= hi)
                    break;
                const uint32_t a = ent[u] & 0x7FFFFFFFu;
                const uint32_t sgn = ent[u] & 0x80000000u;   // the sign bit of s_i(a)
                const uint32_t j = a * m + b;   // first element of the thread in this row
                // decode: with one sketch row the estimate is this bucket's own entry
                float e[VEC];
                if (V1) {
#pragma unroll
                    for (int x = 0; x < VEC; ++x)
                        e[x] = __uint_as_float(__float_as_uint(told[x]) ^ sgn);
                } else {
                    float est[VEC][7];
#pragma unroll
                    for (int y = 0; y < 7; ++y) {
                        float t[VEC];
#pragma unroll
                        for (int x = 0; x < VEC; ++x)
                            t[x] = 0.f;
                        uint32_t in = 0;
                        if (y < v) {
                            in = info[(size_t)y * n + a];
                            if (colok)
                                load_t(((size_t)y * w + (in & 0x7FFFFFFFu)) * m + b, t);
                        }
#pragma unroll
                        for (int x = 0; x < VEC; ++x)
                            est[x][y] = (in >> 31) ? -t[x] : t[x];
                    }
#pragma unroll
                    for (int x = 0; x < VEC; ++x)
                        e[x] = median_small(est[x], v);
                }
                float p[VEC], res[VEC];
#pragma unroll
                for (int x = 0; x < VEC; ++x)
                    p[x] = form_p(V, gv[u][x], e[x]);
                if (QK == CONEF_Q_IDENTITY) {
#pragma unroll
                    for (int x = 0; x < VEC; ++x) {
                        if (i == 0 && colok)
                            msg[j + x] = p[x];
                        res[x] = 0.f;
                    }
                } else if (QK == CONEF_Q_RANDBLOCK) {
#pragma unroll
                    for (int x = 0; x < VEC; ++x) {
                        const uint32_t slot = j + x - blk_start;
                        const bool sel = colok && slot < (uint32_t)L.k;
                        res[x] = sel ? 0.f : p[x];
                        if (i == 0 && sel) {
                            msg[slot] = p[x];
                            if (worker == 0)
                                V.idx[L.idx_off + slot] = j + x;
                        }
                    }
                } else if (QK == CONEF_Q_RANDK) {
                    // membership from the bitmap the selection left (bit i of word w: element 32 w + i);
                    // the thread's VEC elements lie in one word (VEC = 4: j is a multiple of 4)
                    const uint32_t word = colok ? selbits[j >> 5] : 0u;
                    bool sel[VEC];
                    int nsel = 0;
#pragma unroll
                    for (int x = 0; x < VEC; ++x) {
                        sel[x] = (word >> ((j + x) & 31u)) & 1u;
                        res[x] = sel[x] ? 0.f : p[x];
                        nsel += sel[x];
                    }
                    if (i == 0) {   // the CTAs of sketch row 0 meet every matrix row once: they write the message
                        uint32_t slot = nsel ? draw_slot(L, V.wordoff, V.tileoff, word, j) : 0u;
#pragma unroll
                        for (int x = 0; x < VEC; ++x)
                            if (sel[x]) {
                                msg[slot] = p[x];   // message value, ascending index order
                                if (worker == 0)
                                    V.idx[L.idx_off + slot] = j + x;
                                ++slot;
                            }
                    }
                } else {
                    float ph[RK];
#pragma unroll
                    for (int c = 0; c < RK; ++c)
                        ph[c] = c < r ? phat[(size_t)a * r + c] : 0.f;
#pragma unroll
                    for (int x = 0; x < VEC; ++x) {
                        res[x] = p[x];
#pragma unroll
                        for (int c = 0; c < RK; ++c)
                            if (c < r)
                                res[x] = __fmaf_rn(-ph[c], qreg[x][c], res[x]);   // r = p - P_hat Q_i^T
                    }
                }
#pragma unroll
                for (int x = 0; x < VEC; ++x)
                    acc[x] += (double)__uint_as_float(__float_as_uint(res[x]) ^ sgn);   // s_i(a) * r, exact
            }
        }
        if (colok) {
            const size_t dst = ((size_t)i * w + h) * m + b;
            if (VEC == 4)
                rs_store4(Tnew, dst, th, (float)acc[0], (float)acc[1 % VEC], (float)acc[2 % VEC], (float)acc[3 % VEC]);
            else
                rs_store1(Tnew, dst, th, (float)acc[0]);
        }
    }
}

// rs_vec of a tensor chooses the body; both live in one kernel so that one launch covers the model.  (A low-rank Q on one sketch row
// comes here where no tensor takes the walk: 16-byte loads are not possible.)
template <int QK, bool V1>   // V1: one sketch row (the usual setting), no median
__global__ void __launch_bounds__(kRsThreads, V1 && QK == CONEF_Q_LOWRANK ? 5 : 0) k_rowsketch(const __grid_constant__ DevView V)
{
    grid_release();
    const int li = find_layer(V.pfx_rs, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const uint32_t local = blockIdx.x - V.pfx_rs[li];
    const bool vec = L.rs_vec == 4 && V.rs_vec_ok;
    grid_wait();
    if (!(V1 && QK == CONEF_Q_LOWRANK) && vec)
        rs_body<QK, 4, V1>(V, L, li, local);
    else if (L.rs_vec == 4) {
        // 16-byte loads are not possible with this call's gradient pointers: the same tiles,
        // four scalar slabs per vector slab
        const uint32_t slabs4 = (uint32_t)((L.cols + kRsThreads * 4 - 1) / (kRsThreads * 4));
        const uint32_t slabs1 = (uint32_t)((L.cols + kRsThreads - 1) / kRsThreads);
        const uint32_t slab = local % slabs4, rest = local / slabs4;
        for (uint32_t s = slab * 4; s < min(slabs1, slab * 4 + 4); ++s)
            rs_body<QK, 1, V1>(V, L, li, rest * slabs1 + s);
    } else
        rs_body<QK, 1, V1>(V, L, li, local);
}

// ------------------------------------------------------------------ low-rank passes 1 and 2 on a row-sketch state
// The same bucket-major walk (one sketch row, four columns per thread; conef_rswalk.cuh), for tensors whose
// gradients allow 16-byte loads: every matrix row lies in exactly one bucket of sketch row 0, so
// the CTAs of (bucket group, column slab) meet every element once.
//   PASS 1: P_i[a][:] = sum_b p[a][b] Q_{t-1}[b][:]; a warp reduces its 128 columns by shuffles and
//           writes one partial row per (column slab, warp); k_rs_p1_combine adds them in order.
//   PASS 2: Q_i[b][:] = sum_a p[a][b] P_hat[a][:]; a thread accumulates its columns over the rows
//           of the group's buckets and writes one partial row per bucket group, summed in group
//           order by k_lr_pass2_reduce.
// Sums over rows and columns run in bucket order, not index order: like the other factor kernels
// they match the oracle to rounding (fp32, fixed order), not bit for bit.
// RK: the configured rank (2, 4; 8: another one); tensors that rs_exact does not accept take the walk for any rank up to it (with
// room for eight it spilled under these registers: behind a matrix of one row the GPT-2-small list, rank 4, takes 722 us per step instead of 920,
// two of 4096 x 4096, rank 2, two workers 282 instead of 522).
// PASS 3, the step's last, takes the tensors that do not walk along: in a launch of their own behind it they make the step longer (512 x 768,
// 300 x 333 and 768 x 512, rank 4, two workers 244 -> 262 us).  With the walk for any rank up to 8 beside rs_body in k_rowsketch it was 266, the
// GPT-2-small list with 300 x 333 behind it 878 instead of 810, two of 4096 x 4096 around 333 x 4097, rank 2, 1107 instead of 1001.
// CTAs per SM: rank 4 with six, seven and eight (64 registers) on the GPT-2-small list 136 / 115 / 135, 134 / 117 / 127, 142 / 117 / 129 us (with
// the spilling body beside it; 131 / 114 / 125 now);
// rank 2 with seven and eight 65 / 62 / 74, 63 / 59 / 69.
template <int PASS, int RK>
__global__ void __launch_bounds__(kRsThreads, RK == 2 ? 8 : RK == 4 ? 7 : 5) k_rs_pass(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
    __shared__ RwShared S;
    grid_release();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const uint32_t local = blockIdx.x - pfx[li];
    if constexpr (PASS == 3)
        if (L.rs_vec != 4) {
            grid_wait();
            rs_body<CONEF_Q_LOWRANK, 1, true>(V, L, li, local);
            return;
        }
    if constexpr (RK < CONEF_MAX_RANK)
        if (rs_exact(L, RK)) {
            rs_walk<PASS, RK, true>(V, L, local, S);
            return;
        }
    rs_walk<PASS, RK, false>(V, L, local, S);
}

// P_i[a][c] = sum over the (column slab, warp) partials of pass 1, in slab-major order; four consecutive entries per thread
__global__ void __launch_bounds__(256) k_rs_p1_combine(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
    grid_release();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    grid_wait();
    const int worker = blockIdx.y;
    const int64_t nr = L.rows * L.rank;
    const int64_t q = ((int64_t)(blockIdx.x - pfx[li]) * 256 + threadIdx.x) * 4;
    if (q >= nr)
        return;
    const float *__restrict__ ppart = V.ppart + worker * V.ppart_stride + L.pp_off;
    float *__restrict__ out = V.msgp + worker * V.msgp_stride + L.msgp_off;
    if (nr % 4 == 0 && ((L.pp_off | L.msgp_off) & 3) == 0) {
        float4 acc = *(const float4 *)(ppart + q);
#pragma unroll 4
        for (int j = 1; j < L.f_j; ++j) {
            const float4 t = *(const float4 *)(ppart + j * nr + q);
            acc.x = __fadd_rn(acc.x, t.x);
            acc.y = __fadd_rn(acc.y, t.y);
            acc.z = __fadd_rn(acc.z, t.z);
            acc.w = __fadd_rn(acc.w, t.w);
        }
        *(float4 *)(out + q) = acc;
        return;
    }
    for (int64_t x = q; x < min(q + 4, nr); ++x) {
        float acc = ppart[x];
        for (int j = 1; j < L.f_j; ++j)
            acc = __fadd_rn(acc, ppart[j * nr + x]);
        out[x] = acc;
    }
}

}  // namespace conef
