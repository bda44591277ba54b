// Generic sm_100a kernels of the ConEF step.  They are correct for every
// tensor shape and alignment (scalar global accesses only); the tuned kernels
// in conef_fast.cuh take over for the large, aligned tensors.
//
// Arithmetic contract (what makes codes and indices reproducible bit for bit):
// fp32 with explicit __fmaf_rn / __fmul_rn / __fdiv_rn, no fast-math, no
// flush-to-zero; the file is compiled with -fmad=false so that the compiler
// fuses nothing by itself.
#pragma once
#include "conef_common.cuh"

namespace conef {

// ------------------------------------------------------------------ 1-D pass-through
static __global__ void __launch_bounds__(256) k_passthrough(const __grid_constant__ DevView V)
{
    grid_release();
    const int li = find_layer(V.pfx_pass, V.n_layers, blockIdx.x);
    grid_wait();
    pass_tile(V, V.layers[li], blockIdx.x - V.pfx_pass[li]);
}

// ------------------------------------------------------------------ quantiser (S5, C1)
// scale and reciprocal of one block from its absmax; zero block when the
// stored scale is not >= FLT_MIN
__device__ __forceinline__ void quant_scale(float amax, int qmax, int half, float &s, float &inv,
                                            unsigned short &hbits)
{
    s = __fdiv_rn(amax, (float)qmax);
    hbits = 0;
    if (half) {
        s = fminf(s, 65504.0f);
        __half h = __float2half_rn(s);
        hbits = __half_as_ushort(h);
        s = __half2float(h);
    }
    if (!(s >= FLT_MIN)) {
        s = 0.f;
        inv = 0.f;
        hbits = 0;
    } else
        inv = __fdiv_rn(1.0f, s);
}
__device__ __forceinline__ int quant_code(float r, float inv, int qmax)
{
    int c = __float2int_rn(__fmul_rn(r, inv));  // NaN -> 0, out of range saturates
    return max(-qmax, min(qmax, c));
}

// ------------------------------------------------------------------ fused flat step
// One warp per work unit (= quantisation block of 32..256 elements); a lane
// owns unit/32 consecutive elements.  Covers S1+S2+S3+S4+S5 for Q = identity
// and Q = random-k, and S1+S2+S4+S5 ("pass 3") for the low-rank Q.
template <int QK, int CK>
__global__ void __launch_bounds__(kFlatThreads) k_flat(const __grid_constant__ DevView V)
{
    const int li = find_layer(V.pfx_flat, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const int worker = blockIdx.y;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int U = L.unit, E = U >> 5;
    const uint32_t d = (uint32_t)L.d, m = (uint32_t)L.cols;
    uint8_t *st = V.state + worker * V.state_stride;
    const float *__restrict__ g = V.grads[worker] + L.g_off;
    const int64_t unit0 = (int64_t)(blockIdx.x - V.pfx_flat[li]) * kFlatUnitsPerCta;
    const int qmax = (CK == CONEF_C_INT8) ? 127 : 7;

    SketchKeys keys = {};
    if (CK == CONEF_C_COUNTSKETCH)
        keys = sketch_keys(V.seed_c, li, V.cs_rows);
    uint32_t blk_start = 0;
    if (QK == CONEF_Q_RANDBLOCK)
        blk_start = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)V.step), d, (uint32_t)L.k);
    float *__restrict__ msg = V.msgv + worker * V.msgv_stride + L.msgv_off;
    // iConEF-v2: e~ is the k values that the second draw of Q kept; the stored state is q
    constexpr int QD = QK == CONEF_Q_RANDBLOCK ? CONEF_Q_RANDBLOCK : CONEF_Q_RANDK;
    const bool v2 = (QK == CONEF_Q_RANDK || QK == CONEF_Q_RANDBLOCK) && V.iconef == 2;
    const float *__restrict__ ev_old = V.ev_old + worker * V.msgv_stride + L.msgv_off;
    float *__restrict__ ev_new = V.ev_new + worker * V.msgv_stride + L.msgv_off;
    uint32_t blk_startA = 0, blk_startB = 0;
    if (QK == CONEF_Q_RANDBLOCK && v2) {
        blk_startA = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)(V.ev_step + kSecondDraw)), d, (uint32_t)L.k);
        blk_startB = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)(V.step + kSecondDraw)), d, (uint32_t)L.k);
    }
    const int r = L.rank;
    const float *__restrict__ phat = V.phat + L.msgp_off;
    const float *__restrict__ qi = V.msgq + worker * V.msgq_stride + L.msgq_off;

    for (int u = warp; u < kFlatUnitsPerCta; u += kFlatThreads / 32) {
        const int64_t unit = unit0 + u;
        if (unit >= L.nunits)
            break;
        const uint32_t base = (uint32_t)(unit * U) + lane * E;
        // iConEF-v2 with random-k: membership bits of this thread's elements in the two second draws
        // (a thread's E <= 8 elements share one bitmap word) and the slot of its first member
        uint32_t bitsA = 0, bitsB = 0, slotA = 0, slotB = 0;
        if (QK == CONEF_Q_RANDK && v2) {
            if (base < d) {
                const uint32_t emask = (1u << E) - 1u, wi = L.selbits_off + (base >> 5), sh = base & 31u;
                const uint32_t wA = V.ev_valid ? V.selbitsA[wi] : 0u, wB = V.selbitsB[wi];
                bitsA = (wA >> sh) & emask;
                bitsB = (wB >> sh) & emask;
                if (bitsA)
                    slotA = draw_slot(L, V.wordoffA, V.tileoffA, wA, base);
                if (bitsB)
                    slotB = draw_slot(L, V.wordoffB, V.tileoffB, wB, base);
            }
        }
        float val[8], ekeep[8];
        bool selq[8];
        const uint32_t selword = (QK == CONEF_Q_RANDK && base < d) ? V.selbits[L.selbits_off + (base >> 5)] : 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            val[q] = 0.f;
            ekeep[q] = 0.f;
            selq[q] = false;
            const uint32_t j = base + q;
            if (q < E && j < d) {
                float e;
                if (v2) {
                    e = 0.f;
                    if (QK == CONEF_Q_RANDK) {
                        if ((bitsA >> q) & 1u)
                            e = ev_old[slotA + (uint32_t)__popc(bitsA & ((1u << q) - 1u))];
                    } else {
                        uint32_t sl;
                        if (V.ev_valid && draw_member<QD>(L, V.selbitsA, V.wordoffA, V.tileoffA, blk_startA, j, sl))
                            e = ev_old[sl];
                    }
                } else
                    e = decode_elem<CK>(V, L, st, j, keys);
                float p = form_p(V, g[j], e);  // Alg. 2 line 5
                if (has_second<CK>(V))
                    p = __fadd_rn(p, decode_elem<CK>(V, L, st, j, keys, true));  // Alg. 3 line 5: + q
                else if (v2)
                    p = __fadd_rn(p, decode_elem<CK>(V, L, st, j, keys));        // the same line; q is the stored state
                ekeep[q] = e;
                if (QK == CONEF_Q_IDENTITY) {
                    msg[j] = p;
                    val[q] = 0.f;
                } else if (QK == CONEF_Q_RANDK) {
                    selq[q] = (selword >> (j & 31u)) & 1u;   // bitmap left by the selection
                    val[q] = p;
                } else if (QK == CONEF_Q_RANDBLOCK) {
                    const uint32_t slot = j - blk_start;   // wraps to a large value below the block
                    if (slot < (uint32_t)L.k) {
                        msg[slot] = p;
                        if (worker == 0)
                            V.idx[L.idx_off + slot] = j;
                        val[q] = 0.f;   // r = p - Delta is zero on a transmitted coordinate
                    } else
                        val[q] = p;
                } else {
                    const uint32_t row = j / m, col = j - row * m;
                    float acc = p;
                    for (int c = 0; c < r; ++c)
                        acc = __fmaf_rn(-phat[(int64_t)row * r + c], qi[(int64_t)col * r + c], acc);
                    val[q] = acc;  // r = p - P_hat Q_i^T
                }
            }
        }
        if (QK == CONEF_Q_RANDK && ((selword >> (base & 31u)) & ((1u << E) - 1u))) {
            uint32_t slot = draw_slot(L, V.wordoff, V.tileoff, selword, base);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (selq[q]) {
                    msg[slot] = val[q];  // message value, ascending index order
                    if (worker == 0)
                        V.idx[L.idx_off + slot] = base + q;
                    ++slot;
                    val[q] = 0.f;  // r = p - Delta is zero on a transmitted coordinate
                }
        }
        if (v2) {
            // Alg. 3 line 12: e~ = Q(r) by a second draw; line 14 then stores q = C(r - e~), and
            // r - e~ is exactly zero where e~ keeps the value
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t j = base + q;
                uint32_t sl;
                if (QK == CONEF_Q_RANDK) {
                    if ((bitsB >> q) & 1u) {
                        ev_new[slotB + (uint32_t)__popc(bitsB & ((1u << q) - 1u))] = val[q];
                        val[q] = 0.f;
                    }
                } else if (q < E && j < d && draw_member<QD>(L, V.selbitsB, V.wordoffB, V.tileoffB, blk_startB, j, sl)) {
                    ev_new[sl] = val[q];
                    val[q] = 0.f;
                }
            }
        }
        // ---- store r through C (Alg. 2 line 9); Alg. 4 line 9 stores C(beta e + r)
        if (V.beta != 0.f) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
                val[q] = __fmaf_rn(V.beta, ekeep[q], val[q]);
        }
        if (CK == CONEF_C_IDENTITY) {
            float *e = (float *)(st + L.a_off);
#pragma unroll
            for (int q = 0; q < 8; ++q)
                if (q < E && base + q < d)
                    e[base + q] = val[q];
            if (has_second<CK>(V)) {   // e~ = r exactly: nothing is left for q
                float *e2 = (float *)(st + L.a2_off);
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (q < E && base + q < d)
                        e2[base + q] = __fsub_rn(val[q], val[q]);
            }
        } else if (CK == CONEF_C_STOCHQUANT) {
            // Eq. 6 with the block's max-norm: level floor(u) or floor(u) + 1, up with probability u - floor(u)
            float amax = 0.f;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                amax = fmaxf(amax, fabsf(val[q]));
            amax = warp_max(amax);
            const float lv = (float)V.levels;
            float s = __fdiv_rn(amax, lv);
            const bool zero = !(s >= FLT_MIN);
            s = zero ? 0.f : s;
            const float inv = zero ? 0.f : __fdiv_rn(1.0f, s);
            if (lane == 0)
                ((float *)(st + L.b_off))[unit] = s;
            // this worker's variates for this tensor and step: a counter-based stream
            const uint64_t stc = stream_key(mix64(V.seed_c + (uint64_t)worker + 1u), (uint64_t)li, (uint64_t)V.step);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t j = base + q;
                if (q < E && j < d) {
                    int c = 0;
                    if (!zero) {
                        float u = __fmul_rn(fabsf(val[q]), inv);
                        u = !(u <= lv) ? lv : u;
                        const float l = floorf(u);
                        const float frac = __fsub_rn(u, l);
                        const float rnd = __fmul_rn((float)(uint32_t)(h64(stc, j) >> 40), 1.0f / 16777216.0f);
                        int lev = (int)l + (rnd < frac ? 1 : 0);
                        lev = min(lev, V.levels);
                        c = val[q] < 0.f ? -lev : lev;
                    }
                    if (V.sq_wide)
                        ((short *)(st + L.a_off))[j] = (short)c;
                    else
                        ((signed char *)(st + L.a_off))[j] = (signed char)c;
                }
            }
        } else if (CK == CONEF_C_COUNTSKETCH) {
            float *S = (float *)(V.state_new + worker * V.state_stride + L.a_off);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t j = base + q;
                if (q < E && j < d && val[q] != 0.f) {
                    uint32_t lo, width;
                    sketch_window(V, L, j, lo, width);
#pragma unroll
                    for (int i = 0; i < 7; ++i)
                        if (i < V.cs_rows) {
                            uint64_t h = h64(keys.st[i], j);
                            uint64_t b = lo + (((h >> 32) * (uint64_t)width) >> 32);
                            atomicAdd(&S[(int64_t)i * L.w + (int64_t)b], (h & 1) ? -val[q] : val[q]);
                        }
                }
            }
        } else {
            // e~ = C(r); with iConEF-v1 a second round stores q = C(r - e~) (Alg. 3 lines 10, 14)
            const int rounds = has_second<CK>(V) ? 2 : 1;
            for (int lev = 0; lev < rounds; ++lev) {
                const int64_t aoff = lev ? L.a2_off : L.a_off, boff = lev ? L.b2_off : L.b_off;
                float amax = 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    amax = fmaxf(amax, fabsf(val[q]));
                amax = warp_max(amax);
                float s, inv;
                unsigned short hb;
                quant_scale(amax, qmax, V.scale_half, s, inv, hb);
                if (lane == 0) {
                    if (V.scale_half)
                        ((unsigned short *)(st + boff))[unit] = hb;
                    else
                        ((float *)(st + boff))[unit] = s;
                }
                int cq[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    cq[q] = quant_code(val[q], inv, qmax);
                if (CK == CONEF_C_INT8) {
                    signed char *codes = (signed char *)(st + aoff);
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        if (q < E && base + q < d)
                            codes[base + q] = (signed char)cq[q];
                } else {
                    uint8_t *codes = st + aoff;
#pragma unroll
                    for (int q = 0; q < 8; q += 2)
                        if (q < E && base + q < d) {
                            int lo = cq[q] & 0xF;
                            int hi = (base + q + 1 < d) ? (cq[q + 1] & 0xF) : 0;
                            codes[(base + q) >> 1] = (uint8_t)(lo | (hi << 4));
                        }
                }
                if (lev + 1 < rounds) {
#pragma unroll
                    for (int q = 0; q < 8; ++q)
                        val[q] = __fsub_rn(val[q], __fmul_rn((float)cq[q], s));   // what the first state misses
                }
            }
        }
    }
}

// ------------------------------------------------------------------ low-rank pass 1 (generic)
// P_i = M_i Q_{t-1}: one warp per row, lanes stride over the columns.
template <int CK>
__global__ void __launch_bounds__(256) k_lr_pass1(const __grid_constant__ DevView V)
{
    const int li = find_layer(V.pfx_p1, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const int worker = blockIdx.y;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t m = (uint32_t)L.cols;
    const int r = L.rank;
    const uint8_t *st = V.state + worker * V.state_stride;
    const float *__restrict__ g = V.grads[worker] + L.g_off;
    const float *__restrict__ Q = V.qprev + L.msgq_off;
    float *__restrict__ P = V.msgp + worker * V.msgp_stride + L.msgp_off;
    SketchKeys keys = {};
    if (CK == CONEF_C_COUNTSKETCH)
        keys = sketch_keys(V.seed_c, li, V.cs_rows);
    const int64_t row0 = (int64_t)(blockIdx.x - V.pfx_p1[li]) * kP1RowsPerCta;
    for (int rr = 0; rr < kP1RowsPerCta / 8; ++rr) {
        const int64_t row = row0 + warp * (kP1RowsPerCta / 8) + rr;
        if (row >= L.rows)
            break;
        float acc[CONEF_MAX_RANK];
#pragma unroll
        for (int c = 0; c < CONEF_MAX_RANK; ++c)
            acc[c] = 0.f;
        for (uint32_t col = lane; col < m; col += 32) {
            const uint32_t j = (uint32_t)row * m + col;
            float p = form_p(V, g[j], decode_elem<CK>(V, L, st, j, keys));
            if (has_second<CK>(V))
                p = __fadd_rn(p, decode_elem<CK>(V, L, st, j, keys, true));
#pragma unroll
            for (int c = 0; c < CONEF_MAX_RANK; ++c)
                if (c < r)
                    acc[c] = __fmaf_rn(p, Q[(int64_t)col * r + c], acc[c]);
        }
#pragma unroll
        for (int c = 0; c < CONEF_MAX_RANK; ++c)
            if (c < r) {
                float s = warp_sum(acc[c]);
                if (lane == 0)
                    P[row * r + c] = s;
            }
    }
}

// ------------------------------------------------------------------ P-reduce + Gram-Schmidt
__device__ __forceinline__ double block_sum_double(double v, double *sh)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();  // sh may still be read from the previous call
    if (lane == 0)
        sh[warp] = v;
    __syncthreads();
    double t = (lane < (int)(blockDim.x >> 5)) ? sh[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;  // the same value in every thread
}

// One CTA per compressed tensor: P_bar = sum over workers (worker order);
// modified Gram-Schmidt on its columns, left to right, dot products and norms
// accumulated in fp64 and rounded once.
__global__ void __launch_bounds__(1024) k_gram_schmidt(const __grid_constant__ DevView V,
                                                       float *__restrict__ out_sum)
{
    __shared__ double sh[32];
    const int li = find_layer(V.pfx_gs, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const int64_t n = L.rows;
    const int r = L.rank;
    float *__restrict__ pbar = V.pbar + L.msgp_off;
    float *__restrict__ ph = V.phat + L.msgp_off;
    for (int64_t q = threadIdx.x; q < n * r; q += blockDim.x) {
        float acc = V.msgp[L.msgp_off + q];
        for (int i = 1; i < V.n_workers; ++i)
            acc = __fadd_rn(acc, V.msgp[i * V.msgp_stride + L.msgp_off + q]);
        pbar[q] = acc;
        ph[q] = acc;
        if (out_sum)
            out_sum[L.msgp_off + q] = acc;
    }
    __syncthreads();
    for (int c = 0; c < r; ++c) {
        for (int cp = 0; cp < c; ++cp) {
            double part = 0.0;
            for (int64_t a = threadIdx.x; a < n; a += blockDim.x)
                part += (double)ph[a * r + cp] * (double)ph[a * r + c];
            const float dotf = (float)block_sum_double(part, sh);
            for (int64_t a = threadIdx.x; a < n; a += blockDim.x)
                ph[a * r + c] = __fmaf_rn(-dotf, ph[a * r + cp], ph[a * r + c]);
            __syncthreads();
        }
        double part = 0.0;
        for (int64_t a = threadIdx.x; a < n; a += blockDim.x)
            part += (double)ph[a * r + c] * (double)ph[a * r + c];
        const float nu = (float)sqrt(block_sum_double(part, sh));
        const bool dead = !(nu >= FLT_MIN);
        for (int64_t a = threadIdx.x; a < n; a += blockDim.x)
            ph[a * r + c] = dead ? 0.f : __fdiv_rn(ph[a * r + c], nu);
        __syncthreads();
    }
}

// ------------------------------------------------------------------ low-rank pass 2 (generic)
// Q_i = M_i^T P_hat: a thread owns one column and runs down a tile of rows;
// the per-tile partials are summed in tile order by k_lr_pass2_reduce, so the
// result does not depend on scheduling.
template <int CK>
__global__ void __launch_bounds__(kP2ColsPerCta) k_lr_pass2(const __grid_constant__ DevView V)
{
    const int li = find_layer(V.pfx_p2, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const int worker = blockIdx.y;
    const uint32_t m = (uint32_t)L.cols;
    const int r = L.rank;
    const int local = blockIdx.x - V.pfx_p2[li];
    const int ncoltiles = (int)((m + kP2ColsPerCta - 1) / kP2ColsPerCta);
    const int rt = local / ncoltiles, ct = local - rt * ncoltiles;
    const uint32_t col = ct * kP2ColsPerCta + threadIdx.x;
    if (col >= m)
        return;
    const uint8_t *st = V.state + worker * V.state_stride;
    const float *__restrict__ g = V.grads[worker] + L.g_off;
    const float *__restrict__ ph = V.phat + L.msgp_off;
    SketchKeys keys = {};
    if (CK == CONEF_C_COUNTSKETCH)
        keys = sketch_keys(V.seed_c, li, V.cs_rows);
    float acc[CONEF_MAX_RANK];
#pragma unroll
    for (int c = 0; c < CONEF_MAX_RANK; ++c)
        acc[c] = 0.f;
    const int64_t rend = min((int64_t)L.rows, (int64_t)(rt + 1) * kP2RowsPerTile);
    for (int64_t row = (int64_t)rt * kP2RowsPerTile; row < rend; ++row) {
        const uint32_t j = (uint32_t)row * m + col;
        float p = form_p(V, g[j], decode_elem<CK>(V, L, st, j, keys));
        if (has_second<CK>(V))
            p = __fadd_rn(p, decode_elem<CK>(V, L, st, j, keys, true));
#pragma unroll
        for (int c = 0; c < CONEF_MAX_RANK; ++c)
            if (c < r)
                acc[c] = __fmaf_rn(p, ph[row * r + c], acc[c]);
    }
    float *__restrict__ part = V.part + worker * V.part_stride + L.part_off;
#pragma unroll
    for (int c = 0; c < CONEF_MAX_RANK; ++c)
        if (c < r)
            part[((int64_t)rt * m + col) * r + c] = acc[c];
}

// Q_i = sum over the row tiles' partials, in tile order: four consecutive (column, c) entries per
// thread, 16-byte loads where the tensor's offsets allow, the loads of four tiles in flight
constexpr int kQ2PerCta = 1024;
// A tensor with many tiles (tall ones; the bucket groups of a row sketch): the chain of sums is long, and the few CTAs
// that kQ2PerCta leaves it waited for four loads at a time.  A CTA then takes kQ2Few entries; its warps bring 64 tiles at
// a time into shared memory, the next ones while one thread per entry adds those.
// GPT-2-small list on a row sketch (628 bucket groups for the embedding): 77 -> 17 us; odd recurrent layers (131 tiles) 20 -> 7.
constexpr int kQ2Many = 32, kQ2Few = 128;
__device__ __forceinline__ void q2_reduce_many(const DevView &V, const LayerDesc &L, int64_t q0)
{
    constexpr int ROUND = 64, PER = ROUND / 8;   // tiles at a time, of which a thread brings PER
    __shared__ __align__(16) float sum[ROUND][kQ2Few];
    const int worker = blockIdx.y, tid = threadIdx.x;
    const int64_t mr = L.cols * L.rank;
    const int64_t ntiles = (V.fast_on && L.fast) ? L.p2_rows_fast : L.p2_rows_generic;
    const float *__restrict__ part = V.part + worker * V.part_stride + L.part_off;
    float *__restrict__ out = V.msgq + worker * V.msgq_stride + L.msgq_off;
    const int n = (int)min((int64_t)kQ2Few, mr - q0);
    if (mr % 4 != 0 || ((V.part_stride | L.part_off) & 3) != 0) {
        if (tid < n) {
            float acc = part[q0 + tid];
#pragma unroll 8
            for (int64_t t = 1; t < ntiles; ++t)
                acc = __fadd_rn(acc, part[t * mr + q0 + tid]);
            out[q0 + tid] = acc;
        }
        return;
    }
    const int c4 = (tid & 31) * 4, ty = tid >> 5;
    float4 v[PER];
    auto fetch = [&](int64_t t0) {
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int64_t t = t0 + ty + 8 * u;
            v[u] = t < ntiles && c4 < n ? __ldcs((const float4 *)(part + t * mr + q0 + c4)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
    };
    fetch(0);
    float acc = 0.f;
    for (int64_t t0 = 0; t0 < ntiles; t0 += ROUND) {
        if (t0)
            __syncthreads();   // (the previous tiles are added)
#pragma unroll
        for (int u = 0; u < PER; ++u)
            *(float4 *)&sum[ty + 8 * u][c4] = v[u];
        __syncthreads();
        if (t0 + ROUND < ntiles)
            fetch(t0 + ROUND);
        if (tid < kQ2Few) {
            const int have = (int)min((int64_t)ROUND, ntiles - t0);
            int t = 0;
            if (t0 == 0)
                acc = sum[t++][tid];
            for (; t + 8 <= have; t += 8) {
                float x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    x[u] = sum[t + u][tid];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    acc = __fadd_rn(acc, x[u]);
            }
            for (; t < have; ++t)
                acc = __fadd_rn(acc, sum[t][tid]);
        }
    }
    if (tid < n)
        out[q0 + tid] = acc;
}
__global__ void __launch_bounds__(256) k_lr_pass2_reduce(const __grid_constant__ DevView V)
{
    grid_release();
    const int li = find_layer(V.pfx_q2, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    grid_wait();
    const int worker = blockIdx.y;
    const int64_t mr = L.cols * L.rank;
    if (L.q2_per == kQ2Few) {
        q2_reduce_many(V, L, (int64_t)(blockIdx.x - V.pfx_q2[li]) * kQ2Few);
        return;
    }
    const int64_t q = ((int64_t)(blockIdx.x - V.pfx_q2[li]) * 256 + threadIdx.x) * 4;
    if (q >= mr)
        return;
    const int64_t ntiles = (V.fast_on && L.fast) ? L.p2_rows_fast : L.p2_rows_generic;
    const float *__restrict__ part = V.part + worker * V.part_stride + L.part_off;
    float *out = V.msgq + worker * V.msgq_stride + L.msgq_off;
    if (mr % 4 == 0 && ((V.part_stride | L.part_off | V.msgq_stride | L.msgq_off) & 3) == 0) {
        const float4 *p4 = (const float4 *)(part + q);
        const int64_t step = mr / 4;
        float4 acc = p4[0];
        int64_t t = 1;
        for (; t + 4 <= ntiles; t += 4) {
            const float4 a = p4[t * step], b = p4[(t + 1) * step], c = p4[(t + 2) * step], d = p4[(t + 3) * step];
            acc.x = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc.x, a.x), b.x), c.x), d.x);
            acc.y = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc.y, a.y), b.y), c.y), d.y);
            acc.z = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc.z, a.z), b.z), c.z), d.z);
            acc.w = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc.w, a.w), b.w), c.w), d.w);
        }
        for (; t < ntiles; ++t) {
            const float4 a = p4[t * step];
            acc.x = __fadd_rn(acc.x, a.x);
            acc.y = __fadd_rn(acc.y, a.y);
            acc.z = __fadd_rn(acc.z, a.z);
            acc.w = __fadd_rn(acc.w, a.w);
        }
        *(float4 *)(out + q) = acc;
        return;
    }
    for (int64_t j = q; j < min(q + 4, mr); ++j) {
        float acc = part[j];
        for (int64_t t = 1; t < ntiles; ++t)
            acc = __fadd_rn(acc, part[t * mr + j]);
        out[j] = acc;
    }
}

// ------------------------------------------------------------------ aggregate (S6)
// out[j] = ((m_0[j] + m_1[j]) + ...) in worker order; optionally also the mean
__global__ void __launch_bounds__(256) k_reduce_workers(const float *__restrict__ base,
                                                        int64_t stride, int n_workers, int64_t len,
                                                        float *__restrict__ out,
                                                        float *__restrict__ mean_out, float nf)
{
    grid_release();
    grid_wait();
    base = fresh(base);
    for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < len; j += (int64_t)gridDim.x * 256) {
        float acc = base[j];
        for (int i = 1; i < n_workers; ++i)
            acc = __fadd_rn(acc, base[i * stride + j]);
        if (out)
            out[j] = acc;
        if (mean_out)
            mean_out[j] = __fdiv_rn(acc, nf);
    }
}

// ------------------------------------------------------------------ decode alone
template <int CK>
__global__ void __launch_bounds__(256) k_decompress(const __grid_constant__ DevView V, int worker,
                                                    float *__restrict__ out)
{
    const int li = find_layer(V.pfx_flat, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const uint8_t *st = V.state + worker * V.state_stride;
    SketchKeys keys = {};
    if (CK == CONEF_C_COUNTSKETCH)
        keys = sketch_keys(V.seed_c, li, V.cs_rows);
    const int64_t j0 = (int64_t)(blockIdx.x - V.pfx_flat[li]) * kFlatUnitsPerCta * L.unit;
    const int64_t j1 = min(L.d, j0 + (int64_t)kFlatUnitsPerCta * L.unit);
    for (int64_t j = j0 + threadIdx.x; j < j1; j += 256)
    {
        float e = decode_elem<CK>(V, L, st, (uint32_t)j, keys);
        if (has_second<CK>(V))
            e = __fadd_rn(e, decode_elem<CK>(V, L, st, (uint32_t)j, keys, true));   // e~ + q
        if (V.iconef == 2) {   // e~ (the k values of the draw that stored them) + q
            float ev = 0.f;
            uint32_t sl;
            if (V.ev_valid) {
                const float *evp = V.ev_old + worker * V.msgv_stride + L.msgv_off;
                if (V.qkind == CONEF_Q_RANDBLOCK) {
                    const uint32_t bs = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)(V.ev_step + kSecondDraw)),
                                                        (uint32_t)L.d, (uint32_t)L.k);
                    if (draw_member<CONEF_Q_RANDBLOCK>(L, V.selbitsA, V.wordoffA, V.tileoffA, bs, (uint32_t)j, sl))
                        ev = evp[sl];
                } else if (draw_member<CONEF_Q_RANDK>(L, V.selbitsA, V.wordoffA, V.tileoffA, 0u, (uint32_t)j, sl))
                    ev = evp[sl];
            }
            e = __fadd_rn(ev, e);
        }
        out[L.e_off + j] = e;
    }
}

}  // namespace conef
