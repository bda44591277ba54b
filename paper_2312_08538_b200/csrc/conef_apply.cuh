// Model update from the summed messages (Alg. 2 lines 7-8): x <- x - Delta_t, Delta_t the mean
// over workers of Q's outputs.  HBM-bound: x is read and written once (8 B per parameter; the
// random-k case touches only the k shared coordinates).
#pragma once
#include "conef_kernels.cuh"

namespace conef {

constexpr int kApplyThreads = 256;
constexpr int kApplyTile = 4096;      // elements per CTA where the update is dense and elementwise
constexpr int kApplySparse = 1024;    // message values per CTA where it is sparse: four per thread, all in flight

// Low-rank tiles: a CTA's threads are laid out as ap_tx column groups (of ap_vec columns) by ap_ty
// rows; a thread keeps its columns' rows of Q in registers and walks ap_rpt rows, ap_ty apart.
inline void apply_classify(LayerDesc &L)
{
    L.ap_vec = ((L.cols | L.g_off) & 3) == 0 ? 4 : ((L.cols | L.g_off) & 1) == 0 ? 2 : 1;
    const int64_t ncg = (L.cols + L.ap_vec - 1) / L.ap_vec;
    // column tiles of equal width: as few as leave at most 7 % of the threads idle, else the best of eight
    const int64_t ct0 = (ncg + kApplyThreads - 1) / kApplyThreads;
    double best = 0.0;
    for (int64_t ct = ct0; ct < ct0 + 8 && best < 0.93; ++ct) {
        const int64_t tx = (ncg + ct - 1) / ct, ty = kApplyThreads / tx;
        const double used = (double)(tx * ty) / kApplyThreads * (double)ncg / (double)(ct * tx);
        if (used > best && (tx >= 16 || ct == ct0)) {
            best = used;
            L.ap_tx = (int32_t)tx;
            L.ap_ty = (int32_t)ty;
            L.ap_ct = (int32_t)ct;
        }
    }
    // a thread loads rank * 4 bytes per column before its first row: many rows amortise that on large
    // tensors, few keep the SMs busy on small ones
    L.ap_rpt = L.d >= (1 << 22) ? 64 : L.d >= (1 << 20) ? 32 : L.d >= (1 << 17) ? 16 : 8;
}

// tiles per tensor, in the order the kernel decodes them
inline int64_t apply_tiles(LayerDesc &L, int qkind)
{
    if (!L.compressed || qkind == CONEF_Q_IDENTITY)
        return (L.d + kApplyTile - 1) / kApplyTile;
    if (qkind == CONEF_Q_RANDK || qkind == CONEF_Q_RANDBLOCK)
        return (L.k + kApplySparse - 1) / kApplySparse;
    apply_classify(L);
    const int64_t rows = (int64_t)L.ap_ty * L.ap_rpt;
    return L.ap_ct * ((L.rows + rows - 1) / rows);
}

// x[a][b] -= sum_c P_hat[a][c] Qmean[b][c] (an fma chain over ascending c) on a tile.  RK: the rank, or
// 0 for any rank; VEC columns per thread; B rows of x are loaded before the first is used; FV: rows
// of the factors lie on 16-byte boundaries.  HBM-bound (8 bytes per element).  GPT-2-XL list, rank 4:
// one column per thread and 16 rows one after the other took 3.76 ms (3.3 TB/s); four columns and
// eight rows in flight take 2.09 ms (6.0 TB/s); four rows in flight 2.21 ms, eight under a
// 64-register cap (spills) 3.1 ms.  GPT-2-small list, rank 8: 324 -> 193 us.  Odd recurrent layers (33279 x 650 among
// them), rank 2: one column per thread 60 us, two where rows lie on 8-byte boundaries 48 us.
template <int RK, int VEC, int B, bool FV>
__device__ __forceinline__ void apply_lowrank(const DevView &V, const LayerDesc &L, uint32_t tile, float *__restrict__ xs,
                                              bool aligned)
{
    constexpr int RM = RK ? RK : CONEF_MAX_RANK;
    const int r = RK ? RK : L.rank;
    const uint32_t gtx = L.ap_tx, gty = L.ap_ty, gct = L.ap_ct;
    const uint32_t ty = threadIdx.x / gtx, tx = threadIdx.x - ty * gtx;
    const uint32_t rt = tile / gct, ct = tile - rt * gct;
    const uint32_t b = (ct * gtx + tx) * VEC, m = (uint32_t)L.cols;
    if (ty >= gty || b >= m)
        return;
    const float *__restrict__ phat = V.phat + L.msgp_off;
    auto load_row = [&](const float *p, float (&out)[RM]) {
        if (FV) {
#pragma unroll
            for (int c = 0; c + 4 <= RM; c += 4) {
                const float4 t = load_global((const float4 *)(p + c));
                out[c] = t.x; out[c + 1] = t.y; out[c + 2] = t.z; out[c + 3] = t.w;
            }
        } else {
#pragma unroll
            for (int c = 0; c < RM; ++c)
                out[c] = (RK || c < r) ? load_global(p + c) : 0.f;
        }
    };
    float q[VEC][RM];
    {
        const float *__restrict__ qm = V.qprev + L.msgq_off + (size_t)b * r;
#pragma unroll
        for (int v = 0; v < VEC; ++v)
            load_row(qm + v * r, q[v]);
    }
    auto load = [&](const float *p, float (&xv)[VEC]) {
        if (VEC == 4 && aligned) {
            const float4 t = *(const float4 *)p;
            xv[0] = t.x; xv[1 % VEC] = t.y; xv[2 % VEC] = t.z; xv[3 % VEC] = t.w;
        } else if (VEC == 2 && aligned) {
            const float2 t = *(const float2 *)p;
            xv[0] = t.x; xv[1 % VEC] = t.y;
        } else {
#pragma unroll
            for (int v = 0; v < VEC; ++v)
                xv[v] = p[v];
        }
    };
    auto update = [&](const float (&ph)[RM], float (&xv)[VEC]) {
#pragma unroll
        for (int v = 0; v < VEC; ++v) {
            float dl = 0.f;
#pragma unroll
            for (int c = 0; c < RM; ++c)
                if (RK || c < r)
                    dl = __fmaf_rn(ph[c], q[v][c], dl);
            xv[v] = __fsub_rn(xv[v], dl);
        }
    };
    auto store = [&](float *p, const float (&xv)[VEC]) {
        if (VEC == 4 && aligned) {
            *(float4 *)p = make_float4(xv[0], xv[1 % VEC], xv[2 % VEC], xv[3 % VEC]);
        } else if (VEC == 2 && aligned) {
            *(float2 *)p = make_float2(xv[0], xv[1 % VEC]);
        } else {
#pragma unroll
            for (int v = 0; v < VEC; ++v)
                p[v] = xv[v];
        }
    };
    const uint32_t rows = (uint32_t)L.rows, span = gty * (uint32_t)L.ap_rpt;
    uint32_t a = rt * span + ty;
    const uint32_t a1 = min(rows, (rt + 1) * span);
    float *xp = xs + (size_t)a * m + b;
    const float *pp = phat + (size_t)a * r;
    const size_t step = (size_t)gty * m;
    const uint32_t pstep = gty * r;
    // Rows of P_hat come AHEAD rows before their use and ahead of the stores of x in between, which may write them for all that
    // the compiler knows.  Loaded when due they waited for each store: rank 4, GPT-2-XL list, one worker 2.70 ms, two ahead
    // 2.06 (all eight ahead spill: 2.72); rank 8, GPT-2-small list 207 us, one ahead 213, two 195, four 188.
    constexpr int AHEAD = RM <= 2 || B < 4 ? B : RM <= 4 ? 2 : 4;
    static_assert(B % AHEAD == 0, "a row's place in the ring is a constant");
    for (; a + (B - 1) * gty < a1; a += B * gty) {
        float xv[B][VEC], ph[AHEAD][RM];
#pragma unroll
        for (int u = 0; u < B; ++u)
            load(xp + u * step, xv[u]);
#pragma unroll
        for (int u = 0; u < AHEAD; ++u)
            load_row(pp + u * pstep, ph[u]);
#pragma unroll
        for (int u = 0; u < B; ++u) {
            update(ph[u % AHEAD], xv[u]);
            if (u + AHEAD < B)
                load_row(pp + (u + AHEAD) * pstep, ph[u % AHEAD]);
            store(xp + u * step, xv[u]);
        }
        xp += B * step;
        pp += B * pstep;
    }
    for (; a < a1; a += gty) {
        float xv[VEC], ph[RM];
        load(xp, xv);
        load_row(pp, ph);
        update(ph, xv);
        store(xp, xv);
        xp += step;
        pp += pstep;
    }
}

// R: the configured rank of a low-rank Q (1, 2, 4, 8; 0: another one), or -1 for the other compressors
template <int R>
__global__ void __launch_bounds__(kApplyThreads, R == 8 ? 2 : 3)
k_apply(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx, float *__restrict__ x,
        const float *__restrict__ sum_values, const float *__restrict__ sum_dense1d)
{
    grid_release();
    int li = find_layer(pfx, V.n_layers, blockIdx.x);
    if (R >= 0)
        grid_wait(li);
    const LayerDesc &L = V.layers[li];
    const uint32_t tile = blockIdx.x - pfx[li];
    if (R < 0)
        grid_wait();
    sum_values = fresh(sum_values);
    sum_dense1d = fresh(sum_dense1d);
    float *__restrict__ xs = x + L.g_off;
    const float nw = V.n_workers_f;
    if (!L.compressed || (R < 0 && V.qkind == CONEF_Q_IDENTITY)) {
        const size_t at = (size_t)tile * kApplyTile;
        const float *__restrict__ sum = (L.compressed ? sum_values + L.msgv_off : sum_dense1d + L.msg1d_off) + at;
        float *__restrict__ xt = xs + at;
        const int n = (int)min((int64_t)kApplyTile, L.d - (int64_t)at);
        if (n == kApplyTile && (((uintptr_t)xt | (uintptr_t)sum) & 15) == 0) {
            float4 xv[4], sv[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                xv[u] = ((const float4 *)xt)[u * kApplyThreads + threadIdx.x];
                sv[u] = ((const float4 *)sum)[u * kApplyThreads + threadIdx.x];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                ((float4 *)xt)[u * kApplyThreads + threadIdx.x] =
                    make_float4(__fsub_rn(xv[u].x, __fdiv_rn(sv[u].x, nw)), __fsub_rn(xv[u].y, __fdiv_rn(sv[u].y, nw)),
                                __fsub_rn(xv[u].z, __fdiv_rn(sv[u].z, nw)), __fsub_rn(xv[u].w, __fdiv_rn(sv[u].w, nw)));
        } else {
#pragma unroll 4
            for (int q = threadIdx.x; q < n; q += kApplyThreads)
                xt[q] = __fsub_rn(xt[q], __fdiv_rn(sum[q], nw));
        }
        return;
    }
    if constexpr (R < 0) {
        // indices are distinct: no race.  Bound by the 32-byte sectors of x that hold one value each
        const float *__restrict__ sum = sum_values + L.msgv_off;
        const uint32_t *__restrict__ idx = V.idx + L.idx_off;
        constexpr int B = kApplySparse / kApplyThreads;
        uint32_t j[B];
        float sv[B], xv[B];
        bool in[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
            const int64_t s = (int64_t)tile * kApplySparse + u * kApplyThreads + threadIdx.x;
            in[u] = s < L.k;
            j[u] = in[u] ? idx[s] : 0u;
            sv[u] = in[u] ? sum[s] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < B; ++u)
            xv[u] = in[u] ? xs[j[u]] : 0.f;
#pragma unroll
        for (int u = 0; u < B; ++u)
            if (in[u])
                xs[j[u]] = __fsub_rn(xv[u], __fdiv_rn(sv[u], nw));
    } else {
        // Delta = P_hat Qmean^T, Qmean = the warm start left by the reduction of the Q messages.
        // Tensors thinner than the configured rank take the run-time rank.
        const bool exact = R > 0 && L.rank == R;
        const bool fv = ((L.msgp_off | L.msgq_off) & 3) == 0;
        const bool aligned = ((uintptr_t)xs & (L.ap_vec == 2 ? 7 : 15)) == 0;
        constexpr int RX = R > 0 ? R : 0;
        if (L.ap_vec == 4) {
            if (exact && R >= 4 && fv)
                apply_lowrank<RX, 4, 8, (R >= 4)>(V, L, tile, xs, aligned);
            else if (exact && R < 4)
                apply_lowrank<RX, 4, 4, false>(V, L, tile, xs, aligned);
            else
                apply_lowrank<0, 4, 1, false>(V, L, tile, xs, aligned);
        } else if (L.ap_vec == 2) {
            if (exact)
                apply_lowrank<RX, 2, 8, false>(V, L, tile, xs, aligned);
            else
                apply_lowrank<0, 2, 2, false>(V, L, tile, xs, aligned);
        } else {
            if (exact)
                apply_lowrank<RX, 1, 8, false>(V, L, tile, xs, false);
            else
                apply_lowrank<0, 1, 8, false>(V, L, tile, xs, false);
        }
    }
}

inline void apply_launch(int qkind, int rank, const DevView &V, const int32_t *pfx, int tiles, float *x, const float *sum_values,
                         const float *sum_dense1d, cudaStream_t s)
{
    const int r = qkind != CONEF_Q_LOWRANK ? -1 : rank == 1 || rank == 2 || rank == 4 || rank == 8 ? rank : 0;
    switch (r) {
    case -1: launch(k_apply<-1>, dim3(tiles), kApplyThreads, 0, s, V, pfx, x, sum_values, sum_dense1d); break;
    case 1: launch(k_apply<1>, dim3(tiles), kApplyThreads, 0, s, V, pfx, x, sum_values, sum_dense1d); break;
    case 2: launch(k_apply<2>, dim3(tiles), kApplyThreads, 0, s, V, pfx, x, sum_values, sum_dense1d); break;
    case 4: launch(k_apply<4>, dim3(tiles), kApplyThreads, 0, s, V, pfx, x, sum_values, sum_dense1d); break;
    case 8: launch(k_apply<8>, dim3(tiles), kApplyThreads, 0, s, V, pfx, x, sum_values, sum_dense1d); break;
    default: launch(k_apply<0>, dim3(tiles), kApplyThreads, 0, s, V, pfx, x, sum_values, sum_dense1d);
    }
}

// the same for sketches stored in binary16: fp32 sum of the workers' values, one division, stored
// like an update (saturated, nearest even)
__global__ void __launch_bounds__(256) k_error_reset_half(uint8_t *__restrict__ state, int64_t stride_bytes, int n_workers,
                                                          float nw, int64_t halves)
{
    for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < halves; j += (int64_t)gridDim.x * 256) {
        float acc = __half2float(((const __half *)state)[j]);
        for (int i = 1; i < n_workers; ++i)
            acc = __fadd_rn(acc, __half2float(((const __half *)(state + i * stride_bytes))[j]));
        const unsigned short h = rs_to_half(__fdiv_rn(acc, nw));
        for (int i = 0; i < n_workers; ++i)
            ((unsigned short *)(state + i * stride_bytes))[j] = h;
    }
}

}  // namespace conef

namespace conef {

// Error reset for a linear C: every worker's state becomes the mean over workers (sum in worker
// order, one division).  `words` floats per worker.
__global__ void __launch_bounds__(256) k_error_reset(uint8_t *__restrict__ state, int64_t stride_bytes, int n_workers,
                                                     float nw, int64_t words)
{
    for (int64_t j = (int64_t)blockIdx.x * 256 + threadIdx.x; j < words; j += (int64_t)gridDim.x * 256) {
        float acc = ((const float *)state)[j];
        for (int i = 1; i < n_workers; ++i)
            acc = __fadd_rn(acc, ((const float *)(state + i * stride_bytes))[j]);
        acc = __fdiv_rn(acc, nw);
        for (int i = 0; i < n_workers; ++i)
            ((float *)(state + i * stride_bytes))[j] = acc;
    }
}

}  // namespace conef
