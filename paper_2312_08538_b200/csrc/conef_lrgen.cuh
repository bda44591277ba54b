// Low-rank passes on an int8 / int4 error state for the shapes and ranks that the kernels of conef_fast.cuh
// do not take: any width, any alignment, any rank (Sec. 5.2; Alg. 2, and Alg. 4 with beta).
//
//   pass 1  P_i = M_i Q_{t-1}     a warp takes four rows (small models: one), its lanes neighbouring columns
//   pass 2  Q_i = M_i^T P_hat     a warp takes 32 columns and runs down 256 rows (two columns per lane: 168 us instead
//                                 of 140 below)
//   pass 3  r = p - P_hat Q_i^T, absmax, requantise, store: a warp takes 256 consecutive elements (whole
//           quantisation blocks), lane l the elements l, l + 32, ...
//
// Neighbouring lanes always have neighbouring elements, so that every load is a run of contiguous memory
// whatever the width of the matrix, and no load depends on 16-byte alignment.  The rank is a template
// parameter, the factors' rows come as vectors through L1, and every warp has 8 to 16 independent loads in
// flight.  Bound by instruction issue and latency (rank 2, int4: 32, 31 and 47 thread instructions per element,
// issue slots 46, 45 and 74 % busy, DRAM at a quarter of its rate).
//
// The order of every sum is part of the result: a factor that moves by one rounding moves a stored int4
// code by a whole quantum now and then, and the steps that follow amplify it (a reversed sum over the row
// tiles alone: 1e-4 to 6e-4 of the outputs' norm after a few steps).  It is that of the kernels for every
// codec (conef_kernels.cuh), so a row's columns and a tile's rows are not shared out among warps.
//
// A recurrent model's odd layers (24.9 M elements, two workers, int4, rank 2): 222 / 286 / 395 us for the
// three passes on the kernels for every codec (one element and a run-time rank at a time), 125 / 140 / 112 us
// here.
#pragma once
#include "conef_fast.cuh"

namespace conef {

constexpr int kGenThreads = 256;
constexpr int kGenCols = 32;     // pass 2: columns per warp
constexpr int kGenChunk = 256;   // pass 3: elements per warp and step
constexpr int kGenCtas = kPlanSMs * 6;   // CTAs a pass should have at least, where tiles can be made smaller

// tile sizes for a model: rows per warp of pass 1 (4 or 1), steps per tile of pass 3, and whether a whole CTA takes a
// tile of pass 2 (gen_p2_cta)
struct GenPlan {
    int nr = 4, it = 16, coop = 0;
};
// Below this many warps of pass 2 a CTA takes a tile.  Steps without and with it, int8 / int4, ranks 1, 2 and 4: 20 k to 1 M
// elements over all workers (50 to 270 warps) 48.6 -> 38.9, 44.9 -> 34.0, 54.8 -> 38.2 us, 5.1 M (1026 warps) 102 -> 83 us;
// 15 M (2040) 135 -> 137 us, 45 M (4900) 420 -> 451, 50 M (7300) 447 -> 474.
constexpr int64_t kGenCoop = kPlanSMs * 12;
// rows: matrix rows of all workers, chunks: 256-element chunks.  Four rows share a row of Q, one row makes four
// times the warps.  Steps with one and with four rows per warp, int4, rank 2: 3000 x 651 69.1 and 73.0 us,
// 13000 x 651 91.3 and 92.5, 4001 x 6003 173 and 291; four matrices 40000 x 47 139 and 113, of four workers 444
// and 323; 60000 x 333 of four workers 577 and 540.
// tiles2: warps of pass 2.
inline GenPlan gen_plan(int64_t rows, int64_t chunks, int64_t tiles2)
{
    GenPlan G;
    G.coop = tiles2 < kGenCoop;
    if (rows / 32 < kGenCtas)
        G.nr = 1;
    while (G.it > 1 && chunks / (8 * G.it) < kGenCtas)
        G.it /= 2;
    return G;
}
inline bool gen_takes(const LayerDesc &L, int ckind) { return (ckind == CONEF_C_INT8 || ckind == CONEF_C_INT4) && L.d < (1ll << 31); }
inline void gen_classify(LayerDesc &L, const GenPlan &G)
{
    L.g_nr = G.nr;
    L.g_it = G.it;
    // pass 3: a CTA's eight warps take eight neighbouring chunks and step down about one matrix row at a
    // time (wide matrices) or eight chunks on (narrow ones), so that the same rows of Q_i stay in L1
    const int64_t pr = std::max<int64_t>(1, (L.cols + kGenChunk / 2) / kGenChunk);
    L.g_step = (int32_t)(pr <= 8 ? 8 : pr);
    L.g_groups = (int32_t)((L.g_step + 7) / 8);
    const int64_t nc = (L.d + kGenChunk - 1) / kGenChunk;
    L.g_t1 = (int32_t)((L.rows + 8 * L.g_nr - 1) / (8 * L.g_nr));
    L.g_coop = G.coop;
    L.g_t2 = (int32_t)(((L.rows + kP2RowsPerTile - 1) / kP2RowsPerTile) * ((L.cols + kGenCols - 1) / kGenCols));
    if (!G.coop)
        L.g_t2 = (L.g_t2 + 7) / 8;
    L.g_t3 = (int32_t)((nc + (int64_t)L.g_step * L.g_it - 1) / ((int64_t)L.g_step * L.g_it));
}

// a row of a factor; R = 0: any rank
template <int R>
__device__ __forceinline__ void factor_row(const float *__restrict__ p, int r, float (&out)[R ? R : CONEF_MAX_RANK])
{
    if constexpr (R == 4 || R == 8) {
#pragma unroll
        for (int c = 0; c < R; c += 4) {
            const float4 t = load_global((const float4 *)(p + c));
            out[c] = t.x; out[c + 1] = t.y; out[c + 2] = t.z; out[c + 3] = t.w;
        }
    } else if constexpr (R == 2) {
        const float2 t = load_global((const float2 *)p);
        out[0] = t.x; out[1] = t.y;
    } else if constexpr (R == 1) {
        out[0] = load_global(p);
    } else {
#pragma unroll
        for (int c = 0; c < CONEF_MAX_RANK; ++c)
            out[c] = c < r ? load_global(p + c) : 0.f;
    }
}
// float(code) from a code's byte or nibble
template <int CK>
__device__ __forceinline__ float code_value(uint32_t raw)
{
    constexpr bool INT4 = CK == CONEF_C_INT4;
    const uint32_t u = INT4 ? ((raw & 0xFu) ^ 8u) : ((raw & 0xFFu) ^ 0x80u);
    return __fsub_rn(__uint_as_float(0x4B000000u | u), INT4 ? 8388616.f : 8388736.f);
}
template <int CK>
__device__ __forceinline__ uint32_t code_raw(const uint8_t *__restrict__ codes, uint32_t j)
{
    return CK == CONEF_C_INT4 ? (uint32_t)load_global(codes + (j >> 1)) >> (4 * (j & 1u)) : (uint32_t)load_global(codes + j);
}
__device__ __forceinline__ float gen_scale(const uint8_t *__restrict__ b, uint32_t blk, bool half)
{
    return half ? __half2float(__ushort_as_half(load_global((const unsigned short *)b + blk))) : load_global((const float *)b + blk);
}

template <int CK, int R, int NR>   // NR: rows per warp
__device__ __forceinline__ void gen_p1_body(const DevView &V, const LayerDesc &L, uint32_t tile)
{
    constexpr int RM = R ? R : CONEF_MAX_RANK, P1U = NR == 1 ? 6 : RM > 4 ? 2 : 3;   // column groups in flight
    const int r = R ? R : L.rank, worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t m = (uint32_t)L.cols, n = (uint32_t)L.rows;
    const uint32_t row0 = (tile * 8u + warp) * NR;
    const uint8_t *__restrict__ st = fresh(V.state + worker * V.state_stride);
    const uint8_t *__restrict__ codes = st + L.a_off, *__restrict__ scales = st + L.b_off;
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off), *__restrict__ Q = fresh(V.qprev + L.msgq_off);
    const int shift = 31 - __clz(L.unit);
    const bool half = V.scale_half != 0;
    const float lr = V.lr, omb = V.omb;
    uint32_t jb[NR];   // (rows past the end repeat the last one and are not stored)
#pragma unroll
    for (int i = 0; i < NR; ++i)
        jb[i] = min(row0 + i, n - 1) * m;
    float acc[NR][RM];
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
        for (int c = 0; c < RM; ++c)
            acc[i][c] = 0.f;
    auto columns = [&](uint32_t col, auto count) {
        constexpr int N = decltype(count)::value;
        float gv[N][NR], sc[N][NR];
        uint32_t w[N][NR];
#pragma unroll
        for (int u = 0; u < N; ++u)
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const uint32_t j = jb[i] + col + u * 32;
                gv[u][i] = load_global(g + j);
                w[u][i] = code_raw<CK>(codes, j);
                sc[u][i] = gen_scale(scales, j >> shift, half);
            }
#pragma unroll
        for (int u = 0; u < N; ++u) {
            float q[RM];
            factor_row<R>(Q + (size_t)(col + u * 32) * r, r, q);
#pragma unroll
            for (int i = 0; i < NR; ++i) {
                const float p = __fmaf_rn(lr, gv[u][i], __fmul_rn(omb, __fmul_rn(code_value<CK>(w[u][i]), sc[u][i])));   // Alg. 2 (4) line 5
#pragma unroll
                for (int c = 0; c < RM; ++c)
                    acc[i][c] = __fmaf_rn(p, q[c], acc[i][c]);
            }
        }
    };
    uint32_t col = lane;
    for (; col + (P1U - 1) * 32 < m; col += P1U * 32)
        columns(col, IntC<P1U>());
    for (; col < m; col += 32)
        columns(col, IntC<1>());
    // totals of column idx end up in the lanes whose bits below `plain` are zero
    int idx = 0, hh = RM, plain = 32;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1)
        if (hh > 1) {
            hh >>= 1;
            if (lane & o)
                idx += hh;
            plain = o;
        }
    const bool writer = (lane & (plain - 1)) == 0 && idx < r;
    float *__restrict__ P = V.msgp + worker * V.msgp_stride + L.msgp_off;
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        warp_reduce_many<RM>(acc[i], lane);
        if (writer && row0 + i < n)
            P[(size_t)(row0 + i) * r + idx] = acc[i][0];
    }
}

template <int CK, int R>
__device__ __forceinline__ void gen_p2_body(const DevView &V, const LayerDesc &L, uint32_t tile)
{
    constexpr int RM = R ? R : CONEF_MAX_RANK, K = kGenCols / 32, U = RM > 4 ? 4 : 8;   // columns per lane, rows in flight
    const int r = R ? R : L.rank, worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t m = (uint32_t)L.cols, n = (uint32_t)L.rows;
    const uint32_t task = tile * 8u + warp, ct = (m + kGenCols - 1) / kGenCols, rt = task / ct, c0 = (task - rt * ct) * kGenCols + lane;
    const uint32_t r_lo = rt * (uint32_t)kP2RowsPerTile, r_hi = min(n, r_lo + (uint32_t)kP2RowsPerTile);
    if (r_lo >= n)
        return;   // (no CTA-wide barrier below)
    const uint8_t *__restrict__ st = fresh(V.state + worker * V.state_stride);
    const uint8_t *__restrict__ codes = st + L.a_off, *__restrict__ scales = st + L.b_off;
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off), *__restrict__ ph = fresh(V.phat + L.msgp_off);
    const int shift = 31 - __clz(L.unit);
    const bool half = V.scale_half != 0;
    const float lr = V.lr, omb = V.omb;
    uint32_t col[K];   // (columns past the end repeat the last one and are not stored)
#pragma unroll
    for (int k = 0; k < K; ++k)
        col[k] = min(c0 + 32 * k, m - 1);
    float acc[K][RM];
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
        for (int c = 0; c < RM; ++c)
            acc[k][c] = 0.f;
    auto rows = [&](uint32_t a, auto count) {
        constexpr int N = decltype(count)::value;
        float gv[N][K], sc[N][K];
        uint32_t w[N][K];
#pragma unroll
        for (int u = 0; u < N; ++u)
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const uint32_t j = (a + u) * m + col[k];
                gv[u][k] = load_global(g + j);
                w[u][k] = code_raw<CK>(codes, j);
                sc[u][k] = gen_scale(scales, j >> shift, half);
            }
#pragma unroll
        for (int u = 0; u < N; ++u) {
            float pr[RM];
            factor_row<R>(ph + (size_t)(a + u) * r, r, pr);
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float p = __fmaf_rn(lr, gv[u][k], __fmul_rn(omb, __fmul_rn(code_value<CK>(w[u][k]), sc[u][k])));
#pragma unroll
                for (int c = 0; c < RM; ++c)
                    acc[k][c] = __fmaf_rn(p, pr[c], acc[k][c]);
            }
        }
    };
    uint32_t a = r_lo;
    for (; a + U <= r_hi; a += U)
        rows(a, IntC<U>());
    for (; a < r_hi; ++a)
        rows(a, IntC<1>());
    float *part = V.part + worker * V.part_stride + L.part_off + (size_t)rt * m * r;   // added in order by k_lr_pass2_reduce
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (c0 + 32 * k < m) {
#pragma unroll
            for (int c = 0; c < RM; ++c)
                if (R || c < r)
                    part[(size_t)(c0 + 32 * k) * r + c] = acc[k][c];
        }
}

// The same tile by a whole CTA, for models whose tiles do not fill the SMs: the eight warps form p of 32 rows each in shared
// memory, then a warp per column of the factor adds down the rows, in the order of gen_p2_body.  There a warp walks the
// 256 rows eight at a time, 32 waits for memory one after the other, however small the model.
constexpr size_t kGenCoopSmem = (size_t)kP2RowsPerTile * (32 + CONEF_MAX_RANK) * 4;
template <int CK, int R>
__device__ __forceinline__ void gen_p2_cta(const DevView &V, const LayerDesc &L, uint32_t tile, float *smem)
{
    constexpr int U = 16;   // rows in flight per warp
    const int r = R ? R : L.rank, worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t m = (uint32_t)L.cols, n = (uint32_t)L.rows;
    const uint32_t ct = (m + kGenCols - 1) / kGenCols, rt = tile / ct, c0 = (tile - rt * ct) * kGenCols + lane;
    const uint32_t r_lo = rt * (uint32_t)kP2RowsPerTile, have = min(n - r_lo, (uint32_t)kP2RowsPerTile);
    const uint8_t *__restrict__ st = fresh(V.state + worker * V.state_stride);
    const uint8_t *__restrict__ codes = st + L.a_off, *__restrict__ scales = st + L.b_off;
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off), *__restrict__ ph = fresh(V.phat + L.msgp_off) + (size_t)r_lo * r;
    const int shift = 31 - __clz(L.unit);
    const bool half = V.scale_half != 0;
    const float lr = V.lr, omb = V.omb;
    float *const p = smem, *const phs = smem + kP2RowsPerTile * 32;   // [row][column], [row][c]
    for (uint32_t x = threadIdx.x; x < have * r; x += kGenThreads)
        phs[x] = load_global(ph + x);
    const uint32_t col = min(c0, m - 1);   // (columns past the end repeat the last one and are not stored)
    for (uint32_t a0 = warp; a0 < have; a0 += 8 * U) {
        float gv[U], sc[U];
        uint32_t w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {   // (rows past the end repeat the last one)
            const uint32_t j = (r_lo + min(a0 + 8 * u, have - 1)) * m + col;
            gv[u] = load_global(g + j);
            w[u] = code_raw<CK>(codes, j);
            sc[u] = gen_scale(scales, j >> shift, half);
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (a0 + 8 * u < have)
                p[(a0 + 8 * u) * 32 + lane] = __fmaf_rn(lr, gv[u], __fmul_rn(omb, __fmul_rn(code_value<CK>(w[u]), sc[u])));
    }
    __syncthreads();
    if (warp < r && c0 < m) {
        float acc = 0.f;
        uint32_t a = 0;
        for (; a + 8 <= have; a += 8) {
            float x[8], y[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                x[u] = p[(a + u) * 32 + lane];
                y[u] = phs[(a + u) * r + warp];
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                acc = __fmaf_rn(x[u], y[u], acc);
        }
        for (; a < have; ++a)
            acc = __fmaf_rn(p[a * 32 + lane], phs[a * r + warp], acc);
        V.part[worker * V.part_stride + L.part_off + ((size_t)rt * m + c0) * r + warp] = acc;
    }
}

template <int CK, int R, int KB>
__device__ __forceinline__ void gen_p3_body(const DevView &V, const LayerDesc &L, uint32_t tile, uint8_t *bytes)
{
    constexpr int RM = R ? R : CONEF_MAX_RANK, K = kGenChunk / 32;
    const int bs = KB ? (KB == 8 ? 3 : KB == 4 ? 2 : KB == 2 ? 1 : 0) : 26 - __clz(L.unit);   // 32 << bs elements per block (KB << 5, or as configured)
    const int NB = K >> bs;
    constexpr bool INT4 = CK == CONEF_C_INT4;
    constexpr int NW = INT4 ? 1 : 2;   // code words per lane
    const int r = R ? R : L.rank, worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t m = (uint32_t)L.cols, d = (uint32_t)L.d;
    const uint32_t step = L.g_step, groups = L.g_groups, nc = (d + kGenChunk - 1) / kGenChunk;
    const uint32_t tt = tile / groups, cpos = (tile - tt * groups) * 8 + warp;   // place among the chunks of a step
    if (cpos >= step)
        return;   // (no CTA-wide barrier below)
    uint8_t *st = V.state + worker * V.state_stride;
    uint32_t *codes = (uint32_t *)(st + L.a_off);
    uint8_t *scales = st + L.b_off;
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off), *__restrict__ ph = fresh(V.phat + L.msgp_off);
    const float *__restrict__ Q = fresh(V.msgq + worker * V.msgq_stride + L.msgq_off);
    const bool half = V.scale_half != 0;
    const float lr = V.lr, omb = V.omb, beta = V.beta;
    uint8_t *mine = bytes + warp * kGenChunk;
    const uint32_t nblk = (uint32_t)L.nunits;

    uint32_t ch = tt * (uint32_t)L.g_it * step + cpos;
    // row and column of the chunk's first element, and how they move from step to step
    uint32_t row = (ch * kGenChunk) / m, col = ch * kGenChunk - row * m;
    const uint32_t drow = (step * kGenChunk) / m, dcol = step * kGenChunk - drow * m;
    float gn[K], sn = 0.f;
    uint32_t wn[NW];
    auto fetch = [&](uint32_t c) {   // (32-bit offsets: d < 2^31)
        const uint32_t j = c * kGenChunk + lane;
        if (c < nc) {
            if (j + 32 * (K - 1) - lane + 31u < d) {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    gn[k] = __ldcs(g + j + 32 * k);
            } else {
#pragma unroll
                for (int k = 0; k < K; ++k)
                    gn[k] = j + 32 * k < d ? __ldcs(g + j + 32 * k) : 0.f;
            }
#pragma unroll
            for (int x = 0; x < NW; ++x)   // (the state's arrays are padded to 256 bytes)
                wn[x] = codes[c * (32 * NW) + 32 * x + lane];
            const uint32_t b = c * NB + lane;
            sn = 0.f;
            if (lane < NB && b < nblk)
                sn = half ? __half2float(__ushort_as_half(((const unsigned short *)scales)[b])) : ((const float *)scales)[b];
        }
    };
    fetch(ch);
    for (int it = 0; it < L.g_it && ch < nc; ++it, ch += step) {
        float gv[K];
        uint32_t w[NW];
#pragma unroll
        for (int k = 0; k < K; ++k)
            gv[k] = gn[k];
#pragma unroll
        for (int x = 0; x < NW; ++x)
            w[x] = wn[x];
        const float sv = sn;
        if (it + 1 < L.g_it)
            fetch(ch + step);
        const uint32_t j0 = ch * kGenChunk + lane;
        float res[K], ek[K];
#pragma unroll
        for (int k = 0; k < K; ++k) {
            // element 32 k + lane: its word is another lane's
            uint32_t raw;
            if (INT4)
                raw = __shfl_sync(0xffffffffu, w[0], 4 * k + (lane >> 3)) >> (4 * (lane & 7));
            else
                raw = __shfl_sync(0xffffffffu, w[NW == 2 ? k / 4 : 0], 8 * (k & 3) + (lane >> 2)) >> (8 * (lane & 3));
            const float s = __shfl_sync(0xffffffffu, sv, k >> bs);
            ek[k] = __fmul_rn(code_value<CK>(raw), s);
            res[k] = __fmaf_rn(lr, gv[k], __fmul_rn(omb, ek[k]));   // Alg. 2 (4) line 5
        }
        // r = p - P_hat Q_i^T
        if (col + (kGenChunk - 1) < m && (ch + 1) * kGenChunk <= d) {   // one matrix row
            float pr[RM];
            factor_row<R>(ph + (size_t)row * r, r, pr);
            const float *q0 = Q + (size_t)(col + lane) * r;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                float q[RM];
                factor_row<R>(q0 + 32 * k * r, r, q);
#pragma unroll
                for (int c = 0; c < RM; ++c)
                    if (R || c < r)
                        res[k] = __fmaf_rn(-pr[c], q[c], res[k]);
            }
        } else {
            uint32_t cc = col + lane, rr = row;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                if (cc >= m) {
                    const uint32_t t = m >= 32 ? 1u : cc / m;
                    cc -= t * m;
                    rr += t;
                }
                if (j0 + 32 * k < d) {
                    float pr[RM], q[RM];
                    factor_row<R>(ph + (size_t)rr * r, r, pr);
                    factor_row<R>(Q + (size_t)cc * r, r, q);
#pragma unroll
                    for (int c = 0; c < RM; ++c)
                        if (R || c < r)
                            res[k] = __fmaf_rn(-pr[c], q[c], res[k]);
                } else {
                    res[k] = ek[k] = 0.f;
                }
                cc += 32;
            }
        }
        if (beta != 0.f) {   // Alg. 4 line 9 stores C(beta e + r)
#pragma unroll
            for (int k = 0; k < K; ++k)
                res[k] = __fmaf_rn(beta, ek[k], res[k]);
        }
        // block maxima: lane b takes block b's
        float amax = 0.f;
        if constexpr (KB != 0) {
#pragma unroll
            for (int b = 0; b < K / KB; ++b) {
                float x = 0.f;
#pragma unroll
                for (int k = 0; k < KB; ++k)
                    x = fmaxf(x, fabsf(res[b * KB + k]));
                const float y = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(x)));   // (not negative: ordered like integers)
                amax = lane == b ? y : amax;
            }
        } else {
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const float x = fmaxf(0.f, fabsf(res[k]));   // (a NaN counts as nothing, as above)
                const float y = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(x)));
                amax = lane == k >> bs ? fmaxf(amax, y) : amax;
            }
        }
        float s, inv;
        unsigned short hb = 0;
        if (half)
            block_scale<CK, true>(amax, s, inv, hb);
        else
            block_scale<CK, false>(amax, s, inv, hb);
        constexpr float qm = INT4 ? 7.f : 127.f;
        const bool clamp = __any_sync(0xffffffffu, !(__fmul_rn(amax, inv) < qm + 0.49f));   // (see quant_pack8)
#pragma unroll
        for (int k = 0; k < K; ++k) {
            float x = __fmul_rn(res[k], __shfl_sync(0xffffffffu, inv, k >> bs));
            if (clamp)
                x = fminf(fmaxf(x, -qm), qm);
            mine[32 * k + lane] = (uint8_t)__float_as_uint(__fadd_rn(x, 12582912.0f));   // the low byte is the code
        }
        const uint32_t b = ch * NB + lane;
        if (lane < NB && b < nblk) {
            if (half)
                ((unsigned short *)scales)[b] = hb;
            else
                ((float *)scales)[b] = s;
        }
        __syncwarp();
        if (INT4) {
            const uint2 v = *(const uint2 *)(mine + 8 * lane);
            auto four = [](uint32_t x) {   // four bytes' low nibbles -> 16 bits
                x &= 0x0F0F0F0Fu;
                x |= x >> 4;
                return __byte_perm(x, 0u, 0x4420);
            };
            codes[ch * 32 + lane] = four(v.x) | (four(v.y) << 16);
        } else {
#pragma unroll
            for (int x = 0; x < NW; ++x)
                codes[ch * 64 + 32 * x + lane] = *(const uint32_t *)(mine + 128 * x + 4 * lane);
        }
        __syncwarp();
        row += drow;
        col += dcol;
        if (col >= m) {
            col -= m;
            ++row;
        }
    }
}

// R: the configured rank (1, 2, 4, 8; 0: another one).  Tensors thinner than it, and those behind them whose
// factors are off the vector loads' alignment, take the run-time rank.
template <int PASS, int CK, int R, int KB>
__global__ void __launch_bounds__(kGenThreads, PASS == 2 || R == 8 || R == 0 ? 3 : 4) k_gen_pass(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
    __shared__ __align__(16) uint8_t bytes[PASS == 3 ? 8 * kGenChunk : 16];
    extern __shared__ __align__(16) float gen_smem[];
    grid_release();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const uint32_t tile = blockIdx.x - pfx[li];
    grid_wait();
    if (PASS == 1 && !L.compressed) {   // (a 1-D tensor: its message in the same launch)
        pass_tile(V, L, tile);
        return;
    }
    constexpr int VW = R == 8 ? 4 : R ? R : 1;   // floats per vector load
    const bool exact = R != 0 && L.rank == R && ((L.msgp_off | L.msgq_off) & (VW - 1)) == 0;
    if (PASS == 1) {
        if (R && exact) {
            if (L.g_nr == 4)
                gen_p1_body<CK, R, 4>(V, L, tile);
            else
                gen_p1_body<CK, R, 1>(V, L, tile);
        } else {
            for (int x = 0; x < L.g_nr; ++x)
                gen_p1_body<CK, 0, 1>(V, L, tile * (uint32_t)L.g_nr + x);
        }
    } else if (PASS == 2) {
        if (L.g_coop) {
            if (R && exact)
                gen_p2_cta<CK, R>(V, L, tile, gen_smem);
            else
                gen_p2_cta<CK, 0>(V, L, tile, gen_smem);
        } else if (R && exact) {
            gen_p2_body<CK, R>(V, L, tile);
        } else {
            gen_p2_body<CK, 0>(V, L, tile);
        }
    } else {
        if (R && exact)
            gen_p3_body<CK, R, KB>(V, L, tile, bytes);
        else
            gen_p3_body<CK, 0, KB>(V, L, tile, bytes);
    }
}

// launcher (conef_lrgen.cu); coop: the plan's
cudaError_t gen_launch(int pass, int ckind, int rank, int unit, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, bool coop);

}  // namespace conef
