// Low-rank passes on an int8 / int4 error state for the shapes and ranks that the kernels of conef_fast.cuh
// do not take: any width, any alignment, any rank (Sec. 5.2; Alg. 2, and Alg. 4 with beta).
//
//   pass 1  P_i = M_i Q_{t-1}     a warp takes four rows (rank 8: two; small models: one), its lanes neighbouring columns
//   pass 2  Q_i = M_i^T P_hat     128, 64 or 32 threads take as many columns, one each, and run down 256 rows
//   pass 3  r = p - P_hat Q_i^T, absmax, requantise, store: a warp takes 512 (256) consecutive elements, whole
//           quantisation blocks
//
// Where sums are formed neighbouring lanes have neighbouring elements, whatever the width of the matrix, so that every load of
// the gradient and of a factor is a run of contiguous memory and none depends on 16-byte alignment.  Codes are decoded (and
// in pass 3 formed) a word of eight elements per lane on the codes' own alignment, which goes through shared memory: loaded by
// the lane of each element, a code's byte and its scale were two more loads and ten more instructions per element.  The
// gradient of the next rows or chunk is loaded as this one's registers fall free.
//
// The order of every sum is part of the result: a factor that moves by one rounding moves a stored int4
// code by a whole quantum now and then, and the steps that follow amplify it (a reversed sum over the row
// tiles alone: 1e-4 to 6e-4 of the outputs' norm after a few steps).  It is that of the kernels for every
// codec (conef_kernels.cuh), so a row's columns and a tile's rows are not shared out among warps.
//
// A recurrent model's odd layers (28.4 M elements, two workers, int4, rank 2): 94 / 107 / 118 us for the three passes with a lane
// loading the code of its own element, 62 / 73 / 78 us now: 20, 22 and 31 instead of 32, 31 and 47 instructions per element, DRAM
// at half of its rate.  Step and update, before and now: that list 387 -> 286 us; 4001 x 6003, int8, rank 4, four workers 360 -> 325;
// 25 M elements of width 4096 and 1024, int4, rank 1, two workers 300 -> 226; odd matrices, int8, rank 8, four workers 718 -> 545.
#pragma once
#include "conef_fast.cuh"

namespace conef {

constexpr int kGenThreads = 256;
constexpr int kGenCols = 32;     // pass 2: columns of a tile that a CTA takes (gen_p2_cta)
constexpr int kGenChunk = 512;   // pass 3: elements per warp and step, or half as many (kGenChunkElems)
constexpr int kGenCtas = kPlanSMs * 6;   // CTAs a pass should have at least, where tiles can be made smaller

// rows per warp of pass 1 on all but small models (two at rank 8, whose sums alone take 32 registers at four)
__host__ __device__ constexpr int gen_p1_rows(int rank) { return rank > 4 ? 2 : 4; }
// tile sizes for a model: rows per warp of pass 1 (gen_p1_rows or 1), steps per tile of pass 3, and whether a whole CTA takes a
// tile of pass 2 (gen_p2_cta)
struct GenPlan {
    int nr = 1, it = 16, chunk = kGenChunk / 2, coop = 0;
};
// Below this many tiles of 32 columns (all workers) a CTA takes one.  Steps with a CTA per tile and with a column per thread: 512 tiles,
// rank 4, int4 52.6 and 58.9 us; 1026, int8, rank 2 78.9 and 77.5; 1481, int8, rank 4 152 and 146; 1580, int8, rank 1 116.0 and 108.7.
constexpr int64_t kGenCoop = kPlanSMs * 6;
// rows: matrix rows, elems: elements, of all workers.  Four rows share a row of Q, one row makes four
// times the warps.  Steps with one and with four rows per warp, int4, rank 2: 3000 x 651 69.1 and 73.0 us,
// 13000 x 651 91.3 and 92.5, 4001 x 6003 173 and 291; four matrices 40000 x 47 139 and 113, of four workers 444
// and 323; 60000 x 333 of four workers 577 and 540.
// tiles2: tiles of 32 columns of pass 2.
// Elements (all workers) from which a lane of pass 3 has sixteen instead of eight.  Steps with eight and with sixteen, rank 4, int4: 0.5 M
// 32.2 and 35.3 us, 2 M 37.9 and 37.0, 8 M 87.0 and 85.1, 32 M 218 and 204; int8: 18 M of odd widths 238 and 229, 96 M of one
// 6003 wide 320 and 328, odd ones at rank 8 558 and 549.
constexpr int64_t kGenChunkElems = 1'500'000;
inline GenPlan gen_plan(int rank, int64_t rows, int64_t elems, int64_t tiles2)
{
    const int64_t chunks = elems / (kGenChunk / 2);
    GenPlan G;
    G.coop = tiles2 < kGenCoop;
    if (elems >= kGenChunkElems)
        G.chunk = kGenChunk;
    if (rows / 32 >= kGenCtas)
        G.nr = gen_p1_rows(rank);
    while (G.it > 1 && chunks / (8 * G.it) < kGenCtas)
        G.it /= 2;
    return G;
}
inline bool gen_takes(const LayerDesc &L, int ckind) { return (ckind == CONEF_C_INT8 || ckind == CONEF_C_INT4) && L.d < (1ll << 31); }
// Whether a tensor takes the kernels with its rank as a constant: it has the configured rank, and its factors are aligned for
// the vector loads of their rows
__host__ __device__ __forceinline__ bool gen_exact(const LayerDesc &L, int rank)
{
    return (rank == 1 || rank == 2 || rank == 4 || rank == 8) && L.rank == rank && ((L.msgp_off | L.msgq_off) & ((rank == 8 ? 4 : rank) - 1)) == 0;
}
// the rank that a configuration's kernels are made for
__host__ __device__ constexpr int gen_rank(int rank) { return rank <= 2 ? rank : rank <= 4 ? 4 : 8; }
// Threads per tile of pass 2 and columns per tile: equal tiles whose words (one more than the columns make where a row starts
// within a word) are two per thread; the largest that leaves as few threads idle as any other, give or take 5 %.
inline void gen_p2_split(int64_t cols, int32_t &threads, int32_t &width)
{
    double best = 0.0;
    for (int t = 128; t >= 32; t /= 2) {
        const int64_t most = cols % 8 == 0 ? t : t - 7, ct = (cols + most - 1) / most;
        int64_t w = (cols + ct - 1) / ct;
        if (cols % 8 == 0)
            w = (w + 7) / 8 * 8;
        const double used = (double)cols / (double)((cols + w - 1) / w * t);
        if (used > best + 0.05) {
            best = used;
            threads = t;
            width = (int32_t)w;
        }
    }
}
inline void gen_classify(LayerDesc &L, const GenPlan &G, int cfg_rank)
{
    L.g_nr = G.nr;
    L.g_it = G.it;
    // pass 3: a CTA's eight warps take eight neighbouring chunks and step down about one matrix row at a
    // time (wide matrices) or eight chunks on (narrow ones), so that the same rows of Q_i stay in L1
    L.g_chunk = G.chunk == kGenChunk && gen_exact(L, cfg_rank) ? kGenChunk : kGenChunk / 2;
    if (L.g_chunk == kGenChunk)
        L.g_it = (G.it + 1) / 2;
    const int64_t pr = std::max<int64_t>(1, (L.cols + L.g_chunk / 2) / L.g_chunk);
    L.g_step = (int32_t)(pr <= 8 ? 8 : pr);
    L.g_groups = (int32_t)((L.g_step + 7) / 8);
    const int64_t nc = (L.d + L.g_chunk - 1) / L.g_chunk;
    L.g_t1 = (int32_t)((L.rows + 8 * L.g_nr - 1) / (8 * L.g_nr));
    const int64_t rt = (L.rows + kP2RowsPerTile - 1) / kP2RowsPerTile;
    if (G.coop) {
        L.g_p2t = 0;
        L.g_p2w = kGenCols;
        L.g_t2 = (int32_t)(rt * ((L.cols + kGenCols - 1) / kGenCols));
    } else {
        gen_p2_split(L.cols, L.g_p2t, L.g_p2w);
        const int64_t tasks = rt * ((L.cols + L.g_p2w - 1) / L.g_p2w);
        L.g_t2 = (int32_t)((tasks * L.g_p2t + kGenThreads - 1) / kGenThreads);
    }
    L.g_t3 = (int32_t)((nc + (int64_t)L.g_step * L.g_it - 1) / ((int64_t)L.g_step * L.g_it));
}

// bytes of shared memory of a CTA of pass 2
inline size_t gen_p2_smem(const LayerDesc &L, int cfg_rank);

// Ranks as template arguments: R > 0 is the rank, R < 0 stands for any up to -R
__host__ __device__ constexpr int gen_most(int R) { return R < 0 ? -R : R; }
// a row of a factor
template <int R, int AT = 0>   // AT: rows behind p
__device__ __forceinline__ void factor_row(const float *p, int r, float (&out)[gen_most(R)])
{
    if constexpr (R == 4 || R == 8) {
        const float4 t = load_global_at<AT * R * 4>((const float4 *)p);
        out[0] = t.x; out[1] = t.y; out[2] = t.z; out[3] = t.w;
        if constexpr (R == 8) {
            const float4 v = load_global_at<AT * R * 4 + 16>((const float4 *)p);
            out[4] = v.x; out[5] = v.y; out[6] = v.z; out[7] = v.w;
        }
    } else if constexpr (R == 2) {
        const float2 t = load_global_at<AT * 8>((const float2 *)p);
        out[0] = t.x; out[1] = t.y;
    } else if constexpr (R == 1) {
        out[0] = load_global_at<AT * 4>(p);
    } else {
        p += (size_t)AT * r;
#pragma unroll
        for (int c = 0; c < -R; ++c)
            out[c] = c < r ? load_global(p + c) : 0.f;
    }
}
// Eight consecutive elements of the stored error, as loaded: the elements 8 q .. 8 q + 7 of a tensor are whole code words
// and lie in one quantisation block.
struct GenWords {
    uint32_t w0, w1, s;   // code words, bits of the scale
};
template <int CK, bool HALF>
__device__ __forceinline__ GenWords gen_fetch(const uint8_t *__restrict__ codes, const uint8_t *__restrict__ scales, uint32_t q, int qshift)
{
    GenWords w;
    if (CK == CONEF_C_INT4) {
        w.w0 = load_global((const uint32_t *)codes + q);
        w.w1 = 0;
    } else {
        const uint2 t = load_global((const uint2 *)codes + q);
        w.w0 = t.x;
        w.w1 = t.y;
    }
    w.s = HALF ? (uint32_t)load_global((const unsigned short *)scales + (q >> qshift)) : load_global((const uint32_t *)scales + (q >> qshift));
    return w;
}
// ... decoded (Alg. 4, PARTIAL: times 1 - beta), to shared memory.  Eight lanes' first 16 bytes would lie in half of the banks,
// so every other four lanes (swap) store their second half first.
template <int CK, bool HALF, bool PARTIAL>
__device__ __forceinline__ void gen_decode(const GenWords &w, float omb, float *dst, bool swap)
{
    float e[8];
    uint32_t w0 = w.w0, w1 = w.w1;
    if (CK == CONEF_C_INT4) {
        w0 = swap ? __byte_perm(w0, 0u, 0x1032) : w0;
    } else {
        w0 = swap ? w.w1 : w.w0;
        w1 = swap ? w.w0 : w.w1;
    }
    decode8<CK, HALF>(w0, w1, scale_const<CK, HALF>(HALF ? __half2float(__ushort_as_half((unsigned short)w.s)) : __uint_as_float(w.s)), e);
    if (PARTIAL) {
#pragma unroll
        for (int x = 0; x < 8; ++x)
            e[x] = __fmul_rn(omb, e[x]);
    }
    *(float4 *)(dst + (swap ? 4 : 0)) = make_float4(e[0], e[1], e[2], e[3]);
    *(float4 *)(dst + (swap ? 0 : 4)) = make_float4(e[4], e[5], e[6], e[7]);
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

// Floats of shared memory per warp of pass 1: a chunk of gen_p1_cols columns of each row, and eight for where it starts
__host__ __device__ constexpr int gen_p1_cols(int nr) { return nr == 4 ? 128 : 256; }
__host__ __device__ constexpr int gen_p1_floats(int nr) { return nr * (gen_p1_cols(nr) + 8); }
constexpr size_t kGenP1Smem = 8 * gen_p1_floats(4) * 4;

// P_i of NR rows from the lanes' sums
template <int RM, int NR>
__device__ __forceinline__ void gen_p1_store(float (&acc)[NR][RM], float *__restrict__ P, uint32_t row0, uint32_t n, int r)
{
    const int lane = threadIdx.x & 31;
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
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        warp_reduce_many<RM>(acc[i], lane);
        if (writer && row0 + i < n)
            P[(size_t)(row0 + i) * r + idx] = acc[i][0];
    }
}

// NR rows per warp, a chunk of columns at a time.  The lanes decode the chunk's codes a word each, eight elements on their own
// alignment whatever that of the row, into shared memory, whose last eight elements are the next chunk's first.
template <int CK, bool HALF, bool PARTIAL, int R, int NR>
__device__ __forceinline__ void gen_p1_body(const DevView &V, const LayerDesc &L, uint32_t tile, float *smem)
{
    constexpr int RM = gen_most(R), CH = gen_p1_cols(NR), U = CH / 32, PITCH = CH + 8, GR = CH / 8, NG = NR * GR / 32;
    const int r = R > 0 ? R : L.rank, worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t m = (uint32_t)L.cols, n = (uint32_t)L.rows;
    const uint32_t row0 = (tile * 8u + warp) * NR;
    if (row0 >= n)
        return;   // (no CTA-wide barrier below)
    const uint8_t *__restrict__ st = fresh(V.state + worker * V.state_stride);
    const uint8_t *__restrict__ codes = st + L.a_off, *__restrict__ scales = st + L.b_off;
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off), *__restrict__ Q = fresh(V.qprev + L.msgq_off);
    const int qshift = 28 - __clz(L.unit);
    const uint32_t last = ((uint32_t)L.d - 1) >> 3;   // the tensor's last code word
    const float lr = V.lr, omb = V.omb;
    float *const buf = smem + warp * gen_p1_floats(NR);
    const float *gp[NR], *eb[NR];   // (rows past the end repeat the last one and are not stored)
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const uint32_t j = min(row0 + i, n - 1) * m;
        gp[i] = g + j + lane;
        eb[i] = buf + i * PITCH + (j & 7u) + lane;
    }
    // this lane's words of the chunk: the same place in rows 2 x + lane / 16 (one row: x is 0)
    const bool swap = (lane & 4) != 0;
    uint32_t word[NG];
    float *const put = buf + (lane / GR) * PITCH + 8 + 8 * (lane % GR);
#pragma unroll
    for (int x = 0; x < NG; ++x)
        word[x] = ((min(row0 + 32 / GR * x + lane / GR, n - 1) * m) >> 3) + 1 + lane % GR;
    float acc[NR][RM];
#pragma unroll
    for (int i = 0; i < NR; ++i)
#pragma unroll
        for (int c = 0; c < RM; ++c)
            acc[i][c] = 0.f;
    GenWords w[NG];
    auto fetch = [&] {
#pragma unroll
        for (int x = 0; x < NG; ++x) {
            w[x] = gen_fetch<CK, HALF>(codes, scales, min(word[x], last), qshift);
            word[x] += GR;
        }
    };
    fetch();
    float gv[NR][U];
    static_for<U>([&](auto uc) {
        constexpr int u = decltype(uc)::value;
#pragma unroll
        for (int i = 0; i < NR; ++i)
            gv[i][u] = 32 * u + lane < m ? load_global_at<128 * u>(gp[i]) : 0.f;
    });
    if (lane < NR)   // the word that a row begins in
        gen_decode<CK, HALF, PARTIAL>(gen_fetch<CK, HALF>(codes, scales, (min(row0 + lane, n - 1) * m) >> 3, qshift), omb, buf + lane * PITCH, false);
    const float *Qp = Q + (size_t)lane * r;
    auto chunk = [&](uint32_t left, auto whole_c) {   // left: columns of the row from this chunk on
        constexpr bool WHOLE = decltype(whole_c)::value != 0;
#pragma unroll
        for (int x = 0; x < NG; ++x)
            gen_decode<CK, HALF, PARTIAL>(w[x], omb, put + 32 / GR * x * PITCH, swap);
        if (WHOLE)
            fetch();
        __syncwarp();
        static_for<U>([&](auto uc) {
            constexpr int u = decltype(uc)::value;
            if (WHOLE || 32 * u + lane < left) {
                float q[RM];
                factor_row<R, 32 * u>(Qp, r, q);
#pragma unroll
                for (int i = 0; i < NR; ++i) {
                    const float p = __fmaf_rn(lr, gv[i][u], eb[i][32 * u]);   // Alg. 2 (4) line 5
#pragma unroll
                    for (int c = 0; c < RM; ++c)
                        acc[i][c] = __fmaf_rn(p, q[c], acc[i][c]);
                    if (WHOLE && CH + 32 * u + lane < left)   // the next chunk's
                        gv[i][u] = load_global_at<4 * CH + 128 * u>(gp[i]);
                }
            }
        });
        if (WHOLE) {
#pragma unroll
            for (int i = 0; i < NR; ++i)
                gp[i] += CH;
            Qp += (size_t)CH * r;
            __syncwarp();
            if (NR * 8 == 32 || lane < NR * 8)
                buf[(lane >> 3) * PITCH + (lane & 7)] = buf[(lane >> 3) * PITCH + CH + (lane & 7)];
            __syncwarp();
        }
    };
    uint32_t left = m;
    for (; left >= CH; left -= CH)
        chunk(left, IntC<1>());
    if (left)
        chunk(left, IntC<0>());
    __syncwarp();
    gen_p1_store<RM, NR>(acc, V.msgp + worker * V.msgp_stride + L.msgp_off, row0, n, r);
}

// The same for rows of at most kGenNarrow columns, eight words whatever their place within the first: a lane has one word.
// 140 k rows of 33 to 47 columns, rank 2, int4, four workers: 67 us instead of 95.
constexpr int kGenNarrow = 57;
template <int CK, bool HALF, bool PARTIAL, int R, int NR>
__device__ __forceinline__ void gen_p1_narrow(const DevView &V, const LayerDesc &L, uint32_t tile, float *smem)
{
    constexpr int PITCH = 64;
    const int worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t m = (uint32_t)L.cols, n = (uint32_t)L.rows;
    const uint32_t row0 = (tile * 8u + warp) * NR;
    if (row0 >= n)
        return;   // (no CTA-wide barrier below)
    const uint8_t *__restrict__ st = fresh(V.state + worker * V.state_stride);
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off), *__restrict__ Q = fresh(V.qprev + L.msgq_off);
    const float lr = V.lr;
    float *const buf = smem + warp * (NR * PITCH);
    const bool in0 = lane < m, in1 = lane + 32u < m;
    float gv[NR][2];
    uint32_t off[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const uint32_t j = min(row0 + i, n - 1) * m;   // (rows past the end repeat the last one and are not stored)
        off[i] = j & 7u;
        gv[i][0] = in0 ? load_global(g + j + lane) : 0.f;
        gv[i][1] = in1 ? load_global(g + j + lane + 32) : 0.f;
    }
    if (lane < NR * 8) {
        const uint32_t j = min(row0 + (lane >> 3), n - 1) * m;
        const GenWords w = gen_fetch<CK, HALF>(st + L.a_off, st + L.b_off, min((j >> 3) + (lane & 7), ((uint32_t)L.d - 1) >> 3), 28 - __clz(L.unit));
        gen_decode<CK, HALF, PARTIAL>(w, V.omb, buf + 8 * lane, (lane & 4) != 0);
    }
    float q[2][R];
    if (in0)
        factor_row<R>(Q + (size_t)lane * R, R, q[0]);
    if (in1)
        factor_row<R>(Q + (size_t)(lane + 32) * R, R, q[1]);
    __syncwarp();
    float acc[NR][R];
#pragma unroll
    for (int i = 0; i < NR; ++i) {
        const float *const e = buf + i * PITCH + off[i] + lane;
#pragma unroll
        for (int c = 0; c < R; ++c)
            acc[i][c] = 0.f;
#pragma unroll
        for (int u = 0; u < 2; ++u)
            if (u ? in1 : in0) {
                const float p = __fmaf_rn(lr, gv[i][u], e[32 * u]);   // Alg. 2 (4) line 5
#pragma unroll
                for (int c = 0; c < R; ++c)
                    acc[i][c] = __fmaf_rn(p, q[u][c], acc[i][c]);
            }
    }
    __syncwarp();
    gen_p1_store<R, NR>(acc, V.msgp + worker * V.msgp_stride + L.msgp_off, row0, n, R);
}

// A tile of pass 2 (kP2RowsPerTile rows by up to g_p2w columns) by g_p2t threads, a column each, which meet at barrier `bar` and
// go down the rows sixteen at a time: each decodes two code words of the sixteen rows into shared memory, then walks its column.
constexpr int kGenP2Rows = 16;
// (rows are T + (cols & 7) floats apart, so that every element keeps its place within eight)
__host__ __device__ constexpr int gen_p2_floats(int t, int rank) { return 2 * kGenP2Rows * (t + 8 + rank); }
// a row of a factor in shared memory
template <int R>
__device__ __forceinline__ void factor_row_smem(const float *p, float (&out)[R])
{
    if constexpr (R == 4 || R == 8) {
#pragma unroll
        for (int c = 0; c < R; c += 4) {
            const float4 t = *(const float4 *)(p + c);
            out[c] = t.x; out[c + 1] = t.y; out[c + 2] = t.z; out[c + 3] = t.w;
        }
    } else if constexpr (R == 2) {
        const float2 t = *(const float2 *)p;
        out[0] = t.x; out[1] = t.y;
    } else {
        out[0] = p[0];
    }
}
template <int CK, bool HALF, bool PARTIAL, int R, bool PAD = true>   // PAD: with any rank, rows of P_hat on their vectors' boundaries in shared memory
__device__ __forceinline__ void gen_p2_body(const DevView &V, const LayerDesc &L, uint32_t tile, float *smem)
{
    constexpr int RM = gen_most(R), S = kGenP2Rows, KP = (S * RM + 31) / 32;
    const int r = R > 0 ? R : L.rank, worker = blockIdx.y;
    const uint32_t T = (uint32_t)L.g_p2t, lt = 31 - __clz(T);   // threads of a tile
    const uint32_t part_of = threadIdx.x >> lt, tid = threadIdx.x & (T - 1), bar = part_of + 1;
    const uint32_t m = (uint32_t)L.cols, n = (uint32_t)L.rows, wd = (uint32_t)L.g_p2w;
    const uint32_t task = tile * (kGenThreads >> lt) + part_of, ct = (m + wd - 1) / wd, rt = task / ct, c0 = (task - rt * ct) * wd;
    const uint32_t r_lo = rt * (uint32_t)kP2RowsPerTile;
    if (r_lo >= n)
        return;   // (all threads of a tile together)
    const uint32_t have = min(n - r_lo, (uint32_t)kP2RowsPerTile), cols = min(wd, m - c0);
    const uint8_t *__restrict__ st = fresh(V.state + worker * V.state_stride);
    const uint8_t *__restrict__ codes = st + L.a_off, *__restrict__ scales = st + L.b_off;
    const float *__restrict__ ph = fresh(V.phat + L.msgp_off) + (size_t)r_lo * r;
    const int qshift = 28 - __clz(L.unit);
    const uint32_t last = ((uint32_t)L.d - 1) >> 3;
    const float lr = V.lr, omb = V.omb;
    const uint32_t pitch = T + (m & 7u), stage_floats = S * (T + 8);
    float *es = smem + part_of * gen_p2_floats(T, RM), *phs = es + 2 * stage_floats;   // (the stage that is written next)
    int32_t flip = (int32_t)stage_floats, flip_p = S * RM;
    // this thread's words: one of row `dr` of sixteen and one of row dr + 8 (8 m elements are m words on)
    const uint32_t dr = tid >> (lt - 3), dq = tid & ((T >> 3) - 1);
    const bool swap = (tid & 4) != 0;
    uint32_t word = (((r_lo + dr) * m + c0) >> 3) + dq;
    const uint32_t put = (((c0 & 7u) + dr * pitch) & ~7u) + 8 * dq;
    const bool mine = tid < cols;
    const float *gp = fresh(V.grads[worker] + L.g_off) + (size_t)r_lo * m + c0 + (mine ? tid : 0u);
    float acc[RM];
#pragma unroll
    for (int c = 0; c < RM; ++c)
        acc[c] = 0.f;
    GenWords w[2];
    float phn[KP];
    auto fetch = [&](uint32_t a) {   // rows from a on
        w[0] = gen_fetch<CK, HALF>(codes, scales, min(word, last), qshift);
        w[1] = gen_fetch<CK, HALF>(codes, scales, min(word + m, last), qshift);
        word += 2 * m;
#pragma unroll
        for (int x = 0; x < KP; ++x) {
            const uint32_t at = tid + x * T;
            if constexpr (R > 0 || !PAD) {
                if (at < S * r)
                    phn[x] = a * r + at < have * r ? load_global(ph + a * r + at) : 0.f;
            } else {
                const uint32_t row = a + at / RM, c = at % RM;
                if (at < S * RM)
                    phn[x] = row < have && c < r ? load_global(ph + row * r + c) : 0.f;
            }
        }
    };
    fetch(0);
    float gv[S];
#pragma unroll
    for (int u = 0; u < S; ++u) {   // (rows past the end are not used)
        gv[u] = u < have ? load_global(gp) : 0.f;
        gp += m;
    }
    for (uint32_t a = 0; a < have; a += S) {
        gen_decode<CK, HALF, PARTIAL>(w[0], omb, es + put, swap);
        gen_decode<CK, HALF, PARTIAL>(w[1], omb, es + put + 8 * pitch, swap);
#pragma unroll
        for (int x = 0; x < KP; ++x)
            if (tid + x * T < S * (PAD ? RM : r))
                phs[tid + x * T] = phn[x];
        if (a + S < have)
            fetch(a + S);
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(T) : "memory");   // (a stage is written again two barriers on)
        if (mine) {
            const float *ep = es + (c0 & 7u) + tid;
            auto row = [&](int u) {
                const float p = __fmaf_rn(lr, gv[u], *ep);   // Alg. 2 (4) line 5
                ep += pitch;
                float pr[RM];
                if constexpr (R > 0 || PAD) {
                    factor_row_smem<RM>(phs + u * RM, pr);
                } else {
#pragma unroll
                    for (int c = 0; c < RM; ++c)
                        pr[c] = c < r ? phs[u * r + c] : 0.f;
                }
#pragma unroll
                for (int c = 0; c < RM; ++c)
                    acc[c] = __fmaf_rn(p, pr[c], acc[c]);
            };
            if (a + 2 * S <= have) {   // with the next rows' gradient
#pragma unroll
                for (int u = 0; u < S; ++u) {
                    row(u);
                    gv[u] = load_global(gp);
                    gp += m;
                }
            } else if (a + S <= have) {
#pragma unroll
                for (int u = 0; u < S; ++u) {
                    row(u);
                    if (a + S + u < have)
                        gv[u] = load_global(gp);
                    gp += m;
                }
            } else {
#pragma unroll
                for (int u = 0; u < S; ++u)
                    if (a + u < have)
                        row(u);
            }
        }
        es += flip;
        phs += flip_p;
        flip = -flip;
        flip_p = -flip_p;
    }
    if (mine) {
        float *part = V.part + worker * V.part_stride + L.part_off + ((size_t)rt * m + c0 + tid) * r;   // added in order by k_lr_pass2_reduce
#pragma unroll
        for (int c = 0; c < RM; ++c)
            if (R > 0 || c < r)
                part[c] = acc[c];
    }
}

// kP2RowsPerTile rows by kGenCols columns by a whole CTA, for models whose tiles do not fill the SMs: the eight warps form p of 32 rows
// each in shared memory, then a warp per column of the factor adds down the rows, in the order of gen_p2_body.  There a tile waits for memory
// at each of its sixteen stages, however small the model (times: kGenCoop).
constexpr size_t kGenCoopSmem = (size_t)kP2RowsPerTile * (32 + CONEF_MAX_RANK) * 4;
template <int CK, int R>
__device__ __forceinline__ void gen_p2_cta(const DevView &V, const LayerDesc &L, uint32_t tile, float *smem)
{
    constexpr int U = 16;   // rows in flight per warp
    const int r = R > 0 ? R : L.rank, worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
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

inline size_t gen_p2_smem(const LayerDesc &L, int cfg_rank)
{
    if (L.g_p2t == 0)
        return kGenCoopSmem;
    return (size_t)(kGenThreads / L.g_p2t) * gen_p2_floats(L.g_p2t, gen_rank(cfg_rank)) * 4;
}

// Pass 3 takes 32 * E elements per warp at a time.  E consecutive ones are a lane's where codes are decoded and quantised (a block
// is unit / E lanes), between which the residual is formed element by element with neighbouring lanes on neighbouring elements:
// through shared memory.  What is done once per lane and block (scales, addresses, the search for the maximum) is half of all
// instructions at E = 8.
//
// A lane's pieces of 16 bytes are accessed in an order that starts at piece `rot`, so that eight lanes meet all banks; its
// codes are turned accordingly.
constexpr size_t kGenP3Smem = 8 * kGenChunk * 4;
template <int CK, int E>
struct GenTurn {
    static constexpr bool INT4 = CK == CONEF_C_INT4;
    static constexpr int NW = INT4 ? E / 8 : E / 4;   // code words
    uint32_t a, b;   // int4: byte selectors of the words; int8: whether to turn by one and by two words
    // to the order that starts at piece rot, or back from it
    __device__ __forceinline__ GenTurn(int rot)
    {
        if (INT4 && E == 8) {
            a = rot ? 0x1032u : 0x3210u;
            b = 0;
        } else if (INT4) {
            a = rot == 0 ? 0x3210u : rot == 1 ? 0x5432u : rot == 2 ? 0x7654u : 0x1076u;
            b = rot == 0 ? 0x7654u : rot == 1 ? 0x1076u : rot == 2 ? 0x3210u : 0x5432u;
        } else {
            a = rot & 1;
            b = rot & 2;
        }
    }
    __device__ __forceinline__ void turn(const uint32_t (&w)[NW], uint32_t (&o)[NW]) const
    {
        if constexpr (INT4) {
            o[0] = __byte_perm(w[0], w[NW - 1], a);
            if (NW == 2)
                o[NW - 1] = __byte_perm(w[0], w[NW - 1], b);
        } else {
            uint32_t t[NW];
#pragma unroll
            for (int i = 0; i < NW; ++i)
                t[i] = a ? w[(i + 1) % NW] : w[i];
#pragma unroll
            for (int i = 0; i < NW; ++i)
                o[i] = NW == 4 && b ? t[(i + 2) % NW] : t[i];
        }
    }
};
template <int CK, bool HALF, bool PARTIAL, int R, int E>
__device__ __forceinline__ void gen_p3_body(const DevView &V, const LayerDesc &L, uint32_t tile, float *smem)
{
    constexpr int RM = gen_most(R), K = E, NW = GenTurn<CK, E>::NW, CH = 32 * E;
    constexpr bool INT4 = CK == CONEF_C_INT4;
    const int lpb = L.unit / E;   // lanes per quantisation block
    const int r = R > 0 ? R : L.rank, worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t m = (uint32_t)L.cols, n = (uint32_t)L.rows, d = (uint32_t)L.d;
    const uint32_t step = L.g_step, groups = L.g_groups, nc = (d + CH - 1) / CH;
    const uint32_t tt = tile / groups, cpos = (tile - tt * groups) * 8 + warp;   // place among the chunks of a step
    if (cpos >= step)
        return;   // (no CTA-wide barrier below)
    uint8_t *const st = V.state + worker * V.state_stride;
    uint8_t *const codes = st + L.a_off, *const scales = st + L.b_off;
    const float *__restrict__ g = fresh(V.grads[worker] + L.g_off), *__restrict__ ph = fresh(V.phat + L.msgp_off);
    const float *__restrict__ Q = fresh(V.msgq + worker * V.msgq_stride + L.msgq_off);
    const float lr = V.lr, omb = V.omb, beta = V.beta;
    const int bshift = 31 - __clz(L.unit), rot = E == 16 ? (lane >> 1) & 3 : (lane >> 2) & 1;
    const GenTurn<CK, E> to(rot), back((E / 4 - rot) & (E / 4 - 1));
    float *const buf = smem + warp * CH, *const mine = buf + E * lane;
    int at[E / 4];
#pragma unroll
    for (int x = 0; x < E / 4; ++x)
        at[x] = 4 * ((rot + x) & (E / 4 - 1));

    uint32_t ch = tt * (uint32_t)L.g_it * step + cpos;
    if (ch >= nc)
        return;
    // row and column of the chunk's first element, and how they move from step to step
    uint32_t row = (ch * CH) / m, col = ch * CH - row * m;
    const uint32_t drow = (step * CH) / m, dcol = step * CH - drow * m;
    uint32_t w[NW], sw = 0;   // code words and the bits of their scale
#pragma unroll
    for (int x = 0; x < NW; ++x)
        w[x] = 0;
    auto fetch_codes = [&](uint32_t c) {   // (plain loads: this kernel stores to these arrays)
        const uint32_t j = c * CH + E * lane;
        if (j < d) {
            const uint8_t *const at_j = codes + (INT4 ? j >> 1 : j);
            if (NW == 1) {
                w[0] = *(const uint32_t *)at_j;
            } else if (NW == 2) {
                const uint2 t = *(const uint2 *)at_j;
                w[0] = t.x; w[1 % NW] = t.y;
            } else {
                const uint4 t = *(const uint4 *)at_j;
                w[0] = t.x; w[1 % NW] = t.y; w[2 % NW] = t.z; w[3 % NW] = t.w;
            }
            sw = HALF ? (uint32_t)((const unsigned short *)scales)[j >> bshift] : ((const uint32_t *)scales)[j >> bshift];
        }
    };
    float gv[K];
    auto fetch_tail = [&](uint32_t c) {   // the gradient of a chunk that is not full
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const uint32_t j = c * CH + 32 * k + lane;
            gv[k] = j < d ? load_stream_at<0>(g + j) : 0.f;
        }
    };
    fetch_codes(ch);
    if ((ch + 1) * CH <= d) {
        const float *const gj = g + ch * CH + lane;
        static_for<K>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            gv[k] = load_stream_at<128 * k>(gj);
        });
    } else {
        fetch_tail(ch);
    }
    for (int it = 0; it < L.g_it && ch < nc; ++it) {
        {
            uint32_t t[NW];
            to.turn(w, t);
            const ScaleConst<CK> sc = scale_const<CK, HALF>(HALF ? __half2float(__ushort_as_half((unsigned short)sw)) : __uint_as_float(sw));
#pragma unroll
            for (int x = 0; x < E / 8; ++x) {
                float e[8];
                decode8<CK, HALF>(t[INT4 ? x : 2 * x], t[INT4 ? x : (2 * x + 1) % NW], sc, e);
                *(float4 *)(mine + at[2 * x]) = make_float4(e[0], e[1], e[2], e[3]);
                *(float4 *)(mine + at[2 * x + 1]) = make_float4(e[4], e[5], e[6], e[7]);
            }
        }
        const uint32_t nx = ch + step;
        const bool more = it + 1 < L.g_it && nx < nc, more_full = more && (nx + 1) * CH <= d;
        if (more)
            fetch_codes(nx);
        const float *const gj = g + nx * CH + lane;
        __syncwarp();
        // r = p - P_hat Q_i^T; Alg. 4 line 9 stores C(beta e + r)
        auto element = [&](int k, const float (&pr)[RM], const float (&q)[RM]) {
            const float e = buf[32 * k + lane];
            float res = __fmaf_rn(lr, gv[k], PARTIAL ? __fmul_rn(omb, e) : e);   // Alg. 2 (4) line 5
#pragma unroll
            for (int c = 0; c < RM; ++c)
                if (R > 0 || c < r)
                    res = __fmaf_rn(-pr[c], q[c], res);
            if (PARTIAL)
                res = __fmaf_rn(beta, e, res);
            buf[32 * k + lane] = res;
        };
        const bool inside = (ch + 1) * CH <= d;
        if (inside && m - col >= CH) {   // one matrix row
            float pr[RM];
            factor_row<R>(ph + (size_t)row * r, r, pr);
            const float *q0 = Q + (size_t)(col + lane) * r;
            static_for<K>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                float q[RM];
                factor_row<R, 32 * k>(q0, r, q);
                element(k, pr, q);
                load_stream_if<128 * k>(gv[k], gj, more_full);   // the next chunk's
            });
        } else if (inside && m >= CH) {   // two
            float pa[RM], pb[RM];
            factor_row<R>(ph + (size_t)row * r, r, pa);
            factor_row<R>(ph + (size_t)min(row + 1, n - 1) * r, r, pb);
            const int cut = (int)(m - col) - lane;   // elements of the first, from this lane's on
            const float *const qa = Q + (size_t)(col + lane) * r, *const qb = qa - (size_t)m * r;
            static_for<K>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                const bool second = 32 * k >= cut;
                float pr[RM], q[RM];
                factor_row<R, 32 * k>(second ? qb : qa, r, q);
#pragma unroll
                for (int c = 0; c < RM; ++c)
                    pr[c] = second ? pb[c] : pa[c];
                element(k, pr, q);
                load_stream_if<128 * k>(gv[k], gj, more_full);
            });
        } else {
            uint32_t cc = col + lane, rr = row;
            const uint32_t j0 = ch * CH + lane;
            static_for<K>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                if (cc >= m) {
                    const uint32_t t = m >= 32 ? 1u : cc / m;
                    cc -= t * m;
                    rr += t;
                }
                if (j0 + 32 * k < d) {
                    float pr[RM], q[RM];
                    factor_row<R>(ph + (size_t)rr * r, r, pr);
                    factor_row<R>(Q + (size_t)cc * r, r, q);
                    element(k, pr, q);
                } else {
                    buf[32 * k + lane] = 0.f;
                }
                load_stream_if<128 * k>(gv[k], gj, more_full);
                cc += 32;
            });
        }
        if (more && !more_full)
            fetch_tail(nx);
        __syncwarp();
        float res[E / 8][8];
#pragma unroll
        for (int x = 0; x < E / 4; ++x) {
            const float4 t = *(const float4 *)(mine + at[x]);
            res[x >> 1][4 * (x & 1)] = t.x; res[x >> 1][4 * (x & 1) + 1] = t.y; res[x >> 1][4 * (x & 1) + 2] = t.z; res[x >> 1][4 * (x & 1) + 3] = t.w;
        }
        float amax = 0.f;
#pragma unroll
        for (int x = 0; x < E; ++x)
            amax = absmax_nan(amax, res[x >> 3][x & 7]);
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1)
            if (lpb > o)
                amax = absmax_nan(amax, __shfl_xor_sync(0xffffffffu, amax, o));
        float s, inv;
        unsigned short hb = 0;
        block_scale<CK, HALF>(amax, s, inv, hb);
        uint32_t t[E / 4], o[NW];   // (int4: every other word)
        if (__any_sync(0xffffffffu, !(__fmul_rn(amax, inv) < (INT4 ? 7.f : 127.f) + 0.49f))) {   // (see quant_pack8)
            amax = 0.f;
#pragma unroll
            for (int x = 0; x < E; ++x)
                amax = fmaxf(amax, fabsf(res[x >> 3][x & 7]));   // (a NaN counts as nothing)
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1)
                if (lpb > o)
                    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            block_scale<CK, HALF>(amax, s, inv, hb);
#pragma unroll
            for (int x = 0; x < E / 8; ++x)
                quant_pack8<CK, true>(res[x], inv, t[2 * x], t[2 * x + 1]);
        } else {
#pragma unroll
            for (int x = 0; x < E / 8; ++x)
                quant_pack8<CK, false>(res[x], inv, t[2 * x], t[2 * x + 1]);
        }
        const uint32_t j = ch * CH + E * lane;
        uint32_t c[NW];
#pragma unroll
        for (int x = 0; x < NW; ++x)
            c[x] = t[INT4 ? 2 * x : x];
        back.turn(c, o);
        if (j < d) {
            uint8_t *const at_j = codes + (INT4 ? j >> 1 : j);
            if (NW == 1)
                *(uint32_t *)at_j = o[0];
            else if (NW == 2)
                *(uint2 *)at_j = make_uint2(o[0], o[1 % NW]);
            else
                *(uint4 *)at_j = make_uint4(o[0], o[1 % NW], o[2 % NW], o[3 % NW]);
            if ((lane & (lpb - 1)) == 0) {
                if (HALF)
                    ((unsigned short *)scales)[j >> bshift] = hb;
                else
                    ((float *)scales)[j >> bshift] = s;
            }
        }
        __syncwarp();
        ch = nx;
        row += drow;
        col += dcol;
        if (col >= m) {
            col -= m;
            ++row;
        }
    }
}

// R: the configured rank, or the next of 1, 2, 4 and 8 above it (gen_rank).  Tensors of another rank than R, and those behind them whose
// factors are off the vector loads' alignment, take the body for any rank up to R.  That was one for any rank up to 8 with a row per warp in pass
// 1; steps of the recurrent layers of odd widths, before and now: rank 3 608 and 407 us (int8), 596 and 383 (int4), rank 5 641 and 527, rank 7 681 and
// 551, behind a matrix of one row rank 4, int8, 711 and 444, rank 2, int4, 557 and 338.  As a function that is not inlined
// it takes no registers from the body with the rank as a constant, but both were slower: rank 3 439, rank 7 651, rank 8 511 instead of 496.
// R < 0: of models with such tensors (rank -R); R > 0: of those without, whose kernels have the one body alone (rank 2, int8 296 us
// with both and 288 with one, rank 8, int4 501 and 473).  BOTH:
// rank 8 on int8 alone compiles to slower code in its own kernel, though it spills less (4001 x 6003, four workers, fp16 scales: pass 1 286 instead of 260 us,
// pass 2 174 instead of 141; steps 883 and 831), so that it keeps the other body beside it, a row per warp and P_hat's rows as they come.
template <int PASS, int CK, bool HALF, bool PARTIAL, int R>
__device__ __forceinline__ void gen_tile(const DevView &V, const LayerDesc &L, uint32_t tile, float *smem)
{
    constexpr int K = gen_most(R);
    constexpr bool BOTH = CK == CONEF_C_INT8 && R == 8;
    const bool exact = (R > 0 && !BOTH) || gen_exact(L, K);
    if constexpr (BOTH && PASS != 3) {
        if (!exact) {
            if constexpr (PASS == 1) {
                for (int x = 0; x < L.g_nr; ++x)
                    gen_p1_body<CK, HALF, PARTIAL, -K, 1>(V, L, tile * (uint32_t)L.g_nr + x, smem);
            } else if (L.g_p2t == 0) {
                gen_p2_cta<CK, -K>(V, L, tile, smem);
            } else {
                gen_p2_body<CK, HALF, PARTIAL, -K, false>(V, L, tile, smem);
            }
            return;
        }
    }
    if constexpr (PASS == 1) {
        if (exact) {
            if (L.g_nr > 1 && L.cols <= kGenNarrow)
                gen_p1_narrow<CK, HALF, PARTIAL, K, gen_p1_rows(K)>(V, L, tile, smem);
            else if (L.g_nr > 1)
                gen_p1_body<CK, HALF, PARTIAL, K, gen_p1_rows(K)>(V, L, tile, smem);
            else
                gen_p1_body<CK, HALF, PARTIAL, K, 1>(V, L, tile, smem);
            return;
        }
        if (L.g_nr > 1)
            gen_p1_body<CK, HALF, PARTIAL, R, gen_p1_rows(K)>(V, L, tile, smem);
        else
            gen_p1_body<CK, HALF, PARTIAL, R, 1>(V, L, tile, smem);
    } else if constexpr (PASS == 2) {
        if (L.g_p2t == 0) {
            if (exact)
                gen_p2_cta<CK, K>(V, L, tile, smem);
            else
                gen_p2_cta<CK, R>(V, L, tile, smem);
        } else if (exact) {
            gen_p2_body<CK, HALF, PARTIAL, K>(V, L, tile, smem);
        } else {
            gen_p2_body<CK, HALF, PARTIAL, R>(V, L, tile, smem);
        }
    } else {
        if (!exact)
            gen_p3_body<CK, HALF, PARTIAL, -K, 8>(V, L, tile, smem);
        else if (L.g_chunk == kGenChunk)
            gen_p3_body<CK, HALF, PARTIAL, K, 16>(V, L, tile, smem);
        else
            gen_p3_body<CK, HALF, PARTIAL, K, 8>(V, L, tile, smem);
    }
}

// CTAs per SM that the registers have to allow for.  Pass 3 on int8 with four and with three of them, steps on the recurrent layers of odd widths (28.4 M
// elements, two workers): rank 1 292 and 289 us, 2 302 and 297, 3 489 and 456, 4 350 and 343 (104 and 16 bytes spilled); rank 8 with
// three and two 493 and 497.
__host__ __device__ constexpr int gen_ctas(int pass, int ckind, int rank)
{
    if (pass == 2)
        return 3;
    if (pass == 1)
        return rank == 8 ? 3 : 4;
    return rank == 8 ? 2 + (ckind == CONEF_C_INT8) : 3;
}
template <int PASS, int CK, bool HALF, bool PARTIAL, int R>
__global__ void __launch_bounds__(kGenThreads, gen_ctas(PASS, CK, gen_most(R))) k_gen_pass(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
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
    gen_tile<PASS, CK, HALF, PARTIAL, R>(V, L, tile, gen_smem);
}

// launcher (conef_lrgen.cu, the variants by codec in two more files); exact: every tensor is gen_exact; smem2: the most that a tensor's CTAs of pass 2 need
cudaError_t gen_launch(int pass, int ckind, int rank, bool exact, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, size_t smem2);

template <int CK>
cudaError_t gen_launch_codec(int pass, int rank, bool exact, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s, size_t smem2);
extern template cudaError_t gen_launch_codec<CONEF_C_INT8>(int, int, bool, const DevView &, const int32_t *, int, cudaStream_t, size_t);
extern template cudaError_t gen_launch_codec<CONEF_C_INT4>(int, int, bool, const DevView &, const int32_t *, int, cudaStream_t, size_t);

}  // namespace conef
