// P-reduce + orthonormalisation of P_bar on a thread-block cluster.
//
// One cluster per compressed tensor: CTA k of the cluster keeps rows
// [k * rows_per_cta, ...) of P_bar in registers (up to 8 rows per thread), so
// nothing goes back to memory between the sum over workers and P_hat.
// P_hat is the orthonormal factor of the QR factorisation with a positive
// diagonal, the one left-to-right (modified) Gram-Schmidt produces.  It is
// computed through the Gram matrix: G = P_bar^T P_bar needs ONE reduction
// over the tensor (fp64 across threads: per warp by shuffles, per CTA through
// shared memory, across the cluster by reading the other CTAs' shared memory
// in rank order, so the result does not depend on scheduling), its Cholesky
// factor L is formed in fp64 by one warp, a row per lane, and every row solves
// P_hat L^T = P_bar in fp64.  Against Gram-Schmidt column by column (r
// reductions) the GPT-2-small list went from 0.20 to 0.06 ms and P_hat agrees
// with the oracle's Gram-Schmidt to 4e-6 (relative Frobenius).
//
// Bound by latency: trips to L2 and to the other CTAs, the chain of square roots and divisions, and the shuffles of the Gram
// matrix.  With every value's own butterfly, rounds without a row, one thread's Cholesky and a trip per worker for the few
// rows of a thread, rank 8 took 39 and 40 us on the GPT-2-small list (28 and 36 now); steps of small models at rank 8: 512 x 768 and
// 768 x 512, int4, four workers 77 -> 65 us, 501 x 333 and 77 x 999, int8 56 -> 46.  Rank 4 as before (ten values instead of 36).
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <float.h>

#include <utility>

#include "conef_internal.h"
#include "conef_kernels.cuh"

namespace conef {

namespace cg = cooperative_groups;

constexpr int kGsThreads = 512;
// rows per thread: 8 rows of rank up to 8 fit the 128 registers a 512-thread CTA may use
__host__ __device__ constexpr int gs_rows(int R) { return R <= 8 ? 8 : 4; }
__host__ __device__ constexpr int gs_rows_per_cta(int R) { return kGsThreads * gs_rows(R); }

// Sums over a warp's lanes of NV doubles per lane (a power of two), each to dst[base + its place]: halves are exchanged, so that every
// value is added along the tree of a butterfly (the order does not depend on NV).
template <int NV>
__device__ __forceinline__ void gs_reduce(double (&t)[NV], int lane, double *dst)
{
    int n = NV, idx = 0, plain = 32;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
        if (n > 1) {
            n >>= 1;
            const bool up = (lane & o) != 0;
#pragma unroll
            for (int i = 0; i < NV / 2; ++i)
                if (i < n) {
                    const double send = up ? t[i] : t[i + n], keep = up ? t[i + n] : t[i];
                    t[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
                }
            idx += up ? n : 0;
            plain = o;
        } else {
            t[0] += __shfl_xor_sync(0xffffffffu, t[0], o);
        }
    }
    if ((lane & (plain - 1)) == 0)
        dst[idx] = t[0];
}
// entries [E0, E0 + NV) of the Gram matrix of a warp's rows: entry j (j + 1) / 2 + c is the sum of v[.][c] v[.][j]
template <int R, int ROWS, int E0, int NV>
__device__ __forceinline__ void gs_gram(const float (&v)[ROWS][R], int rounds, int lane, double *warp_g)
{
    double t[NV];
#pragma unroll
    for (int x = 0; x < NV; ++x)
        t[x] = 0.0;
#pragma unroll
    for (int k = 0; k < ROWS; ++k)
        if (k < rounds) {
#pragma unroll
            for (int j = 0; j < R; ++j)
#pragma unroll
                for (int c = 0; c <= j; ++c)
                    if (j * (j + 1) / 2 + c >= E0 && j * (j + 1) / 2 + c < E0 + NV)   // products of two floats are exact in fp64
                        t[j * (j + 1) / 2 + c - E0] = fma((double)v[k][c], (double)v[k][j], t[j * (j + 1) / 2 + c - E0]);
        }
    gs_reduce<NV>(t, lane, warp_g + E0);
}

template <int R>
__global__ void __launch_bounds__(kGsThreads, 1)
k_gs_cluster(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx, float *__restrict__ out_sum)
{
    constexpr int kGsRows = gs_rows(R);
    cg::cluster_group cluster = cg::this_cluster();
    const unsigned csize = cluster.num_blocks();
    const unsigned crank = cluster.block_rank();
    grid_release();
    const int tile = blockIdx.x / csize;         // one cluster per tensor of this launch
    const int li = find_layer(pfx, V.n_layers, tile);
    const LayerDesc *Lp = V.layers + li;
    const int64_t n = Lp->rows;
    const int r = Lp->rank;                      // r <= R
    const int64_t off = Lp->msgp_off;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t rows_per_cta = (n + csize - 1) / csize;
    const int64_t row_lo = crank * rows_per_cta;
    const int64_t row_hi = min(n, row_lo + rows_per_cta);
    // rounds of kGsThreads rows in which this warp has any
    const int64_t mine = row_hi - row_lo - warp * 32;
    const int rounds = mine <= 0 ? 0 : (int)min((int64_t)kGsRows, (mine + kGsThreads - 1) / kGsThreads);

    grid_wait();
    // P_bar = ((P_0 + P_1) + P_2) + ... in worker order.  All of a worker's values are loaded
    // before any is used and nothing is stored until the sum is complete, so that the loads of a
    // round are in flight together (one round trip to L2 per worker instead of one per value).
    float v[kGsRows][R];
#pragma unroll
    for (int k = 0; k < kGsRows; ++k)
#pragma unroll
        for (int c = 0; c < R; ++c)
            v[k][c] = 0.f;
    constexpr int KB = R > 4 ? 2 : 8;   // rows loaded per round (registers)
    const bool whole = r == R && (off & 3) == 0 && (V.msgp_stride & 3) == 0;
    if (rounds <= 1) {   // (one row per thread at most: of four workers together)
        const int64_t a = row_lo + tid;
        for (int i = 0; rounds == 1 && i < V.n_workers; i += 4) {
            float x[4][R];
#pragma unroll
            for (int y = 0; y < 4; ++y) {
                const bool in = i + y < V.n_workers && a < row_hi;
                const float *__restrict__ src = fresh(V.msgp + (int64_t)(in ? i + y : 0) * V.msgp_stride + off);
                if (whole) {
#pragma unroll
                    for (int c = 0; c < R; c += 4) {
                        const float4 t = in ? load_global((const float4 *)(src + a * R + c)) : make_float4(0.f, 0.f, 0.f, 0.f);
                        x[y][c] = t.x; x[y][c + 1] = t.y; x[y][c + 2] = t.z; x[y][c + 3] = t.w;
                    }
                } else {
#pragma unroll
                    for (int c = 0; c < R; ++c)
                        x[y][c] = in && c < r ? load_global(src + a * r + c) : 0.f;
                }
            }
#pragma unroll
            for (int y = 0; y < 4; ++y)
                if (i + y < V.n_workers) {
#pragma unroll
                    for (int c = 0; c < R; ++c)
                        v[0][c] = i + y == 0 ? x[y][c] : __fadd_rn(v[0][c], x[y][c]);
                }
        }
    } else
    for (int i = 0; i < V.n_workers; ++i) {
        const float *__restrict__ src = fresh(V.msgp + i * V.msgp_stride + off);
#pragma unroll
        for (int k0 = 0; k0 < kGsRows; k0 += KB) {
            float x[KB][R];
            if (whole) {
                // full rank: a row is R contiguous, 16-byte aligned floats
#pragma unroll
                for (int k = 0; k < KB; ++k) {
                    const int64_t a = row_lo + (int64_t)(k0 + k) * kGsThreads + tid;
#pragma unroll
                    for (int c = 0; c < R; c += 4) {
                        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (a < row_hi)
                            t = load_global((const float4 *)(src + a * R + c));
                        x[k][c] = t.x; x[k][c + 1] = t.y; x[k][c + 2] = t.z; x[k][c + 3] = t.w;
                    }
                }
            } else {
#pragma unroll
                for (int k = 0; k < KB; ++k) {
                    const int64_t a = row_lo + (int64_t)(k0 + k) * kGsThreads + tid;
#pragma unroll
                    for (int c = 0; c < R; ++c)
                        x[k][c] = (a < row_hi && c < r) ? load_global(src + a * r + c) : 0.f;
                }
            }
#pragma unroll
            for (int k = 0; k < KB; ++k)
#pragma unroll
                for (int c = 0; c < R; ++c)
                    v[k0 + k][c] = i == 0 ? x[k][c] : __fadd_rn(v[k0 + k][c], x[k][c]);
        }
    }
    const bool vec = r == R && (off & 3) == 0;
#pragma unroll
    for (int k = 0; k < kGsRows; ++k) {
        const int64_t a = row_lo + (int64_t)k * kGsThreads + tid;
        if (a < row_hi) {
            if (vec) {
#pragma unroll
                for (int c = 0; c < R; c += 4) {
                    const float4 t = make_float4(v[k][c], v[k][c + 1], v[k][c + 2], v[k][c + 3]);
                    *(float4 *)(V.pbar + off + a * R + c) = t;
                    if (out_sum) {
                        if (((uintptr_t)out_sum & 15) == 0)
                            *(float4 *)(out_sum + off + a * R + c) = t;
                        else {
                            out_sum[off + a * R + c] = t.x; out_sum[off + a * R + c + 1] = t.y;
                            out_sum[off + a * R + c + 2] = t.z; out_sum[off + a * R + c + 3] = t.w;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int c = 0; c < R; ++c)
                    if (c < r) {
                        V.pbar[off + a * r + c] = v[k][c];
                        if (out_sum)
                            out_sum[off + a * r + c] = v[k][c];
                    }
            }
        }
    }

    // The orthonormal factor through the Gram matrix: P_bar = P_hat L^T with L the Cholesky factor of
    // G = P_bar^T P_bar, which is the same P_hat as left-to-right Gram-Schmidt gives (both are the
    // QR factorisation with a positive diagonal), but needs ONE reduction over the tensor instead of
    // one per column.  G is accumulated in fp64 throughout (Cholesky-QR squares the condition
    // number: fp32 partial sums lost a 4 x 4 P_bar of condition 2e3), factored in fp64 by one
    // warp, and every row is solved in fp64.  A column whose
    // pivot is not >= FLT_MIN as a float is dead: it becomes zero and takes no part afterwards.
    constexpr int NG = R * (R + 1) / 2;          // entries (j, c), c <= j, at j (j + 1) / 2 + c
    __shared__ double warp_g[kGsThreads / 32][NG];
    __shared__ double cta_g[NG];
    __shared__ double Ls[NG];
    __shared__ double invd[R];
    static_assert(R == 4 || R == 8, "the entries in groups of powers of two");
    if (R == 4) {
        gs_gram<R, kGsRows, 0, 8>(v, rounds, lane, warp_g[warp]);
        gs_gram<R, kGsRows, 8, 2>(v, rounds, lane, warp_g[warp]);
    } else {
        gs_gram<R, kGsRows, 0, 16>(v, rounds, lane, warp_g[warp]);
        gs_gram<R, kGsRows, 16, 16>(v, rounds, lane, warp_g[warp]);
        gs_gram<R, kGsRows, 32, 4>(v, rounds, lane, warp_g[warp]);
    }
    __syncthreads();
    if (tid < NG) {
        double t = 0.0;
#pragma unroll
        for (int w = 0; w < kGsThreads / 32; ++w)
            t += warp_g[w][tid];
        cta_g[tid] = t;
    }
    cluster.sync();   // every CTA's partial Gram matrix is in its shared memory
    if (tid < NG) {
        double t = 0.0;
        for (unsigned k0 = 0; k0 < csize; k0 += 8) {   // rank order; the loads of eight CTAs' in flight together
            double x[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
                x[k] = k0 + k < csize ? *cluster.map_shared_rank(&cta_g[tid], k0 + k) : 0.0;
#pragma unroll
            for (int k = 0; k < 8; ++k)
                t = k0 + k < csize ? t + x[k] : t;
        }
        Ls[tid] = t;
    }
    auto left = cluster.barrier_arrive();   // this CTA reads no other's shared memory any more
    __syncthreads();
    if (warp == 0) {   // lane j: row j of L
        double row[R];
#pragma unroll
        for (int c = 0; c < R; ++c)
            row[c] = c <= lane && lane < R ? Ls[lane * (lane + 1) / 2 + c] : 0.0;
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const double sd = sqrt(__shfl_sync(0xffffffffu, row[k], k));
            const bool dead = !((float)sd >= FLT_MIN);   // also a negative or NaN pivot
            const double inv = dead ? 0.0 : 1.0 / sd;
            row[k] = dead ? 0.0 : lane == k ? sd : row[k] * inv;
            if (lane == k)
                invd[k] = inv;
#pragma unroll
            for (int c = k + 1; c < R; ++c)
                row[c] -= row[k] * __shfl_sync(0xffffffffu, row[k], c);
        }
        if (lane < R) {
#pragma unroll
            for (int c = 0; c < R; ++c)
                if (c <= lane)
                    Ls[lane * (lane + 1) / 2 + c] = row[c];
        }
    }
    __syncthreads();
    // P_hat[a][c] = (P_bar[a][c] - sum_{k<c} L[c][k] P_hat[a][k]) / L[c][c]
#pragma unroll
    for (int k = 0; k < kGsRows; ++k)
        if (k < rounds) {
            double x[R];
#pragma unroll
            for (int c = 0; c < R; ++c) {
                double t = (double)v[k][c];
#pragma unroll
                for (int kk = 0; kk < c; ++kk)
                    t -= Ls[c * (c + 1) / 2 + kk] * x[kk];
                x[c] = t * invd[c];
                v[k][c] = (float)x[c];
            }
        }
#pragma unroll
    for (int k = 0; k < kGsRows; ++k) {
        const int64_t a = row_lo + (int64_t)k * kGsThreads + tid;
        if (a < row_hi) {
            if (vec) {
#pragma unroll
                for (int c = 0; c < R; c += 4)
                    *(float4 *)(V.phat + off + a * R + c) = make_float4(v[k][c], v[k][c + 1], v[k][c + 2], v[k][c + 3]);
            } else {
#pragma unroll
                for (int c = 0; c < R; ++c)
                    if (c < r)
                        V.phat[off + a * r + c] = v[k][c];
            }
        }
    }
    cluster.barrier_wait(std::move(left));   // no CTA leaves while its shared memory may still be read
}

// Launch over `tiles` tensors (prefix table pfx) with the given cluster size.
template <int R>
inline cudaError_t gs_launch(const DevView &V, const int32_t *pfx, int tiles, int cluster_size, float *out_sum,
                             cudaStream_t s)
{
    if (tiles <= 0)
        return cudaSuccess;
    static bool allowed[64] = {};
    return launch_cluster(k_gs_cluster<R>, tiles, cluster_size, kGsThreads, s, allowed, V, pfx, out_sum);
}

}  // namespace conef
