// The selection kernels of a context (method and measurements: conef_select.cuh).
#pragma once
#include "conef_select.cuh"

namespace conef {

// select_finish for a tensor of at most kSelTailTiles tiles, word offsets included: its bitmap is
// completed in shared memory (16 words per thread), so that nothing but the list and the bitmap
// itself is waited for
__device__ __forceinline__ uint32_t select_finish_short(SelectSharedTiles &S, const SelectWindow &W, const uint2 *list, uint32_t nlist,
                                                        uint32_t *bits, uint32_t *tileoff, uint16_t *wordoff, uint32_t ntiles)
{
    constexpr int PER = kSelTailWords / kSelThreads;   // a tile is 16 threads' words
    static_assert(PER == 16, "half a warp per tile");
    const int tid = threadIdx.x, lane = tid & 31;
    const uint32_t w0 = tid * PER;
    const bool mine = w0 < ntiles * (kHistTile / 32);
    uint32_t below = 0;
    if (mine) {
#pragma unroll
        for (int x = 0; x < PER; x += 8) {
            uint32_t v[8];
            load_cg(bits + w0 + x, v);
#pragma unroll
            for (int y = 0; y < 8; ++y) {
                S.words[w0 + x + y] = v[y];
                below += __popc(v[y]);
            }
        }
    }
    const auto get = [list](uint32_t x) { return load_cg(&list[x]); };
    if (select_threshold(S, W, get, nlist, below) == 0xFFFFFFFFu)
        return 0xFFFFFFFFu;
    select_listed(S, W, get, nlist, [&](uint32_t j) { atomicOr(&S.words[j >> 5], 1u << (j & 31u)); });
    __syncthreads();
    uint32_t word[PER], cnt = 0, total;
#pragma unroll
    for (int x = 0; x < PER; ++x) {
        word[x] = mine ? S.words[w0 + x] : 0u;
        cnt += __popc(word[x]);
    }
    uint32_t run = block_exclusive(cnt, S.wsum, total);
    const uint32_t start = __shfl_sync(0xffffffffu, run, lane & 16);   // of this thread's tile
    if (mine) {
        if ((tid & 15) == 0)
            tileoff[tid >> 4] = run;
        run -= start;
#pragma unroll
        for (int x = 0; x < PER; x += 8) {
            uint32_t pair[4];
#pragma unroll
            for (int y = 0; y < 8; ++y) {
                pair[y / 2] = y % 2 ? pair[y / 2] | (run << 16) : run;
                run += __popc(word[x + y]);
            }
            *(uint4 *)(wordoff + w0 + x) = make_uint4(pair[0], pair[1], pair[2], pair[3]);
            *(uint4 *)(bits + w0 + x) = make_uint4(word[x], word[x + 1], word[x + 2], word[x + 3]);
            *(uint4 *)(bits + w0 + x + 4) = make_uint4(word[x + 4], word[x + 5], word[x + 6], word[x + 7]);
        }
    }
    return total;
}

// One CTA hashes V.sel_tiles tiles of 8192 elements (1, 2, 4 or 8: several on large models, where the
// search for the tensor, the fence and the ticket would otherwise take as long as the hashing; 210 M
// elements 308 -> 240 us); a warp hashes a run of 1024 elements per tile, 32 (one bitmap word) per lane
// at a time.
__global__ void __launch_bounds__(kSelThreads, 5) k_rk_select(const __grid_constant__ DevView V)
{
    __shared__ SelectSharedTiles S;
    __shared__ uint32_t s_n, s_base, s_cnt[8], s_last, s_listed;
    grid_release();
    const int li = find_layer(V.pfx_hist, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    const uint32_t d = (uint32_t)L.d, lo = L.sel_lo, hi = L.sel_hi, T = (uint32_t)V.sel_tiles;
    const uint32_t tile0 = (blockIdx.x - V.pfx_hist[li]) * T, ncta = (uint32_t)(V.pfx_hist[li + 1] - V.pfx_hist[li]);
    const uint32_t ntiles = (uint32_t)((L.d + kHistTile - 1) / kHistTile);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t st = stream_key(V.seed_q, (uint64_t)li, (uint64_t)V.step);
    uint32_t *ctr = V.sel + L.sel_off;   // listed elements and finished CTAs: zero between selections
    uint2 *list = (uint2 *)V.cand + L.cand_off;
    uint32_t *bits = V.selbits + L.selbits_off;
    uint32_t *tileoff = V.tileoff + L.tileoff_off;
    uint16_t *wordoff = V.wordoff + L.wordoff_off;
    const bool windowed = d > (uint32_t)kSelShortTensor;
    const uint32_t cap = V.sel_how == CONEF_SELECT_FULL ? 1u : L.cand_cap;

    S.hist[tid] = 0;   // the bins of select_threshold
    if (tid < 8)
        s_cnt[tid] = 0;
    if (tid == 0)
        s_n = 0;
    __syncthreads();
    if (windowed) {
        const uint32_t w0 = tile0 * (kHistTile / 32) + warp * T * 32u + lane;   // this lane's first bitmap word
        uint32_t cnt = 0;
        for (uint32_t i = 0; i < T; ++i) {
            const uint32_t w = w0 + i * 32u;
            if (w * 32ull >= d)
                break;
            const uint32_t j0 = w * 32u;
            uint32_t inside;
            const uint32_t word = select_word(st, j0, d, lo, hi, inside);
            for (uint32_t m = inside; m; m &= m - 1) {   // the few inside the window
                const uint32_t j = j0 + (uint32_t)__ffs(m) - 1u;
                const uint2 e = make_uint2(hash32(st, j), V.sel_how == CONEF_SELECT_STALE ? 0xFFFFFFFFu : j);
                const uint32_t pos = atomicAdd(&s_n, 1u);
                if (pos < (uint32_t)kSelList) {
                    ((uint2 *)S.keys)[pos] = e;
                } else {   // (not expected: the list of a CTA holds several times the usual number)
                    grid_wait();
                    const uint32_t g = select_claim(ctr, 1u);
                    if (g < cap)
                        list[g] = e;
                }
            }
            if (i == 0)
                grid_wait();   // (the first tile is hashed while the kernel ahead ends)
            bits[w] = word;
            cnt += __popc(word);
        }
        grid_wait();
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if (lane == 0 && cnt)
            atomicAdd(&s_cnt[(warp * T) >> 3], cnt);   // a warp's words lie in one tile
        __syncthreads();
        const uint32_t n = min(s_n, (uint32_t)kSelList);
        if (tid == 0)
            s_base = n ? select_claim(ctr, n) : 0u;
        if (tid < T && tile0 + tid < ntiles)
            tileoff[tile0 + tid] = s_cnt[tid];
        __syncthreads();
        for (uint32_t x = tid; x < n; x += kSelThreads)
            if (s_base + x < cap)
                list[s_base + x] = ((uint2 *)S.keys)[x];
    } else {
        grid_wait();
    }
    __threadfence();
    __syncthreads();
    if (tid == 0)
        s_last = select_ticket(ctr, ncta, s_listed);   // (one thread's answer: the barriers below depend on it)
    __syncthreads();
    if (!s_last)
        return;

    // ---- the CTA that finishes the tensor
    const uint32_t k = (uint32_t)L.k, nlist = s_listed;
    const SelectWindow W{lo, hi, d, k, L.sel_scale, V.status};
    uint32_t total = 0xFFFFFFFFu;
    if (windowed && nlist <= cap && V.sel_how != CONEF_SELECT_MISS)
        total = ntiles <= (uint32_t)kSelTailTiles
                    ? select_finish_short(S, W, list, nlist, bits, tileoff, wordoff, ntiles)
                    : select_finish<kHistTile>(S, W, list, nlist, tileoff, ntiles,
                                               [&](uint32_t j) { atomicOr(&bits[j >> 5], 1u << (j & 31u)); });
    if (total == 0xFFFFFFFFu) {
        __syncthreads();
        select_exact(S, st, d, k);
        if (S.bad && tid == 0) {
            atomicOr(V.status, ST_SELECT_FAILED);
            S.tau = 0;
        }
        __syncthreads();
        const uint64_t tau = S.tau;
        for (uint32_t t = 0; t < ntiles; ++t) {
            if (tid == 0)
                s_cnt[0] = 0;
            __syncthreads();
            const uint64_t j0 = (uint64_t)t * kHistTile + tid * 32u;
            uint32_t word = 0;
            for (uint32_t q = 0; q < 32 && j0 + q < d; ++q)
                if ((((uint64_t)hash32(st, j0 + q) << 32) | (j0 + q)) <= tau)
                    word |= 1u << q;
            if (j0 < d)
                bits[j0 >> 5] = word;
            const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(word));
            if (lane == 0 && c)
                atomicAdd(&s_cnt[0], c);
            __syncthreads();
            if (tid == 0)
                tileoff[t] = s_cnt[0];
        }
        __threadfence();
        __syncthreads();
        total = scan_counts(tileoff, ntiles, S.wsum);
        if (ntiles <= (uint32_t)kSelTailTiles)
            for (uint32_t t = warp; t < ntiles; t += kSelThreads / 32)
                select_offsets(bits, wordoff, t);
    }
    if (tid == 0) {
        if (total != k)
            atomicOr(V.status, ST_COUNT_MISMATCH);
        ctr[0] = ctr[1] = 0;
    }
}

// The same for models all of whose tensors have at most kSelClusterTiles tiles: a cluster per tensor, no counters,
// one pass.
static __global__ void __launch_bounds__(kSelThreads) k_rk_select_cluster(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
    __shared__ SelectCluster S;
    grid_release();
    const uint32_t csize = cooperative_groups::this_cluster().num_blocks(), rank = cooperative_groups::this_cluster().block_rank();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x / csize);
    const LayerDesc &L = V.layers[li];
    const uint32_t d = (uint32_t)L.d, k = (uint32_t)L.k;
    const uint64_t st = stream_key(V.seed_q, (uint64_t)li, (uint64_t)V.step);
    const SelectResult R = select_in_cluster(S, st, d, k, L.sel_lo, L.sel_hi, L.sel_scale, V.sel_how);
    grid_wait();
    if (rank == 0 && threadIdx.x == 0) {
        if (R.failed)
            atomicOr(V.status, ST_SELECT_FAILED);
        if (R.total != k)
            atomicOr(V.status, ST_COUNT_MISMATCH);
    }
    if (rank * (uint32_t)kHistTile >= d)
        return;
    uint32_t all;
    const uint32_t before = block_exclusive(__popc(R.word), S.wsum, all), w = rank * (kHistTile / 32) + threadIdx.x;
    V.selbits[L.selbits_off + w] = R.word;   // (the arrays cover whole tiles; words past the tensor are zero)
    V.wordoff[L.wordoff_off + w] = (uint16_t)before;
    if (threadIdx.x == 0)
        V.tileoff[L.tileoff_off + rank] = R.first;
}

// word offsets of the tensors with more than kSelTailTiles tiles: a warp per tile
__global__ void __launch_bounds__(kSelThreads) k_rk_offsets(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
    grid_release();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    grid_wait();
    const uint32_t tile = (blockIdx.x - pfx[li]) * (kSelThreads / 32) + (threadIdx.x >> 5);
    if ((int64_t)tile * kHistTile < L.d)
        select_offsets(V.selbits + L.selbits_off, V.wordoff + L.wordoff_off, tile);
}

}  // namespace conef
