// Random-k selection (S3a): the shared index set S_t = the k smallest keys (hash32(j) << 32 | j) of a
// tensor, which depends on (seed, tensor, step) only.
//
// Every element is hashed ONCE.  The k-th smallest of d uniform hashes lies within a few standard
// deviations, sqrt(k (1 - k/d)) ranks, of rank k, so the window [lo, hi] of hash values that holds it
// is known before anything is hashed (select_window; six deviations and a margin: missed with
// probability below 1e-8 per tensor and step).  The hashing pass marks the elements below the window
// in a bitmap and lists the few inside it (about 12 sqrt(k)); the CTA that finishes a tensor last
// picks the exact threshold key among those, marks the members of the list, and turns the tiles' counts
// into message offsets.  Where the window missed, and for tensors so short that it would hold most
// of the tensor, that CTA finds the threshold by a radix select that hashes the tensor again.
//
// Consumers read the bitmap (bit i of word w: element 32 w + i is a member) and
//   slot(j) = tileoff[j / 8192] + wordoff[j / 32] + members of j's word below j.
//
// Bound by the integer pipe, no memory traffic to speak of.  Transformer-big list (210 M elements): a three-level radix
// select that hashed everything three times took 1.26 ms in ten launches; this takes 0.2 ms in two.
#pragma once
#include <cooperative_groups.h>

#include "conef_common.cuh"

namespace conef {

constexpr int kSelThreads = 256;
constexpr int kSelBins = 2048;
constexpr int kSelShortTensor = 1024;   // up to here the window is not used
constexpr int kSelTailTiles = 16;       // tensors of at most this many tiles: the last CTA also writes the offsets
constexpr int kSelList = 2304;          // window entries a CTA holds in shared memory (a tensor of kSelTailTiles expects 2204 at most)
constexpr int kSelTiles = 1280;         // tile counts it holds there
constexpr int kSelTailWords = kSelTailTiles * kHistTile / 32;

// shared memory of the CTA that finds a tensor's threshold
struct SelectShared {
    uint32_t hist[kSelBins];
    uint64_t keys[kSelList];
    uint32_t wsum[kSelThreads / 32], wsum2[kSelThreads / 32];
    uint64_t tau;
    uint32_t bin, rem, n, bad;
};
// ... and of the CTA that finishes a tensor
struct SelectSharedTiles : SelectShared {
    union {
        uint32_t tiles[kSelTiles];
        uint32_t words[kSelTailWords];
    };
};

// A tensor's counters, one 64-bit word: listed elements in the low half, CTAs that have finished in the high
// half.  A CTA's ticket thus also tells how many elements were listed before it.
using SelectCtr = unsigned long long;
__device__ __forceinline__ uint32_t select_claim(uint32_t *ctr, uint32_t n) { return (uint32_t)atomicAdd((SelectCtr *)ctr, (SelectCtr)n); }
// thread 0 only; whether this CTA is the last of ncta, and the elements listed by all of them
__device__ __forceinline__ bool select_ticket(uint32_t *ctr, uint32_t ncta, uint32_t &listed)
{
    const SelectCtr before = atomicAdd((SelectCtr *)ctr, 1ull << 32);
    listed = (uint32_t)before;
    if ((uint32_t)(before >> 32) != ncta - 1)
        return false;
    __threadfence();   // (with the barrier that follows, for the whole CTA)
    return true;
}

// The 32 elements from j0 on (a multiple of 32, below d): bits of those whose hash is below the window [lo, hi],
// and of those inside it.  lo is even and hi odd, so the lowest bit of the hash does not matter.
__device__ __forceinline__ uint32_t select_word(uint64_t st, uint32_t j0, uint32_t d, uint32_t lo, uint32_t hi, uint32_t &inside)
{
    // bit q is the carry of h + (2^32 - bound), i.e. h >= bound
    uint32_t not_below = 0, above = 0;
    const uint32_t nlo = 0u - lo, nhi = 0u - (hi + 1u);
    const uint64_t z0 = st + kGolden * ((uint64_t)j0 + 1);
#pragma unroll
    for (int q = 31; q >= 0; --q) {
        const uint32_t h = hash32_but_lowest_of(z0 + kGolden * (uint64_t)q);
        asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %2, %3;\n\taddc.u32 %0, %0, %0;\n\t"
            "add.cc.u32 t, %2, %4;\n\taddc.u32 %1, %1, %1;\n\t}"
            : "+r"(not_below), "+r"(above) : "r"(h), "r"(nlo), "r"(nhi));
    }
    const uint32_t exist = d - j0 >= 32u ? 0xFFFFFFFFu : (1u << (d - j0)) - 1u;
    const uint32_t word = lo ? ~not_below & exist : 0u;
    inside = ~above & ~word & exist;
    return word;
}

// exclusive prefix over the CTA's threads of v; total: the sum over all threads; FRESH: wsum is not in use
template <bool FRESH = false>
__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t *wsum, uint32_t &total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o)
            inc += n;
    }
    if (!FRESH)
        __syncthreads();   // wsum may still be read from the previous call
    if (lane == 31)
        wsum[warp] = inc;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kSelThreads / 32; ++w) {
        const uint32_t t = wsum[w];
        before += w < warp ? t : 0u;
        all += t;
    }
    total = all;
    return before + inc - v;
}

// The bin of the histogram that holds rank `rank` (1-based) and the rank within it; S.bad when none does.
__device__ __forceinline__ void select_bin(SelectShared &S, uint32_t rank)
{
    constexpr int PER = kSelBins / kSelThreads;
    const int tid = threadIdx.x;
    if (tid == 0)
        S.bad = 1u;
    uint32_t c[PER], sum = 0, total;
#pragma unroll
    for (int x = 0; x < PER; ++x)
        sum += c[x] = S.hist[tid * PER + x];
    uint32_t before = block_exclusive(sum, S.wsum, total);
    if (before < rank && rank <= before + sum) {
#pragma unroll
        for (int x = 0; x < PER; ++x) {
            if (before < rank && rank <= before + c[x]) {
                S.bin = tid * PER + x;
                S.rem = rank - before;
                S.bad = 0u;
            }
            before += c[x];
        }
    }
    __syncthreads();
}

// S.tau = the key of rank `rank` (1-based) among the S.n keys in S.keys
__device__ __forceinline__ void select_key(SelectShared &S, uint32_t rank)
{
    const uint32_t n = S.n;
    if (n > (uint32_t)kSelList || rank == 0 || rank > n) {
        if (threadIdx.x == 0)
            S.bad = 1u;
    } else {
        for (uint32_t x = threadIdx.x; x < n; x += kSelThreads) {
            const uint64_t me = S.keys[x];
            uint32_t below = 0;
            for (uint32_t y = 0; y < n; ++y)
                below += S.keys[y] < me;
            if (below == rank - 1)   // keys are distinct
                S.tau = me;
        }
    }
    __syncthreads();
}

// A tensor's window, its k and d (scale: see select_window), and where a list that holds anything but
// elements of the window is reported (null: nowhere)
struct SelectWindow {
    uint32_t lo, hi, d, k;
    uint64_t scale;
    int32_t *status;
    // Whether a list entry can be one of this tensor's; no entry is used as an index before this is known.
    // (Calls that share one scratch and overlap see one another's entries.  A form without load_cg read shared
    // memory out of bounds: an entry that was written lies inside the window, and select_window's scale
    // then gives a bin below kSelThreads, so that entry had been read before it was written.)
    __device__ __forceinline__ bool holds(uint2 e) const { return e.x - lo <= hi - lo && e.y < d; }
    // Result of a list that failed: as if the window had missed, so that the tensor is hashed again.  All
    // threads of the CTA take it.
    __device__ __forceinline__ uint32_t stale() const
    {
        if (status && threadIdx.x == 0)
            atomicOr(status, ST_LIST_STALE);
        return 0xFFFFFFFFu;
    }
};

// The threshold among the window's elements, get(x) for x < nlist.  `below_mine`: the calling thread's share of the
// number of elements below the window.  The caller has zeroed S.hist[0 .. kSelThreads) and synchronised.  Returns
// the number of elements below the window, or 0xFFFFFFFF where the window does not hold the threshold;
// S.tau is the threshold key (0 when no listed element belongs).
template <class Get>
__device__ __forceinline__ uint32_t select_threshold(SelectShared &S, const SelectWindow &W, Get get, uint32_t nlist, uint32_t below_mine)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t lo = W.lo, k = W.k;
    const bool shared = nlist <= (uint32_t)kSelList;
    bool stale = false;
    if (shared) {
        // one linear bin per thread; the few keys of the bin that holds the rank are compared
        auto bin_of = [&](uint32_t h) { return (uint32_t)(((uint64_t)(h - lo) * W.scale) >> 32); };
#pragma unroll 4
        for (uint32_t x = tid; x < nlist; x += kSelThreads) {
            const uint2 e = get(x);
            S.keys[x] = ((uint64_t)e.x << 32) | e.y;
            if (W.holds(e))
                atomicAdd(&S.hist[bin_of(e.x)], 1u);
            else
                stale = true;
        }
        if (tid == 0) {
            S.n = 0;
            S.bad = 1u;
            S.tau = 0;
        }
        if (__syncthreads_or(stale))
            return W.stale();
        const uint32_t c = S.hist[tid];
        uint32_t inc = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t n = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o)
                inc += n;
        }
        below_mine = __reduce_add_sync(0xffffffffu, below_mine);
        if (lane == 31) {
            S.wsum[warp] = inc;
            S.wsum2[warp] = below_mine;
        }
        __syncthreads();
        uint32_t before = inc - c, below = 0;
#pragma unroll
        for (int w = 0; w < kSelThreads / 32; ++w) {
            before += w < warp ? S.wsum[w] : 0u;
            below += S.wsum2[w];
        }
        if (below > k || k - below > nlist)
            return 0xFFFFFFFFu;
        const uint32_t rank = k - below;
        if (rank == 0)
            return below;
        if (before < rank && rank <= before + c) {
            S.bin = tid;
            S.rem = rank - before;
        }
        __syncthreads();
        const uint32_t bin = S.bin;
        for (uint32_t x = tid; x < nlist; x += kSelThreads) {
            const uint64_t key = S.keys[x];
            if (bin_of((uint32_t)(key >> 32)) == bin)
                S.hist[kSelThreads + min(atomicAdd(&S.n, 1u), (uint32_t)(kSelBins - kSelThreads - 1))] = x;   // (its place, not its count)
        }
        __syncthreads();
        const uint32_t np = S.n;
        if (np > (uint32_t)(kSelBins - kSelThreads - 1))
            return 0xFFFFFFFFu;
        for (uint32_t x = tid; x < np; x += kSelThreads) {
            const uint64_t me = S.keys[S.hist[kSelThreads + x]];
            uint32_t smaller = 0;
            for (uint32_t y = 0; y < np; ++y)
                smaller += S.keys[S.hist[kSelThreads + y]] < me;
            if (smaller == S.rem - 1) {   // keys are distinct
                S.tau = me;
                S.bad = 0u;
            }
        }
        __syncthreads();
        return S.bad ? 0xFFFFFFFFu : below;
    }
    // a longer list stays in L2: two passes over it, 2048 bins
    const uint64_t scale8 = W.scale * (kSelBins / kSelThreads);
    auto bin_of = [&](uint32_t h) { return (uint32_t)(((uint64_t)(h - lo) * scale8) >> 32); };
    for (int b = kSelThreads + tid; b < kSelBins; b += kSelThreads)
        S.hist[b] = 0;
    if (tid == 0)
        S.tau = 0;
    uint32_t below;
    block_exclusive(below_mine, S.wsum, below);   // (synchronises)
    if (below > k || k - below > nlist)
        return 0xFFFFFFFFu;
    if (below == k)
        return below;
#pragma unroll 8
    for (uint32_t x = tid; x < nlist; x += kSelThreads) {
        const uint2 e = get(x);
        if (W.holds(e))
            atomicAdd(&S.hist[bin_of(e.x)], 1u);
        else
            stale = true;
    }
    if (__syncthreads_or(stale))
        return W.stale();
    select_bin(S, k - below);
    if (S.bad)
        return 0xFFFFFFFFu;
    const uint32_t bin = S.bin;
    if (tid == 0)
        S.n = 0;
    __syncthreads();
#pragma unroll 8
    for (uint32_t x = tid; x < nlist; x += kSelThreads) {
        const uint2 e = get(x);
        if (bin_of(e.x) == bin) {
            const uint32_t pos = atomicAdd(&S.n, 1u);
            if (pos < (uint32_t)kSelList)
                S.keys[pos] = ((uint64_t)e.x << 32) | e.y;
        }
    }
    __syncthreads();
    select_key(S, S.rem);
    return S.bad ? 0xFFFFFFFFu : below;
}

// calls f(j) for the listed elements that belong to the set; j < d, also where the list changed after
// select_threshold looked at it
template <class Get, class F>
__device__ __forceinline__ void select_listed(SelectShared &S, const SelectWindow &W, Get get, uint32_t nlist, F f)
{
    const uint64_t tau = S.tau;
    if (nlist <= (uint32_t)kSelList) {
        for (uint32_t x = threadIdx.x; x < nlist; x += kSelThreads)
            if (S.keys[x] <= tau)
                f((uint32_t)S.keys[x]);
    } else {
#pragma unroll 4
        for (uint32_t x = threadIdx.x; x < nlist; x += kSelThreads) {
            const uint2 e = get(x);
            if ((((uint64_t)e.x << 32) | e.y) <= tau && e.y < W.d)
                f(e.y);
        }
    }
}

// The threshold key of rank k over all d elements by one CTA: 11 + 11 + 10 bits of the hash, then the
// index among the elements that share the threshold's hash.
static __device__ __noinline__ void select_exact(SelectShared &S, uint64_t st, uint32_t d, uint32_t k)
{
    const int tid = threadIdx.x;
    uint32_t prefix = 0, rank = k;
#pragma unroll 1
    for (int level = 0; level < 3; ++level) {
        for (int b = tid; b < kSelBins; b += kSelThreads)
            S.hist[b] = 0;
        __syncthreads();
        for (uint64_t j = tid; j < d; j += kSelThreads) {
            const uint32_t h = hash32(st, j);
            if (level == 0)
                atomicAdd(&S.hist[h >> 21], 1u);
            else if (level == 1) {
                if ((h >> 21) == prefix)
                    atomicAdd(&S.hist[(h >> 10) & 2047u], 1u);
            } else if ((h >> 10) == prefix)
                atomicAdd(&S.hist[h & 1023u], 1u);
        }
        __syncthreads();
        select_bin(S, rank);
        if (S.bad)
            return;
        prefix = level == 0 ? S.bin : level == 1 ? (prefix << 11) | S.bin : (prefix << 10) | S.bin;
        rank = S.rem;
        __syncthreads();
    }
    if (tid == 0)
        S.n = 0;
    __syncthreads();
    for (uint64_t j = tid; j < d; j += kSelThreads)
        if (hash32(st, j) == prefix) {
            const uint32_t pos = atomicAdd(&S.n, 1u);
            if (pos < (uint32_t)kSelList)
                S.keys[pos] = ((uint64_t)prefix << 32) | (uint32_t)j;
        }
    __syncthreads();
    select_key(S, rank);
}

// ---- a tensor of at most kSelClusterTiles tiles: a cluster, one tile per CTA
// Without it a selection is a chain of trips to L2 (a place in the list, a fence, the ticket, the bitmap and the list read
// back) whatever the tensor's size.
// Everything is exchanged through the CTAs' shared memory, and nothing in global memory is touched before the
// result is written, so that all of it can run while the kernel ahead in the stream ends.
constexpr int kSelClusterTiles = 16;
// All clusters of a launch have the size that the largest tensor needs, so small tensors beside a large one leave most of
// their CTAs idle, and those of many tensors do not fit the SMs together.  Selection and step of one worker on the GPU, clusters
// and k_rk_select, one tensor of 16 tiles beside small ones: 11 (176 CTAs idle) 11.5 and 15.1 us, 19 (285) 14.4 and 15.4, 23
// (345) 14.2 and 15.7, 31 (465) 18.6 and 15.6, 300 (4500) 76.7 and 20.8; of 8 tiles: 39 (273) 12.3 and 13.8, 43 (301) 14.8 and
// 14.0, 1000 (7000) 116 and 37.  Tensors of 16 tiles, none idle: 20 (320 CTAs) 20.5 and 23.0, 40 (640) 30.8 and 33.4, 60 (960)
// 40.5 and 39.3, 200 (3200) 110 and 94.  Clusters of one CTA are faster throughout (1000 tensors 38.4 and 40.0).
constexpr int64_t kSelClusterIdle = kPlanSMs * 2, kSelClusterCtas = kPlanSMs * 5;
constexpr int kSelMine = 1024;   // window elements of a CTA: expected 607 at most (d = 8192, k = d / 2), or a whole short tensor
struct SelectCluster : SelectShared {
    uint2 mine[kSelMine];
    uint32_t words[kSelThreads];
    uint32_t n_mine, below;                                       // this CTA's elements inside the window and below it
    uint32_t base[kSelClusterTiles + 1], cnt[kSelClusterTiles];   // of the CTA that finds the threshold: the lists' places, members listed
    uint64_t r_tau;                                               // what that CTA writes into all of them: the threshold key,
    uint32_t r_first, r_total, r_found;                           // members before this CTA's tile and in all, whether the window held
};
struct SelectResult {
    uint32_t word, first, total;   // this thread's 32 elements, members before this CTA's tile, members of the tensor
    bool failed;
};
// how: CONEF_SELECT_*; with STALE, of which there is nothing here (no list outlives the call), as with MISS
__device__ __forceinline__ SelectResult select_in_cluster(SelectCluster &S, uint64_t st, uint32_t d, uint32_t k, uint32_t lo, uint32_t hi,
                                                          uint64_t scale, int how)
{
    static_assert(kHistTile == 32 * kSelThreads, "a word per thread");
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const uint32_t rank = cluster.block_rank(), csize = cluster.num_blocks();
    const int tid = threadIdx.x, lane = tid & 31;
    if (d <= (uint32_t)kSelShortTensor) {   // the window is everything
        lo = 0u;
        hi = 0xFFFFFFFFu;
        scale = 256u;
    }
    const SelectWindow W{lo, hi, d, k, scale, nullptr};
    const uint32_t room = how == CONEF_SELECT_FULL ? 1u : (uint32_t)kSelMine;
    S.hist[tid] = 0;   // the bins of select_threshold
    if (tid == 0)
        S.n_mine = S.below = 0;
    __syncthreads();
    const uint32_t j0 = rank * (uint32_t)kHistTile + tid * 32u;
    uint32_t word = 0;
    if (j0 < d) {
        uint32_t inside;
        word = select_word(st, j0, d, lo, hi, inside);
        for (; inside; inside &= inside - 1) {
            const uint32_t j = j0 + (uint32_t)__ffs(inside) - 1u, pos = atomicAdd(&S.n_mine, 1u);
            if (pos < room)
                S.mine[pos] = make_uint2(hash32(st, j), j);
        }
    }
    const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(word));
    if (lane == 0 && c)
        atomicAdd(&S.below, c);
    cluster.sync();
    if (rank == 0) {
        uint32_t below = 0, n = 0;
        if (tid < 32) {   // (a CTA per lane)
            if ((uint32_t)tid < csize) {
                n = *cluster.map_shared_rank(&S.n_mine, tid);
                below = *cluster.map_shared_rank(&S.below, tid);
            }
            const bool full = __any_sync(0xffffffffu, n > room);
            uint32_t inc = n;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o)
                    inc += t;
            }
            if (tid < kSelClusterTiles) {
                S.base[tid] = inc - n;
                S.cnt[tid] = 0;
            }
            if (tid == kSelClusterTiles - 1) {
                S.base[kSelClusterTiles] = inc;
                S.r_found = !full && (how == CONEF_SELECT_NORMAL || how == CONEF_SELECT_FULL);
            }
        }
        __syncthreads();
        const uint32_t nlist = S.base[kSelClusterTiles];
        auto owner = [&](uint32_t x) {   // the CTA that listed entry x
            uint32_t r = 0;
#pragma unroll
            for (uint32_t o = kSelClusterTiles / 2; o; o /= 2)
                r += x >= S.base[r + o] ? o : 0u;
            return r;
        };
        auto get = [&](uint32_t x) {
            const uint32_t r = owner(x);
            return cluster.map_shared_rank(S.mine, r)[x - S.base[r]];
        };
        const bool found = S.r_found && select_threshold(S, W, get, nlist, below) != 0xFFFFFFFFu;
        __syncthreads();
        if (found) {
            const uint64_t tau = S.tau;
            for (uint32_t x = tid; x < nlist; x += kSelThreads) {
                uint64_t key;
                if (nlist <= (uint32_t)kSelList) {
                    key = S.keys[x];
                } else {
                    const uint2 e = get(x);
                    key = ((uint64_t)e.x << 32) | e.y;
                }
                if (key <= tau)
                    atomicAdd(&S.cnt[owner(x)], 1u);
            }
            __syncthreads();
        } else {
            select_exact(S, st, d, k);
            __syncthreads();
        }
        if (tid < 32) {
            const uint32_t m = found && (uint32_t)tid < csize ? below + S.cnt[tid & (kSelClusterTiles - 1)] : 0u;
            uint32_t inc = m;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o)
                    inc += t;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, inc, 31);
            if ((uint32_t)tid < csize) {
                SelectCluster *to = cluster.map_shared_rank(&S, tid);
                to->r_tau = found || !S.bad ? S.tau : 0u;
                to->r_first = inc - m;
                to->r_total = total;
                to->r_found = found ? 1u : S.bad ? 2u : 0u;
            }
        }
    }
    cluster.sync();
    SelectResult R;
    const uint64_t tau = S.r_tau;
    R.failed = S.r_found == 2u;
    if (S.r_found == 1u) {
        S.words[tid] = word;
        __syncthreads();
        for (uint32_t x = tid; x < S.n_mine; x += kSelThreads) {
            const uint2 e = S.mine[x];
            if ((((uint64_t)e.x << 32) | e.y) <= tau)
                atomicOr(&S.words[(e.y >> 5) & (kSelThreads - 1)], 1u << (e.y & 31u));
        }
        __syncthreads();
        R.word = S.words[tid];
        R.first = S.r_first;
        R.total = S.r_total;
    } else {   // the threshold is known, but not from the window: every element once more
        word = 0;
        for (uint32_t q = 0; q < 32 && j0 < d && j0 + q < d; ++q)
            if ((((uint64_t)hash32(st, j0 + q) << 32) | (j0 + q)) <= tau)
                word |= 1u << q;
        R.word = word;
        uint32_t mine;
        block_exclusive(__popc(word), S.wsum, mine);
        if (tid == 0)
            S.below = mine;
        cluster.sync();
        uint32_t n = (uint32_t)lane < csize ? *cluster.map_shared_rank(&S.below, lane) : 0u;
        R.total = __reduce_add_sync(0xffffffffu, n);
        R.first = __reduce_add_sync(0xffffffffu, (uint32_t)lane < rank ? n : 0u);
        cluster.sync();   // (no CTA leaves while its shared memory may still be read)
    }
    return R;
}

// exclusive scan of n counts in place by the CTA; returns the total
__device__ __forceinline__ uint32_t scan_counts(uint32_t *cnt, int64_t n, uint32_t *wsum)
{
    constexpr int PER = 4;
    uint32_t carry = 0;
    for (int64_t base = 0; base < n; base += kSelThreads * PER) {
        const int64_t at = base + (int64_t)threadIdx.x * PER;
        uint32_t c[PER], sum = 0, total;
#pragma unroll
        for (int x = 0; x < PER; ++x)
            sum += c[x] = at + x < n ? load_cg(cnt + at + x) : 0u;
        uint32_t run = carry + block_exclusive(sum, wsum, total);
#pragma unroll
        for (int x = 0; x < PER; ++x) {
            if (at + x < n)
                cnt[at + x] = run;
            run += c[x];
        }
        carry += total;
    }
    __syncthreads();
    return carry;
}

// What the last CTA of a tensor does with the window's elements: finds the threshold, calls mark(j) for
// the listed members and adds them to their tiles' counts (tile = j / TILE), and turns the counts
// into exclusive offsets, in place.  Returns the number of members, or 0xFFFFFFFF where the window
// does not hold the threshold (nothing is marked then).
template <uint32_t TILE, class Mark>
__device__ __forceinline__ uint32_t select_finish(SelectSharedTiles &S, const SelectWindow &W, const uint2 *list, uint32_t nlist,
                                                  uint32_t *cnt, uint32_t ntiles, Mark mark)
{
    const int tid = threadIdx.x;
    const bool shared = ntiles <= (uint32_t)kSelTiles;
    uint32_t mine = 0;
#pragma unroll 4
    for (uint32_t t = tid; t < ntiles; t += kSelThreads) {
        const uint32_t c = load_cg(cnt + t);
        if (shared)
            S.tiles[t] = c;
        mine += c;
    }
    const auto get = [list](uint32_t x) { return load_cg(&list[x]); };
    if (select_threshold(S, W, get, nlist, mine) == 0xFFFFFFFFu)
        return 0xFFFFFFFFu;
    select_listed(S, W, get, nlist, [&](uint32_t j) {
        mark(j);
        atomicAdd(shared ? &S.tiles[j / TILE] : &cnt[j / TILE], 1u);
    });
    if (!shared) {
        __threadfence();
        __syncthreads();
        return scan_counts(cnt, ntiles, S.wsum);
    }
    __syncthreads();
    constexpr uint32_t PER = (kSelTiles + kSelThreads - 1) / kSelThreads;
    uint32_t c[PER], sum = 0, total;
#pragma unroll
    for (uint32_t x = 0; x < PER; ++x)
        sum += c[x] = tid * PER + x < ntiles ? S.tiles[tid * PER + x] : 0u;
    uint32_t run = block_exclusive(sum, S.wsum, total);
#pragma unroll
    for (uint32_t x = 0; x < PER; ++x) {
        if (tid * PER + x < ntiles)
            cnt[tid * PER + x] = run;
        run += c[x];
    }
    return total;
}

// Offsets of the words of one tile of 8192 elements (a warp; 8 words per lane).
__device__ __forceinline__ void select_offsets(const uint32_t *bits, uint16_t *wordoff, uint32_t tile)
{
    const int lane = threadIdx.x & 31;
    const uint32_t w0 = tile * (kHistTile / 32) + lane * 8;
    uint32_t word[8], cnt = 0;   // (the arrays cover whole tiles; words past the tensor are zero)
    load_cg(bits + w0, word);
#pragma unroll
    for (int x = 0; x < 8; ++x)
        cnt += __popc(word[x]);
    uint32_t inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o)
            inc += n;
    }
    uint32_t run = inc - cnt;
    uint32_t pair[4];
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        pair[x / 2] = x % 2 ? pair[x / 2] | (run << 16) : run;
        run += __popc(word[x]);
    }
    *(uint4 *)(wordoff + w0) = make_uint4(pair[0], pair[1], pair[2], pair[3]);
}

}  // namespace conef
