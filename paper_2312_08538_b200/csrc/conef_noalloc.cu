// Allocation-free variant of the random-k index selection.
//
// Who needs it: the side that RECEIVES a random-k message.  To scatter the k
// values back into a dense update it must know the index set S_t, which
// depends only on (seed, tensor, step).  Such a receiver (a parameter server,
// a rank that only applies updates, a hook called from inside another
// framework's step) often holds no ConEF context and is not allowed to touch
// the device allocator: its memory pool is fixed up front, and a cudaMalloc in
// the middle of a step would synchronise the device or fail under memory
// pressure.  The selection needs scratch (a count per tile, the elements near the threshold);
// here that scratch is a fixed array that lives in the library's device image.
#include <cuda_runtime.h>

#include <mutex>

#include "conef_select.cuh"

using namespace conef;

namespace {

constexpr int kNaPer = 8;                                           // consecutive elements per thread
constexpr int kNaTile = kSelThreads * kNaPer;                       // elements per CTA
constexpr int64_t kNaMaxElems = CONEF_NOALLOC_MAX_ELEMS;
constexpr int64_t kNaTiles = kNaMaxElems / kNaTile;
constexpr int64_t kNaList = 16 * 2048 + 256;                        // select_window's room at its largest: d = 2^24, k = d / 2
constexpr int64_t kNaWords = 8 + kNaTiles + 2 * kNaList;            // counters, a count per tile, the window's elements

// The scratch itself.  Every GPU that loads the library holds these ~290 KB
// until the process exits.  In host code the name below is only a handle for
// cudaGetSymbolAddress; it is not a device address.
static __device__ __align__(256) uint32_t g_noalloc_scratch[kNaWords];

// Counter words: elements listed and CTAs that have finished (the second kernel of every call clears
// them, so that whatever calls that overlap did to them is over with the last of those calls), then what
// the first kernel leaves for the second: the threshold key, and whose it is (hash stream, d, k; k = 0: no
// threshold).
enum { NA_LISTED = 0, NA_DONE = 1, NA_TAU_LO = 2, NA_TAU_HI = 3, NA_STREAM_LO = 4, NA_STREAM_HI = 5, NA_D = 6, NA_K = 7 };

struct NaArgs {
    uint32_t *ctr, *cnt;
    uint2 *list;
    uint64_t stream;   // hash stream key of (seed, tensor, step)
    uint32_t d, k, lo, hi, cap, ntiles, how;   // how: CONEF_SELECT_*
    uint64_t scale;
};

// The context's selection (conef_select.cuh) without its bitmap: one pass counts each tile's elements
// below the window and lists those inside; the last CTA finds the threshold and the tiles' offsets.
__global__ void __launch_bounds__(kSelThreads) k_na_select(const NaArgs a)
{
    __shared__ SelectSharedTiles S;
    __shared__ uint32_t s_n, s_base, s_cnt, s_last, s_listed;
    const int tid = threadIdx.x;
    const bool windowed = a.d > (uint32_t)kSelShortTensor;   // (shorter ones come here with CONEF_SELECT_HALF only: see k_na_cluster)
    grid_release();
    S.hist[tid] = 0;   // the bins of select_threshold
    if (tid == 0)
        s_n = s_cnt = 0;
    __syncthreads();
    if (windowed) {
        const uint32_t j0 = blockIdx.x * kNaTile + tid * kNaPer;
        uint32_t below = 0, upto = 0;
        const uint64_t z0 = a.stream + kGolden * ((uint64_t)j0 + 1);
#pragma unroll
        for (uint32_t q = 0; q < kNaPer; ++q) {
            const uint32_t h = hash32_but_lowest_of(z0 + kGolden * q);
            below |= h < a.lo ? 1u << q : 0u;
            upto |= h <= a.hi ? 1u << q : 0u;
        }
        const uint32_t exist = j0 >= a.d ? 0u : a.d - j0 >= kNaPer ? (1u << kNaPer) - 1u : (1u << (a.d - j0)) - 1u;
        for (uint32_t m = upto & ~below & exist; m; m &= m - 1) {
            const uint32_t j = j0 + (uint32_t)__ffs(m) - 1u;
            const uint2 e = make_uint2(hash32(a.stream, j), a.how == CONEF_SELECT_STALE ? 0xFFFFFFFFu : j);
            const uint32_t pos = atomicAdd(&s_n, 1u);
            if (pos < (uint32_t)kSelList) {
                ((uint2 *)S.keys)[pos] = e;
            } else {
                grid_wait();
                const uint32_t g = select_claim(a.ctr, 1u);
                if (g < a.cap)
                    a.list[g] = e;
            }
        }
        below = __popc(below & exist);
        below = __reduce_add_sync(0xffffffffu, below);
        if ((tid & 31) == 0 && below)
            atomicAdd(&s_cnt, below);
        grid_wait();   // (all of that while the kernel ahead ends)
        __syncthreads();
        const uint32_t n = min(s_n, (uint32_t)kSelList);
        if (tid == 0) {
            s_base = n ? select_claim(a.ctr, n) : 0u;
            a.cnt[blockIdx.x] = s_cnt;
        }
        __syncthreads();
        for (uint32_t x = tid; x < n; x += kSelThreads)
            if (s_base + x < a.cap)
                a.list[s_base + x] = ((uint2 *)S.keys)[x];
    } else {
        grid_wait();
    }
    if (tid == 0 && blockIdx.x == 0)
        a.ctr[NA_K] = 0;   // (before this CTA's ticket, so before the last CTA's result)
    __threadfence();
    __syncthreads();
    if (tid == 0)
        s_last = select_ticket(a.ctr, a.ntiles, s_listed);   // (one thread's answer: the barriers below depend on it)
    __syncthreads();
    if (!s_last)
        return;
    const uint32_t nlist = s_listed;
    uint32_t total = 0xFFFFFFFFu;
    if (windowed && nlist <= a.cap && a.how != CONEF_SELECT_MISS)
        total = select_finish<kNaTile>(S, SelectWindow{a.lo, a.hi, a.d, a.k, a.scale, nullptr}, a.list, nlist, a.cnt, a.ntiles, [](uint32_t) {});
    bool failed = false;
    // no listed element belongs: the members are the elements below the window (lo > 0 then)
    if (total != 0xFFFFFFFFu && S.tau == 0 && tid == 0)
        S.tau = ((uint64_t)a.lo << 32) - 1u;
    if (total == 0xFFFFFFFFu) {
        __syncthreads();
        select_exact(S, a.stream, a.d, a.k);
        failed = S.bad != 0;
        const uint64_t tau = failed ? 0 : S.tau;
        for (uint32_t t = 0; t < a.ntiles; ++t) {
            __syncthreads();
            if (tid == 0)
                s_cnt = 0;
            __syncthreads();
            uint32_t c = 0;
            for (uint32_t q = tid; q < kNaTile; q += kSelThreads) {
                const uint32_t j = t * kNaTile + q;
                c += j < a.d && (((uint64_t)hash32(a.stream, j) << 32) | j) <= tau;
            }
            c = __reduce_add_sync(0xffffffffu, c);
            if ((tid & 31) == 0 && c)
                atomicAdd(&s_cnt, c);
            __syncthreads();
            if (tid == 0)
                a.cnt[t] = s_cnt;
        }
        __threadfence();
        __syncthreads();
        total = scan_counts(a.cnt, a.ntiles, S.wsum);
    }
    if (tid == 0) {
        a.ctr[NA_TAU_LO] = (uint32_t)S.tau;
        a.ctr[NA_TAU_HI] = (uint32_t)(S.tau >> 32);
        a.ctr[NA_STREAM_LO] = (uint32_t)a.stream;
        a.ctr[NA_STREAM_HI] = (uint32_t)(a.stream >> 32);
        a.ctr[NA_D] = a.d;
        a.ctr[NA_K] = failed || total != a.k ? 0u : a.k;
    }
}

// The members in ascending order, hashed once more.  A selection that did not come out as exactly k
// coordinates, or whose result is not there (another call's kernels ran in between), is made visible in
// the output itself, since this entry point neither synchronises nor owns a status buffer: nothing is
// written but idx_out[0] = 0xFFFFFFFF, a value no index can take.
__global__ void __launch_bounds__(kSelThreads) k_na_write(const NaArgs a, uint32_t *__restrict__ idx_out)
{
    __shared__ uint32_t wsum[kSelThreads / 32], s_own, s_first;
    __shared__ uint64_t s_tau;
    const uint32_t j0 = blockIdx.x * kNaTile + threadIdx.x * kNaPer;
    grid_release();
    uint32_t h[kNaPer];   // (while the first kernel ends)
#pragma unroll
    for (uint32_t q = 0; q < kNaPer; ++q)
        h[q] = hash32(a.stream, j0 + q);
    grid_wait();
    if (threadIdx.x == 0) {   // (one thread reads them: a CTA has to agree on whether it goes on)
        const uint2 tau = *(const uint2 *)(a.ctr + NA_TAU_LO);
        const uint4 of = *(const uint4 *)(a.ctr + NA_STREAM_LO);
        s_first = a.cnt[blockIdx.x];
        s_tau = ((uint64_t)tau.y << 32) | tau.x;
        s_own = of.x == (uint32_t)a.stream && of.y == (uint32_t)(a.stream >> 32) && of.z == a.d && of.w == a.k;
        if (blockIdx.x == 0)
            a.ctr[NA_DONE] = a.ctr[NA_LISTED] = 0;   // (no CTA of this kernel reads them)
    }
    __syncthreads();
    if (!s_own) {
        if (blockIdx.x == 0 && threadIdx.x == 0)
            idx_out[0] = 0xFFFFFFFFu;
        return;
    }
    const uint64_t tau = s_tau;
    uint32_t in = 0, total;
#pragma unroll
    for (uint32_t q = 0; q < kNaPer; ++q) {
        const uint32_t j = j0 + q;
        if ((((uint64_t)h[q] << 32) | j) <= tau && j < a.d)
            in |= 1u << q;
    }
    uint32_t slot = s_first + block_exclusive<true>(__popc(in), wsum, total);
    for (; in; in &= in - 1, ++slot)
        if (slot < a.k)   // never past the caller's k entries, whatever went wrong before
            idx_out[slot] = j0 + (uint32_t)__ffs(in) - 1u;
}

// Tensors of at most kNaClusterTiles tiles of 8192: one cluster does all of it, without the scratch
// (one launch, and nothing kept between calls).  54 convolutions, of which 19 are that small: 552 -> 408 us with it and
// with the first kernel's hashing ahead of its wait.  Eight calls in a row, a cluster and two kernels, k = d / 100: 1 tile 37 and 58
// us, 8 tiles 37 and 65, 16 tiles 38 and 69 (k = d / 2: 38 and 68, 38 and 80, 38 and 85), so the line is not where the cluster gets
// slower: eight CTAs are what a cluster may have on every device without opting in.
constexpr int kNaClusterTiles = 8;
__global__ void __launch_bounds__(kSelThreads) k_na_cluster(const NaArgs a, uint32_t *__restrict__ idx_out)
{
    __shared__ SelectCluster S;
    grid_release();
    const SelectResult R = select_in_cluster(S, a.stream, a.d, a.k, a.lo, a.hi, a.scale, (int)a.how);
    grid_wait();
    if (R.failed || R.total != a.k) {
        if (blockIdx.x == 0 && threadIdx.x == 0)
            idx_out[0] = 0xFFFFFFFFu;
        return;
    }
    const uint32_t j0 = blockIdx.x * (uint32_t)kHistTile + threadIdx.x * 32u;
    uint32_t all, slot = R.first + block_exclusive(__popc(R.word), S.wsum, all);
    for (uint32_t m = R.word; m; m &= m - 1, ++slot)
        if (slot < a.k)
            idx_out[slot] = j0 + (uint32_t)__ffs(m) - 1u;
}

// device address of the scratch on each device, resolved once per device
std::mutex g_mu;
uint32_t *g_scratch_ptr[64] = {nullptr};

int write_indices(uint64_t seed, int64_t tensor, int64_t step, int64_t d, int64_t k, int how, uint32_t *idx_out, conef_stream stream)
{
    if (d <= 0 || k <= 0 || k > d || tensor < 0 || step < 0 || !idx_out)
        return CONEF_ERR_INVALID_ARG;
    if (d > kNaMaxElems)
        return CONEF_ERR_TOO_LARGE;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64)
        return CONEF_ERR_CUDA;
    uint32_t *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_scratch_ptr[dev]) {
            // set-up, with this device current: turn the symbol into its device address
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p)
                return CONEF_ERR_CUDA;
            g_scratch_ptr[dev] = (uint32_t *)p;
        }
        scratch = g_scratch_ptr[dev];
    }
    if (cudaPeekAtLastError() != cudaSuccess)
        return CONEF_ERR_CUDA;   // an error from before this call is pending: nothing is launched on top of it
    cudaStream_t s = (cudaStream_t)stream;
    NaArgs a;
    a.ctr = scratch;
    a.cnt = scratch + 8;
    a.list = (uint2 *)(scratch + 8 + kNaTiles);
    a.stream = stream_key(seed, (uint64_t)tensor, (uint64_t)step);
    a.d = (uint32_t)d;
    a.k = (uint32_t)k;
    select_window(d, k, a.lo, a.hi, a.cap, a.scale);
    a.how = (uint32_t)how;
    if (how == CONEF_SELECT_FULL)
        a.cap = 1;
    const int64_t ctas = (d + kHistTile - 1) / kHistTile;
    if (ctas <= kNaClusterTiles && how != CONEF_SELECT_HALF) {
        static bool allowed[64] = {};
        const int size = ctas <= 1 ? 1 : ctas <= 2 ? 2 : ctas <= 4 ? 4 : kNaClusterTiles;
        launch_cluster(k_na_cluster, 1, size, kSelThreads, s, allowed, a, idx_out);
        return cudaGetLastError() == cudaSuccess ? CONEF_OK : CONEF_ERR_CUDA;
    }
    a.ntiles = (uint32_t)((d + kNaTile - 1) / kNaTile);
    launch(k_na_select, dim3(a.ntiles), kSelThreads, 0, s, a);
    if (how != CONEF_SELECT_HALF)
        launch(k_na_write, dim3(a.ntiles), kSelThreads, 0, s, a, idx_out);
    return cudaGetLastError() == cudaSuccess ? CONEF_OK : CONEF_ERR_CUDA;
}

}  // namespace

extern "C" int conef_randk_indices_noalloc(uint64_t seed, int64_t tensor, int64_t step, int64_t d, int64_t k,
                                           uint32_t *idx_out, conef_stream stream)
{
    return write_indices(seed, tensor, step, d, k, CONEF_SELECT_NORMAL, idx_out, stream);
}
extern "C" int conef_randk_indices_noalloc_select(uint64_t seed, int64_t tensor, int64_t step, int64_t d, int64_t k,
                                                  int how, uint32_t *idx_out, conef_stream stream)
{
    if (how < CONEF_SELECT_NORMAL || how > CONEF_SELECT_HALF)
        return CONEF_ERR_INVALID_ARG;
    return write_indices(seed, tensor, step, d, k, how, idx_out, stream);
}
