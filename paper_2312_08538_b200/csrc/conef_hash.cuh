// Hashing shared by the selection kernels: the shared random-k index set
// (Sec. 5.3: same seed on every GPU) and the count sketch's h_i, s_i
// (Sec. 4.2.2) come from one 64-bit finalising mixer (splitmix64's) keyed by
// (seed, a, b) and evaluated at the element index.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace conef {

__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z)
{
    z ^= z >> 30;
    z *= 0xBF58476D1CE4E5B9ULL;
    z ^= z >> 27;
    z *= 0x94D049BB133111EBULL;
    z ^= z >> 31;
    return z;
}
constexpr uint64_t kGolden = 0x9E3779B97F4A7C15ULL;
__host__ __device__ __forceinline__ uint64_t stream_key(uint64_t seed, uint64_t a, uint64_t b)
{
    return mix64(mix64(seed + kGolden * (a + 1)) + kGolden * (b + 1));
}
__host__ __device__ __forceinline__ uint64_t h64(uint64_t st, uint64_t j)
{
    return mix64(st + kGolden * (j + 1));
}
__device__ __forceinline__ uint32_t hash32(uint64_t st, uint64_t j) { return (uint32_t)(h64(st, j) >> 32); }
// hash32 without the mixer's last step, which can only flip the lowest bit: comparisons with an even
// bound (x < even) come out the same.  z: st + kGolden * (j + 1), which a caller with a run of consecutive j
// steps along by additions of constants (left to the compiler it was three multiplies per element)
__device__ __forceinline__ uint32_t hash32_but_lowest_of(uint64_t z)
{
    z ^= z >> 30;
    z *= 0xBF58476D1CE4E5B9ULL;
    z ^= z >> 27;
    return (uint32_t)((z * 0x94D049BB133111EBULL) >> 32);
}

// Window [lo, hi] of hash values that holds the k-th smallest of d uniform 32-bit hashes: six
// standard deviations of that rank, sqrt(k (1 - k/d)), and a margin for small k, to either side of
// its expectation; cap: room for the elements inside (12 deviations and twice the margin expected);
// scale: ((h - lo) * scale) >> 32 cuts the window into 256 equal bins
inline void select_window(int64_t d, int64_t k, uint32_t &lo, uint32_t &hi, uint32_t &cap, uint64_t &scale)
{
    const double sd = __builtin_sqrt((double)k * (1.0 - (double)k / (double)d)), half = 6.0 * sd + 16.0;
    const double per = 4294967296.0 / (double)d;   // hash values per rank
    const double a = ((double)k - half) * per, b = ((double)k + half) * per;
    lo = (a > 0.0 ? (uint32_t)a : 0u) & ~1u;                  // even, and hi odd: see hash32_but_lowest
    hi = (b < 4294967295.0 ? (uint32_t)b : 0xFFFFFFFFu) | 1u;
    cap = (uint32_t)(16.0 * sd + 256.0);
    scale = (256ull << 32) / ((uint64_t)(hi - lo) + 1u);
}

// random-block-k: first index of the kept block, uniform on [0, d - k], from the shared stream
__host__ __device__ __forceinline__ uint32_t randblock_start(uint64_t st, uint32_t d, uint32_t k)
{
    return (uint32_t)(((h64(st, 0) >> 32) * ((uint64_t)(d - k) + 1)) >> 32);
}

}  // namespace conef
