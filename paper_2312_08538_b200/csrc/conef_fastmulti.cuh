// One launch per low-rank pass over all tensors of a model of small or middling size (int8 / int4 error state).
//
// The tuned passes (conef_fast.cuh) take CTAs whose size follows from a tensor's width, so a model of many widths
// took a launch per size on side streams, forked and joined by events, and a further launch for the tensors of
// any other shape; with short tiles these cost as much as the passes.  Here every CTA has 256 threads: it holds
// as many tiles of its tensor as fit (f_nsub, each with its own part of shared memory and its own barrier), or
// one tile of the passes for any shape (conef_lrgen.cuh; up to multi_gen elements), or, in pass 1, of a 1-D tensor that passes through.
// What a tile computes, and the order of its sums, is that of those kernels.
// ResNet-50 list (seven widths and one odd convolution), int8, rank 4, four workers: 550 -> 440 us per step and update; six
// aligned matrices of 16 M elements together, int4, one worker 220 -> 182 us, eight workers 500 -> 492.  (64 registers, four CTAs per SM, spill: 577 us on the
// first list; two CTAs: 485 us.)
#pragma once
#include "conef_fast.cuh"
#include "conef_lrgen.cuh"

namespace conef {

constexpr int kMultiThreads = 256;
constexpr size_t kMultiSmem = 72 * 1024;   // shared memory of a CTA's tiles, where more than one shares it: three CTAs per SM
// Iterations per tile of passes 1 and 3 at most (pass 2's are part of the order of its sums).  Shorter tiles are slower, longer ones
// no faster at rank 4.  ResNet-50 list, four workers, int8, 8, 16, 32, 64 iterations and no limit: rank 4 532, 462, 443, 441, 441 us, rank 8
// 731, 606, 563, 554, 555; six matrices of 16 M elements together, eight workers, int4, rank 4: 553, 508, 496, 497, 496.
constexpr int kMultiIt = 32;
// Tensors of any other shape share these launches up to this many of their elements (all workers).  Beyond, they and the 1-D
// tensors have launches of their own (k_gen_pass), with four CTAs per SM instead of three at rank 4, three instead of two at rank 8,
// the block size as a constant in pass 3 and all of L1.  Step and update, one 1024 x 512 matrix beside an odd one of two workers,
// shared and on their own.  Rank 8, int4: 10 M elements 193 and 186 us, 16 M 274 and 267, 20 M 359 and 305, 28 M 412 and 342, 36 M 485
// and 467, 80 M 1032 and 841; int8: 16 M 259 and 287, 24 M 380 and 353, 36 M 451 and 512, 80 M 940 and 893; sixteen odd ones of eight
// workers, 167 M: 1827 and 1479, 1681 and 1586.  Rank 4, int4: 20 M 204 and 215, 40 M 332 and 365, 120 M 846 and 869; int8: 40 M 324 and
// 358, 120 M 820 and 830; those sixteen: 1045 and 1054, 1027 and 976.  (Ups and downs are waves of CTAs.)
constexpr int64_t multi_gen(int rank) { return rank == 8 ? 18'000'000 : 160'000'000; }
constexpr int multi_ctas(int pass, int rank) { return rank == 4 ? 3 : min_ctas(pass, rank); }

// bytes of shared memory of one tile
__host__ __device__ inline size_t multi_tile_bytes(int pass, int rank, int code_words, int scale_bytes, int it, int subs, int threads, int unit)
{
    const size_t b = (size_t)ring_depth(pass, rank) * threads * (32 + 4 * code_words) + fast_stage_bytes(pass, rank, it, subs, threads, unit, scale_bytes, kMultiStageIt);
    return (b + 127) / 128 * 128;
}

// Warps per tile (any divisor of the warps of a period) so that the CTAs are as full as possible, then as many as possible;
// a tile's iterations stay those of the plan.
inline void multi_classify(LayerDesc &L, int ckind, int scale_bytes)
{
    const int64_t nw = L.f_lcm / 256;
    int best = 1;
    for (int w = 1; w <= kFastMaxWarps; ++w)
        if (nw % w == 0 && kFastMaxWarps / w * w >= kFastMaxWarps / best * best)
            best = w;
    L.f_cw = best * 256;
    L.f_threads = best * 32;
    L.f_ncg = (int32_t)(nw / best);
    L.f_it1 = std::min(L.f_it1, kMultiIt);
    L.f_it3 = std::min(L.f_it3, kMultiIt);
    L.f_rt1 = (int32_t)((L.f_niter + L.f_it1 - 1) / L.f_it1);
    L.f_rt3 = (int32_t)((L.f_niter + L.f_it3 - 1) / L.f_it3);
    size_t most = 1;
    const int its[3] = {L.f_it1, L.f_it2, L.f_it3};
    for (int pass = 1; pass <= 3; ++pass)
        most = std::max(most, multi_tile_bytes(pass, L.rank, ckind == CONEF_C_INT4 ? 1 : 2, scale_bytes, its[pass - 1], L.f_subs, L.f_threads, L.unit));
    L.f_nsub = (int32_t)std::max<size_t>(1, std::min<size_t>(kMultiThreads / L.f_threads, kMultiSmem / most));
}

// the launch of one pass: conef_fastmulti.cu.  smem: the most that a CTA's tiles need
cudaError_t multi_launch(int pass, int ckind, int rank, int half, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s,
                         size_t smem);

}  // namespace conef
