// Tuned fused step for Q in {identity, random-k, random-block-k} with an int8 / int4 error state, or the
// stochastic quantiser of Eq. 6 with at most 127 levels (Alg. 2 lines 5, 6, 9 in one kernel): decode,
// p = eta g + e, message, residual, block absmax, requantise, store in place.  ICO = 1 is iConEF-v1
// (Alg. 3): a second state q of the same kind is decoded beside the first, p = (eta g + e~) + q, and the
// store has a second round, q = C(r - decode(e~)).  Takes every size and every 4-byte alignment of the
// gradients.
//
// A lane owns 16 consecutive elements and a warp 512 ("a chunk"), so that one block scale, its
// reciprocal, one copy of codes and one set of addresses serve 16 elements, and a quantisation block (32
// to 256 elements) is an aligned group of 2 to 16 lanes.  Each warp stages its chunks through a ring of its
// own in shared memory by asynchronous 16-byte copies that a warp issues over contiguous memory; the
// 16-byte pieces of the gradient are laid out so that a lane's own pieces come back without bank
// conflicts.  Gradients off a 16-byte boundary are copied from the boundary below and shifted when they
// are read.
//
// The few transmitted coordinates are handled on the staged data before the chunk is computed: their
// p goes to the message, and their gradient and code are zeroed in shared memory, which makes p, and so
// the residual, exactly zero there without a test per element.
//
// HBM-bound (4 + 2 state bytes per element).  Transformer-big list, int8 / 256 / fp32, random-k 1 %, one
// worker: 338 us with eight elements per lane (352 warp instructions per 256 elements, 67 % of the ALU
// pipe's slots: membership tests and selects, prefix sums over lanes, a scale per eight elements),
// 208 us = 6.1 TB/s now (204 instructions).
#pragma once
#include "conef_fast.cuh"

namespace conef {

constexpr int kF16Threads = 256;
constexpr int kF16Chunk = 512;                                     // elements per warp and step
constexpr int kF16PerTile = kHistTile / kF16Chunk;                 // chunks per selection tile
// Stages per warp and CTAs per SM: three and three with one state; with two states (stages a quarter
// larger, more registers) two and four.  Transformer-big list, int8, one worker: 208 us with three and
// three, 219 with two and four; two int8 states on 14.6 M elements of four workers: 91 us with two and
// four, 122 with three and three.
__host__ __device__ constexpr int f16_ring(int ico) { return ico == 1 ? 2 : 3; }
__host__ __device__ constexpr int f16_ctas(int ico) { return ico == 1 ? 4 : 3; }

// Where piece p (16 bytes) of a chunk's gradient lies in its stage.  The pieces of a 128-byte line stay
// within 128 bytes: a layout that spread them over four rows cost an L2 request per piece (0.058
// requests per element now, tag lookups at 26 % of their rate).  The exchange inside a line makes the reads of lanes 64 bytes apart
// free of bank conflicts.
__host__ __device__ constexpr uint32_t f16_slot(uint32_t p) { return p ^ ((p >> 3) & 3u); }

// a warp's stage
template <int CK, int ICO>
struct alignas(128) F16Stage {
    static constexpr int CB = CK == CONEF_C_INT4 ? kF16Chunk / 2 : kF16Chunk;   // bytes of codes
    float4 g[kF16Chunk / 4 + 8];                     // 129 pieces used
    uint8_t codes[ICO == 1 ? 2 : 1][CB];
    // what a lane copies as words: random-k's bitmap words, their offsets (two per word) and the tile's
    // offset, then the block scales of the one or two states
    uint32_t aux[(25 + 32 + 15) / 4 * 4];
};
constexpr int kF16AuxSel = 0, kF16AuxOff = 16, kF16AuxTile = 24, kF16AuxScales = 25;

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ void cp_async16_cg(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
// the first `bytes` of 16 bytes; the rest is filled with zeros
__device__ __forceinline__ void cp_async16_part(void *dst, const void *src, uint32_t bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes) : "memory");
}

// 16 codes as floats 2^23 + bias + code
template <bool INT4>
__device__ __forceinline__ void code_floats(const uint32_t (&w)[INT4 ? 2 : 4], uint32_t (&t)[16])
{
    if (INT4) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            const uint32_t v = w[x] ^ 0x88888888u, lo = v & 0x0F0F0F0Fu, hi = (v >> 4) & 0x0F0F0F0Fu;
#pragma unroll
            for (int q = 0; q < 8; ++q)
                t[8 * x + q] = __byte_perm(q & 1 ? hi : lo, 0x4B000000u, 0x7440u | (q >> 1));
        }
    } else {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const uint32_t v = w[x] ^ 0x80808080u;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                t[4 * x + q] = __byte_perm(v, 0x4B000000u, 0x7440u | q);
        }
    }
}
// codes from the patterns 0x4B400000 + code (rounded values plus 1.5 * 2^23): the low byte or nibble of
// each is the two's complement code
template <bool INT4>
__device__ __forceinline__ void pack_codes(const uint32_t (&t)[16], uint32_t (&w)[INT4 ? 2 : 4])
{
    if (INT4) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {
            // even and odd elements' bytes first, then nibbles
            const uint32_t *v = t + 8 * x;
            const uint32_t lo = __byte_perm(__byte_perm(v[0], v[2], 0x0040), __byte_perm(v[4], v[6], 0x0040), 0x5410);
            const uint32_t hi = __byte_perm(__byte_perm(v[1], v[3], 0x0040), __byte_perm(v[5], v[7], 0x0040), 0x5410);
            w[x] = (lo & 0x0F0F0F0Fu) | ((hi << 4) & 0xF0F0F0F0u);
        }
    } else {
#pragma unroll
        for (int x = 0; x < 4; ++x)
            w[x] = __byte_perm(__byte_perm(t[4 * x], t[4 * x + 1], 0x0040), __byte_perm(t[4 * x + 2], t[4 * x + 3], 0x0040), 0x5410);
    }
}

template <int QK, int CK, bool HALF, int ICO>
__global__ void __launch_bounds__(kF16Threads, f16_ctas(ICO)) k_flat16(const __grid_constant__ DevView V, const int32_t *__restrict__ pfx)
{
    constexpr bool INT4 = CK == CONEF_C_INT4;
    constexpr int DK = CK == CONEF_C_STOCHQUANT ? CONEF_C_INT8 : CK;   // levels decode like int8 codes
    constexpr int kF16Ring = f16_ring(ICO);
    constexpr int NW = INT4 ? 2 : 4, SB = HALF ? 2 : 4, NS = ICO == 1 ? 2 : 1;
    using Stage = F16Stage<CK, ICO>;
    extern __shared__ __align__(128) uint8_t f16_smem[];
    grid_release();
    const int li = find_layer(pfx, V.n_layers, blockIdx.x);
    const LayerDesc &L = V.layers[li];
    if (!L.compressed) {   // (a 1-D tensor: its message in the same launch)
        grid_wait();
        pass_tile(V, L, blockIdx.x - pfx[li]);
        return;
    }
    const int worker = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t d = (uint32_t)L.d;
    const uint32_t tile0 = (blockIdx.x - pfx[li]) * (uint32_t)V.fv_tiles;
    const int shift = 31 - __clz(L.unit), lpb = L.unit >> 4;   // lanes per quantisation block
    uint8_t *st = V.state + worker * V.state_stride;
    uint8_t *codes[2] = {st + L.a_off, st + L.a2_off}, *scales[2] = {st + L.b_off, st + L.b2_off};
    const float *g = V.grads[worker] + L.g_off;
    const uint32_t gs = (uint32_t)((uintptr_t)g >> 2) & 3u;    // floats past the 16-byte boundary
    const float *ga = g - gs;
    float *__restrict__ msg = V.msgv + worker * V.msgv_stride + L.msgv_off;
    const uint32_t *__restrict__ bits = V.selbits + L.selbits_off, *__restrict__ tileoff = V.tileoff + L.tileoff_off;
    const uint16_t *__restrict__ wordoff = V.wordoff + L.wordoff_off;
    uint32_t blk_start = 0;
    if (QK == CONEF_Q_RANDBLOCK)
        blk_start = randblock_start(stream_key(V.seed_q, (uint64_t)li, (uint64_t)V.step), d, (uint32_t)L.k);
    // (read once: the copies' memory clobbers would have them loaded again for every chunk)
    const uint32_t abytes = (uint32_t)L.a_bytes, bbytes = (uint32_t)L.b_bytes, kept = (uint32_t)L.k;
    uint32_t *__restrict__ idx = V.idx + L.idx_off;
    const float lr = V.lr;
    const f32x2 lr2 = pk2(lr, lr);
    Stage *ring = (Stage *)f16_smem + warp * kF16Ring;

    // the warp's chunks: every eighth one of the CTA's tiles
    const uint32_t c0 = tile0 * kF16PerTile + warp, nchunks = (d + kF16Chunk - 1) / kF16Chunk;
    const uint32_t c1 = min(nchunks, (tile0 + (uint32_t)V.fv_tiles) * kF16PerTile);
    // Words of the aux array this lane copies, two at most: word `at` comes from src + (c >> sh) * step.
    // Without random-k the scales come first.
    constexpr int SC0 = QK == CONEF_Q_RANDK ? kF16AuxScales : 0;
    const uint32_t nsc = (uint32_t)(kF16Chunk >> shift) * SB / 4;   // words of scales per chunk and state (a chunk holds an even number of blocks)
    const uint32_t naux = SC0 + NS * nsc;
    struct AuxCopy {
        const uint8_t *src;
        uint32_t step, sh, limit;   // (c >> sh) * step stays below limit
    };
    auto aux_copy = [&](uint32_t at) {
        AuxCopy a;
        a.sh = 0;
        a.limit = 0xFFFFFFFFu;
        if (QK == CONEF_Q_RANDK && at < (uint32_t)kF16AuxOff) {
            a.src = (const uint8_t *)(bits + at);
            a.step = kF16Chunk / 8;
        } else if (QK == CONEF_Q_RANDK && at < (uint32_t)kF16AuxTile) {
            a.src = (const uint8_t *)wordoff + (at - kF16AuxOff) * 4;
            a.step = kF16Chunk / 16;
        } else if (QK == CONEF_Q_RANDK && at == (uint32_t)kF16AuxTile) {
            a.src = (const uint8_t *)tileoff;
            a.step = 4;
            a.sh = 4;   // kF16PerTile chunks per tile
        } else {
            const uint32_t i = at - SC0, x = i >= nsc ? 1u : 0u, w = i - x * nsc;
            a.src = scales[NS == 2 ? x : 0] + w * 4;
            a.step = nsc * 4;
            a.limit = bbytes > w * 4 ? bbytes - w * 4 : 0u;
        }
        return a;
    };
    static_assert(kF16PerTile == 16, "tile of a chunk by a shift");
    const AuxCopy aux0 = aux_copy(lane), aux1 = aux_copy(lane + 32);
    const bool has0 = (uint32_t)lane < naux, has1 = lane + 32u < naux;
    float4 *const my_g = (float4 *)((uint8_t *)ring + f16_slot(lane) * 16);
    constexpr uint32_t CB = Stage::CB;
    auto issue = [&](uint32_t c, int slot) {
        if (c < c1) {
            const uint32_t base = c * (uint32_t)kF16Chunk;
            Stage &S = ring[slot];
            float4 *dst = (float4 *)((uint8_t *)my_g + slot * sizeof(Stage));   // piece i * 32 + lane
            const float *src = ga + base + lane * 4;
            uint8_t *cdst = S.codes[0] + lane * 16;
            const uint32_t cpos = c * CB + lane * 16;
            if (base + kF16Chunk + 4u <= d) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    cp_async16_cg(dst + i * 32, src + i * 128);
                if (gs && lane == 0)   // the piece that holds the chunk's last gs elements
                    cp_async16_cg(&S.g[128], src + 512);
                if (lane < (int)(CB / 16)) {
#pragma unroll
                    for (int x = 0; x < NS; ++x)
                        cp_async16_cg(cdst + x * CB, codes[x] + cpos);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    const int64_t have = (int64_t)d + gs - ((int64_t)base + (i * 32 + lane) * 4);   // floats left from here
                    if (i < 4 || lane == 0)
                        cp_async16_part(i < 4 ? dst + i * 32 : &S.g[128], have > 0 ? src + i * 128 : ga,
                                        have >= 4 ? 16u : have > 0 ? (uint32_t)have * 4u : 0u);
                }
                // (the state's arrays are padded to 256 bytes, and what lies between the tensor's end and the
                // padding is zero)
                if (lane < (int)(CB / 16)) {
#pragma unroll
                    for (int x = 0; x < NS; ++x)
                        cp_async16_part(cdst + x * CB, codes[x] + (cpos < abytes ? cpos : 0u), cpos < abytes ? 16u : 0u);
                }
            }
            const uint32_t o0 = (c >> aux0.sh) * aux0.step;
            if (has0 && o0 < aux0.limit)
                cp_async_small<4>(&S.aux[lane], aux0.src + o0);
            if (naux > 32u) {
                const uint32_t o1 = (c >> aux1.sh) * aux1.step;
                if (has1 && o1 < aux1.limit)
                    cp_async_small<4>(&S.aux[lane + 32], aux1.src + o1);
            }
        }
        cp_async_commit();
    };
    auto scale_of = [&](const Stage &S, int x) {
        const uint32_t b = (uint32_t)(lane * 16) >> shift;
        const uint32_t *sc = S.aux + SC0 + x * nsc;
        if (HALF)
            return __half2float(__ushort_as_half(((const unsigned short *)sc)[b]));
        return __uint_as_float(sc[b]);
    };
    auto compute = [&](uint32_t c, Stage &S) {
        const uint32_t base = c * (uint32_t)kF16Chunk + lane * 16;   // this lane's first element
        const uint32_t left = base < d ? min(d - base, 16u) : 0u;    // ... and how many of them exist
        float s1 = 0.f, s2 = 0.f;
        if (left) {
            s1 = scale_of(S, 0);
            if (ICO == 1)
                s2 = scale_of(S, 1);
        }
        // transmitted coordinates
        uint32_t members = 0, slot = 0;
        if (QK == CONEF_Q_RANDK) {
            const uint32_t word = S.aux[kF16AuxSel + (lane >> 1)], sh = (lane & 1) * 16u;
            members = (word >> sh) & 0xFFFFu;   // (no bits past the tensor)
            if (members)
                slot = S.aux[kF16AuxTile] + ((const unsigned short *)(S.aux + kF16AuxOff))[lane >> 1] + __popc(word & ((1u << sh) - 1u));
        } else if (QK == CONEF_Q_RANDBLOCK) {
            const uint32_t b1 = blk_start + kept;
            if (left && base < b1 && base + left > blk_start) {
                const uint32_t a = max(base, blk_start) - base, e = min(base + left, b1) - base;
                members = ((1u << e) - 1u) & ~((1u << a) - 1u);
                slot = base + a - blk_start;
            }
        }
        if (QK != CONEF_Q_IDENTITY) {
            float *gf = (float *)S.g;
            while (members) {
                const uint32_t q = (uint32_t)__ffs(members) - 1u;
                members &= members - 1u;
                const uint32_t e = lane * 16u + q, f = e + gs;
                float *gp = gf + f16_slot(f >> 2) * 4u + (f & 3u);
                float err[2];
#pragma unroll
                for (int x = 0; x < NS; ++x) {
                    int code;
                    if (INT4) {
                        uint8_t *cp = &S.codes[x][e >> 1];
                        const uint32_t byte = *cp, at = 4u * (e & 1u);
                        code = (int)(((byte >> at) & 0xFu) ^ 8u) - 8;
                        *cp = (uint8_t)(byte & ~(0xFu << at));
                    } else {
                        code = (int)(signed char)S.codes[x][e];
                        S.codes[x][e] = 0;
                    }
                    err[x] = __fmul_rn((float)code, x ? s2 : s1);
                }
                float p = __fmaf_rn(lr, *gp, err[0]);   // Alg. 2 line 5
                if (ICO == 1)
                    p = __fadd_rn(p, err[1]);           // Alg. 3 line 5
                *gp = 0.f;
                msg[slot] = p;
                if (worker == 0)
                    idx[slot] = base + q;
                ++slot;
            }
            asm volatile("" ::: "memory");   // the vector reads below see those stores
        }
        // p of 16 elements, as pairs
        f32x2 p2[8];
        {
            f32x2 g2[8];
            if (gs == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const ulonglong2 v = *(const ulonglong2 *)&S.g[f16_slot(lane * 4 + i)];
                    g2[2 * i] = v.x;
                    g2[2 * i + 1] = v.y;
                }
            } else {
                float v[20];
#pragma unroll
                for (int i = 0; i < 5; ++i) {
                    const float4 t = S.g[f16_slot(lane * 4 + i)];
                    v[4 * i] = t.x; v[4 * i + 1] = t.y; v[4 * i + 2] = t.z; v[4 * i + 3] = t.w;
                }
                if (gs == 1) {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        g2[i] = pk2(v[2 * i + 1], v[2 * i + 2]);
                } else if (gs == 2) {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        g2[i] = pk2(v[2 * i + 2], v[2 * i + 3]);
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        g2[i] = pk2(v[2 * i + 3], v[2 * i + 4]);
                }
            }
            constexpr float off = INT4 ? 8388616.f : 8388736.f;   // 2^23 + bias
            const f32x2 off2 = pk2(-off, -off);
#pragma unroll
            for (int x = 0; x < NS; ++x) {
                uint32_t w[NW], t[16];
                if (INT4) {
                    const uint2 v = *(const uint2 *)(S.codes[x] + lane * 8);
                    w[0] = v.x; w[1] = v.y;
                } else {
                    const uint4 v = *(const uint4 *)(S.codes[x] + lane * 16);
                    w[0] = v.x; w[1] = v.y; w[NW - 2] = v.z; w[NW - 1] = v.w;
                }
                code_floats<INT4>(w, t);
                const float sx = x ? s2 : s1;
                const f32x2 sx2 = pk2(sx, sx);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const f32x2 e2 = mul2(add2(pk2u(t[2 * i], t[2 * i + 1]), off2), sx2);   // float(code) * scale
                    if (x == 0) {
                        p2[i] = fma2(lr2, g2[i], e2);        // Alg. 2 line 5
                    } else {
                        float a, b, qa, qb;                  // (a packed multiply followed by a packed add may be contracted)
                        upk2(p2[i], a, b);
                        upk2(e2, qa, qb);
                        p2[i] = pk2(__fadd_rn(a, qa), __fadd_rn(b, qb));   // Alg. 3 line 5: + q
                    }
                }
            }
        }
        float r[16];
#pragma unroll
        for (int i = 0; i < 8; ++i)
            upk2(p2[i], r[2 * i], r[2 * i + 1]);
        if (QK == CONEF_Q_IDENTITY) {   // everything is sent, nothing is left
            if (left == 16u && ((uintptr_t)(msg + base) & 15) == 0) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    *(float4 *)(msg + base + 4 * i) = make_float4(r[4 * i], r[4 * i + 1], r[4 * i + 2], r[4 * i + 3]);
            } else {
#pragma unroll
                for (int q = 0; q < 16; ++q)
                    if (q < (int)left)
                        msg[base + q] = r[q];
            }
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                p2[i] = 0ull;
                r[2 * i] = r[2 * i + 1] = 0.f;
            }
        }
        // store r through C (Alg. 2 line 9), and with Alg. 3 what that misses
#pragma unroll
        for (int x = 0; x < NS; ++x) {
            float amax = 0.f;
#pragma unroll
            for (int q = 0; q < 16; ++q)
                amax = fmaxf(amax, fabsf(r[q]));
#pragma unroll
            for (int o = 8; o >= 1; o >>= 1)
                if (lpb > o)
                    amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            float s, inv;
            unsigned short hb = 0;
            uint32_t w[NW], t[16];
            if constexpr (CK == CONEF_C_STOCHQUANT) {
                // Eq. 6 with the block's max-norm: level floor(u) or floor(u) + 1, up with probability
                // u - floor(u); the variate of (worker, tensor, step, element) from a counter-based stream
                const float lv = (float)V.levels;
                s = __fdiv_rn(amax, lv);
                const bool zero = !(s >= FLT_MIN);
                s = zero ? 0.f : s;
                inv = zero ? 0.f : __fdiv_rn(1.0f, s);
                const uint64_t stc = stream_key(mix64(V.seed_c + (uint64_t)worker + 1u), (uint64_t)li, (uint64_t)V.step);
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    float u = __fmul_rn(fabsf(r[q]), inv);
                    u = !(u <= lv) ? lv : u;
                    const float l = floorf(u);
                    const float frac = __fsub_rn(u, l);
                    const float rnd = __fmul_rn((float)(uint32_t)(h64(stc, base + q) >> 40), 1.0f / 16777216.0f);
                    int lev = (int)l + (rnd < frac ? 1 : 0);
                    lev = min(lev, V.levels);
                    t[q] = (uint32_t)(zero ? 0 : r[q] < 0.f ? -lev : lev);
                }
            } else {
                block_scale<DK, HALF>(amax, s, inv, hb);
                // |r * inv| <= amax * inv (rounding is monotone): the clamp is needed only where that
                // bound rounds past qmax, which takes a binary16 scale that was rounded down by a lot
                constexpr float qm = INT4 ? 7.f : 127.f;
                const bool clamp = __any_sync(0xffffffffu, !(__fmul_rn(amax, inv) < qm + 0.49f));
                if (x == 0) {
                    const f32x2 inv2 = pk2(inv, inv);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        float a, b;
                        upk2(mul2(p2[i], inv2), a, b);
                        t[2 * i] = __float_as_uint(a);
                        t[2 * i + 1] = __float_as_uint(b);
                    }
                } else {
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        t[q] = __float_as_uint(__fmul_rn(r[q], inv));
                }
                if (clamp) {
#pragma unroll
                    for (int q = 0; q < 16; ++q)
                        t[q] = __float_as_uint(fminf(fmaxf(__uint_as_float(t[q]), -qm), qm));
                }
#pragma unroll
                for (int q = 0; q < 16; ++q)   // (scalar: see above)
                    t[q] = __float_as_uint(__fadd_rn(__uint_as_float(t[q]), 12582912.0f));
            }
            pack_codes<INT4>(t, w);
            if (left) {
                if ((lane & (lpb - 1)) == 0) {
                    if (HALF)
                        ((unsigned short *)scales[x])[base >> shift] = hb;
                    else
                        ((float *)scales[x])[base >> shift] = s;
                }
                uint8_t *dst = codes[x] + (INT4 ? base >> 1 : base);
                if (left == 16u) {
                    if (INT4)
                        *(uint2 *)dst = make_uint2(w[0], w[1]);
                    else
                        *(uint4 *)dst = make_uint4(w[0], w[1], w[NW - 2], w[NW - 1]);
                } else {   // (elements past the end are zero, also the high nibble of an odd last byte)
                    const uint32_t nb = INT4 ? (left + 1) >> 1 : left;
#pragma unroll
                    for (int b = 0; b < NW * 4; ++b)
                        if (b < (int)nb)
                            dst[b] = (uint8_t)(w[b >> 2] >> (8 * (b & 3)));
                }
            }
            if (x + 1 < NS) {
#pragma unroll
                for (int q = 0; q < 16; ++q)   // r - decode(e~)
                    r[q] = __fsub_rn(r[q], __fmul_rn(__fsub_rn(__uint_as_float(t[q]), 12582912.0f), s));
            }
        }
    };
    grid_wait();
#pragma unroll
    for (int i = 0; i < kF16Ring - 1; ++i)
        issue(c0 + i * 8, i);
    int buf = 0;
    for (uint32_t c = c0; c < c1; c += 8) {
        cp_async_wait<kF16Ring - 2>();   // this chunk has landed
        __syncwarp();                    // ... for every lane, and every lane is done with the stage filled next
        issue(c + (kF16Ring - 1) * 8, buf == 0 ? kF16Ring - 1 : buf - 1);
        compute(c, ring[buf]);
        buf = buf + 1 == kF16Ring ? 0 : buf + 1;
    }
    cp_async_wait<0>();
}

// launcher (conef_flat16.cu)
cudaError_t flat16_launch(int qkind, int ckind, int half, const DevView &V, const int32_t *pfx, int tiles, cudaStream_t s);

}  // namespace conef
