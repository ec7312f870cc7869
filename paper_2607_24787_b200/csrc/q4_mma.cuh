// 4-bit weights as mma.sync operands.
//
// A packed row of D weights is D/2 bytes of nibbles (element 2b in the low half of byte b, 2b+1 in the high half) followed by
// D/32 fp16 scales, one per group of 32: weight = scale * (q - 8). Of a 32-bit word of eight nibbles, w & 0x000f000f holds two bf16 numbers
// q * 2^-133 (subnormals: the bits of a bf16 number are linear up to 255) and w & 0x00f000f0 two of 16 q * 2^-133. A packed fma a pair
// takes them to what the other operand is multiplied by: q4_exact to (q - 8) * 2^-6, with the scale left for the sums (fp32 activations),
// q4_weights to the weight rounded to bf16 (bf16 activations). Nine instructions a word of eight; OR-ing in an exponent, subtracting it again
// and shifting three times took eleven. With q itself as the operand and -8 times the sum of the other operand added, five a word did, but
// where that sum is large beside the result (rows of one sign, heavy tails) up to 2.6 times the error of fp32 multiply-adds was left.
#pragma once

#include <cstdint>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "mma_ops.cuh"

namespace spm {

// The 8 * nseg groups of a row (nseg = hidden / 256) are split over the warps evenly, one to four consecutive groups a warp, over as many
// warps as that allows up to sixteen. Fewer warps of more groups each spend fewer instructions on what is done once a tile, but have
// less to hide latencies with (whole steps of the Qwen3 shape, us a layer, eight warps of eight groups -> sixteen of four: one sequence
// 21.9 -> 20.5, 64 sequences 150 -> 142).
constexpr int kQ4MaxWarps = 16;
__host__ __device__ constexpr int q4_groups(int nseg) {
    for (int gb = 1; gb < 4; ++gb)
        if (8 * nseg % gb == 0 && 8 * nseg / gb <= kQ4MaxWarps) return gb;
    return 4;
}
__host__ __device__ constexpr int q4_warps(int nseg) { return 8 * nseg / q4_groups(nseg); }
static_assert(q4_warps(1) == 8 && q4_warps(5) == 10 && q4_warps(7) == 14 && q4_warps(8) == 16, "hidden sizes up to 2048");
__host__ __device__ constexpr int q4_rows_per_warp(int nw) { return (16 + nw - 1) / nw; }
constexpr int kQ4Rows = 16;            // rows of a tile
constexpr int kQ4MaxStages = 8;

__host__ __device__ constexpr uint32_t q4_part_bytes(int D) { return uint32_t(D) / 2 + uint32_t(D) / 16; }      // one packed row

// nibble pairs (i, i + 4), i = 0..3, of a word: even i times 2^-133, odd i times 2^-129
struct Nib4 { uint32_t p[4]; };
__device__ __forceinline__ Nib4 q4_unpack(uint32_t w) {
    const uint32_t h = w >> 8;
    return Nib4{{w & 0x000f000fu, w & 0x00f000f0u, h & 0x000f000fu, h & 0x00f000f0u}};
}
__device__ __forceinline__ __nv_bfloat162 bf2(uint32_t v) { return *reinterpret_cast<const __nv_bfloat162*>(&v); }
__device__ __forceinline__ uint32_t bits2(__nv_bfloat162 v) { return *reinterpret_cast<const uint32_t*>(&v); }
// ... (q - 8) * 2^-6, exact: q 2^-133 * 2^127 - 2^-3
constexpr uint32_t kQ4Up127 = 0x7f007f00u, kQ4Up123 = 0x7d007d00u, kQ4Eight = 0xbe00be00u;      // 2^127, 2^123, -2^-3, twice
constexpr float kQ4ExactUnscale = 64.f;
__device__ __forceinline__ Nib4 q4_exact(uint32_t w) {
    const Nib4 q = q4_unpack(w);
    return Nib4{{bits2(__hfma2(bf2(q.p[0]), bf2(kQ4Up127), bf2(kQ4Eight))), bits2(__hfma2(bf2(q.p[1]), bf2(kQ4Up123), bf2(kQ4Eight))),
                 bits2(__hfma2(bf2(q.p[2]), bf2(kQ4Up127), bf2(kQ4Eight))), bits2(__hfma2(bf2(q.p[3]), bf2(kQ4Up123), bf2(kQ4Eight)))}};
}

// Weights as the tensor cores of ffn_grouped_q4_kernel get them, bf16_rn(bf16_rn(scale) * (q - 8)), times 2^-22: one packed fma on the masked
// nibbles, q 2^-133 * (s 2^111) - 8 s 2^-22, rounds once like that product (all of its operands are exact: s is an fp16 number rounded to
// bf16, at most 2^16). `odd` is `even` over 16. Sums stay at 2^-22 of the result, so results below 2^-100 or so lose bits.
struct Q4Scaled { __nv_bfloat162 even, odd, off; };
constexpr uint32_t kQ4Up111 = 0x77007700u, kQ4Down4 = 0x3d803d80u, kQ4Off = 0xb600b600u, kQ4Down22 = 0x34803480u;      // 2^111, 2^-4, -2^-19, 2^-22, twice
constexpr float kQ4Unscale = 4194304.f;         // 2^22
__device__ __forceinline__ Q4Scaled q4_scaled(__nv_bfloat162 s) {
    const __nv_bfloat162 even = __hmul2(s, bf2(kQ4Up111));
    return Q4Scaled{even, __hmul2(even, bf2(kQ4Down4)), __hmul2(s, bf2(kQ4Off))};
}
__device__ __forceinline__ __nv_bfloat162 q4_bf16_scales(uint32_t halves) { return __float22bfloat162_rn(__half22float2(*reinterpret_cast<const __half2*>(&halves))); }
// PLAIN: subtract, then multiply, for scales that are not finite (the fma would make a NaN of q times infinity minus 8 times infinity)
template <bool PLAIN>
__device__ __forceinline__ Nib4 q4_weights(uint32_t w, const Q4Scaled& s, __nv_bfloat162 plain) {
    if constexpr (PLAIN) {
        Nib4 r;
#pragma unroll
        for (int i = 0; i < 4; ++i) r.p[i] = bits2(__hmul2(__hmul2(bf2(nib_pair(w, i)), plain), bf2(kQ4Down22)));
        return r;
    }
    const Nib4 q = q4_unpack(w);
    return Nib4{{bits2(__hfma2(bf2(q.p[0]), s.even, s.off)), bits2(__hfma2(bf2(q.p[1]), s.odd, s.off)),
                 bits2(__hfma2(bf2(q.p[2]), s.even, s.off)), bits2(__hfma2(bf2(q.p[3]), s.odd, s.off))}};
}
// GB consecutive fp16 scales as pairs of groups (the second half of the last pair is 0 where GB is odd)
template <int GB>
__device__ __forceinline__ void q4_scale_pairs(uint32_t addr, uint32_t (&v)[(GB + 1) / 2]) {
    if constexpr (GB == 4) {
        asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(addr));
    } else if constexpr (GB == 2) {
        v[0] = lds32(addr);
    } else {
#pragma unroll
        for (int i = 0; i < GB; ++i) v[i / 2] = (i & 1) ? v[i / 2] | lds16(addr + 2 * i) << 16 : lds16(addr + 2 * i);
    }
}

// GB consecutive fp16 scales
template <int GB>
__device__ __forceinline__ void q4_scales(uint32_t addr, float (&s)[GB]) {
    if constexpr (GB % 2 == 0) {
        uint32_t v[GB / 2];
        if constexpr (GB == 4) {
            asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v[0]), "=r"(v[1]) : "r"(addr));
        } else {
            v[0] = lds32(addr);
        }
#pragma unroll
        for (int i = 0; i < GB / 2; ++i) {
            const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&v[i]));
            s[2 * i] = f.x; s[2 * i + 1] = f.y;
        }
    } else {
#pragma unroll
        for (int i = 0; i < GB; ++i) s[i] = lds_half(addr + 2 * i);
    }
}

// Phase 1: gate and up (2^-6 of them) of H blocks of eight rows over one warp's groups, for the MMA's eight N columns. A block's gate rows
// are the upper half of M, its up rows the lower, so that the last rows of a share cost blocks of eight and not tiles of sixteen.
// rows: the first row, rows of `pitch` bytes that hold gate, then up; grp0: the warp's first group;
// x: the B operand of each group, four words: nibble pairs 0..3.
// add(acc, c, s0, s1) puts a group's sums c onto acc: gate row g (s0) and up row g (s1).
template <int GB, int H, typename Add>
__device__ __forceinline__ void q4_phase1(uint32_t rows, uint32_t pitch, int D, int grp0, int lane, const uint32_t (&x)[GB][4],
                                          float (&acc)[H][4], Add add) {
    const uint32_t part = q4_part_bytes(D);
    // matrices: gate rows 0-7, up rows 0-7, 16 bytes (a group) each, then those of the next group
    const uint32_t at = rows + uint32_t(lane & 7) * pitch + uint32_t((lane >> 3) & 1) * part + uint32_t(grp0) * 16;
    const uint32_t sc = rows + uint32_t(lane >> 2) * pitch + uint32_t(D / 2 + grp0 * 2);
    float sg[H][GB], su[H][GB];
#pragma unroll
    for (int h = 0; h < H; ++h) {
        q4_scales<GB>(sc + uint32_t(h) * 8 * pitch, sg[h]);
        q4_scales<GB>(sc + uint32_t(h) * 8 * pitch + part, su[h]);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[h][j] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < GB; i += 2)
#pragma unroll
        for (int h = 0; h < H; ++h) {
            const uint4 w = ldsm4(at + uint32_t(h) * 8 * pitch + uint32_t(i + (i + 1 < GB ? (lane >> 4) : 0)) * 16);
            auto group = [&](int j, uint32_t wg, uint32_t wu) {
                const Nib4 a = q4_exact(wg), b = q4_exact(wu);
                float c[4];
                mma_k16_first(c, a.p[0], b.p[0], a.p[1], b.p[1], x[j][0], x[j][1]);
                mma_k16(c, a.p[2], b.p[2], a.p[3], b.p[3], x[j][2], x[j][3]);
                add(acc[h], c, sg[h][j], su[h][j]);
            };
            group(i, w.x, w.y);
            if (i + 1 < GB) group(i + 1 < GB ? i + 1 : i, w.z, w.w);
        }
}

// Phase 2 for one group: y += W_down^T act over the tile's 16 rows (2^-6 of it). lo, hi: transposed matrices of the group's nibbles, rows 0-7
// and 8-15; b0, b1: the activations times the group's scale, rows 2t, 2t + 1 and 2t + 8, 2t + 9. A lane gets the columns 4g .. 4g + 3 of
// the group: y[0][0..1], y[0][2..3], y[1][0..1], y[1][2..3] for N columns 2t, 2t + 1.
__device__ __forceinline__ void q4_phase2(float (&y)[2][4], uint32_t lo, uint32_t hi, uint32_t b0, uint32_t b1) {
    const Nib4 a = q4_exact(lo), b = q4_exact(hi);
    float c0[4], c1[4];
    mma_k16_first(c0, a.p[0], a.p[1], b.p[0], b.p[1], b0, b1);
    mma_k16_first(c1, a.p[2], a.p[3], b.p[2], b.p[3], b0, b1);
#pragma unroll
    for (int i = 0; i < 4; ++i) { y[0][i] += c0[i]; y[1][i] += c1[i]; }
}

// Whether any of a warp's bf16 pairs holds an infinity or a NaN
template <int N>
__device__ __forceinline__ bool q4_any_nonfinite(const uint32_t (&b)[N][2]) {
    __nv_bfloat162 zeros = bf2(0u);            // sums of products with zero
#pragma unroll
    for (int i = 0; i < N; ++i) zeros = __hfma2(bf2(b[i][0]), bf2(0u), __hfma2(bf2(b[i][1]), bf2(0u), zeros));
    return __any_sync(0xffffffffu, (bits2(zeros) & 0x7fff7fffu) != 0);
}

}  // namespace spm
