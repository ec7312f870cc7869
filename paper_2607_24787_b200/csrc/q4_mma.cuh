// 4-bit weights as mma.sync operands.
//
// A packed row of D weights is D/2 bytes of nibbles (element 2b in the low half of byte b, 2b+1 in the high half) followed by
// D/32 fp16 scales, one per group of 32: weight = scale * (q - 8). Of a 32-bit word of eight nibbles, w & 0x000f000f holds two bf16 numbers
// q * 2^-133 (subnormals: the bits of a bf16 number are linear up to 255) and w & 0x00f000f0 two of 16 q * 2^-133, so five
// instructions a word make operands; OR-ing in an exponent, subtracting it again and shifting three times took eleven. The
// other operand is scaled up by a power of two to meet them (below 2^127), that of the odd nibbles by a sixteenth of it. The
// -8 goes in as a C operand: -8 times the sum of the other operand over the group, which an MMA with a constant operand makes.
// The tensor cores multiply bf16 subnormals exactly (probed on B200), so all products are exact in fp32.
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
constexpr uint32_t kQ4OffEven = 0x80088008u, kQ4OffOdd = 0x80808080u;       // -8 and -128 times 2^-133, twice

__host__ __device__ constexpr uint32_t q4_part_bytes(int D) { return uint32_t(D) / 2 + uint32_t(D) / 16; }      // one packed row

// nibble pairs (i, i + 4), i = 0..3, of a word: even i times 2^-133, odd i times 2^-129
struct Nib4 { uint32_t p[4]; };
__device__ __forceinline__ Nib4 q4_unpack(uint32_t w) {
    const uint32_t h = w >> 8;
    return Nib4{{w & 0x000f000fu, w & 0x00f000f0u, h & 0x000f000fu, h & 0x00f000f0u}};
}
// ... the same of q - 8, without an offset to add: for operands that are not finite, where q times them and -8 times them are not
// (q - 8) times them
__device__ __forceinline__ Nib4 q4_unpack_exact(uint32_t w) {
    Nib4 r;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        uint32_t half[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int v = int((w >> (4 * i + 16 * h)) & 15u) - 8;
            half[h] = uint32_t(v < 0 ? 0x8000 : 0) | uint32_t((v < 0 ? -v : v) << (i & 1 ? 4 : 0));
        }
        r.p[i] = half[0] | half[1] << 16;
    }
    return r;
}
template <bool EXACT>
__device__ __forceinline__ Nib4 q4_operands(uint32_t w) {
    if constexpr (EXACT) return q4_unpack_exact(w);
    return q4_unpack(w);
}

// Weights as the tensor cores of ffn_grouped_q4_kernel get them, bf16_rn(bf16_rn(scale) * (q - 8)), times 2^-22: one packed fma on the masked
// nibbles, q 2^-133 * (s 2^111) - 8 s 2^-22, rounds once like that product (all of its operands are exact: s is an fp16 number rounded to
// bf16, at most 2^16). `odd` is `even` over 16.
struct Q4Scaled { __nv_bfloat162 even, odd, off; };
__device__ __forceinline__ __nv_bfloat162 bf2(uint32_t v) { return *reinterpret_cast<const __nv_bfloat162*>(&v); }
__device__ __forceinline__ uint32_t bits2(__nv_bfloat162 v) { return *reinterpret_cast<const uint32_t*>(&v); }
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

// C = {c0, c1, c0, c1}
__device__ __forceinline__ void mma_k16_from(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1, float c0, float c1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %10, %11};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1));
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

// The power of two that takes numbers of at most `bits` (a positive fp32 number's bits) below 2^127, and 2^133 over it. (Beyond
// 2^121 the latter stops at 2^127; such numbers overflow the activation anyway.)
__device__ __forceinline__ int q4_exponent(uint32_t bits) { return min(max(int(bits >> 23) - 127, -1), 120); }
__device__ __forceinline__ float q4_up(int e) { return __uint_as_float(uint32_t(253 - e) << 23); }        // 2^(126 - e)
__device__ __forceinline__ float q4_down(int e) { return __uint_as_float(uint32_t(134 + e) << 23); }      // 2^(7 + e)

// Phase 1 of a tile: gate and up of its rows over one warp's groups, for the MMA's eight N columns.
// rows: the tile's first row, rows of `pitch` bytes that hold gate, then up; grp0: the warp's first group;
// x: the B operand of each group, four words: nibble pairs 0..3; off: the C operand of each group, this lane's columns 2t, 2t + 1.
// add(acc, c, s0, s1) puts a group's sums c onto acc: rows g (s0) and g + 8 (s1).
template <int GB, bool EXACT, typename Add>
__device__ __forceinline__ void q4_phase1(uint32_t rows, uint32_t pitch, int D, int grp0, int lane, const uint32_t (&x)[GB][4], const float (&off)[GB][2],
                                          float (&gate)[4], float (&up)[4], Add add) {
    const uint32_t part = q4_part_bytes(D);
    // matrices: gate rows 0-7, 8-15, up rows 0-7, 8-15, 16 bytes (a group) each
    const uint32_t at = rows + uint32_t((lane & 7) + ((lane >> 3) & 1) * 8) * pitch + uint32_t(lane >> 4) * part + uint32_t(grp0) * 16;
    const uint32_t sc = rows + uint32_t(lane >> 2) * pitch + uint32_t(D / 2 + grp0 * 2);
    float g0[GB], g1[GB], u0[GB], u1[GB];
    q4_scales<GB>(sc, g0);
    q4_scales<GB>(sc + 8 * pitch, g1);
    q4_scales<GB>(sc + part, u0);
    q4_scales<GB>(sc + 8 * pitch + part, u1);
#pragma unroll
    for (int j = 0; j < 4; ++j) gate[j] = up[j] = 0.f;
#pragma unroll
    for (int i = 0; i < GB; ++i) {
        const uint4 w = ldsm4(at + i * 16);
        const Nib4 a = q4_operands<EXACT>(w.x), b = q4_operands<EXACT>(w.y), c = q4_operands<EXACT>(w.z), d = q4_operands<EXACT>(w.w);
        const float o0 = EXACT ? 0.f : off[i][0], o1 = EXACT ? 0.f : off[i][1];
        float cg[4], cu[4];
        mma_k16_from(cg, a.p[0], b.p[0], a.p[1], b.p[1], x[i][0], x[i][1], o0, o1);
        mma_k16_from(cu, c.p[0], d.p[0], c.p[1], d.p[1], x[i][0], x[i][1], o0, o1);
        mma_k16(cg, a.p[2], b.p[2], a.p[3], b.p[3], x[i][2], x[i][3]);
        mma_k16(cu, c.p[2], d.p[2], c.p[3], d.p[3], x[i][2], x[i][3]);
        add(gate, cg, g0[i], g1[i]);
        add(up, cu, u0[i], u1[i]);
    }
}
// ... and its C operand from the B operand
__device__ __forceinline__ void q4_offset(const uint32_t (&x)[4], float (&off)[2]) {
    float c[4];
    mma_k16_first(c, kQ4OffEven, kQ4OffEven, kQ4OffOdd, kQ4OffOdd, x[0], x[1]);
    mma_k16(c, kQ4OffEven, kQ4OffEven, kQ4OffOdd, kQ4OffOdd, x[2], x[3]);
    off[0] = c[0]; off[1] = c[1];
}

// Phase 2 for one group: y += W_down^T act over the tile's 16 rows. lo, hi: transposed matrices of the group's nibbles, rows 0-7 and 8-15;
// b0, b1: the activations times the group's scale, rows 2t, 2t + 1 and 2t + 8, 2t + 9. A lane gets the columns 4g .. 4g + 3 of
// the group: y[0][0..1], y[0][2..3], y[1][0..1], y[1][2..3] for N columns 2t, 2t + 1; the odd ones are sixteen times too large.
template <bool EXACT>
__device__ __forceinline__ void q4_phase2(float (&y)[2][4], uint32_t lo, uint32_t hi, uint32_t b0, uint32_t b1) {
    const Nib4 a = q4_operands<EXACT>(lo), b = q4_operands<EXACT>(hi);
    if constexpr (!EXACT) {
        mma_k16(y[0], kQ4OffEven, kQ4OffOdd, kQ4OffEven, kQ4OffOdd, b0, b1);
        mma_k16(y[1], kQ4OffEven, kQ4OffOdd, kQ4OffEven, kQ4OffOdd, b0, b1);
    }
    mma_k16(y[0], a.p[0], a.p[1], b.p[0], b.p[1], b0, b1);
    mma_k16(y[1], a.p[2], a.p[3], b.p[2], b.p[3], b0, b1);
}

// Whether any of a warp's bf16 pairs holds an infinity or a NaN
template <int N>
__device__ __forceinline__ bool q4_any_nonfinite(const uint32_t (&b)[N][2]) {
    uint32_t top = 0;
#pragma unroll
    for (int i = 0; i < N; ++i) top = __vmaxu2(top, __vmaxu2(b[i][0] & 0x7fff7fffu, b[i][1] & 0x7fff7fffu));
    return __any_sync(0xffffffffu, (top & 0xffffu) >= 0x7f80u || (top >> 16) >= 0x7f80u);
}

// The scale 2^k of phase 2's activations: 2^96 unless an activation of 2^15 or more (65504 is the largest scale) asks for less.
// y is kept in step with it.
struct Q4ActScale {
    float up = 79228162514264337593543950336.f;         // 2^96 ...
    float back = 1.f;                                   // ... and 2^96 over it
    template <int GB>
    __device__ __forceinline__ void fit(float largest, float (&y)[GB][2][4]) {      // largest: of this lane; infinities and NaNs change nothing
        if (!__any_sync(0xffffffffu, largest >= 32768.f)) return;
        const uint32_t bits = __reduce_max_sync(0xffffffffu, isfinite(largest) ? __float_as_uint(largest) : 0u);
        const int e = int(bits >> 23) - 127;
        if (e < 15) return;
        const float want = __uint_as_float(uint32_t(96 - (e - 14) + 127) << 23);       // (e <= 127)
        if (want >= up) return;
        const float step = want / up;                       // both powers of two
        up = want;
        back /= step;
#pragma unroll
        for (int i = 0; i < GB; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int v = 0; v < 4; ++v) y[i][j][v] *= step;
    }
    // four columns of a group from the lane's y of one N column
    __device__ __forceinline__ float4 out(float a, float b, float c, float d) const {
        constexpr float even = 137438953472.f, odd = 8589934592.f;        // 2^(133 - 96) and a sixteenth of it
        return make_float4(a * even * back, b * odd * back, c * even * back, d * odd * back);
    }
};

}  // namespace spm
