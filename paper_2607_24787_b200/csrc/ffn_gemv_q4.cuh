// Slot-indexed SwiGLU expert FFN for decode with 4-bit experts (the paper's on-device setting:
// 4-bit weights, 1.94 MB per DeepSeek-VL2-Tiny expert), one activation row per token.
//
// A blob row j holds the packed gate[j][:], up[j][:] and column j of W_down back to back (q4_mma.cuh has the format). The
// (expert, j) rows of a token are split evenly over the CTAs, as in ffn_gemv_kernel; a CTA takes its rows in tiles of 16, whatever
// experts they belong to, one bulk copy a row.
//
// All arithmetic on weights is mma.sync, with the fp32 operand as the sum of three bf16 numbers (split3) in three columns of N, so
// that nothing is rounded to 16 bits. The warps split the columns in groups of 32 (one scale):
//   Phase 1 (M = eight gate rows and the same up rows; K = the group): the group's scale goes onto the fp32 sum of its 32 products; the warps' sums
// meet in shared memory, a warp takes a row's activation from them.
//   Phase 2 (M = hidden columns, K = the tile's 16 rows): act * scale is the split operand; two groups, whose scales differ, use columns of
// N of their own. y stays in registers for all tiles of the CTA, each column in one warp: no sum over warps.
//
// Why MMAs: with fp32 FMAs the kernel was bound by instruction issue, 27 warp instructions per eight weights and lane, eight of which
// widened halves to floats and eight multiplied; an MMA operand needs nine. A layer of the Qwen3 shape (a step as one kernel; with
// separate launches before) 26.5 -> 18.3 us, of the DeepSeek shape 25.6 -> 16.2; its part of that, 14.6 -> 9 (in rounds of tiles: see q4_tiles).
// What bounds it now: latencies between dependent instructions (half of the issue slots are used), and still instruction issue.
// The tensor cores cut a sum off where fp32 adds round it, always towards zero, so no chain of MMAs is longer than a group (phase 1) or a
// tile (phase 2); longer sums are fp32 adds. (With y in the accumulators for all tiles a CTA of 384 tiles was off by 2.4e-6; 1 % faster.)
// Error against 64 bits, 18 shapes of hidden 256 to 2048, rows that are normal, log-normal, of one sign, with outliers: 0.79 - 0.86 of the
// FMAs' on average, 2.2e-7 of the result at worst (2.7e-7). Activations below 2^-110 lose bits: their third parts end at bf16's last one.
#pragma once

#include <climits>
#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ffn_gemv.cuh"
#include "q4_mma.cuh"
#include "q4_rounds.h"

namespace spm {

// One of the three parts of split3 by a lane that wants only that (p > 2: zero): what is left of a number after the parts before it. What is not
// finite leaves NaNs; guarded: the number itself as the first part, zeros as the others.
struct Q4Part {
    uint32_t m1, m2;               // masks of the parts that go first
    __device__ __forceinline__ explicit Q4Part(int p) : m1(p > 2 ? 0xffffffffu : p >= 1 ? 0xffff0000u : 0u), m2(p >= 2 ? 0xffff0000u : 0u) {}
    template <bool GUARDED>
    __device__ __forceinline__ float left(float v) const {
        float r = v - __uint_as_float(__float_as_uint(v) & m1);
        if (GUARDED && m1 != 0 && !(fabsf(v) < INFINITY)) r = 0.f;
        return r - __uint_as_float(__float_as_uint(r) & m2);
    }
    template <bool GUARDED = false>
    __device__ __forceinline__ uint32_t pair(float a, float b) const {
        return __byte_perm(__float_as_uint(left<GUARDED>(a)), __float_as_uint(left<GUARDED>(b)), 0x7632);
    }
};

// Where the tiles of a CTA are: a ring of stages of kQ4Rows rows, one barrier a stage that completes when all rows of it have been asked for
// and have landed, the phase-1 sums [tile of a round][warps][kQ4Red], gate and up of each row, and the activations [tile of a round][rows].
constexpr int kQ4Red = 33;             // (a lane reads one row's sum of one warp)
static_assert(kQ4MaxStages <= 2 * kQ4Super, "half of a ring is a round");
template <int NW>
struct Q4Ring {
    uint32_t rows, bars, pitch;
    float *red, *act;
    int stages;
    int st = 0, st_in = 0;         // stage of the next tile to use, of the next to fill
    uint32_t ph = 0;
    __device__ __forceinline__ Q4Ring(unsigned char* smem, int D, int n_stages, int thread) : stages(n_stages) {
        pitch = mt_pitch(3 * q4_part_bytes(D), false);
        uint64_t* b = reinterpret_cast<uint64_t*>(smem + size_t(n_stages) * kQ4Rows * pitch);
        rows = smem_u32(smem);
        bars = smem_u32(b);
        red = reinterpret_cast<float*>(b + kQ4MaxStages);
        act = red + (kQ4Super * NW * kQ4Red + 3) / 4 * 4;
        if (thread == 0) {
            for (int s = 0; s < stages; ++s) mbar_init(bars + 8u * s, kQ4Rows);
            fence_barrier_init();
        }
    }
    // The warp's rows (warp, warp + NW) of `count` tiles from `tile` on; row_at(row), called by the whole warp, is null for rows that are
    // not there. The lanes look the rows up side by side, one elected lane asks for them (lanes that ask side by side are taken one by
    // one). `waited`: row_at waits for arrivals, which the lane that waited has seen, but the one that asks reads the bytes: the barrier
    // and the fence hand them on.
    template <typename F>
    __device__ __forceinline__ void fill(int tile, int count, int warp, int lane, uint32_t bytes, bool waited, F row_at) {
        constexpr int kPer = q4_rows_per_warp(NW);
        const int mine = warp + lane % kPer * NW;
        const bool in = lane < count * kPer && mine < kQ4Rows;
        const unsigned long long at = reinterpret_cast<unsigned long long>(row_at(in ? (tile + lane / kPer) * kQ4Rows + mine : INT_MAX));
        if (waited) {
            __syncwarp();
            asm volatile("fence.proxy.async;" ::: "memory");
        }
        for (int k = 0; k < count; ++k) {
#pragma unroll
            for (int r = 0; r < kPer; ++r) {
                const int i = warp + r * NW;
                const unsigned long long src = __shfl_sync(0xffffffffu, at, k * kPer + r);
                if (kQ4Rows % NW != 0 && i >= kQ4Rows) continue;
                if (elect_one()) {
                    if (src) {
                        mbar_arrive_expect_tx(bars + 8u * st_in, bytes);
                        bulk_g2s(rows + uint32_t(st_in * kQ4Rows + i) * pitch, reinterpret_cast<const void*>(src), bytes, bars + 8u * st_in, policy_evict_first());
                    } else {
                        mbar_arrive(bars + 8u * st_in);
                    }
                }
                __syncwarp();
            }
            st_in = st_in + 1 == stages ? 0 : st_in + 1;
        }
    }
};

// B operand of phase 1: the lane's part (N column = part) of the activations of its eight columns in each of the warp's groups.
// get(col, v): eight consecutive fp32 from column col on.
template <int GB, typename F>
__device__ __forceinline__ void q4_operand(uint32_t (&x)[GB][4], int warp, int lane, F get) {
    const int g = lane >> 2, t = lane & 3;
    float v[GB][8], zeros[4] = {0.f, 0.f, 0.f, 0.f};         // (sums of products with zero: NaN where one is not finite)
#pragma unroll
    for (int i = 0; i < GB; ++i) {
        get((warp * GB + i) * 32 + t * 8, v[i]);
#pragma unroll
        for (int q = 0; q < 8; ++q) zeros[q & 3] = fmaf(v[i][q], 0.f, zeros[q & 3]);
    }
    const Q4Part part(g);
    if (__any_sync(0xffffffffu, (zeros[0] + zeros[1]) + (zeros[2] + zeros[3]) != 0.f)) {
#pragma unroll
        for (int i = 0; i < GB; ++i) {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[i][q] = v[i][q] != v[i][q] ? __uint_as_float(0x7fffffffu) : v[i][q];      // (a NaN whose upper half is one too)
#pragma unroll
            for (int q = 0; q < 4; ++q) x[i][q] = part.pair<true>(v[i][q], v[i][q + 4]);
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < GB; ++i)
#pragma unroll
        for (int q = 0; q < 4; ++q) x[i][q] = part.pair(v[i][q], v[i][q + 4]);
}

// The CTA's rows 0 .. span - 1, in rounds of up to four tiles: phase 1 of all of them, the warps' sums meet once, a warp a tile takes the
// activations, phase 2 of all. What bounds a round is the latency between dependent instructions, which several tiles between two barriers
// hide: whole steps of the 4-bit Qwen3 shape (three tiles a CTA), us a layer, 18.1 a tile at a time -> 17.3, DeepSeek shape (four, the last of one
// row) 16.1 -> 13.8. (One barrier a tile, phase 2 a tile behind phase 1: 18.0 and 14.4.) Where the ring holds fewer tiles than the
// CTA has, two neighbouring rounds fill it (q4_rounds.h), so that one is on its way. fill(tile): ask for the warp's rows of a tile; the first
// `stages` tiles have been asked for. weight(row): routing weight. Every thread of the CTA takes part. Returns false, in every
// thread, when a wait ran out (the caller drains and leaves).
template <int GB, int NW, typename Fill, typename Weight>
__device__ __forceinline__ bool q4_tiles(Q4Ring<NW>& ring, const uint32_t (&x)[GB][4], float (&y)[GB][2][4], int D, int span,
                                         int warp, int lane, unsigned long long limit, Fill fill, Weight weight) {
    const int g = lane >> 2, t = lane & 3, grp0 = warp * GB;
    const int tiles = (span + kQ4Rows - 1) / kQ4Rows;
    const uint32_t P = ring.pitch, PART = q4_part_bytes(D);
    Q4Rounds rounds(tiles, ring.stages);
    int before = 0;                  // tiles of the round before
    for (int k = 0; rounds.left > 0;) {
        const int nt = rounds.next(tiles - k);
        int st0 = ring.st;
        auto rows_of = [&](int u) { return ring.rows + uint32_t((st0 + u < ring.stages ? st0 + u : st0 + u - ring.stages) * kQ4Rows) * P; };
        // `whole`: for the case below, a group's three parts added up before the scale goes onto them
        auto phase1 = [&](auto whole, auto blocks, int u) {
            constexpr bool kWhole = decltype(whole)::value;
            constexpr int H = decltype(blocks)::value;
            float acc[H][4];
            q4_phase1<GB, H>(rows_of(u), P, D, grp0, lane, x, acc, [](float (&a)[4], const float (&c)[4], float s0, float s1) {
                if constexpr (kWhole) {
                    float lo = c[0] + c[1], hi = c[2] + c[3];
                    lo += __shfl_xor_sync(0xffffffffu, lo, 1);
                    hi += __shfl_xor_sync(0xffffffffu, hi, 1);
                    a[0] = fmaf(s0, lo, a[0]); a[2] = fmaf(s1, hi, a[2]);
                } else {
                    a[0] = fmaf(s0, c[0], a[0]); a[1] = fmaf(s0, c[1], a[1]);
                    a[2] = fmaf(s1, c[2], a[2]); a[3] = fmaf(s1, c[3], a[3]);
                }
            });
            // columns 0 and 1 are in lane t = 0, column 2 in lane t = 1 (the others hold zeros)
            float* r = ring.red + (u * NW + warp) * kQ4Red + g;
#pragma unroll
            for (int h = 0; h < H; ++h) {
                float vg = acc[h][0] + acc[h][1], vu = acc[h][2] + acc[h][3];
                if constexpr (!kWhole) { vg += __shfl_xor_sync(0xffffffffu, vg, 1); vu += __shfl_xor_sync(0xffffffffu, vu, 1); }
                if (t == 0) { r[8 * h] = vg * kQ4ExactUnscale; r[16 + 8 * h] = vu * kQ4ExactUnscale; }
            }
        };
        // warp u: tile u; even lanes take a row's gate, odd ones its up. True where an activation is not finite.
        auto activations = [&]() -> bool {
            bool odd = false;
            if (warp < nt) {
                const int r = lane >> 1, row = (k + warp) * kQ4Rows + r;
                const float* p = ring.red + warp * NW * kQ4Red + (lane & 1) * 16 + r;
                float sum = 0.f;         // (front to back: the loads overlap, so it takes no longer than shuffles between lanes)
#pragma unroll
                for (int w = 0; w < NW; ++w) sum += p[w * kQ4Red];
                const float up = __shfl_xor_sync(0xffffffffu, sum, 1);
                if ((lane & 1) == 0) {
                    const float act = row < span ? sum / (1.f + expf(-sum)) * up * weight(row) : 0.f;
                    ring.act[warp * kQ4Rows + r] = act;
                    odd = !isfinite(act);
                }
            }
            return odd;
        };
        float a0, a1, a2, a3;            // activations of rows 2t, 2t + 1, 2t + 8, 2t + 9
        auto take = [&](int u) {
            const float* acts = ring.act + u * kQ4Rows;
            const float2 lo = *reinterpret_cast<const float2*>(acts + 2 * t), hi = *reinterpret_cast<const float2*>(acts + 2 * t + 8);
            a0 = lo.x; a1 = lo.y; a2 = hi.x; a3 = hi.y;
        };
        bool ok = true;
        for (int u = 0; u < nt && ok; ++u) {
            ok = __all_sync(0xffffffffu, mbar_wait_bounded(ring.bars + 8u * ring.st, ring.ph, limit));
            if (++ring.st == ring.stages) { ring.st = 0; ring.ph ^= 1; }
            if (span - (k + u) * kQ4Rows > 8) phase1(std::false_type{}, std::integral_constant<int, 2>{}, u);
            else phase1(std::false_type{}, std::integral_constant<int, 1>{}, u);
        }
        if (!__syncthreads_and(ok)) return false;
        // every warp is done with the tiles of the round before this one
        for (int u = k - before; u < k; ++u)
            if (u + ring.stages < tiles) fill(u + ring.stages);
        if (__syncthreads_or(activations())) {
            // An infinite scale times a part that is zero is a NaN where the scale times the sum is an infinity.
            for (int u = 0; u < nt; ++u) {
                take(u);
                if (__any_sync(0xffffffffu, !isfinite(a0 * 0.f + a1 * 0.f + a2 * 0.f + a3 * 0.f)))       // (so in all warps or in none)
                    phase1(std::true_type{}, std::integral_constant<int, 2>{}, u);
            }
            __syncthreads();
            activations();
            __syncthreads();
        }
        for (int u = 0; u < nt; ++u) {
            const int nr = span - (k + u) * kQ4Rows;
            const uint32_t rows = rows_of(u);
            take(u);
            // N columns 0-2: the parts for one group, 4-6: for the next (where there is one)
            const bool second = g >= 4;
            const uint32_t at = rows + 2 * PART + uint32_t((lane & 7) + ((lane >> 3) & 1) * 8) * P + uint32_t(grp0) * 16;
            const uint32_t sc = rows + 2 * PART + uint32_t(2 * t) * P + uint32_t(D / 2 + grp0 * 2);
            float s0[GB], s1[GB], s2[GB], s3[GB];
            q4_scales<GB>(sc, s0);
            q4_scales<GB>(sc + P, s1);
            q4_scales<GB>(sc + 8 * P, s2);
            q4_scales<GB>(sc + 9 * P, s3);
            if (nr < kQ4Rows) {          // rows past the last one hold whatever was there: their activations are 0, so their scales must be finite
#pragma unroll
                for (int i = 0; i < GB; ++i) {
                    s0[i] = 2 * t < nr ? s0[i] : 0.f; s1[i] = 2 * t + 1 < nr ? s1[i] : 0.f;
                    s2[i] = 2 * t + 8 < nr ? s2[i] : 0.f; s3[i] = 2 * t + 9 < nr ? s3[i] : 0.f;
                }
            }
            uint32_t b[(GB + 1) / 2][2];
            const Q4Part part(g & 3);
            auto operand = [&](auto guarded) {
#pragma unroll
                for (int i = 0; i < GB; i += 2) {
                    const int j = i + 1 < GB ? i + 1 : GB - 1;
                    const float v0 = a0 * (second ? s0[j] : s0[i]), v1 = a1 * (second ? s1[j] : s1[i]), v2 = a2 * (second ? s2[j] : s2[i]), v3 = a3 * (second ? s3[j] : s3[i]);
                    b[i / 2][0] = part.pair<decltype(guarded)::value>(v0, v1);
                    b[i / 2][1] = part.pair<decltype(guarded)::value>(v2, v3);
                    if (i + 1 >= GB && second) b[i / 2][0] = b[i / 2][1] = 0u;
                }
            };
            operand(std::false_type{});
            if (q4_any_nonfinite(b)) operand(std::true_type{});
#pragma unroll
            for (int i = 0; i < GB; i += 2) {
                // matrices: rows 0-7 and 8-15 of group i, then of group i + 1; transposed: a lane has four columns of two rows a word
                const uint4 w = ldsm4t(at + uint32_t(i + (i + 1 < GB ? (lane >> 4) : 0)) * 16);
                q4_phase2(y[i], w.x, w.y, b[i / 2][0], b[i / 2][1]);
                if (i + 1 < GB) q4_phase2(y[i + 1 < GB ? i + 1 : i], w.z, w.w, b[i / 2][0], b[i / 2][1]);
            }
        }
        k += nt;
        before = nt;
    }
    return true;
}

// After the last tile: put(column, four consecutive y) for the columns of the warp's groups
template <int GB, typename F>
__device__ __forceinline__ void q4_result(const float (&y)[GB][2][4], int warp, int lane, F put) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int i = 0; i < GB; ++i) {
        float4 o = make_float4(y[i][0][0] + y[i][0][1], y[i][0][2] + y[i][0][3], y[i][1][0] + y[i][1][1], y[i][1][2] + y[i][1][3]);
        o.x += __shfl_xor_sync(0xffffffffu, o.x, 1); o.y += __shfl_xor_sync(0xffffffffu, o.y, 1);
        o.z += __shfl_xor_sync(0xffffffffu, o.z, 1); o.w += __shfl_xor_sync(0xffffffffu, o.w, 1);
        if (t == (i & 1) * 2) put((warp * GB + i) * 32 + g * 4, make_float4(o.x * kQ4ExactUnscale, o.y * kQ4ExactUnscale, o.z * kQ4ExactUnscale, o.w * kQ4ExactUnscale));
    }
}

template <int NSEG, int MAXNB>
__global__ void __launch_bounds__(q4_warps(NSEG) * 32, 1)
ffn_gemv_q4_kernel(const __grid_constant__ FfnArgs<MAXNB> a, const int n_stages) {
    constexpr int D = NSEG * 256, GB = q4_groups(NSEG), NW = q4_warps(NSEG);
    constexpr uint32_t ROWB = 3 * q4_part_bytes(D);
    extern __shared__ __align__(128) unsigned char smem[];
    grid_dep_launch();
    const unsigned long long t_entry = (a.clock && threadIdx.x == 0) ? global_timer_ns() : 0ull;
    const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x) >> 5, 0), lane = threadIdx.x & 31;      // (warp: uniform)
    const int tok = blockIdx.y, G = gridDim.x, c = blockIdx.x, I = a.I;
    const int R = a.entries(tok) * I;
    const int q_rows = R / G, rem_rows = R - q_rows * G;
    const int r_begin = q_rows * c + min(c, rem_rows), span = q_rows + (c < rem_rows ? 1 : 0);
    const unsigned long long limit = a.limit();
    Q4Ring<NW> ring(smem, D, n_stages, threadIdx.x);
    __syncthreads();
    int filled = min(n_stages, (span + kQ4Rows - 1) / kQ4Rows);
    // Everything above is independent of the preceding kernel; with `early` so are the first weight copies (see ffn_gemv_kernel), but for those
    // of shared experts, which are the caller's and may have been written just before. They are the last entries.
    const bool early = a.early && !a.dev_code && (span == 0 || a.code_of(tok, (r_begin + min(span, filled * kQ4Rows) - 1) / I) >= 0);
    auto depend = [&]() {
        grid_dep_wait();
        // window start: kernel entry, or the end of the dependency wait when launched ahead of its predecessor's end
        if (a.clock && threadIdx.x == 0) atomicMin(a.clock, a.dev_code || early ? global_timer_ns() : t_entry);
    };
    if (!early) depend();

    int src_ent = -1;                          // (per lane) entry whose blob was looked up last
    const unsigned char* src_base = nullptr;   // (null: it cannot be served; its rows are skipped)
    bool gave_up = false;
    auto resolve = [&](int ent) -> const unsigned char* {
        const int code = a.code_of(tok, ent);
        if (code < 0) {
            if (-1 - code >= a.n_shared) { atomicOr(a.status, kStatusBadSlot); return nullptr; }
            return a.shared + size_t(-1 - code) * a.blob_bytes;
        }
        if (code >= a.n_slots) { atomicOr(a.status, kStatusBadSlot); return nullptr; }
        // device-side wait for the batch of copies that fills this slot; after one has run out no other is begun
        if (a.ready && (gave_up || !ffn_wait_arrival(a.ready + a.watch[ent], a.want[ent], limit))) {
            gave_up = true;
            atomicOr(a.status, kStatusCopyTimeout);
            return nullptr;
        }
        return a.pool + size_t(code) * a.blob_bytes;
    };
    auto row_at = [&](int row) -> const unsigned char* {
        if (row >= span) return nullptr;
        const int ent = (r_begin + row) / I;
        if (ent != src_ent) { src_ent = ent; src_base = resolve(ent); }
        return src_base ? src_base + size_t(r_begin + row - ent * I) * ROWB : nullptr;
    };
    ring.fill(0, filled, warp, lane, ROWB, a.ready != nullptr, row_at);
    if (early) depend();

    uint32_t x[GB][4];
    const float* xt = a.x + size_t(tok) * D;
    const bool vec = (reinterpret_cast<uintptr_t>(xt) & 15) == 0;       // the caller's rows may start at any float
    q4_operand<GB>(x, warp, lane, [&](int col, float (&v)[8]) {
        if (vec) {
            const float4 lo = *reinterpret_cast<const float4*>(xt + col), hi = *reinterpret_cast<const float4*>(xt + col + 4);
            v[0] = lo.x; v[1] = lo.y; v[2] = lo.z; v[3] = lo.w; v[4] = hi.x; v[5] = hi.y; v[6] = hi.z; v[7] = hi.w;
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = xt[col + q];
        }
    });
    float y[GB][2][4] = {};
    const bool ok = q4_tiles<GB, NW>(ring, x, y, D, span, warp, lane, limit,
        [&](int tile) { ring.fill(tile, 1, warp, lane, ROWB, a.ready != nullptr, row_at); ++filled; },
        [&](int row) {
            const int kk = a.kidx_of(tok, (r_begin + row) / I);
            return kk == 255 ? 1.f : a.w[size_t(tok) * a.K + kk];
        });
    if (!ok) {
        if (lane == 0) atomicOr(a.status, kStatusCopyTimeout);
        // leave no copy in flight into shared memory that is about to be released
        for (int k = max(0, filled - n_stages); k < filled; ++k)
            if (!mbar_wait_bounded(ring.bars + 8u * (k % n_stages), (k / n_stages) & 1, kWaitLimitNs)) break;
    }
    float* out = a.partial + (size_t(tok) * G + c) * D;
    q4_result<GB>(y, warp, lane, [&](int col, float4 v) { *reinterpret_cast<float4*>(out + col) = v; });
    if (a.clock) {
        __syncthreads();
        if (threadIdx.x == 0) atomicMax(a.clock + 1, global_timer_ns());
    }
}

// Ring of a CTA with rows_per_cta rows: all its tiles where they fit beside `reserve` bytes. Returns the bytes of ring, barriers and sums.
inline size_t ffn_gemv_q4_shape(int D, int rows_per_cta, size_t reserve, int* stages) {
    const size_t stage = size_t(kQ4Rows) * mt_pitch(3 * q4_part_bytes(D), false);
    const size_t rest = kQ4MaxStages * 8 + size_t(kQ4Super) * kQ4MaxWarps * kQ4Red * 4 + 16 + size_t(kQ4Super) * kQ4Rows * 4;
    const size_t fit = (kFfnSmemLimit - 1024 - rest - reserve) / stage;
    const int want = rows_per_cta < kQ4Rows ? 1 : (rows_per_cta + kQ4Rows - 1) / kQ4Rows;
    *stages = int(fit < size_t(want) ? fit : size_t(want));
    if (*stages > kQ4MaxStages) *stages = kQ4MaxStages;
    return size_t(*stages) * stage + rest;
}

}  // namespace spm
