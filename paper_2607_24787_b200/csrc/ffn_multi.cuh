// Slot-indexed SwiGLU expert FFN for several sequences with fp32 activations: every expert's weights
// are streamed once per kMtTokens of the tokens that were routed to it.
//
// The batched path where the grouped tcgen05 kernels do not apply (fp32 weights, shared experts, intermediate or hidden
// sizes that do not tile by 128, spm_set_batched_path(1)) and enough expert reads are shared (multi_pays). One GEMV
// per sequence, the other kernel of that path, reads an expert once per token: 16 sequences of the DeepSeek shape
// (1280 x 896, 6 of 64 and 2 shared experts) ask for 880 MB a layer where the distinct experts hold 350 MB.
// Measured there, the kernel's window in a host-free step: 104 us a layer with it, 72 us here (350 MB at the card's copy rate: 54 us; 76 with eight
// warps instead of ten).
//
// Work. An entry is an expert with at most kMtTokens of its tokens. Its rows (row j = gate[j][:], up[j][:] and
// column j of W_down, contiguous in the blob) are taken in blocks of kMtRows; the blocks of all entries, in
// expert order, are split evenly over the CTAs, so a CTA's share is one to a few segments of consecutive
// blocks. A block comes in two ring stages, gate / up rows and W_down rows, with one bulk copy per row and
// rows padded so that eight of them start in different banks.
//
// Arithmetic: mma.sync with operands split so that nothing is rounded to 16 bits. An fp32 activation is the sum
// of three bf16 numbers (8 significant bits each, by truncation, exact); a bf16 or (q - 8) weight is a bf16
// number already and an fp32 weight is split likewise. All products are exact in the tensor core's fp32
// accumulator, which is only trusted with 16 or 32 terms (8 in phase 2) of each part, small parts first, before the
// sum is added to an fp32 register with an ordinary rounded addition. Error against 64 bits over eight shapes of
// all three weight types: 1.9e-7 to 2.2e-7 of the result, with fp32 FMAs (one sequence at a time, sums cut over all 148 CTAs)
// 1.8e-7 to 2.1e-7, geometric mean of the ratio 1.04 (tests/test_gpu_multi.py). With plain fp32 FMAs, columns split over
// the lanes, this kernel needed 944 warp instructions per row of 1280 columns (its rows arrive every 1280 issue slots) and 108 us
// for the layer above; with MMAs about 400.
// mma.sync and not tcgen05: the accumulator has to come back to registers every 16 terms.
//   Phase 1 (M = 8 gate rows over 8 up rows, N = tokens, K = hidden): the warps (eight to twenty) split the columns in groups
// of 32; a lane ends up with gate and up of the same (row, token); the warps' sums meet in shared memory.
//   Phase 2 (M = hidden, N = tokens, K = the block's 8 rows): the same groups of columns; y stays in registers
// for the whole segment and is written once, to slot (segment, token) of `partial`.
//   The phases are one block apart: while the warps' sums of block i become activations, phase 2 of block i - 1
// runs, and one CTA barrier a block is enough. What bounds it now is the chain of latencies of a block: HBM is busy half of
// the time and a quarter of the issue slots are used; with two to three blocks in the ring, copies and arithmetic overlap only in part.
// mt_combine_kernel adds a token's experts in k order, each over its segments in CTA order. Every sum has
// a fixed order given the routing of the whole call, so results are bitwise reproducible. They depend on the call in the last
// bits: how many tokens share an expert picks one of two summation orders (NS), and the even split of all entries' blocks says
// where an expert's sum is cut. (With one GEMV per sequence they depend on the sequence's own routing and nb.)
//
// The routing is turned into entries inside the kernel, by every CTA for itself (counts by shared-memory
// atomics, a prefix sum over the experts, token lists by ballot): 1 - 2 us in place of a planning kernel and
// its launch gap.
#pragma once

#include <type_traits>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "ffn_gemv.cuh"
#include "mma_ops.cuh"

namespace spm {

constexpr int kMtTokens = 8;          // tokens of an entry: N of the MMAs
constexpr int kMtRows = 8;            // rows of a block: gate and up rows together are M of the first MMA
constexpr int kMtMaxStages = 8;
constexpr int kMtMaxPairs = SPM_MAX_BATCH * SPM_MAX_TOPK;

struct Q4Tag {};                      // weight type of packed 4-bit rows

struct MtArgs {
    const unsigned char* pool;      // slot pool of this layer
    const unsigned char* shared;    // shared-expert blobs of this layer (may be null)
    const float* x;                 // [nb][D] router input
    const float* w;                 // [nb][K] routing weights
    float* partial;                 // [(CTAs + entries) * kMtTokens][D], see mt_partial_rows
    int32_t* map;                   // {entries, -, -, -, [nb][SPM_MAX_TOPK][2] of each (token, k) pair entry | position << 16 (< 0: none), and
                                    //   its expert's slot (shared expert s: -1 - s)}
    int* status;
    unsigned long long* clock;      // optional {first CTA past its dependency wait, latest CTA end} in ns (globaltimer)
    const int32_t* dev_ids;         // [nb][K] expert ids left in device memory by the routing kernel, with
    const short* dev_slot;          //   [n] slot of each expert; null: `ids` and `slot` below
    unsigned long long blob_bytes, wait_limit_ns;
    int D, I, K, n, nb, n_slots, n_shared;     // n_shared: 0 in every wave but the first
    short ids[kMtMaxPairs];
    short slot[SPM_MAX_EXPERTS];               // < 0: not in this wave
};

// Even split of R blocks over G CTAs: CTA c takes q blocks, the first R % G one more. (By cost, a block of an entry with
// three MMAs a tile counting 4 : 3 against one with one, the layer above took 83 us instead of 77: a block costs its
// latency, not its MMAs.)
struct MtSplit {
    int q, rem;
    __device__ MtSplit(int R, int G) : q(R / G), rem(R - (R / G) * G) {}
    __device__ int begin(int c) const { return q * c + min(c, rem); }
    __device__ int cta_of(int b) const {
        const int cut = rem * (q + 1);
        return b < cut ? b / (q + 1) : rem + (b - cut) / q;
    }
};

// barrier wait that gives up after a limit, or as soon as another warp of the CTA has given up
__device__ __forceinline__ bool mt_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, unsigned long long limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_timer_ns();
    for (;;) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (global_timer_ns() - t0 > limit_ns) {
            *abort_flag = 1;
            atomicOr(status, kStatusCopyTimeout);
            return false;
        }
    }
}

// Chain of the NS products of one A tile with a B operand's parts, small parts first
template <int NS>
__device__ __forceinline__ void mma_chain_k16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, const uint32_t (&b0)[NS], const uint32_t (&b1)[NS]) {
    mma_k16_first(c, a0, a1, a2, a3, b0[NS - 1], b1[NS - 1]);
#pragma unroll
    for (int p = NS - 2; p >= 0; --p) mma_k16(c, a0, a1, a2, a3, b0[p], b1[p]);
}
template <int NS>
__device__ __forceinline__ void mma_chain_k8(float (&c)[4], uint32_t a0, uint32_t a1, const uint32_t (&b)[NS]) {
    mma_k8_first(c, a0, a1, b[NS - 1]);
#pragma unroll
    for (int p = NS - 2; p >= 0; --p) mma_k8(c, a0, a1, b[p]);
}

// The parts of a B operand {a, b} that a lane holds. NS = 3 (up to eight tokens): all three, the MMAs' N is the token, one
// MMA per part. NS = 1 (up to two tokens): the lane's own, N is part * 2 + token, one MMA for all parts.
template <int NS>
__device__ __forceinline__ void b_parts(float a, float b, int lane, uint32_t (&out)[NS]) {
    const Split3 v = split3(a, b);
    if constexpr (NS == 3) {
#pragma unroll
        for (int p = 0; p < 3; ++p) out[p] = v.part[p];
    } else {
        const int p = lane >> 3;
        out[0] = p == 0 ? v.part[0] : p == 1 ? v.part[1] : p == 2 ? v.part[2] : 0u;
    }
}

// Per weight type: where a lane's operands come from. Lane (g, t) = (lane / 4, lane % 4). A group is 32 columns.
//   weight(part, col) * scale(part, D, group): a value of one matrix's part of a blob row, for mt_plain_y
//   phase1: acc[0..1] += gate row g, acc[2..3] += up row g, for N columns 2t, 2t + 1
//   phase2: y[tile][0..1] += hidden column ycol(g, tile), y[tile][2..3] += ycol(g + 8, tile), for N columns 2t, 2t + 1
// x[kb][q] is the B operand of K-block kb: the activations of columns xcol(t, kb, q, 0 / 1) of the lane's token.
template <typename WT> struct MtWeight;

template <> struct MtWeight<uint16_t> {      // bf16
    static __device__ __forceinline__ float silu(float v) { return __fdividef(v, 1.f + __expf(-v)); }      // (as in the batch-1 kernels of each type)
    static __host__ __device__ constexpr uint32_t part_bytes(int D) { return uint32_t(D) * 2; }
    static __device__ __forceinline__ int xcol(int t, int kb, int q, int half) { return kb * 16 + 2 * t + 8 * q + half; }
    static __device__ __forceinline__ int ycol(int m, int tile) { return tile * 16 + m; }
    static __device__ __forceinline__ float weight(const unsigned char* part, int col) { return __uint_as_float(uint32_t(reinterpret_cast<const uint16_t*>(part)[col]) << 16); }
    static __device__ __forceinline__ float scale(const unsigned char*, int, int) { return 1.f; }
    template <int NS>
    static __device__ __forceinline__ void phase1(uint32_t rows, uint32_t stride, int D, int grp, int lane, const uint32_t (&x)[2][2][NS], float (&acc)[4]) {
        const int mat = lane >> 3;             // matrices: gate k 0-7, up k 0-7, gate k 8-15, up k 8-15
        const uint32_t at = rows + uint32_t(lane & 7) * stride + uint32_t(mat & 1) * part_bytes(D) + uint32_t(grp * 32 + (mat >> 1) * 8) * 2;
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) {
            const uint4 a = ldsm4(at + kb * 32);
            float c[4];
            mma_chain_k16<NS>(c, a.x, a.y, a.z, a.w, x[kb][0], x[kb][1]);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] += c[i];
        }
    }
    template <int NS>
    static __device__ __forceinline__ void phase2(uint32_t rows, uint32_t stride, int, int grp, int lane, float2, const uint32_t (&act)[NS], float (&y)[2][4]) {
        const uint4 a = ldsm4t(rows + uint32_t(lane & 7) * stride + uint32_t(grp * 32 + (lane >> 3) * 8) * 2);
        float c0[4], c1[4];
        mma_chain_k8<NS>(c0, a.x, a.y, act);
        mma_chain_k8<NS>(c1, a.z, a.w, act);
#pragma unroll
        for (int i = 0; i < 4; ++i) { y[0][i] += c0[i]; y[1][i] += c1[i]; }
    }
};

template <> struct MtWeight<float> {         // both operands in three parts: nine products
    static __device__ __forceinline__ float silu(float v) { return __fdividef(v, 1.f + __expf(-v)); }
    static __host__ __device__ constexpr uint32_t part_bytes(int D) { return uint32_t(D) * 4; }
    static __device__ __forceinline__ int xcol(int t, int kb, int q, int half) { return kb * 16 + 2 * t + 8 * q + half; }
    static __device__ __forceinline__ int ycol(int m, int tile) { return tile * 16 + m; }
    static __device__ __forceinline__ float weight(const unsigned char* part, int col) { return reinterpret_cast<const float*>(part)[col]; }
    static __device__ __forceinline__ float scale(const unsigned char*, int, int) { return 1.f; }
    template <int NS>
    static __device__ __forceinline__ void phase1(uint32_t rows, uint32_t stride, int D, int grp, int lane, const uint32_t (&x)[2][2][NS], float (&acc)[4]) {
        const uint32_t at = rows + uint32_t(lane >> 2) * stride + uint32_t(grp * 32 + 2 * (lane & 3)) * 4;
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) {
            Split3 a[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {      // gate k, up k, gate k + 8, up k + 8
                const float2 v = ldsf2(at + uint32_t(i & 1) * part_bytes(D) + kb * 64 + (i >> 1) * 32);
                a[i] = split3(v.x, v.y);
            }
            float c[4];
            mma_k16_first(c, a[0].part[2], a[1].part[2], a[2].part[2], a[3].part[2], x[kb][0][NS - 1], x[kb][1][NS - 1]);
#pragma unroll
            for (int s = NS; s >= 0; --s)      // smallest products first
#pragma unroll
                for (int p = 2; p >= 0; --p)
                    if (s - p >= 0 && s - p < NS)
                        mma_k16(c, a[0].part[p], a[1].part[p], a[2].part[p], a[3].part[p], x[kb][0][s - p], x[kb][1][s - p]);
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[i] += c[i];
        }
    }
    template <int NS>
    static __device__ __forceinline__ void phase2(uint32_t rows, uint32_t stride, int, int grp, int lane, float2, const uint32_t (&act)[NS], float (&y)[2][4]) {
        const uint32_t at = rows + uint32_t(2 * (lane & 3)) * stride + uint32_t(grp * 32 + (lane >> 2)) * 4;
#pragma unroll
        for (int tile = 0; tile < 2; ++tile) {
            Split3 a[2];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                const uint32_t p = at + uint32_t(tile * 16 + i * 8) * 4;
                a[i] = split3(ldsf(p), ldsf(p + stride));
            }
            float c[4];
            mma_k8_first(c, a[0].part[2], a[1].part[2], act[NS - 1]);
#pragma unroll
            for (int s = NS; s >= 0; --s)
#pragma unroll
                for (int p = 2; p >= 0; --p)
                    if (s - p >= 0 && s - p < NS) mma_k8(c, a[0].part[p], a[1].part[p], act[s - p]);
#pragma unroll
            for (int i = 0; i < 4; ++i) y[tile][i] += c[i];
        }
    }
};

template <> struct MtWeight<Q4Tag> {         // (q - 8) through the MMA, a group's scale on its fp32 sum (phase 1) or on the activation (phase 2)
    static __device__ __forceinline__ float silu(float v) { return v / (1.f + expf(-v)); }
    static __host__ __device__ constexpr uint32_t part_bytes(int D) { return uint32_t(D) / 2 + uint32_t(D) / 16; }
    // lane t's K positions are the eight weights of word t of the group's 16 bytes, in the order they unpack
    static __device__ __forceinline__ int xcol(int t, int kb, int q, int half) { return t * 8 + 2 * kb + q + 4 * half; }
    // ... and its M positions four nibbles of half a word
    static __device__ __forceinline__ int ycol(int m, int tile) { return (m & 3) * 8 + ((m >> 2) & 1) * 4 + 2 * tile + (m >> 3); }
    static __device__ __forceinline__ float weight(const unsigned char* part, int col) { return float(((part[col >> 1] >> (4 * (col & 1))) & 15) - 8); }
    static __device__ __forceinline__ float scale(const unsigned char* part, int D, int grp) { return __half2float(reinterpret_cast<const __half*>(part + D / 2)[grp]); }
    template <int NS>
    static __device__ __forceinline__ void phase1(uint32_t rows, uint32_t stride, int D, int grp, int lane, const uint32_t (&x)[2][2][NS], float (&acc)[4]) {
        const uint32_t row = rows + uint32_t(lane >> 2) * stride, PART = part_bytes(D);
        const uint32_t wg = lds32(row + grp * 16 + (lane & 3) * 4), wu = lds32(row + PART + grp * 16 + (lane & 3) * 4);
        const float sg = lds_half(row + D / 2 + grp * 2), su = lds_half(row + PART + D / 2 + grp * 2);
        // (one chain, small parts of both halves first: a rounding less than two chains and a sum)
        float c[4];
#pragma unroll
        for (int p = NS - 1; p >= 0; --p)
#pragma unroll
            for (int kb = 0; kb < 2; ++kb) {
                const uint32_t a0 = nib_pair(wg, 2 * kb), a1 = nib_pair(wu, 2 * kb), a2 = nib_pair(wg, 2 * kb + 1), a3 = nib_pair(wu, 2 * kb + 1);
                if (p == NS - 1 && kb == 0) mma_k16_first(c, a0, a1, a2, a3, x[kb][0][p], x[kb][1][p]);
                else mma_k16(c, a0, a1, a2, a3, x[kb][0][p], x[kb][1][p]);
            }
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = fmaf(i < 2 ? sg : su, c[i], acc[i]);
    }
    template <int NS>
    static __device__ __forceinline__ void phase2(uint32_t rows, uint32_t stride, int D, int grp, int lane, float2 act, const uint32_t (&)[NS], float (&y)[2][4]) {
        const int g = lane >> 2;
        const uint32_t row = rows + uint32_t(2 * (lane & 3)) * stride;
        const uint32_t at = row + grp * 16 + (g & 3) * 4 + (g >> 2) * 2, sc = row + D / 2 + grp * 2;
        const uint32_t w = lds16(at) | (lds16(at + stride) << 16);          // four nibbles of row 2t, four of row 2t + 1
        uint32_t b[NS];
        b_parts<NS>(act.x * lds_half(sc), act.y * lds_half(sc + stride), lane, b);
#pragma unroll
        for (int tile = 0; tile < 2; ++tile) {
            float c[4];
            mma_chain_k8<NS>(c, nib_pair(w, 2 * tile), nib_pair(w, 2 * tile + 1), b);
#pragma unroll
            for (int i = 0; i < 4; ++i) y[tile][i] += c[i];
        }
    }
};

template <typename WT, int GB, int NW>       // GB: groups of 32 columns per warp; NW: warps
__global__ void __launch_bounds__(NW * 32, 1)
ffn_multi_kernel(const __grid_constant__ MtArgs a, const int n_stages) {
    static_assert(NW >= kMtRows && NW % 2 == 0, "a warp feeds, and sums up, a row of a block");
    constexpr int kMtWarps = NW, kMtThreads = NW * 32;
    using W = MtWeight<WT>;
    extern __shared__ __align__(128) unsigned char smem[];
    const int D = a.D, I = a.I, n = a.n, n_pairs = a.nb * a.K, n_grp = D / 32;
    const uint32_t PART = W::part_bytes(D), GU = mt_pitch(2 * PART, sizeof(WT) == 4), DN = mt_pitch(PART, sizeof(WT) == 4);      // row pitches
    const uint32_t dn_ring = uint32_t(n_stages) * kMtRows * GU;                // the gate / up ring, then the W_down ring
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + dn_ring + uint32_t(n_stages) * kMtRows * DN);
    float* red = reinterpret_cast<float*>(bars + 2 * kMtMaxStages);            // [2][warps][128] phase-1 sums
    float* actv = red + 2 * kMtWarps * 128;                                    // [2][token][row]
    int* start = reinterpret_cast<int*>(actv + 2 * kMtTokens * kMtRows);           // [n] tokens of each expert, then its first entry
    int& s_entries = start[n];
    int& s_routed = start[n + 1];
    int& s_abort = start[n + 2];
    short* ids = reinterpret_cast<short*>(start + n + 4);                      // [n_pairs]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t ring = smem_u32(smem), gu_bar = smem_u32(bars), dn_bar = gu_bar + 8 * kMtMaxStages;

    grid_dep_launch();
    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) { mbar_init(gu_bar + 8 * s, kMtRows); mbar_init(dn_bar + 8 * s, kMtRows); }
        s_abort = 0;
        fence_barrier_init();
    }
    for (int e = threadIdx.x; e < n; e += kMtThreads) start[e] = 0;

    const bool early = a.dev_ids == nullptr;
    const int per_shared = (a.nb + kMtTokens - 1) / kMtTokens, NB = (I + kMtRows - 1) / kMtRows;
    const unsigned long long limit = a.wait_limit_ns ? a.wait_limit_ns : kWaitLimitNs;
    int n_routed = 0, b_begin = 0, steps = 0;
    // expert of an entry (>= n: shared expert) and which run of kMtTokens of its tokens it holds
    auto expert_of = [&](int u, int& chunk) -> int {
        if (u >= n_routed) {
            const int s = (u - n_routed) / per_shared;
            chunk = u - n_routed - s * per_shared;
            return n + s;
        }
        int lo = 0, hi = n;             // last expert whose first entry is <= u (experts without tokens share their successor's number)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (start[mid] <= u) lo = mid; else hi = mid;
        }
        chunk = u - start[lo];
        return lo;
    };

    // ---- The warps also fill the rings, warp i row i of every block. (All of a block's copies from one warp held up the
    // block's barrier: 112 us a layer.)
    struct Feed { int n, st, u, row; const unsigned char* src; };     // blocks issued, stage of the next, its entry, this warp's row of it
    Feed fgu{}, fdn{};
    const uint64_t pol = policy_evict_first();
    bool feeding = false;
    auto feed = [&](Feed& f, uint32_t ring_at, uint32_t bar, uint32_t pitch, uint32_t off, uint32_t bytes) {
        if (!feeding || f.n >= steps || warp >= kMtRows) return;
        if (!f.src || f.row >= NB * kMtRows) {
            if (f.src) { ++f.u; f.row = warp; }
            int chunk;
            const int e = expert_of(f.u, chunk);
            if (e >= n) {
                f.src = a.shared + size_t(e - n) * a.blob_bytes;
            } else {
                const int slot = a.dev_slot ? a.dev_slot[e] : a.slot[e];
                if (slot < 0 || slot >= a.n_slots) {        // nothing more is issued; every wait of the CTA ends once the flag is seen
                    if (lane == 0) { atomicOr(a.status, kStatusBadSlot); *reinterpret_cast<volatile int*>(&s_abort) = 1; }
                    feeding = false;
                    return;
                }
                f.src = a.pool + size_t(slot) * a.blob_bytes;
            }
        }
        if (elect_one()) {
            if (f.row < I) {
                mbar_arrive_expect_tx(bar + 8 * f.st, bytes);
                bulk_g2s(ring_at + uint32_t(f.st * kMtRows + warp) * pitch, f.src + size_t(f.row) * (3 * PART) + off, bytes, bar + 8 * f.st, pol);
            } else {
                mbar_arrive(bar + 8 * f.st);
            }
        }
        __syncwarp();
        ++f.n;
        f.row += kMtRows;
        f.st = f.st + 1 == n_stages ? 0 : f.st + 1;
    };
    auto feed_gu = [&]() { feed(fgu, ring, gu_bar, GU, 0, 2 * PART); };
    auto feed_dn = [&]() { feed(fdn, ring + dn_ring, dn_bar, DN, 2 * PART, PART); };
    const int g = lane >> 2, t = lane & 3;
    // a warp's groups are warp, warp + NW, ...: the same number for every warp but with fp32 weights, where a
    // warp without a last group computes group 0 there and drops it: straight-line code, so that the MMA chains interleave.
    const bool has_last = sizeof(WT) != 4 || warp + (GB - 1) * kMtWarps < n_grp;
    const int last_grp = has_last ? warp + (GB - 1) * kMtWarps : 0;
    bool dead = false;
    int st1 = 0, st2 = 0;                     // stages of the next block in either ring, and their phases
    uint32_t ph1 = 0, ph2 = 0;

    // One segment: `seg` blocks from block blk0 of entry u on, this CTA's blocks k, k + 1, ...; `mine`: see below
    auto segment = [&](auto parts, int k, int u, int blk0, int seg, int e, int ntok, int mine) {
        constexpr int NS = decltype(parts)::value;
        uint32_t x[GB][2][2][NS];
        float y[GB][2][4];
        const int n_tok = NS == 3 ? g : g & 1;             // token of this lane's N column as a B operand
        {
            const int p = __shfl_sync(0xffffffffu, mine, min(n_tok, ntok - 1));
            const float* xt = a.x + size_t(e >= n ? p : p / a.K) * D;
#pragma unroll
            for (int i = 0; i < GB; ++i) {
                const int grp = warp + i * kMtWarps;
                const bool on = grp < n_grp && n_tok < ntok;
#pragma unroll
                for (int kb = 0; kb < 2; ++kb)
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        b_parts<NS>(on ? xt[grp * 32 + W::xcol(t, kb, q, 0)] : 0.f, on ? xt[grp * 32 + W::xcol(t, kb, q, 1)] : 0.f, lane, x[i][kb][q]);
#pragma unroll
                for (int tile = 0; tile < 2; ++tile)
#pragma unroll
                    for (int v = 0; v < 4; ++v) y[i][tile][v] = 0.f;
            }
        }
        // Role in the meeting of the warps' phase-1 sums: warp i < 8 does row i. NS = 3: eight tokens, gate or up, half of the
        // warps each. NS = 1: two tokens, gate or up, the three parts of every eighth warp each.
        const int m_row = warp, m_tok = lane & (NS == 3 ? 7 : 1), m_up = (lane >> (NS == 3 ? 3 : 1)) & 1;
        const float* m_at = red + (NS == 3 ? (lane >> 4) * (kMtWarps / 2) * 128 + (m_row * 4 + (m_tok >> 1)) * 4 + (m_tok & 1) + 2 * m_up
                                           : (lane >> 2) * 128 + m_row * 16 + m_tok + 2 * m_up);
        const int wp = __shfl_sync(0xffffffffu, mine, min(m_tok, ntok - 1));
        const float wt = e >= n ? 1.f : a.w[wp];
        const float* act_at = actv + n_tok * kMtRows + 2 * t;
        // phase 1 of block s and phase 2 of block s - 1 side by side, one barrier in between
        auto step = [&](auto first, auto last, int s) {         // `first` / `last`: no phase 2 / no phase 1 (straight-line code in between)
            constexpr bool kP1 = !decltype(last)::value, kP2 = !decltype(first)::value;
            const int i1 = k + s, i2 = i1 - 1;                  // numbers of the two blocks in this CTA's share
            const int nr1 = I - (blk0 + s) * kMtRows;           // rows left in the expert from block i1 on
            if constexpr (kP1) {
                if (!dead) dead = !__all_sync(0xffffffffu, mt_wait(gu_bar + 8 * st1, ph1, &s_abort, a.status, limit));
                const uint32_t rows = ring + uint32_t(st1) * kMtRows * GU;
                if (++st1 == n_stages) { st1 = 0; ph1 ^= 1; }
                float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                for (int i = 0; i + 1 < GB; ++i) W::template phase1<NS>(rows, GU, D, warp + i * kMtWarps, lane, x[i], acc);
                if constexpr (sizeof(WT) == 4) {
                    float end[4] = {0.f, 0.f, 0.f, 0.f};
                    W::template phase1<NS>(rows, GU, D, last_grp, lane, x[GB - 1], end);
#pragma unroll
                    for (int i = 0; i < 4; ++i) acc[i] += has_last ? end[i] : 0.f;
                } else {
                    W::template phase1<NS>(rows, GU, D, last_grp, lane, x[GB - 1], acc);
                }
                *reinterpret_cast<float4*>(red + (i1 & 1) * kMtWarps * 128 + warp * 128 + lane * 4) = make_float4(acc[0], acc[1], acc[2], acc[3]);
            }
            if constexpr (kP2) {
                if (!dead) dead = !__all_sync(0xffffffffu, mt_wait(dn_bar + 8 * st2, ph2, &s_abort, a.status, limit));
                const int nr2 = nr1 + kMtRows;
                if (nr2 < kMtRows) {        // rows past the expert's last one: their activations are 0, so their W_down must be finite
                    for (int i = threadIdx.x; i < (kMtRows - nr2) * int(PART / 16); i += kMtThreads) {
                        const int r = i / int(PART / 16), o = i - r * int(PART / 16);
                        *reinterpret_cast<uint4*>(smem + dn_ring + uint32_t(st2 * kMtRows + nr2 + r) * DN + o * 16) = make_uint4(0, 0, 0, 0);
                    }
                    fence_proxy_async();    // ordered before the copy that refills the stage
                }
            }
            __syncthreads();
            // every warp is done with the gate / up rows of block i1 and with the W_down rows of block i2 - 1
            if (!dead) {
                if constexpr (kP1) feed_gu();
                if (i1 >= 2 && fdn.n < i1 - 1 + n_stages) feed_dn();
            }
            if (kP1 && warp < kMtRows) {
                float v;
                const float* from = m_at + (i1 & 1) * (kMtWarps * 128);
                if constexpr (NS == 3) {
                    // Pairs first: a chain over more warps rounds more often. Error against 64 bits, mean of 22 shapes: chains over eight
                    // warps 2.151e-7, over as many as now 2.159e-7 (3 % more on some shapes), in pairs 2.125e-7; and a shorter chain of
                    // latencies (0.5 us a layer).
                    float p[kMtWarps / 2];
#pragma unroll
                    for (int i = 0; i < kMtWarps / 2; ++i) p[i] = from[i * 128];
#pragma unroll
                    for (int d = 1; d < kMtWarps / 2; d *= 2)
#pragma unroll
                        for (int i = 0; i + d < kMtWarps / 2; i += 2 * d) p[i] += p[i + d];
                    v = p[0];
                } else {
                    v = 0.f;
#pragma unroll
                    for (int w = 0; w < kMtWarps; w += 8) {
                        const bool on = kMtWarps % 8 == 0 || w + (lane >> 2) < kMtWarps;
                        float p = 0.f;
#pragma unroll
                        for (int i = 0; i < 3; ++i) p += on ? from[w * 128 + i * 4] : 0.f;
                        v += p;
                    }
                }
                if constexpr (NS == 1) {
                    v += __shfl_xor_sync(0xffffffffu, v, 4);
                    v += __shfl_xor_sync(0xffffffffu, v, 8);
                }
                v += __shfl_xor_sync(0xffffffffu, v, 16);
                const float up = __shfl_xor_sync(0xffffffffu, v, NS == 3 ? 8 : 2);
                if (lane < (NS == 3 ? 8 : 2))
                    actv[(i1 & 1) * kMtTokens * kMtRows + m_tok * kMtRows + m_row] = m_row < nr1 && m_tok < ntok ? W::silu(v) * up * wt : 0.f;
            }
            if constexpr (kP2) {
                const float2 act = *reinterpret_cast<const float2*>(act_at + (i2 & 1) * kMtTokens * kMtRows);
                uint32_t actb[NS];
                b_parts<NS>(act.x, act.y, lane, actb);
                const uint32_t rows = ring + dn_ring + uint32_t(st2) * kMtRows * DN;
#pragma unroll
                for (int i = 0; i < GB; ++i) W::template phase2<NS>(rows, DN, D, i + 1 < GB ? warp + i * kMtWarps : last_grp, lane, act, actb, y[i]);
                if (++st2 == n_stages) { st2 = 0; ph2 ^= 1; }
            }
        };
        using T = std::true_type;
        using F = std::false_type;
        step(T{}, F{}, 0);
        for (int s = 1; s < seg; ++s) step(F{}, F{}, s);
        step(F{}, T{}, seg);
        float* out = a.partial + size_t(int(blockIdx.x) + u) * kMtTokens * D;
#pragma unroll
        for (int i = 0; i < GB; ++i) {
            const int grp = warp + i * kMtWarps;
#pragma unroll
            for (int tile = 0; tile < 2; ++tile)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    float o = y[i][tile][v];
                    int tl = 2 * t + (v & 1);
                    if constexpr (NS == 1) {                // the parts' sums are in the lanes t = 0, 1, 2 (3: zero)
                        o += __shfl_xor_sync(0xffffffffu, o, 1);
                        o += __shfl_xor_sync(0xffffffffu, o, 2);
                        tl = t == 0 ? v & 1 : kMtTokens;
                    }
                    if (tl < ntok && grp < n_grp) out[size_t(tl) * D + grp * 32 + W::ycol(g + 8 * (v >> 1), tile)] = o;
                }
        }
    };

    // With the routing among the launch arguments the plan and the first weight copies need not wait for the preceding kernel.
    auto depend = [&]() {
        grid_dep_wait();
        if (a.clock && threadIdx.x == 0) atomicMin(a.clock, global_timer_ns());
    };
    if (!early) depend();
    __syncthreads();
    for (int i = threadIdx.x; i < n_pairs; i += kMtThreads) {
        int e = a.dev_ids ? __ldcg(a.dev_ids + i) : int(a.ids[i]);
        if (!a.dev_ids && a.slot[e] < 0) e = -1;
        ids[i] = short(e);
        if (e >= 0) atomicAdd(&start[e], 1);
    }
    __syncthreads();
    if (warp == 0) {            // tokens per expert -> entries before the expert
        int run = 0;
        for (int e0 = 0; e0 < n; e0 += 32) {
            const int e = e0 + lane;
            const int c = e < n ? (start[e] + kMtTokens - 1) / kMtTokens : 0;
            int pc = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, pc, o);
                if (lane >= o) pc += t;
            }
            if (e < n) start[e] = run + pc - c;
            run += __shfl_sync(0xffffffffu, pc, 31);
        }
        if (lane == 0) { s_routed = run; s_entries = run + a.n_shared * per_shared; }
    }
    __syncthreads();
    const int U = s_entries;
    n_routed = s_routed;
    const MtSplit split(U * NB, int(gridDim.x));
    b_begin = split.begin(int(blockIdx.x));
    steps = split.begin(int(blockIdx.x) + 1) - b_begin;
    fgu.u = b_begin / NB;
    fgu.row = (b_begin - fgu.u * NB) * kMtRows + warp;
    fdn = fgu;
    feeding = true;
    for (int i = 0; i < n_stages; ++i) { feed_gu(); feed_dn(); }
    if (early) depend();                 // activations and routing weights come from the preceding kernel

    if (blockIdx.x == 0) {
        if (threadIdx.x == 0) a.map[0] = s_entries;
        for (int i = threadIdx.x; i < a.nb * SPM_MAX_TOPK; i += kMtThreads) {
            const int t = i / SPM_MAX_TOPK, k = i % SPM_MAX_TOPK;
            if (k < a.K ? ids[t * a.K + k] < 0 : k >= a.K + a.n_shared) a.map[4 + 2 * i] = -1;      // not in this wave
        }
    }
    for (int k = 0; k < steps;) {
        const int b = b_begin + k, u = b / NB, blk0 = b - u * NB, seg = min(steps - k, NB - blk0);
        int chunk;
        const int e = expert_of(u, chunk);
        int ntok, mine = 0;           // lane l < ntok: pair (routed) or token (shared) of position l, in (token, k) order
        if (e >= n) {
            ntok = min(kMtTokens, a.nb - chunk * kMtTokens);
            mine = chunk * kMtTokens + min(lane, ntok - 1);
        } else {
            const int lo = chunk * kMtTokens;
            int seen = 0;
            for (int i0 = 0; i0 < n_pairs && seen < lo + kMtTokens; i0 += 32) {
                const unsigned m = __ballot_sync(0xffffffffu, i0 + lane < n_pairs && ids[i0 + lane] == e);
                const int want = lo + lane - seen, c = __popc(m);          // this lane's position inside this word of pairs
                if (want >= 0 && want < c && lane < kMtTokens) mine = i0 + int(__fns(m, 0, want + 1));
                seen += c;
            }
            ntok = min(kMtTokens, seen - lo);
        }
        if (blk0 == 0 && warp == 0 && lane < ntok) {        // the CTA with an entry's first block says where its pairs are
            const int tk = e >= n ? mine : mine / a.K, kk = e >= n ? a.K + (e - n) : mine - tk * a.K;
            int32_t* pair = a.map + 4 + 2 * (tk * SPM_MAX_TOPK + kk);
            pair[0] = u | (lane << 16);
            pair[1] = e >= n ? n - 1 - e : a.dev_slot ? a.dev_slot[e] : a.slot[e];
        }
        if (ntok <= 2) segment(std::integral_constant<int, 1>{}, k, u, blk0, seg, e, ntok, mine);
        else segment(std::integral_constant<int, 3>{}, k, u, blk0, seg, e, ntok, mine);
        k += seg;
    }
    // Wind-down after a wait ran out or a slot was bad: leave no copy in flight into shared memory that is about to be
    // released. (The flag is raised ahead of a barrier of the loop above, so the whole CTA sees it here.) A warp that gave up
    // stopped feeding, others went on until they saw the flag, and a stage completes only with the arrivals of all eight warps:
    // the warps agree on the last block that any of them fed and arrive, without a copy, for the blocks up to it. Such
    // a block's stage is free to take them: whoever fed the block had waited for the stage's block before it.
    if (*reinterpret_cast<volatile int*>(&s_abort)) {
        __syncthreads();
        if (threadIdx.x == 0) { s_entries = 0; s_routed = 0; }
        __syncthreads();
        if (lane == 0) { atomicMax(&s_entries, fgu.n); atomicMax(&s_routed, fdn.n); }
        __syncthreads();
        const int n_gu = s_entries, n_dn = s_routed;
        if (warp < kMtRows && elect_one()) {
            for (int i = fgu.n; i < n_gu; ++i) mbar_arrive(gu_bar + 8 * (i % n_stages));
            for (int i = fdn.n; i < n_dn; ++i) mbar_arrive(dn_bar + 8 * (i % n_stages));
        }
        // the drain has a bound of its own: a short limit of the caller must not end it early
        const unsigned long long t0 = global_timer_ns();
        auto drain = [&](uint32_t bar, int n_fed) {
            for (int i = max(0, n_fed - n_stages); i < n_fed; ++i) {
                const unsigned long long spent = global_timer_ns() - t0;
                mbar_wait_bounded(bar + 8 * (i % n_stages), (i / n_stages) & 1, spent < kWaitLimitNs ? kWaitLimitNs - spent : 0);
            }
        };
        drain(gu_bar, n_gu);
        drain(dn_bar, n_dn);
    }
    if (a.clock) {
        __syncthreads();
        if (threadIdx.x == 0) atomicMax(a.clock + 1, global_timer_ns());
    }
}

// Four columns of one token's y of one expert by plain fp32 multiply-adds, one warp together: the sums that the GEMV per
// sequence takes. For operands that are not finite. The split arithmetic marks those (its result is Inf or NaN: no finite
// sum contains one) but does not keep them apart: an infinity times an empty lower part of the other operand is NaN, and
// a NaN whose payload is in its low 16 bits is an infinity in the first part. (Behind the segments in ffn_multi_kernel, the
// same code cost the hot loop up to 60 registers; here it costs nothing.)
template <typename WT>
__device__ __noinline__ float4 mt_plain_y(const unsigned char* blob, int I, int D, const float* x, float wt, int d) {
    using W = MtWeight<WT>;
    const uint32_t PART = W::part_bytes(D);
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int j = 0; j < I; ++j) {
        const unsigned char *gate = blob + size_t(j) * (3 * PART), *up = gate + PART, *down = up + PART;
        float pg = 0.f, pu = 0.f;
        for (int g = int(threadIdx.x & 31); g < D / 32; g += 32) {
            float dg = 0.f, du = 0.f;
            for (int i = g * 32; i < g * 32 + 32; ++i) {
                dg = fmaf(W::weight(gate, i), x[i], dg);
                du = fmaf(W::weight(up, i), x[i], du);
            }
            pg = fmaf(W::scale(gate, D, g), dg, pg);
            pu = fmaf(W::scale(up, D, g), du, pu);
        }
        pg = warp_sum(pg);
        pu = warp_sum(pu);
        if (d < D) {
            const float s = W::silu(pg) * pu * wt * W::scale(down, D, d / 32);
            y.x = fmaf(s, W::weight(down, d), y.x);
            y.y = fmaf(s, W::weight(down, d + 1), y.y);
            y.z = fmaf(s, W::weight(down, d + 2), y.z);
            y.w = fmaf(s, W::weight(down, d + 3), y.w);
        }
    }
    return y;
}

struct MtCombineArgs {
    const float* partial;
    const int32_t* map;
    float* h;                       // [nb][D]
    const unsigned char *pool, *shared;
    const float *x, *w;             // as in MtArgs
    unsigned long long* clock;
    unsigned long long blob_bytes;
    int KS, G, I, D, K, n_slots, n_shared;      // KS: experts of a token in this wave's launch (K + shared), G: CTAs of ffn_multi_kernel
};

// h[t][d] += sum over the token's experts of this wave, in k order, of their segments' partial rows in CTA order.
// Block = (32 groups of four columns) x (K + n_shared experts); kMtAhead loads of a thread are in flight together.
constexpr int kMtAhead = 8;
template <typename WT>
static __global__ void mt_combine_kernel(const __grid_constant__ MtCombineArgs a) {
    __shared__ float4 part[SPM_MAX_TOPK][32];
    grid_dep_launch();
    grid_dep_wait();
    if (a.clock && threadIdx.x == 0) atomicMin(a.clock, global_timer_ns());
    const int D = a.D, t = blockIdx.y, c = threadIdx.x & 31, k = threadIdx.x >> 5;
    const int d = (blockIdx.x * 32 + c) * 4;
    // (the number of entries and the residual are on their way with the pair's place: where they are needed they would cost a latency each:
    // 0.1 - 0.8 us a layer, fp32 1024 x 250 49 -> 47.6)
    const int32_t code = a.map[4 + 2 * (t * SPM_MAX_TOPK + k)], entries = a.map[0];
    float* hp = a.h + size_t(t) * D + d;
    const bool mine = k == 0 && d < D, vec = (reinterpret_cast<uintptr_t>(hp) & 15) == 0;       // the caller's rows may start at any float (spm_moe_ffn)
    float4 tot = make_float4(0.f, 0.f, 0.f, 0.f), acc = tot;
    if (mine) tot = vec ? *reinterpret_cast<const float4*>(hp) : make_float4(hp[0], hp[1], hp[2], hp[3]);
    if (code >= 0 && d < D) {
        const int u = code & 0xffff, tl = code >> 16, NB = (a.I + kMtRows - 1) / kMtRows;
        const MtSplit split(entries * NB, a.G);
        const int c0 = split.cta_of(u * NB), total = split.cta_of(u * NB + NB - 1) - c0 + 1;
        const float* p = a.partial + (size_t(c0 + u) * kMtTokens + size_t(tl)) * D + d;
        for (int i0 = 0; i0 < total; i0 += kMtAhead) {
            float4 v[kMtAhead];
#pragma unroll
            for (int i = 0; i < kMtAhead; ++i)
                v[i] = i0 + i < total ? __ldcg(reinterpret_cast<const float4*>(p + size_t(i0 + i) * kMtTokens * D)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < kMtAhead; ++i) { acc.x += v[i].x; acc.y += v[i].y; acc.z += v[i].z; acc.w += v[i].w; }
        }
    }
    if (code >= 0) {            // (one pair per warp)
        const float probe = fmaf(acc.x, 0.f, fmaf(acc.y, 0.f, fmaf(acc.z, 0.f, acc.w * 0.f)));       // NaN unless all four are finite
        if (__any_sync(0xffffffffu, probe != 0.f)) {
            const int slot = a.map[5 + 2 * (t * SPM_MAX_TOPK + k)];
            if (slot < a.n_slots && -1 - slot < a.n_shared)
                acc = mt_plain_y<WT>(slot < 0 ? a.shared + size_t(-1 - slot) * a.blob_bytes : a.pool + size_t(slot) * a.blob_bytes, a.I, D, a.x + size_t(t) * D,
                                     k < a.K ? a.w[size_t(t) * a.K + k] : 1.f, d);
        }
    }
    part[k][c] = acc;
    __syncthreads();
    if (mine) {
        float4 sum = part[0][c];
        for (int kk = 1; kk < a.KS; ++kk) { const float4 p = part[kk][c]; sum.x += p.x; sum.y += p.y; sum.z += p.z; sum.w += p.w; }
        tot.x += sum.x; tot.y += sum.y; tot.z += sum.z; tot.w += sum.w;
        if (vec) *reinterpret_cast<float4*>(hp) = tot;
        else { hp[0] = tot.x; hp[1] = tot.y; hp[2] = tot.z; hp[3] = tot.w; }
    }
    if (a.clock) {
        __syncthreads();
        if (threadIdx.x == 0) atomicMax(a.clock + 1, global_timer_ns());
    }
}

// Largest number of entries: every routed expert's last entry may be partly filled, plus the shared ones
inline int mt_max_entries(int nb, int K, int n, int n_shared) {
    const int pairs = nb * K;
    return (pairs < n ? pairs : n) + pairs / kMtTokens + n_shared * ((nb + kMtTokens - 1) / kMtTokens);
}
inline size_t mt_partial_rows(int ctas, int nb, int K, int n, int n_shared) {
    return size_t(ctas + mt_max_entries(nb, K, n, n_shared)) * kMtTokens;
}
// Ring stages that fit beside the rest of the shared memory, and its total
inline int mt_stages(size_t row_bytes, bool fp32, int n, int n_pairs, int warps, size_t* smem) {
    const size_t rest = 2 * kMtMaxStages * 8 + 2 * (size_t(warps) * 128 + kMtTokens * kMtRows) * 4 + size_t(n + 4) * 4 + size_t(n_pairs) * 2;
    const size_t stage = size_t(kMtRows) * (mt_pitch(uint32_t(row_bytes) / 3 * 2, fp32) + mt_pitch(uint32_t(row_bytes) / 3, fp32));
    size_t s = (kFfnSmemLimit - rest) / stage;
    if (s > size_t(kMtMaxStages)) s = kMtMaxStages;
    *smem = s * stage + rest;
    return int(s);
}

}  // namespace spm
