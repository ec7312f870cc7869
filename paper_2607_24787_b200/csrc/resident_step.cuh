// One decode step of one sequence whose experts are all in HBM, as one kernel: routing, adapter and expert FFN of every layer.
//
// A host-free batch-1 step used to be two launches a layer (routing kernel, expert GEMV). What a layer of the Qwen3 shape spent
// its 26 us on: 14.5 in the GEMV, 9.1 in a routing kernel on the 8 SMs of one cluster (3.4 of them to pull 148 partial rows, 1.2 MB,
// through one GPC's port), 3.4 between the kernels. Here every CTA keeps its SM for the whole step and the routing is split over
// all of them; three exchanges a layer take the place of the launches:
//
//   partial rows   each CTA's sum over its share of the (expert, row) pairs -> the CTAs that own 16 columns of the hidden row each
//   hidden row     16 updated columns of each owner                         -> every CTA, which normalises the row for itself
//   logits         router and adapter rows, one warp each, over all CTAs    -> every CTA, which does the Top-K for itself
//
// A value travels as an 8-byte word {fp32, tag of the exchange}, so that it needs no flag and no fence: whoever reads a word with
// the tag of this layer has the value (8-byte accesses are single). A hop costs one store and one load through L2, about a
// microsecond; the logits, which have a writer each, have a 128-byte line each (sixteen writers to a line that all SMs poll took 4 us).
// One buffer per exchange is enough: a CTA overwrites a word one layer later, when it holds data that every reader of
// the old word contributed to after reading it.
//
// A layer of the Qwen3 shape now takes 19.5 us, of the DeepSeek shape 15.3 (21): the FFN 11.5 - 13 and 8 - 10 with the slowest SM 2 us
// behind the mean, and a chain of latencies of 6 (partial rows 1.4, hidden row 1, norm and dot products 1.5, logits 1.1, Top-K 0.6, first
// copies 0.5). With 4-bit experts 16.3 and 13.1, 6 and 4.5 of which are the tiles.
//
// The arithmetic, the orders of all sums and the split of the rows are those of router_adapter_kernel and ffn_gemv_kernel, so the
// outputs have the same bits as host-driven steps. The adapter's ranking, which only the host reads, is done by the last
// CTA (which owns no columns where there are fewer than 16 a CTA) while the others exchange the hidden row.
//
// Registers: nine or ten warps leave a thread 168, sixteen 128. Instances that spill: hidden 1280 of bf16 (68 bytes stored and loaded),
// hidden 1792 and 2048 of 4 bits (116 / 148 and 128 / 160); 16 bytes at 1280 of 4 bits.
//
// The CTAs wait for one another, so the launch is cooperative (one CTA per SM, all resident or none). Every wait is
// bounded: a CTA that gives up raises a flag that the others' waits look at, and all of them return with nothing in flight.
#pragma once

#include "ffn_gemv.cuh"
#include "ffn_gemv_q4.cuh"
#include "router_adapter.cuh"

namespace spm {

// Warps of a CTA: as many as the GEMV may take (those it does not use only route). Rows of 9216 bytes and more leave it eight at most,
// whose threads then have 255 registers. Rows of five segments have one more than the GEMV takes: the 320 quads of a hidden row of 1280
// bf16 then are one a thread (DeepSeek shape 15.8 -> 15.45 us a layer; twelve warps 15.8. Ten or twelve warps at fewer segments: within 2 %
// either way). fp32 rows of five segments, 640 columns, have half as many quads and take as long with nine warps (8.93 : 8.91 us a layer,
// 512 rows, 4 of 64).
constexpr int step_warps(int nseg, bool q4) { return q4 ? q4_warps(nseg) : nseg >= 6 ? 8 : nseg == 5 ? kFfnMaxWarps + 1 : kFfnMaxWarps; }
constexpr int kStatusStepTimeout = 16;            // status bit (1 to 8: expert and routing kernels)
constexpr int kStepCols = 16;                     // columns of the hidden row that an owner adds up
constexpr int kStepMaxCtas = kReduceGroupsR * kReduceChunkR;
constexpr unsigned long long kStepStartNs = 30000000000ull;     // default limit of the first exchange: kernels of other streams may hold SMs until then

struct StepArgs {
    const float* h_in;              // [D]
    float* h_out;                   // [D], may be h_in
    const float* gamma;             // [L][D]
    const void* router_w;           // [L][n][D]
    const void* adapter_a;          // [L - 1][r][D]
    const void* adapter_b;          // [L - 1][n][r]
    const unsigned char* pools;     // [L] pools of pool_bytes
    const unsigned char* shared;    // [L][n_shared] blobs (may be null)
    const short* slot_map;          // [L][n]
    unsigned long long* part;       // exchange: [CTAs][D] ...
    unsigned long long* hx;         // [D] ...
    unsigned long long* zx;         // [n + r][z_stride], words {fp32 bits, tag << 32}
    int z_stride;                   // 16, a line of its own for each writer, where there is room
    unsigned* abort_word;           // tag0 of a launch that gave up
    Mailbox* mailbox;               // [L]
    int* status;
    unsigned long long pool_bytes, blob_bytes, wait_limit_ns;
    uint32_t tag0;                  // layer l's exchanges carry tag0 + l, different from what any word holds before
    int I, K, n, r, L, n_slots, n_shared;
    int nw, depth;                  // GEMV warps and rows of a warp's ring (4-bit experts: -, tiles of the CTA's ring)
    uint32_t ring_bytes;            // shared memory ahead of the routing arrays
    int renorm, predict, xs_in_ring;
    float eps;
};

__device__ __forceinline__ unsigned long long ll_word(float v, uint32_t tag) { return (static_cast<unsigned long long>(tag) << 32) | __float_as_uint(v); }
__device__ __forceinline__ float ll_value(unsigned long long w) { return __uint_as_float(uint32_t(w)); }
__device__ __forceinline__ void ll_store(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void ll_store2(unsigned long long* p, unsigned long long v0, unsigned long long v1) {
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(v0), "l"(v1) : "memory");
}
__device__ __forceinline__ unsigned long long ll_load(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void ll_load2(const unsigned long long* p, unsigned long long& v0, unsigned long long& v1) {
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(v0), "=l"(v1) : "l"(p) : "memory");
}

// Bound of a thread's polling: true when the limit has run out or another CTA has given up.
struct StepSpin {
    const StepArgs& a;
    unsigned long long limit, t0 = 0;
    int polls = 0;
    __device__ StepSpin(const StepArgs& args, unsigned long long limit_ns) : a(args), limit(limit_ns) {}
    __device__ __forceinline__ bool give_up() {
        if ((++polls & 15) != 0) return false;          // (a poll takes half a microsecond; the exchanges some three)
        unsigned flag;
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(flag) : "l"(a.abort_word) : "memory");
        if (flag == a.tag0) return true;
        const unsigned long long now = global_timer_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 <= limit) return false;
        raise(a);
        return true;
    }
    static __device__ __forceinline__ void raise(const StepArgs& a) {
        atomicOr(a.status, kStatusStepTimeout);
        asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(a.abort_word), "r"(a.tag0) : "memory");
    }
};

// Elements of k[j0..j1) that come before e in (key descending, index ascending); j0 a multiple of 4, k 16-byte aligned.
__device__ __forceinline__ int count_before(const int* k, int j0, int j1, int e) {
    const int ke = k[e];
    int c0 = 0, c1 = 0, c2 = 0, c3 = 0, j = j0;
#pragma unroll 4
    for (; j + 4 <= j1; j += 4) {
        const int4 t = *reinterpret_cast<const int4*>(k + j);
        const int d = e - j;
        c0 += t.x > ke - int(0 < d);
        c1 += t.y > ke - int(1 < d);
        c2 += t.z > ke - int(2 < d);
        c3 += t.w > ke - int(3 < d);
    }
    for (; j < j1; ++j) c0 += k[j] > ke - int(j < e);
    return c0 + c1 + c2 + c3;
}

// Shared memory behind the GEMV's ring and barriers, in floats: [normalised row][n logits][n probabilities, or sums of the owned columns]
// [r adapter hidden][scratch 32][16 residuals][experts and weights of the chosen, 2 x 16][slot map, shorts]
__host__ __device__ constexpr size_t step_route_bytes(int D, int n, int r, bool xs_in_ring) {
    const size_t n4 = (size_t(n) + 3) & ~size_t(3), sums = size_t(kReduceGroupsR) * kStepCols;
    return sizeof(float) * ((xs_in_ring ? 0 : size_t(D)) + n4 + (n4 > sums ? n4 : sums) + ((size_t(r) + 3) & ~size_t(3)) + 32 + kStepCols + 2 * SPM_MAX_TOPK) +
           n4 * sizeof(short);
}

template <typename WT, int NSEG, bool Q4>
__global__ void __launch_bounds__(step_warps(NSEG, Q4) * 32, 1)
resident_step_kernel(const __grid_constant__ StepArgs a) {
    constexpr int kStepWarps = step_warps(NSEG, Q4), kStepThreads = kStepWarps * 32;
    static_assert(kStepThreads >= kRouterThreads, "the hidden row is normalised by the routing kernel's number of threads");
    constexpr int VEC = 16 / int(sizeof(WT));
    constexpr int D = NSEG * 32 * VEC;
    constexpr uint32_t ROWB = Q4 ? 3 * q4_part_bytes(D) : 3u * D * uint32_t(sizeof(WT));
    constexpr int GB = Q4 ? q4_groups(NSEG) : 1;
    constexpr int NV4 = (D / 4 + kRouterThreads - 1) / kRouterThreads;     // float4s of the hidden row per routing thread

    extern __shared__ __align__(128) unsigned char smem[];
    const int tid = threadIdx.x, wi = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;      // (wi: uniform)
    const int G = gridDim.x, c = blockIdx.x, n = a.n, I = a.I, nw = a.nw, depth = a.depth;
    const int n4 = (n + 3) & ~3;
    unsigned char* ring = smem + size_t(wi < nw ? wi : 0) * depth * ROWB;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + size_t(nw) * depth * ROWB);
    float* route = reinterpret_cast<float*>(smem + a.ring_bytes);
    float* xs = a.xs_in_ring ? reinterpret_cast<float*>(smem) : route;
    float* zs = route + (a.xs_in_ring ? 0 : D);
    float* ps = zs + n4;
    float* us = ps + max(n4, kReduceGroupsR * kStepCols);
    float* scratch = us + ((a.r + 3) & ~3);
    float* hres = scratch + 32;             // residual of the owned columns
    int* isel = reinterpret_cast<int*>(hres + kStepCols);
    float* s_w = reinterpret_cast<float*>(isel + SPM_MAX_TOPK);
    short* smap = reinterpret_cast<short*>(s_w + SPM_MAX_TOPK);

    // even split of the (expert, j) rows over the CTAs, then over the warps, as in ffn_gemv_kernel
    const GemvShare share(I, a.K + a.n_shared, Q4 ? 0 : a.n_shared, c, G);
    const int r_begin = share.r_begin, span = share.span;
    const int my_n = wi < nw && span > wi ? (span - wi + nw - 1) / nw : 0;
    const uint32_t bar0 = smem_u32(bars + (wi < nw ? wi : 0) * depth), ring0 = smem_u32(ring);
    // The warp's first rows of a layer are looked up by a lane each, which knows where they are but for the slot. The first n_early, of shared
    // experts, are asked for ahead of the routing, while the ring has nothing else to do (DeepSeek shape, two shared experts of eight:
    // 17.9 -> 16.2 us a layer).
    const int n_first = min(depth, my_n);
    const int n_early = Q4 || a.xs_in_ring ? 0 : min(n_first, share.n_shared_rows > wi ? (share.n_shared_rows - wi + nw - 1) / nw : 0);
    int first_ent, first_j;
    if constexpr (Q4) {              // (a tile's rows go round the warps)
        constexpr int kPer = q4_rows_per_warp(kStepWarps);
        share.row(min(lane / kPer * kQ4Rows + wi + lane % kPer * kStepWarps, max(span - 1, 0)), first_ent, first_j);
    } else {
        share.row(wi + min(lane, max(n_first - 1, 0)) * nw, first_ent, first_j);
    }
    const unsigned long long limit = a.wait_limit_ns ? a.wait_limit_ns : kWaitLimitNs;
    Q4Ring<kStepWarps> tiles(smem, D, Q4 ? depth : 0, tid);         // (4-bit experts)
    if (!Q4 && wi < nw && lane == 0) {
        for (int d = 0; d < depth; ++d) mbar_init(bar0 + 8u * d, 1);
        fence_barrier_init();
    }
    const bool owner = c * kStepCols < D, ranks = c == G - 1;
    if (owner && tid < kStepCols) hres[tid] = a.h_in[c * kStepCols + tid];

    // what routing reads of a layer: this warp's first weight row, the gain, the slot map
    const int my_row = c + G * wi;
    uint4 v[NSEG];
    float4 gv[NV4];
    short slot0 = 0;
    auto row_ptr = [&](int l, int row) {
        return row < n ? static_cast<const WT*>(a.router_w) + (size_t(l) * n + row) * D
                       : static_cast<const WT*>(a.adapter_a) + (size_t(l) * a.r + (row - n)) * D;
    };
    auto load_row = [&](int l, int row, int rows) {
        const uint4* p = reinterpret_cast<const uint4*>(row_ptr(l, row < rows ? row : 0));
#pragma unroll
        for (int it = 0; it < NSEG; ++it) v[it] = row < rows ? __ldg(p + it * 32 + lane) : make_uint4(0, 0, 0, 0);
    };
    auto rows_of = [&](int l) { return n + (a.predict && l <= a.L - 2 ? a.r : 0); };
    auto preload = [&](int l) {
        load_row(l, my_row, rows_of(l));
#pragma unroll
        for (int i = 0; i < NV4; ++i) {
            const int at = (i * kRouterThreads + tid) * 4;
            if (tid < kRouterThreads && at < D) gv[i] = __ldg(reinterpret_cast<const float4*>(a.gamma + size_t(l) * D + at));
        }
        if (tid < n) slot0 = __ldg(a.slot_map + size_t(l) * n + tid);
    };
    preload(0);

    int st_in = 0, st_out = 0;          // ring stages of the next copy and the next row, and the phase of the latter
    uint32_t ph = 0;
    // The row at `src` into the next stage of the warp's ring, by one elected lane with operands that are the same in the warp (lanes that
    // ask side by side are taken one by one; this took the DeepSeek shape from 19.3 to 17.8 us a layer). A bad slot's row is whatever
    // was there: the status word says so.
    auto ask = [&](const unsigned char* src) {
        if (elect_one()) {
            if (src) {
                mbar_arrive_expect_tx(bar0 + 8u * st_in, ROWB);
                bulk_g2s(ring0 + uint32_t(st_in) * ROWB, src, ROWB, bar0 + 8u * st_in, policy_evict_first());
            } else {
                mbar_arrive(bar0 + 8u * st_in);
            }
        }
        __syncwarp();
        st_in = st_in + 1 == depth ? 0 : st_in + 1;
    };
    auto ask_early = [&](int l) {
        for (int i = 0; i < n_early; ++i) {
            const int e = __shfl_sync(0xffffffffu, first_ent, i) - a.K, j = __shfl_sync(0xffffffffu, first_j, i);
            ask(a.shared + (size_t(l) * a.n_shared + e) * a.blob_bytes + size_t(j) * ROWB);
        }
    };
    __syncwarp();
    ask_early(0);
    // Leaves no copy of the `asked` last ones in flight
    auto drain = [&](int asked) {
        for (; asked > 0; --asked) {
            if (!mbar_wait_bounded(bar0 + 8u * st_out, ph, kWaitLimitNs)) break;
            st_out = st_out + 1 == depth ? 0 : st_out + 1;
            if (st_out == 0) ph ^= 1;
        }
    };
    for (int l = 0; l < a.L; ++l) {
        const uint32_t tag = a.tag0 + uint32_t(l);
        const int rows = rows_of(l);
        int dead = 0;

        // ---- hidden row -> normalised row, in every CTA (the sums of router_adapter_kernel) ----
        float4 hv[NV4];
        if (tid < kRouterThreads) {
            if (l == 0) {
#pragma unroll
                for (int i = 0; i < NV4; ++i) {
                    const int at = (i * kRouterThreads + tid) * 4;
                    if (at < D) hv[i] = *reinterpret_cast<const float4*>(a.h_in + at);
                }
            } else {
                StepSpin spin(a, limit);
                unsigned long long w[NV4][4];
#pragma unroll
                for (int i = 0; i < NV4; ++i)
#pragma unroll
                    for (int q = 0; q < 4; ++q) w[i][q] = 0ull;
                for (;;) {
                    bool missing = false;
#pragma unroll
                    for (int i = 0; i < NV4; ++i) {
                        const int at = (i * kRouterThreads + tid) * 4;
                        if (at >= D) continue;
#pragma unroll
                        for (int q = 0; q < 4; q += 2)
                            if (uint32_t(w[i][q] >> 32) != tag || uint32_t(w[i][q + 1] >> 32) != tag) {
                                ll_load2(a.hx + at + q, w[i][q], w[i][q + 1]);
                                missing = true;
                            }
                    }
                    if (!missing) break;
                    if (spin.give_up()) { dead = 1; break; }
                }
#pragma unroll
                for (int i = 0; i < NV4; ++i) hv[i] = make_float4(ll_value(w[i][0]), ll_value(w[i][1]), ll_value(w[i][2]), ll_value(w[i][3]));
            }
        }
        float ss = 0.f;
        if (tid < kRouterThreads) {
#pragma unroll
            for (int i = 0; i < NV4; ++i)
                if ((i * kRouterThreads + tid) * 4 < D) {
                    ss = fmaf(hv[i].x, hv[i].x, ss); ss = fmaf(hv[i].y, hv[i].y, ss);
                    ss = fmaf(hv[i].z, hv[i].z, ss); ss = fmaf(hv[i].w, hv[i].w, ss);
                }
        }
        ss = block_reduce(ss, scratch, false);
        const float inv = 1.0f / sqrtf(ss / float(D) + a.eps);
        if (tid < kRouterThreads) {
#pragma unroll
            for (int i = 0; i < NV4; ++i) {
                const int at = (i * kRouterThreads + tid) * 4;
                if (at < D)
                    *reinterpret_cast<float4*>(xs + at) = make_float4(hv[i].x * gv[i].x * inv, hv[i].y * gv[i].y * inv, hv[i].z * gv[i].z * inv, hv[i].w * gv[i].w * inv);
            }
        }
        if (tid < n) smap[tid] = slot0;
        for (int e = tid + kStepThreads; e < n; e += kStepThreads) smap[e] = a.slot_map[size_t(l) * n + e];
        if (__syncthreads_or(dead)) { drain(n_early); return; }

        // ---- logits: one warp per router or adapter row ----
        for (int row = my_row; row < rows; row += G * kStepWarps) {
            if (row != my_row) load_row(l, row, rows);
            float acc = 0.f;
#pragma unroll
            for (int it = 0; it < NSEG; ++it) {
                float f[VEC];
                unpack16(v[it], f);
#pragma unroll
                for (int q = 0; q < VEC; q += 4) {
                    const float4 t = *reinterpret_cast<const float4*>(xs + (it * 32 + lane) * VEC + q);
                    acc = fmaf(f[q], t.x, acc); acc = fmaf(f[q + 1], t.y, acc);
                    acc = fmaf(f[q + 2], t.z, acc); acc = fmaf(f[q + 3], t.w, acc);
                }
            }
            acc = warp_sum(acc);
            if (lane == 0) ll_store(a.zx + row * a.z_stride, ll_word(acc, tag));
        }
        // the GEMV's copy of the row: like one 16-byte weight vector per lane and segment, or as an MMA operand
        float xr[Q4 ? 1 : NSEG][VEC];
        uint32_t xq[GB][4];
        if constexpr (Q4) {
            q4_operand<GB>(xq, wi, lane, [&](int col, float (&f)[8]) {
                const float4 lo = *reinterpret_cast<const float4*>(xs + col), hi = *reinterpret_cast<const float4*>(xs + col + 4);
                f[0] = lo.x; f[1] = lo.y; f[2] = lo.z; f[3] = lo.w; f[4] = hi.x; f[5] = hi.y; f[6] = hi.z; f[7] = hi.w;
            });
        } else {
#pragma unroll
            for (int s = 0; s < NSEG; ++s)
#pragma unroll
                for (int q = 0; q < VEC; q += 4) {
                    const float4 t = *reinterpret_cast<const float4*>(xs + (s * 32 + lane) * VEC + q);
                    xr[s][q] = t.x; xr[s][q + 1] = t.y; xr[s][q + 2] = t.z; xr[s][q + 3] = t.w;
                }
        }
        for (int i = tid; i < rows; i += kStepThreads) {
            StepSpin spin(a, l == 0 && !a.wait_limit_ns ? kStepStartNs : limit);
            unsigned long long w;
            while (uint32_t((w = ll_load(a.zx + i * a.z_stride)) >> 32) != tag)
                if (spin.give_up()) { dead = 1; break; }
            float z = ll_value(w);
            if (i >= n) { us[i - n] = z; continue; }
            if (!isfinite(z)) {          // ids are meaningless then; keep the ordering total so that every rank is filled
                if (c == 0) atomicOr(a.status, kStatusNonFinite);
                z = -3.0e38f;
            }
            ps[i] = z;
            reinterpret_cast<int*>(zs)[i] = order_key(z);
        }
        if (a.xs_in_ring) fence_proxy_async();      // the row was written and read where copies are about to land
        if (__syncthreads_or(dead)) { drain(n_early); return; }

        // ---- Top-K; then the first weight copies go out, and the routing weights are computed behind them ----
        int sel = 0, top_key = 0;           // lane k: the k-th expert; key of the first
        // Every warp ranks for itself, or two threads an expert count what comes before it, and a barrier. The first pays for 4 bits, whose
        // rows are then looked up ahead, for fp32 rows of 1024 (both up to 128 experts), and with ten warps (up to 64; of 128 either takes
        // as long); elsewhere it is the longer way to the first copies. Whole steps, us a layer, counting : every warp with two keys a lane
        // (with four): DeepSeek shape (6 of 64) 15.7 : 15.4 (15.5), 1280 x 512 (4 of 24) 11.2 : 11.0; 512 x 768 (6 and a shared one of 64)
        // 9.2 : 9.2 (9.5), 768 x 512 (6 of 64) 9.2 : 9.3 (9.4), 256 x 512 (6 of 64) 6.8 : 7.0 (7.25); fp32, four keys, 1024 x 200 (8 of
        // 128) 9.9 : 9.5, 1024 x 128 (2 of 16) 6.7 : 6.6, 896 x 200 (8 of 128) 9.4 : 9.5, 768 x 128 (2 of 16) 6.6 : 6.8.
        constexpr bool kWideFp32 = sizeof(WT) == 4 && NSEG == 8;
        constexpr int kFew = 64, kRanked = Q4 || kWideFp32 ? kTopKeys * 32 : NSEG == 5 ? kFew : 0;
        auto key_of = [&](int e) { return reinterpret_cast<const int*>(zs)[e]; };
        if (kRanked > 0 && n <= kRanked) {
            if (Q4 || wi < nw)
                sel = kRanked <= kFew || (Q4 && n <= kFew) ? warp_top_k<kFew / 32>(n, a.K, lane, key_of, top_key)
                                                           : warp_top_k<kTopKeys>(n, a.K, lane, key_of, top_key);
        } else {                            // two threads an expert count what comes before it
            const int half_n = (n / 2) & ~3;
            for (int u0 = 0; u0 < 2 * n; u0 += kStepThreads) {
                const int u = u0 + tid, e = u >> 1;
                int rk = u < 2 * n ? count_before(reinterpret_cast<const int*>(zs), (u & 1) ? half_n : 0, (u & 1) ? n : half_n, e) : 0;
                rk += __shfl_xor_sync(0xffffffffu, rk, 1);
                if (u < 2 * n && (u & 1) == 0 && rk < a.K) isel[rk] = e;
            }
            __syncthreads();
            if (lane < a.K) sel = isel[lane];
            top_key = reinterpret_cast<const int*>(zs)[isel[0]];
        }
        // lane k: slot of entry k, routed or shared (negative)
        const int code_of = lane >= a.K ? a.K - 1 - lane : smap[sel] >= 0 ? smap[sel] : 1 << 20;       // no slot: fails the range check below
        if (c == 0 && wi == 0 && lane < a.K) a.mailbox[l].ids[lane] = tagged(tag & 0xffffu, sel);
        auto blob = [&](int ent) -> const unsigned char* {          // by whole warps; null after a bad slot number
            const int code = __shfl_sync(0xffffffffu, code_of, ent);
            if (code >= a.n_slots) { atomicOr(a.status, kStatusBadSlot); return nullptr; }
            return code < 0 ? a.shared + (size_t(l) * a.n_shared + size_t(-1 - code)) * a.blob_bytes
                            : a.pools + size_t(l) * a.pool_bytes + size_t(code) * a.blob_bytes;
        };
        auto row_at = [&](int row) -> const unsigned char* {        // (4-bit experts)
            const int ent = row < span ? (r_begin + row) / I : 0;
            const unsigned char* base = blob(ent);
            return base && row < span ? base + size_t(r_begin + row - ent * I) * ROWB : nullptr;
        };
        int n_in = n_first;                 // rows that the warp has asked for
        if constexpr (Q4) {
            tiles.fill(0, min(depth, (span + kQ4Rows - 1) / kQ4Rows), wi, lane, ROWB, false, [&](int row) -> const unsigned char* {
                const unsigned char* base = blob(first_ent);
                return base && row < span ? base + size_t(first_j) * ROWB : nullptr;
            });
        } else {       // (the lanes look the rows up side by side)
            const unsigned char* base = blob(first_ent);
            const unsigned long long at = base ? reinterpret_cast<unsigned long long>(base + size_t(first_j) * ROWB) : 0ull;
            for (int i = n_early; i < n_first; ++i) ask(reinterpret_cast<const unsigned char*>(__shfl_sync(0xffffffffu, at, i)));
        }
        // Routing weights: the router tail's softmax over all experts, by every warp for itself. The four butterflies are the sums
        // of that tail's four warps, added in their order.
        float wk = 1.f;                     // lane k: weight of entry k
        if (Q4 ? wi == 0 : wi < nw) {
            const float top = key_value(top_key);
            float part[4] = {0.f, 0.f, 0.f, 0.f};
            for (int e0 = 0; e0 < n; e0 += 128)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (e0 + q * 32 + lane < n) part[q] += expf(ps[e0 + q * 32 + lane] - top);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int q = 0; q < 4; ++q) part[q] += __shfl_xor_sync(0xffffffffu, part[q], o);
            const float sum = ((part[0] + part[1]) + part[2]) + part[3];
            const float p = lane < a.K ? expf(ps[sel] - top) / sum : 0.f;
            float tot = 0.f;
            for (int k = 0; k < a.K; ++k) tot += __shfl_sync(0xffffffffu, p, k);
            if (lane < a.K) wk = a.renorm ? p / tot : p;
            if (Q4 && lane < SPM_MAX_TOPK) s_w[lane] = wk;
        }

        // ---- expert FFN: this CTA's rows, as in ffn_gemv_kernel ----
        unsigned long long* out = a.part + size_t(c) * D;
        auto send = [&](int col, float4 y) {        // four consecutive columns of the CTA's partial row
            ll_store2(out + col, ll_word(y.x, tag), ll_word(y.y, tag));
            ll_store2(out + col + 2, ll_word(y.z, tag), ll_word(y.w, tag));
        };
        if constexpr (Q4) {
            float y[GB][2][4] = {};
            if (!q4_tiles<GB, kStepWarps>(tiles, xq, y, D, span, wi, lane, limit, [&](int tile) { tiles.fill(tile, 1, wi, lane, ROWB, false, row_at); },
                                          [&](int row) { return s_w[(r_begin + row) / I]; })) {
                if (tid == 0) StepSpin::raise(a);
                // leave no copy in flight: the tile that was waited for and those asked for since
                int st = tiles.st == 0 ? depth - 1 : tiles.st - 1;
                uint32_t phase = tiles.st == 0 ? tiles.ph ^ 1 : tiles.ph;
                do {
                    mbar_wait_bounded(tiles.bars + 8u * st, phase, kWaitLimitNs);
                    if (++st == depth) { st = 0; phase ^= 1; }
                } while (st != tiles.st_in);
                return;
            }
            q4_result<GB>(y, wi, lane, send);
            // (a CTA without rows has met no barrier since the logits: its warps may still be ranking them and adding up their exponentials,
            // where sums of the owned columns and the adapter's logits are about to go)
            if (span == 0) __syncthreads();
        } else {
            uint64_t ya[NSEG][VEC / 2];
#pragma unroll
            for (int s = 0; s < NSEG; ++s)
#pragma unroll
                for (int q = 0; q < VEC / 2; ++q) ya[s][q] = 0ull;
            int done = 0;
            for (; done < n_in; ++done) {
                if (!__all_sync(0xffffffffu, mbar_wait_bounded(bar0 + 8u * st_out, ph, limit))) {
                    if (lane == 0) StepSpin::raise(a);
                    dead = 1;
                    break;
                }
                int ent, j;
                share.row(wi + done * nw, ent, j);
                gemv_row<WT, NSEG>(ring0 + uint32_t(st_out) * ROWB + lane * 16, xr, __shfl_sync(0xffffffffu, wk, ent), ya);
                __syncwarp();
                st_out = st_out + 1 == depth ? 0 : st_out + 1;
                if (st_out == 0) ph ^= 1;
                if (n_in < my_n) {
                    share.row(wi + n_in * nw, ent, j);
                    const unsigned char* base = blob(ent);
                    ask(base ? base + size_t(j) * ROWB : nullptr);
                    ++n_in;
                }
            }
            if (dead) drain(n_in - done);
            if (wi < nw && !dead) gemv_stage_y<NSEG>(ring, lane, ya);
            if (__syncthreads_or(dead)) return;

            // ---- partial rows -> owned columns -> hidden row of the next layer ----
            {
                constexpr int Q = VEC / 4;
                const size_t ring_stride = size_t(depth) * ROWB;
                for (int p = tid; p < D / 4; p += kStepThreads) {
                    const float4 y = gemv_sum_warps(smem + size_t(p) * sizeof(float4), ring_stride, nw);
                    const int s = p / (32 * Q), h = (p / 32) % Q, ln = p % 32;
                    send(s * 32 * VEC + ln * VEC + 4 * h, y);
                }
                fence_proxy_async();            // the ring held partial sums: ordered before the next layer's copies
                if (a.n_shared > 0 && l + 1 < a.L) {
                    __syncthreads();
                    ask_early(l + 1);
                }
            }
        }
        if (l + 1 < a.L) preload(l + 1);
        if (owner && tid < kReduceGroupsR * kStepCols) {
            // the combine kernel's order: kReduceGroupsR runs of consecutive rows, each front to back, the runs in order, the residual last
            const int g = tid / kStepCols, col = tid % kStepCols;
            const int per = (G + kReduceGroupsR - 1) / kReduceGroupsR;
            const int c0 = g * per, cnt = min(G, c0 + per) - c0;
            const unsigned long long* p = a.part + size_t(c0) * D + c * kStepCols + col;
            unsigned long long w[kReduceChunkR];
#pragma unroll
            for (int i = 0; i < kReduceChunkR; ++i) w[i] = i < cnt ? ll_load(p + size_t(i) * D) : 0ull;
            StepSpin spin(a, limit);
            for (;;) {
                bool missing = false;
#pragma unroll
                for (int i = 0; i < kReduceChunkR; ++i)
                    if (i < cnt && uint32_t(w[i] >> 32) != tag) {
                        w[i] = ll_load(p + size_t(i) * D);
                        missing = true;
                    }
                if (!missing) break;
                if (spin.give_up()) break;          // (raised: the next exchange ends the launch)
            }
            float acc = 0.f;
#pragma unroll
            for (int i = 0; i < kReduceChunkR; ++i) acc += ll_value(w[i]);
            ps[g * kStepCols + col] = acc;
            asm volatile("bar.sync 3, %0;" ::"n"(kReduceGroupsR * kStepCols) : "memory");
            if (tid < kStepCols) {
                float tot = ps[tid];
#pragma unroll
                for (int i = 1; i < kReduceGroupsR; ++i) tot += ps[i * kStepCols + tid];
                tot += hres[tid];
                hres[tid] = tot;
                if (l + 1 < a.L) ll_store(a.hx + c * kStepCols + tid, ll_word(tot, tag + 1));
                else a.h_out[c * kStepCols + tid] = tot;
            }
        }
        if (ranks && rows > n && tid >= 128 && tid < 256) {      // the adapter's tail, as in router_adapter_kernel
            const WT* B = static_cast<const WT*>(a.adapter_b) + size_t(l) * n * a.r;
            for (int e = tid - 128; e < n; e += 128) {
                float acc = 0.f;
                for (int q = 0; q < a.r; ++q) acc = fmaf(load_weight(B, size_t(e) * a.r + q), us[q], acc);
                if (!isfinite(acc)) {
                    atomicOr(a.status, kStatusNonFinite);
                    acc = -3.0e38f;
                }
                zs[e] = acc;
            }
            asm volatile("bar.sync 2, 128;" ::: "memory");
            half_softmax(zs, n, scratch + 16, 2);
            Mailbox* mb = a.mailbox + l;
            for (int e = tid - 128; e < n; e += 128) {
                const int rk = rank_of_key(reinterpret_cast<const int*>(zs), n, e);
                mb->order[rk] = tagged(tag & 0xffffu, e);
                mb->scores[e] = zs[e];
            }
        }
    }
}

}  // namespace spm
