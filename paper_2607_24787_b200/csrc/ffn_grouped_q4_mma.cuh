// Batched decode with 4-bit experts, few tokens an expert: the grouped SwiGLU expert FFN with the unpacked weights going from
// registers straight into mma.sync.
//
// Takes the place of ffn_grouped_q4_kernel (tcgen05) where an expert has few tokens, which is the rule in decode: 64 sequences of
// the Qwen3 shape give an expert about four. There the tensor cores idle either way, and what the tcgen05 kernel spends its time on
// is the way of an operand: unpack, store to tensor or shared memory, fence, hand-shake, 1050 cycles for an item that HBM
// delivers in 340. An mma.sync operand is where the unpacking leaves it, in the registers of the lane that needs it. A layer of a whole
// host-free step of that shape: 197 -> 146 us (HBM time of its experts: 49; 142 with exact weights and the scale on the activations,
// which rounds elsewhere than the tcgen05 kernel: outputs of 64 sequences then moved by 1e-2 where a near-tied Top-K choice tipped), 133 with
// TMA boxes and split tasks (below), 125 with shorter routing, gather and combine kernels around it.
// What bounds it now: instruction issue and dependent-issue latency, 99,000 instructions a scheduler at 0.56 a cycle; the packed bf16
// multiply-adds of the unpacking run at half rate (FMA pipe 45 %, ALU 42 % of active cycles).
//
// Work. A task is 128 intermediate rows of an expert (GgUnit) for up to kMqTokens of its tokens; CTA b runs the tasks b, b + grid, ...
// of all experts in order (a hot expert's runs of tokens go to different CTAs), but for the last one to two tasks a CTA, which are split
// evenly by tiles. A task that falls to two CTAs is begun by the first of them ahead of all else, which leaves its sums, unrounded, where
// the result goes, and finished by the second after all else: a chain of sums is the same whoever adds, so outputs have the same bits. (760
// tasks of 64 sequences of the Qwen3 shape on 148 CTAs: six for some, where an even share is 5.1; 137.5 -> 133 us a layer; 16 sequences
// 87.6 -> 82, 8: 66.5 -> 60.3. 64 of 60 experts lose 1 %, two sequences, which give no CTA a second task, 0.6 us.)
// Tasks are split, too, where the kernel waits for copies of experts. What a CTA begins first may then be of an expert that is on its way,
// and holds up the rest; but so may any task of a list in order, and a wave's copies are one arrival. Offloaded steps of the Qwen3 shape
// with device-side waits, us a layer, split : in order: 4 sequences, 120 slots 109 : 115, 16 sequences, 96 slots 997 : 1004, 64 sequences,
// 32 slots 4982 : 4999.
// A task goes through its rows in tiles of 16; the warps split the columns in groups of 32 (one scale), GB consecutive groups a warp.
//   Phase 1 (M = 16 gate rows, then 16 up rows; N = tokens; K = 32 columns, two MMAs). The warps' sums meet in shared memory.
//   Phase 2 (M = 16 hidden columns, N = tokens, K = 16 rows): the warp's own columns. y stays in the accumulators for the whole task.
// Phase 2 is one tile behind phase 1, so that one CTA barrier a tile is enough. A tile comes as three boxes of 16 rows by TMA, gate and up into one
// ring, W_down into another. Where 16 rows of a part would start in the same banks (hidden a multiple of 512) a box is 16 bytes wider
// than the part, which pads the rows. (Two bulk copies a row, asked for by all warps: 80 of some 640 instructions of a warp and tile. 64
// sequences of the Qwen3 shape 146 -> 137.5 us a layer.)
//
// A token's result depends on its own row and the expert only (a column of the MMAs), so outputs do not depend on waves, batch
// mates or the CTA. What is rounded is what the tcgen05 kernel rounds: scales, products of scale and q - 8, token rows and activations,
// to bf16; sums are fp32. The two kernels differ in the order of the sums alone.
#pragma once

#include <type_traits>

#include "ffn_grouped.cuh"
#include "ffn_multi.cuh"
#include "q4_mma.cuh"

namespace spm {

constexpr int kMqTokens = 8;                  // tokens of a task: N of the MMAs
constexpr int kMqTiles = kGgTileRows / kQ4Rows;
constexpr int kMqRed = 264;                   // pitch of a warp's phase-1 sums: 256 floats, the next warp's eight banks on
constexpr int kMqAct = 24;                     // pitch of a token's activations (bf16): 12 banks, so that eight tokens' pairs of rows have banks of their own
constexpr int kMqMaxTasks = 512;              // tasks of a CTA (two more where some are split)
constexpr int kMqTaskSlots = kMqMaxTasks + 4;

struct MqArgs {
    const __nv_bfloat16* xs;        // sorted token rows, columns 8g .. 8g + 7 in the order 0 4 1 5 2 6 3 7
    GgArgs g;
};
struct MqTask { int slot, jt_n, row, unit, span; };   // global slot, 128-row tile * 16 + tokens, first token row, unit, first tile | end << 8
static_assert(kMqTaskSlots * sizeof(MqTask) % 16 == 0, "sums behind the tasks are stored four at a time");

// Tasks of a CTA at worst: every expert's last run partly filled
inline int mq_max_tasks(int nb, int K, int n, int n_jt, int grid) {
    const int pairs = nb * K, runs = (pairs < n ? pairs : n) + pairs / kMqTokens;
    return (runs * n_jt + grid - 1) / grid;
}
inline size_t mq_rest_bytes(int n) {
    return 2 * kQ4MaxStages * 8 + 2 * size_t(kQ4MaxWarps) * kMqRed * 4 + 2 * kMqTokens * kMqAct * 2 + 2 * kMqTokens * 4 + 16 +
           size_t(kMqTaskSlots) * sizeof(MqTask) + size_t(n + 1) * 4;
}
inline int mq_stages(int D, int n, size_t* smem) {
    const size_t stage = 3 * size_t(kQ4Rows) * mt_pitch(q4_part_bytes(D), false);
    size_t s = (kFfnSmemLimit - mq_rest_bytes(n)) / stage;
    if (s > size_t(kQ4MaxStages)) s = kQ4MaxStages;
    *smem = s * stage + mq_rest_bytes(n);
    return int(s);
}

// Whether any of a warp's scales is infinite or a NaN, from sums of scale times zero
__device__ __forceinline__ bool mq_nonfinite(__nv_bfloat162 zeros) { return __any_sync(0xffffffffu, (bits2(zeros) & 0x7fff7fffu) != 0); }

// Phase 1 of a tile: gate and up of its rows (2^-22 of them) over one warp's groups, for the MMA's eight token columns.
// rows: the tile's first gate row, rows of `pitch` bytes, kQ4Rows of gate, then of up; x: the B operand of each group, nibble pairs 0..3.
template <int GB>
__device__ __forceinline__ void mq_phase1(uint32_t rows, uint32_t pitch, int D, int grp0, int lane, const uint32_t (&x)[GB][4], float (&gate)[4], float (&up)[4]) {
    const uint32_t part = kQ4Rows * pitch;
    // matrices: gate rows 0-7, 8-15, up rows 0-7, 8-15, 16 bytes (a group) each
    const uint32_t at = rows + uint32_t((lane & 7) + ((lane >> 3) & 1) * 8) * pitch + uint32_t(lane >> 4) * part + uint32_t(grp0) * 16;
    const uint32_t sc = rows + uint32_t(lane >> 2) * pitch + uint32_t(D / 2 + grp0 * 2);
    constexpr int GP = (GB + 1) / 2;
    __nv_bfloat162 s[4][GP], zeros = bf2(0u);            // gate rows g and g + 8, up rows g and g + 8: pairs of groups
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        uint32_t v[GP];
        q4_scale_pairs<GB>(sc + uint32_t(r & 1) * 8 * pitch + uint32_t(r >> 1) * part, v);
#pragma unroll
        for (int i = 0; i < GP; ++i) { s[r][i] = q4_bf16_scales(v[i]); zeros = __hfma2(s[r][i], bf2(0u), zeros); }
    }
    auto run = [&](auto plain) {
#pragma unroll
        for (int i = 0; i < GB; ++i) {
            const uint4 w4 = ldsm4(at + i * 16);
            const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
            Nib4 a[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const __nv_bfloat162 one = (i & 1) ? __high2bfloat162(s[r][i / 2]) : __low2bfloat162(s[r][i / 2]);
                a[r] = q4_weights<decltype(plain)::value>(w[r], q4_scaled(one), one);
            }
            mma_k16(gate, a[0].p[0], a[1].p[0], a[0].p[1], a[1].p[1], x[i][0], x[i][1]);
            mma_k16(up, a[2].p[0], a[3].p[0], a[2].p[1], a[3].p[1], x[i][0], x[i][1]);
            mma_k16(gate, a[0].p[2], a[1].p[2], a[0].p[3], a[1].p[3], x[i][2], x[i][3]);
            mma_k16(up, a[2].p[2], a[3].p[2], a[2].p[3], a[3].p[3], x[i][2], x[i][3]);
        }
    };
    if (mq_nonfinite(zeros)) run(std::true_type{});
    else run(std::false_type{});
}
// Phase 2: y += W_down^T act over the tile's 16 rows (2^-22 of it). b0, b1: the activations of rows 2t, 2t + 1 and 2t + 8, 2t + 9. A lane
// gets the columns 4g .. 4g + 3 of each group: y[0][0..1], y[0][2..3], y[1][0..1], y[1][2..3] for tokens 2t, 2t + 1.
template <int GB>
__device__ __forceinline__ void mq_phase2(uint32_t rows, uint32_t pitch, int D, int grp0, int lane, uint32_t b0, uint32_t b1, float (&y)[GB][2][4]) {
    const uint32_t at = rows + uint32_t((lane & 7) + ((lane >> 3) & 1) * 8) * pitch + uint32_t(grp0) * 16;
    const uint32_t sc = rows + uint32_t(2 * (lane & 3)) * pitch + uint32_t(D / 2 + grp0 * 2);
    constexpr int GP = (GB + 1) / 2;
    uint32_t v[4][GP];                       // rows 2t, 2t + 1, 2t + 8, 2t + 9
    q4_scale_pairs<GB>(sc, v[0]);
    q4_scale_pairs<GB>(sc + pitch, v[1]);
    q4_scale_pairs<GB>(sc + 8 * pitch, v[2]);
    q4_scale_pairs<GB>(sc + 9 * pitch, v[3]);
    __nv_bfloat162 s[2][GB], zeros = bf2(0u);            // a group's scales of two rows
#pragma unroll
    for (int i = 0; i < GB; ++i)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            s[r][i] = q4_bf16_scales(__byte_perm(v[2 * r][i / 2], v[2 * r + 1][i / 2], (i & 1) ? 0x7632 : 0x5410));
            zeros = __hfma2(s[r][i], bf2(0u), zeros);
        }
    auto run = [&](auto plain) {
        constexpr bool kPlain = decltype(plain)::value;
#pragma unroll
        for (int i = 0; i < GB; i += 2) {
            // matrices: rows 0-7 and 8-15 of group i, then of group i + 1; transposed: a lane has four columns of two rows a word
            const uint4 w = ldsm4t(at + uint32_t(i + (i + 1 < GB ? (lane >> 4) : 0)) * 16);
            auto group = [&](int j, uint32_t lo, uint32_t hi) {
                const Nib4 a = q4_weights<kPlain>(lo, q4_scaled(s[0][j]), s[0][j]), b = q4_weights<kPlain>(hi, q4_scaled(s[1][j]), s[1][j]);
                mma_k16(y[j][0], a.p[0], a.p[1], b.p[0], b.p[1], b0, b1);
                mma_k16(y[j][1], a.p[2], a.p[3], b.p[2], b.p[3], b0, b1);
            };
            group(i, w.x, w.y);
            if (i + 1 < GB) group(i + 1 < GB ? i + 1 : i, w.z, w.w);
        }
    };
    if (mq_nonfinite(zeros)) run(std::true_type{});
    else run(std::false_type{});
}

template <int NSEG>
__global__ void __launch_bounds__(q4_warps(NSEG) * 32, 1)
ffn_grouped_q4_mma_kernel(const __grid_constant__ CUtensorMap rowmap, const __grid_constant__ MqArgs m, const int n_stages) {
    constexpr int D = NSEG * 256, GB = q4_groups(NSEG), NW = q4_warps(NSEG);
    constexpr uint32_t PART = q4_part_bytes(D), PITCH = mt_pitch(PART, false), BOX = kQ4Rows * PITCH;      // a box: 16 rows of a part
    extern __shared__ __align__(128) unsigned char smem[];
    const GgArgs& a = m.g;
    const uint32_t dn_ring = uint32_t(n_stages) * 2 * BOX;                    // the gate / up ring, then the W_down ring
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + dn_ring + uint32_t(n_stages) * BOX);
    MqTask* tasks = reinterpret_cast<MqTask*>(bars + 2 * kQ4MaxStages);
    float* red = reinterpret_cast<float*>(tasks + kMqTaskSlots);                  // [2][warps] phase-1 sums
    __nv_bfloat16* actv = reinterpret_cast<__nv_bfloat16*>(red + 2 * NW * kMqRed);      // [2][token][row]
    float* s_w = reinterpret_cast<float*>(actv + 2 * kMqTokens * kMqAct);     // [2 tasks][token]
    int& s_abort = *reinterpret_cast<int*>(s_w + 2 * kMqTokens);
    int* runs = &s_abort + 4;                                                 // [experts + 1] runs of tokens before each expert
    const int warp = __shfl_sync(0xffffffffu, int(threadIdx.x) >> 5, 0), lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;      // (warp: uniform)
    const uint32_t ring = smem_u32(smem), gu_bar = smem_u32(bars), dn_bar = gu_bar + 8 * kQ4MaxStages;
    const unsigned long long limit = a.wait_limit_ns ? a.wait_limit_ns : kWaitLimitNs;

    grid_dep_launch();
    if (threadIdx.x == 0) {
        for (int s = 0; s < n_stages; ++s) { mbar_init(gu_bar + 8 * s, 1); mbar_init(dn_bar + 8 * s, 1); }
        s_abort = 0;
        fence_barrier_init();
    }
    grid_dep_wait();
    if (a.clock && threadIdx.x == 0) atomicMin(a.clock, global_timer_ns());

    // ---- the CTA's tasks ----
    const int n_jt = a.I / kGgTileRows, n_exp = (a.n_units_dev ? __ldcg(a.n_units_dev) : a.n_units) / n_jt;
    for (int e = threadIdx.x; e < n_exp; e += NW * 32) runs[e + 1] = (__ldcg(&a.units[e * n_jt].ntok) + kMqTokens - 1) / kMqTokens;
    __syncthreads();
    if (warp == 0) {
        int run = 0;
        for (int e0 = 0; e0 < n_exp; e0 += 32) {
            int v = e0 + lane < n_exp ? runs[e0 + lane + 1] : 0;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, v, o);
                if (lane >= o) v += u;
            }
            if (e0 + lane < n_exp) runs[e0 + lane + 1] = run + v;
            run += __shfl_sync(0xffffffffu, v, 31);
        }
        if (lane == 0) runs[0] = 0;
    }
    __syncthreads();
    const int n_all = n_exp > 0 ? runs[n_exp] * n_jt : 0, G = int(gridDim.x);
    // Rounds of whole tasks, then the tiles s .. e of the tasks from `split` on: a head (the last of these tasks, begun here), which goes
    // first, whole tasks, a tail (the first of them, begun by the CTA before), which goes last.
    const int c = int(blockIdx.x), rounds = max(n_all / G - 1, 0), split = rounds * G;
    int s = 0, e = c < n_all ? kMqTiles : 0, first = c;
    if (n_all >= G) {
        const int tiles = (n_all - split) * kMqTiles, q = tiles / G, rem = tiles - q * G;
        s = q * c + min(c, rem);
        e = s + q + (c < rem ? 1 : 0);
        first = split + s / kMqTiles;
        e -= s / kMqTiles * kMqTiles;
        s %= kMqTiles;
    }
    const int head = e % kMqTiles ? 1 : 0, tail = s ? 1 : 0, whole = e / kMqTiles - tail;
    const int n_tasks = min(kMqMaxTasks + 2, head + rounds + whole + tail), n_tiles = e - s + rounds * kMqTiles;
    for (int i = threadIdx.x; i < n_tasks; i += NW * 32) {
        const int j = i - head - rounds;             // >= 0: a whole task of the split ones, or the tail
        const int task = i < head ? first + e / kMqTiles : j < 0 ? c + (i - head) * G : j < whole ? first + tail + j : first;
        const int span = i < head ? (e % kMqTiles) << 8 : (j == whole ? s : 0) | kMqTiles << 8;
        const int run = task / n_jt, jt = task - run * n_jt;
        int lo = 0, hi = n_exp;              // the expert whose runs hold this one
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (runs[mid] <= run) lo = mid; else hi = mid;
        }
        const int4 v = __ldcg(reinterpret_cast<const int4*>(a.units + lo * n_jt + jt));      // GgUnit{slot, jt, row0, ntok}
        const int tok = (run - runs[lo]) * kMqTokens;
        tasks[i] = MqTask{v.x, v.y * 16 + min(kMqTokens, v.w - tok), v.z + tok, lo * n_jt + jt, span};
    }
    __syncthreads();

    // ---- The last warp fills the rings ----
    struct Feed { int task, tile, end, n, st, row; };  // next tile, its task's end; tiles asked for; stage of the next; the tile's row of the map
    const uint64_t pol = policy_evict_first();
    bool feeding = warp == NW - 1;
    auto open = [&](Feed& f, bool wait) {
        if (!feeding || f.task >= n_tasks) return;
        const MqTask k = tasks[f.task];
        f.tile = k.span & 255;
        f.end = k.span >> 8;
        f.row = k.slot * a.I + (k.jt_n >> 4) * kGgTileRows + f.tile * kQ4Rows;
        if (wait && a.unit_wait) {       // the expert's copy may still be on its way
            const GgWait uw = a.unit_wait[k.unit];
            const GgAbort ab{&s_abort, a.status, limit};
            if (uw.watch >= 0 && !__all_sync(0xffffffffu, gg_wait_arrival(a.ready + uw.watch, uw.want, ab))) feeding = false;
        }
    };
    auto feed = [&](Feed& f, uint32_t ring_at, uint32_t bar, int part, int parts, bool wait) {
        if (!feeding || f.task >= n_tasks) return;
        if (elect_one()) {
            mbar_arrive_expect_tx(bar + 8 * f.st, uint32_t(parts) * BOX);
            for (int i = 0; i < parts; ++i)
                tma_load_2d_hint(ring_at + uint32_t(f.st * parts + i) * BOX, &rowmap, (part + i) * int(PART / 8), f.row, bar + 8 * f.st, pol);
        }
        __syncwarp();
        ++f.n;
        f.st = f.st + 1 == n_stages ? 0 : f.st + 1;
        f.row += kQ4Rows;
        if (++f.tile < f.end) return;
        ++f.task;
        open(f, wait);
    };
    Feed fgu{0, 0, 0, 0, 0, 0}, fdn = fgu;
    auto feed_gu = [&]() { feed(fgu, ring, gu_bar, 0, 2, true); };
    auto feed_dn = [&]() { feed(fdn, ring + dn_ring, dn_bar, 2, 1, false); };     // (never ahead of the other)
    open(fgu, true);
    open(fdn, false);
    for (int i = 0; i < n_stages; ++i) { feed_gu(); feed_dn(); }

    // ---- tiles: phase 1 of tile k, phase 2 of tile k - 1 ----
    const int grp0 = warp * GB;
    uint32_t x[GB][4];
    float y[GB][2][4];
    auto load_x = [&](int task) {           // token rows, and the routing weights, of the task that phase 1 comes to
        const MqTask k = task < n_tasks ? tasks[task] : MqTask{0, 0, 0, 0, 0};
        const bool on = g < (k.jt_n & 15);
        const __nv_bfloat16* p = m.xs + size_t(k.row + g) * D + grp0 * 32 + t * 8;
#pragma unroll
        for (int i = 0; i < GB; ++i) {
            const uint4 v = on ? __ldcg(reinterpret_cast<const uint4*>(p + i * 32)) : make_uint4(0, 0, 0, 0);
            x[i][0] = v.x; x[i][1] = v.y; x[i][2] = v.z; x[i][3] = v.w;
        }
        if (threadIdx.x < kMqTokens) s_w[(task & 1) * kMqTokens + threadIdx.x] = int(threadIdx.x) < (k.jt_n & 15) ? __ldcg(a.wrow + k.row + threadIdx.x) : 0.f;
    };
    auto clear_y = [&]() {
#pragma unroll
        for (int i = 0; i < GB; ++i)
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
                for (int v = 0; v < 4; ++v) y[i][j][v] = 0.f;
    };
    load_x(0);
    clear_y();
    bool dead = false;
    int st1 = 0, st2 = 0;
    uint32_t ph1 = 0, ph2 = 0;
    // Tile k is tile k % 8 of the CTA's task k / 8: a head counts as the last tiles of its eight, so that all tasks end at multiples of
    // eight but the tail, the last, which ends with the loop.
    const int k0 = head ? kMqTiles - e % kMqTiles : 0, k1 = k0 + n_tiles;
    auto finish = [&](int task, float unscale) {            // a lane has four consecutive columns of two tokens
        const MqTask kk = tasks[task];
        const int n_tok = kk.jt_n & 15;
        float* out = a.partial + (size_t(kk.jt_n >> 4) * a.rows_cap + kk.row) * D + grp0 * 32 + g * 4;
#pragma unroll
        for (int i = 0; i < GB; ++i) {
            if (2 * t < n_tok)
                *reinterpret_cast<float4*>(out + size_t(2 * t) * D + i * 32) =
                    make_float4(y[i][0][0] * unscale, y[i][0][2] * unscale, y[i][1][0] * unscale, y[i][1][2] * unscale);
            if (2 * t + 1 < n_tok)
                *reinterpret_cast<float4*>(out + size_t(2 * t + 1) * D + i * 32) =
                    make_float4(y[i][0][1] * unscale, y[i][0][3] * unscale, y[i][1][1] * unscale, y[i][1][3] * unscale);
        }
    };
    for (int k = k0; k <= k1 && n_tiles > 0; ++k) {
        const bool p1 = k < k1, p2 = k > k0;
        const int task1 = k / kMqTiles;
        if (p1) {
            if (!dead) dead = !__all_sync(0xffffffffu, mt_wait(gu_bar + 8 * st1, ph1, &s_abort, a.status, limit));
            const uint32_t rows = ring + uint32_t(st1) * 2 * BOX;
            if (++st1 == n_stages) { st1 = 0; ph1 ^= 1; }
            float ag[4] = {}, au[4] = {};
            mq_phase1<GB>(rows, PITCH, D, grp0, lane, x, ag, au);
            float* r = red + ((k & 1) * NW + warp) * kMqRed + lane * 4;
            *reinterpret_cast<float4*>(r) = make_float4(ag[0], ag[1], ag[2], ag[3]);
            *reinterpret_cast<float4*>(r + 128) = make_float4(au[0], au[1], au[2], au[3]);
            if (k % kMqTiles == kMqTiles - 1) load_x(task1 + 1);        // the next task's rows are on their way while this tile is finished
        }
        if (p2 && !dead) dead = !__all_sync(0xffffffffu, mt_wait(dn_bar + 8 * st2, ph2, &s_abort, a.status, limit));
        __syncthreads();
        // every warp is done with the gate / up rows of tile k and with the W_down rows of tile k - 2
        if (!dead) {
            if (p1) feed_gu();
            if (k >= k0 + 2 && fdn.n < k - k0 - 1 + n_stages) feed_dn();
        }
        // 128 (row, token) pairs, one a lane of four warps (with eight pairs in each of sixteen warps, the exponential and the division cost every
        // warp a tile's time: 64 sequences of the Qwen3 shape 155 us a layer against 146)
        if (p1 && warp < 4) {
            const int pair = warp * 32 + lane;
            const float* r = red + (k & 1) * NW * kMqRed + pair;
            float vg = 0.f, vu = 0.f;
#pragma unroll
            for (int w = 0; w < NW; ++w) { vg += r[w * kMqRed]; vu += r[w * kMqRed + 128]; }
            vg *= kQ4Unscale;
            vu *= kQ4Unscale;
            const int row = (pair >> 4) + 8 * ((pair >> 1) & 1), tok = 2 * ((pair >> 2) & 3) + (pair & 1);
            actv[((k & 1) * kMqTokens + tok) * kMqAct + row] = __float2bfloat16_rn(vg / (1.f + expf(-vg)) * vu * s_w[(task1 & 1) * kMqTokens + tok]);
        }
        if (!p2) continue;
        {
            const __nv_bfloat16* av = actv + (((k - 1) & 1) * kMqTokens + g) * kMqAct + 2 * t;
            const uint32_t b0 = *reinterpret_cast<const uint32_t*>(av), b1 = *reinterpret_cast<const uint32_t*>(av + 8);
            mq_phase2<GB>(ring + dn_ring + uint32_t(st2) * BOX, PITCH, D, grp0, lane, b0, b1, y);
            if (++st2 == n_stages) { st2 = 0; ph2 ^= 1; }
        }
        if ((k - 1) % kMqTiles == kMqTiles - 1) {
            const int task2 = (k - 1) / kMqTiles;
            finish(task2, task2 < head ? 1.f : kQ4Unscale);
            if (task2 < head) {              // the next CTA goes on from here
                __threadfence();
                __syncwarp();
                if (lane == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(a.act_ready + blockIdx.x) : "memory");
            }
            clear_y();
            if (tail && task2 == n_tasks - 2) {
                const GgAbort ab{&s_abort, a.status, limit};
                if (!dead) dead = !__all_sync(0xffffffffu, gg_wait_count(a.act_ready + blockIdx.x - 1, NW, ab));
                const MqTask kk = tasks[task2 + 1];
                const int n_tok = kk.jt_n & 15;
                const float* in = a.partial + (size_t(kk.jt_n >> 4) * a.rows_cap + kk.row) * D + grp0 * 32 + g * 4;
#pragma unroll
                for (int i = 0; i < GB; ++i) {
                    const float* p = in + size_t(2 * t) * D + i * 32;
#pragma unroll
                    for (int q = 0; q < 4; ++q) {        // (one by one: loaded four at a time, they would want other registers than as sums of the MMAs)
                        if (2 * t < n_tok) asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(y[i][q >> 1][(q & 1) * 2]) : "l"(p + q));
                        if (2 * t + 1 < n_tok) asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(y[i][q >> 1][(q & 1) * 2 + 1]) : "l"(p + D + q));
                    }
                }
            }
        }
    }
    if (tail) finish(n_tasks - 1, kQ4Unscale);
    // Wind-down after a wait ran out: the warp that asked waits for what is in flight.
    __syncthreads();
    if (warp == NW - 1 && *reinterpret_cast<volatile int*>(&s_abort)) {
        const unsigned long long t0 = global_timer_ns();
        auto drain = [&](uint32_t bar, int n_fed) {
            for (int i = max(0, n_fed - n_stages); i < n_fed; ++i) {
                const unsigned long long spent = global_timer_ns() - t0;
                mbar_wait_bounded(bar + 8 * (i % n_stages), (i / n_stages) & 1, spent < kWaitLimitNs ? kWaitLimitNs - spent : 0);
            }
        };
        drain(gu_bar, fgu.n);
        drain(dn_bar, fdn.n);
    }
    if (a.clock) {
        __syncthreads();
        if (threadIdx.x == 0) atomicMax(a.clock + 1, global_timer_ns());
    }
}

}  // namespace spm
