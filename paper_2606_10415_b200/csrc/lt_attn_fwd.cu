// Attention forward for sm_100a: O = softmax(scale Q K^T [+ causal mask]) V and the row
// log-sum-exp.  It produces the forward state the backward needs (the paper's Algorithm 1
// takes saved probability tiles; this library keeps LSE and rebuilds P in the backward).
//
// One CTA per (batch, query head, pair of neighbouring 128-row query tiles).  Warp 0 streams
// K_j / V_j tiles with TMA through one ring, warp 1 issues S = Q_i K_j^T and O += P V_j on the
// tcgen05 tensor cores, and each query tile has its own group of four softmax warps (one thread
// per query row), so that the tensor cores work on one tile of the pair while the other tile's
// scores are exponentiated.  S, P and O live in tensor memory.
// The running row maximum is only raised when it grew by more than 2^8 since the output
// was last rescaled, so most key tiles need no pass over O.
#include <float.h>
#include <math.h>

#include <algorithm>
#include <mutex>

#include "../../include/lt_attn_debug.h"
#include "lt_common.cuh"
#include "lt_host.h"

namespace lt {

constexpr int kFwdTileRows = 128;
constexpr int kFwdBoxBytes = 128 * 128;
constexpr float kFwdLog2e = 1.4426950408889634f;
constexpr float kFwdLn2 = 0.6931471805599453f;
// three warpgroups: control (producer warp, issuer warp, two warps that only fill up the group) and 2 x 4
// softmax warps; the control group hands most of its registers to the softmax warps, each of whose threads
// keeps the 128 scores of a query row in registers
constexpr int kFwdThreads = 384;
constexpr int kFwdSoftmaxWarp0 = 4;
constexpr int kFwdRegsAtLaunch = 168, kFwdRegsControl = 80, kFwdRegsSoftmax = 208;
static_assert(kFwdRegsAtLaunch * kFwdThreads <= 65536 && 128 * kFwdRegsControl + 256 * kFwdRegsSoftmax <= 65536,
              "register shares exceed the register file");
constexpr float kFwdRescaleLog2 = 8.f;        // P <= 2^8 stays far inside fp16 range

enum {
    kWaitFwdQ = 301, kWaitFwdKV = 302, kWaitFwdEmpty = 303, kWaitFwdS = 304, kWaitFwdP = 305,
    kWaitFwdO = 306, kWaitFwdSFree = 307, kWaitFwdTurn = 308, kWaitFwdDone = 309, kWaitFwdMerge = 310
};

template <int D>
struct __align__(1024) FwdSmem {
    static constexpr int kBoxes = D / 64;
    static constexpr int kTile = kBoxes * kFwdBoxBytes;
    uint8_t q[2][kTile];   // the pair's two query tiles
    static constexpr int kSlots = D == 128 ? 5 : 8;
    uint8_t kv[kSlots][kTile];   // ring of key and value tiles, in the order of their use
    uint64_t bar_q[2], bar_kv_full[kSlots], bar_kv_empty[kSlots];
    uint64_t bar_s_full[2], bar_s_free, bar_p_ready[2], bar_p_half[2], bar_o_done[2], bar_exp[4], bar_done, bar_merge;
    float2 merge[kFwdTileRows];  // (split keys) maximum and sum of the odd key tiles' half, per query row
    uint32_t tmem_base;
    int abort_flag;
};

static_assert(sizeof(FwdSmem<128>) + 1024 <= 232448, "shared memory (with room to align it) exceeds the 227 KB per-block limit");

struct FwdParams {
    float *lse;
    unsigned int *status;
    int B, Hq, Hkv, S, causal;
    float scale;
};

// Twelve warps: a producer, an issuer (and two idle ones, so that registers can be resized by groups of four), and four
// softmax warps for each of the two chains.
//
// A CTA runs two chains S -> softmax -> P V -> S side by side (index t).  Normally they are the two query tiles of a pair
// over the same key tiles; kSplitKeys: the even and the odd key tiles of one query tile, whose two softmaxes are put
// together at the end (each chain has its own maximum, sum and O).  That is twice the CTAs with half as long a walk, for
// grids that leave multiprocessors idle or wait for a few long walks: splits_keys().
//
// What bounds it: the exponential unit, 1 024 cycles per tile of 128 x 128 scores, with the softmax warps' other work (load,
// maximum, store, hand-offs: about 1 300 cycles a tile) that two warps per scheduler hide only in part; a step of both chains takes
// about 3 000 cycles, the exponential unit and the tensor cores (2 048 cycles a step at D = 128) are each busy for two thirds
// of it, and in long runs the power limit.  Hence the layout of tensor memory: the softmax warps hold a tile's scores in
// registers as soon as they are there, so the chains share one region of scores and P has columns of its own; a chain's next
// scores are formed under its softmax instead of behind its product P V.  (With S and P of a chain in one region a step took 3 600
// cycles, most of it the chain softmax -> P V -> S.)  us, a region per chain / this (heads, S, D; causal unless noted; calls on
// end): 32, 4096, 128 160 / 147; 32, 1024, 128 21.3 / 17.5; 32, 3000, 128 101 / 86; 8, 300, 128 8.0 / 7.2; 64 of 1531, 64 unmasked 74.8 / 67.7;
// 128 of 333, 64 17.4 / 15.5; 2, 129, 64 5.46 / 5.22.
// Tried with this layout: the second chain's first scores in columns of their own, so that both chains' first ones are formed at
// once (equal for short calls, 2-4 % slower for long ones at D = 128).  Tried before the score region was shared: two warps per row and
// tile, 16 softmax warps with a vote on the maximum (11 % slower: they wait for each other); the maximum found during the
// first quarter's exponentials (3 % slower); both chains started at once (2 % slower); a fifth of the exponentials as
// polynomials (no gain, at a smaller share of the unit's time than now).
template <int D, bool kBf16, bool kSplitKeys, bool kOneCopy>
__global__ void __launch_bounds__(kFwdThreads, 1)
fwd_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
           const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_o, const FwdParams p) {
    using Smem = FwdSmem<D>;
    constexpr int kBoxes = D / 64;
    constexpr uint32_t kTileBytes = Smem::kTile;
    constexpr uint32_t kTmemCols = 512;
    constexpr uint32_t kColS = 0;     // scores of one chain at a time
    constexpr uint32_t kColP = 128;   // chain t: P at columns [128 + 64 t, 192 + 64 t)
    constexpr uint32_t kColO = 256;   // chain t: O at columns [256 + D t, 256 + D t + D)

    extern __shared__ uint8_t smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;

    // heavy (late) query-tile pairs get the low block ids
    const int n_tiles = (p.S + kFwdTileRows - 1) / kFwdTileRows;  // the last tile may be ragged
    const int n_pairs = (n_tiles + 1) / 2;
    const int n_bh = p.B * p.Hq;
    const int n_groups = kSplitKeys ? n_tiles : n_pairs;  // of query tiles, one to a CTA
    const int pr = p.causal ? (n_groups - 1 - blockIdx.x / n_bh) : (blockIdx.x / n_bh);
    const int bh = blockIdx.x % n_bh;
    const int b = bh / p.Hq;
    const int h = bh % p.Hq;
    const int g = h / (p.Hq / p.Hkv);
    const int i0 = kSplitKeys ? pr : 2 * pr;
    const int n_keys = p.causal ? i0 + 1 : n_tiles;  // key tiles of query tile i0
    const bool has_b = kSplitKeys ? n_keys > 1 : (i0 + 1) < n_tiles;  // the second chain exists
    // last step of chain t (a key tile; split keys: key tile 2 j + t); -1 when there is no second chain
    const int j_last0 = kSplitKeys ? (n_keys + 1) / 2 - 1 : n_keys - 1;
    const int j_last1 = kSplitKeys ? n_keys / 2 - 1 : has_b ? (p.causal ? i0 + 1 : n_tiles - 1) : -1;
    const int n_q = kSplitKeys ? 1 : has_b ? 2 : 1;              // query tiles

    if (tid == 0) {
        sm.abort_flag = 0;
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            mbar_init(&sm.bar_q[t], 1);
            mbar_init(&sm.bar_s_full[t], 1);
            mbar_init(&sm.bar_p_ready[t], 4);
            mbar_init(&sm.bar_p_half[t], 4);
            mbar_init(&sm.bar_o_done[t], 1);
        }
        for (int x = 0; x < Smem::kSlots; ++x) {
            mbar_init(&sm.bar_kv_full[x], 1);
            mbar_init(&sm.bar_kv_empty[x], 1);
        }
        mbar_init(&sm.bar_s_free, 4);
        for (int x = 0; x < 4; ++x) mbar_init(&sm.bar_exp[x], 1);
        mbar_init(&sm.bar_done, 1);
        mbar_init(&sm.bar_merge, 128);
        mbar_fence_init();
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
        tma_prefetch_desc(&map_o);
    }
    if (warp == 0) {
        tmem_alloc(&sm.tmem_base, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    volatile int *abort_flag = &sm.abort_flag;
    // (The set-up above, and the softmax warps' first pass below, run under the tail of the predecessor in the stream; its
    // results are read, and O and LSE written, only behind grid_dependency_wait().)

    // The tensor-core work in its order: score products are numbered by (step, chain); number m is issued when the softmax
    // warps hold the scores of number m - 1 in registers, the products with V of number m - 2 come behind it.  on_s and
    // on_pv get (step, chain, whether it is the first and the last to use the step's key or value tile) and return false to leave.
    // (Behind the end of the first chain of a pair, its last product with V goes ahead, so that its output can be stored.)
    // Two forms of the same walk (fwd_plan has the rule).  One loop with one copy of either kind of work is a sixth of the code: it is the faster one at
    // D = 64, and at D = 128 where an SM runs one or two CTAs of short walks out of a cold instruction cache; unrolled over the
    // chains, with the chain a constant, a product takes fewer instructions to issue, which counts where products are twice as
    // long and many.  us, one copy / unrolled (heads, S, D): 32, 1024, 128 17.9 / 18.9; 128 of 333, 64 15.8 / 16.8; 32, 4096, 64
    // 106.7 / 108.0; on the other side 32, 4096, 128 140.5 / 137.5; 128 / 16 of 4 096, 128 534 / 509; 4, 8000, 128 63.6 / 61.4.
    auto walk = [&](auto on_s, auto on_pv) -> bool {
        auto first = [&](int j, int t) { return kSplitKeys || t == (j <= j_last0 ? 0 : 1); };
        auto last = [&](int j, int t) { return kSplitKeys || t == (j <= j_last1 ? 1 : 0); };
        if constexpr (!kOneCopy) {
            int m = 0, j1 = 0, t1 = 0, j2 = 0, t2 = 0;  // numbers m - 1 and m - 2
            const int j_end = j_last0 > j_last1 ? j_last0 : j_last1;
            for (int j = 0; j <= j_end; ++j) {
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (j > (t == 0 ? j_last0 : j_last1)) continue;
                    const bool ahead = !kSplitKeys && j > j_last0;
                    if (ahead && m >= 2 && !on_pv(j2, t2, first(j2, t2), last(j2, t2))) return false;
                    if (!on_s(m, j, t, first(j, t), last(j, t))) return false;
                    if (!ahead && m >= 2 && !on_pv(j2, t2, first(j2, t2), last(j2, t2))) return false;
                    j2 = j1; t2 = t1;
                    j1 = j; t1 = t;
                    ++m;
                }
            }
            if (m >= 2 && !on_pv(j2, t2, first(j2, t2), last(j2, t2))) return false;
            return on_pv(j1, t1, first(j1, t1), last(j1, t1));
        }
        const int n = j_last0 + j_last1 + 2;
        int s = 0, sj = 0, st = 0, v = 0, vj = 0, vt = 0;  // next score product, next product with V
        auto advance = [&](int &j, int &t) {
            if (t == 0 && j <= j_last1) { t = 1; return; }
            ++j;
            t = j <= j_last0 ? 0 : 1;
        };
        while (v < n) {
            if (s < n && s - v <= (!kSplitKeys && sj > j_last0 ? 1 : 2)) {
                if (!on_s(s, sj, st, first(sj, st), last(sj, st))) return false;
                advance(sj, st);
                ++s;
            } else {
                if (!on_pv(vj, vt, first(vj, vt), last(vj, vt))) return false;
                advance(vj, vt);
                ++v;
            }
        }
        return true;
    };
    if (warp < kFwdSoftmaxWarp0) {
        warpgroup_regs_set<kFwdRegsControl, kFwdRegsAtLaunch>();
        if (warp == 0) {
            // ------------------------------------------------------------------ producer
            if (lane == 0) {
                grid_dependency_wait();
                if (blockIdx.x == 0) p.status[kStatusWordTimeout] = 0u;  // (a wait gives up after a second at the earliest)
                for (int t = 0; t < n_q; ++t) {
                    mbar_arrive_expect_tx(&sm.bar_q[t], kTileBytes);
#pragma unroll
                    for (int x = 0; x < kBoxes; ++x)
                        tma_load_4d(sm.q[t] + x * kFwdBoxBytes, &map_q, &sm.bar_q[t], x * 64, (i0 + t) * kFwdTileRows, h, b);
                }
                int fill = 0, slot = 0, round = 0;  // fill = round * kSlots + slot: tiles whose loads were started
                auto load = [&](const CUtensorMap *map, int j, int t) -> bool {
                    const int row0 = (kSplitKeys ? 2 * j + t : j) * kFwdTileRows;  // inside the head; rows past S arrive as zeros
                    if (round > 0 && !mbar_wait(&sm.bar_kv_empty[slot], (round - 1) & 1, abort_flag, p.status, kWaitFwdEmpty)) return false;
                    mbar_arrive_expect_tx(&sm.bar_kv_full[slot], kTileBytes);
#pragma unroll
                    for (int x = 0; x < kBoxes; ++x)
                        tma_load_4d(sm.kv[slot] + x * kFwdBoxBytes, map, &sm.bar_kv_full[slot], x * 64, row0, g, b);
                    ++fill;
                    if (++slot == Smem::kSlots) slot = 0, ++round;
                    return true;
                };
                const bool ok = walk([&](int, int j, int t, bool first, bool) { return !first || load(&map_k, j, t); },
                                     [&](int j, int t, bool first, bool) { return !first || load(&map_v, j, t); });
                if (!ok || *abort_flag) {
                    // somebody gave up: wait (bounded) for the copies in flight before the CTA exits
                    for (int t = 0; t < n_q; ++t)
                        for (int w = 0; w < (1 << 16) && !mbar_try_wait(&sm.bar_q[t], 0); ++w) {}
                    for (int f = fill > Smem::kSlots ? fill - Smem::kSlots : 0; f < fill; ++f)
                        for (int w = 0; w < (1 << 16) && !mbar_try_wait(&sm.bar_kv_full[f % Smem::kSlots], (f / Smem::kSlots) & 1); ++w) {}
                }
            }
        } else if (warp == 1) {
            // ------------------------------------------------------------------ MMA issuer
            // The whole warp walks the loop, so that counters, wait results (voted) and descriptor arithmetic are
            // warp-uniform; one elected lane issues the products and commits.
            const bool leader = elect_one();
            auto wait_all = [&](uint64_t *bar, uint32_t parity, uint64_t *bar_b, uint32_t parity_b, int code) {
                return mbar_wait_warp(bar, parity, bar_b, parity_b, abort_flag, p.status, code);
            };
            constexpr uint32_t kSlotStep = kTileBytes >> 4;  // (products with a slot number are 32-bit ones)
            int slot = 0, round = 0;  // the ring's next tile
            int k_slot = 0, k_round = 0, v_slot = 0, v_round = 0;  // the tiles in use
            auto next_tile = [&](bool first, int &mine, int &mine_round) {
                if (!first) return;
                mine = slot;
                mine_round = round;
                if (++slot == Smem::kSlots) slot = 0, ++round;
            };
            // descriptors of slot 0; the next slot follows one tile later
            const uint64_t dQ0 = desc_kmajor(smem_u32(sm.q[0])), dK0 = desc_kmajor(smem_u32(sm.kv[0]));
            const uint64_t dV0 = desc_mnmajor(smem_u32(sm.kv[0]), kFwdBoxBytes);
            auto koff = [](int kk) -> uint64_t { return static_cast<uint64_t>((kk >> 2) * (kFwdBoxBytes >> 4) + (kk & 3) * 2); };
            auto roff = [](int kk) -> uint64_t { return static_cast<uint64_t>(kk * (2048 >> 4)); };
            constexpr uint32_t idesc_s = make_idesc(128, 128, false, false, kBf16);
            constexpr uint32_t idesc_o = make_idesc(128, D, false, true, kBf16);
            if (wait_all(&sm.bar_q[0], 0, n_q < 2 ? nullptr : &sm.bar_q[1], 0, kWaitFwdQ))
                walk(
                    [&](int m, int j, int t, bool first, bool last) -> bool {
                        // chain t's scores, in the one score region
                        next_tile(first, k_slot, k_round);
                        if (!wait_all(&sm.bar_kv_full[k_slot], k_round & 1, m > 0 ? &sm.bar_s_free : nullptr, (m - 1) & 1,
                                      both_codes(kWaitFwdKV, kWaitFwdSFree))) return false;
                        tc_fence_after_sync();
                        if (leader) {
                            const uint64_t dQ = dQ0 + static_cast<uint32_t>(kSplitKeys ? 0 : t) * kSlotStep, dK = dK0 + static_cast<uint32_t>(k_slot) * kSlotStep;
#pragma unroll
                            for (int kk = 0; kk < D / 16; ++kk) umma_ss(tmem + kColS, dQ + koff(kk), dK + koff(kk), idesc_s, kk > 0);
                            umma_commit(&sm.bar_s_full[t]);
                            if (last) umma_commit(&sm.bar_kv_empty[k_slot]);
                        }
                        return true;
                    },
                    [&](int j, int t, bool first, bool last) -> bool {
                        // O_t (+)= P_t V, P_t read from tensor memory; the keys of a tile in two halves of 64, so that the
                        // first half's products run while the softmax warps exponentiate the second half (quarters were
                        // measured too and lost to the extra hand-offs)
                        next_tile(first, v_slot, v_round);
                        const uint64_t dV = dV0 + static_cast<uint32_t>(v_slot) * kSlotStep;
#pragma unroll
                        for (int half = 0; half < 2; ++half) {
                            if (!wait_all(half == 0 ? &sm.bar_p_half[t] : &sm.bar_p_ready[t], j & 1, half == 0 ? &sm.bar_kv_full[v_slot] : nullptr,
                                          v_round & 1, half == 0 ? both_codes(kWaitFwdP, kWaitFwdKV) : kWaitFwdP)) return false;
                            tc_fence_after_sync();
                            if (leader) {
#pragma unroll
                                for (int kk = 4 * half; kk < 4 * half + 4; ++kk)
                                    umma_ts(tmem + kColO + t * D, tmem + kColP + t * 64 + kk * 8, dV + roff(kk), idesc_o, (j > 0) | (kk > 0));
                                if (half == 1) {
                                    umma_commit(&sm.bar_o_done[t]);
                                    if (last) umma_commit(&sm.bar_kv_empty[v_slot]);
                                }
                            }
                        }
                        return true;
                    });
            // every product issued above has finished before tensor memory is released
            if (leader) umma_commit(&sm.bar_done);
            if (!wait_all(&sm.bar_done, 0, nullptr, 0, kWaitFwdDone))
                for (int w = 0; w < (1 << 16) && !mbar_try_wait(&sm.bar_done, 0); ++w) {}
        }
    } else {
        // ------------------------------------------------------------------ softmax warps
        warpgroup_regs_set<kFwdRegsSoftmax, kFwdRegsAtLaunch>();
        const int t = (warp - kFwdSoftmaxWarp0) >> 2;   // which query tile of the pair
        const int quad = warp & 3;                      // tensor-memory lane quadrant of this warp
        const int row = quad * 32 + lane;               // query row inside the tile
        const int j_last = t == 0 ? j_last0 : j_last1;
        const int i = kSplitKeys ? i0 : i0 + t;
        const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
        const uint32_t tS = tmem + lane_base + kColS;
        const uint32_t tP = tmem + lane_base + kColP + t * 64;
        const uint32_t tO = tmem + lane_base + kColO + t * D;
        const float scale_log2 = p.scale * kFwdLog2e;
        // last visible key of a masked tile: the row's own index on a causal diagonal tile, the end of
        // the sequence on the ragged last key tile without a causal mask
        const int tail_keys = p.S - (n_tiles - 1) * kFwdTileRows;
        const int last_key = p.causal ? row : tail_keys - 1;
        float m_used = -INFINITY;  // the maximum the stored P, l and O are relative to
        float l = 0.f;             // running sum of exp2(score - m_used)
        bool ok = true;
        // Pass -1 works on whatever tensor memory holds and leaves nothing behind: it brings the loop's instructions into the
        // instruction cache while the first tiles are on their way (a first tile took 3 400 cycles instead of 1 450).  It takes longer
        // than tiles out of L2 do: a forward behind another kernel and on new inputs gains by it, one of many on the same inputs loses,
        // and short walks of split keys lose either way.  us, with it / without (heads, S, D): forward and backward in turn on
        // changing inputs: 128 of 333, 64 50.3 / 50.7; 8 of 64, 64 13.8 / 14.0; 32, 1024, 128 65.7 / 66.0; 8, 192, 128 24.0 / 23.7; forward calls alone: 8, 192, 64
        // 6.02 / 5.46; 32 of 64, 64 5.30 / 5.11; 32, 1024, 64 16.1 / 15.2; 8, 192, 128 6.68 / 6.33; 128 of 333, 64 15.7 / 15.4.
        const bool warm_up = !kSplitKeys || (D == 128 && n_tiles >= 8);
        for (int j = warm_up && t == 0 ? -1 : 0; j <= j_last; ++j) {
            if (j >= 0 && !(ok = mbar_wait_warp(&sm.bar_s_full[t], j & 1, nullptr, 0, abort_flag, p.status, kWaitFwdS))) break;
            tc_fence_after_sync();
            // the whole score row of this key tile stays in registers
            uint32_t sc[128];
#pragma unroll
            for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, *reinterpret_cast<uint32_t(*)[32]>(&sc[c * 32]));
            tmem_wait_ld();
            // the other chain's scores may follow
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0 && j >= 0) mbar_arrive(&sm.bar_s_free);
            const int key_tile = kSplitKeys ? 2 * j + t : j;
            if (p.causal ? key_tile == i : key_tile == n_tiles - 1 && tail_keys < kFwdTileRows) {
                __syncwarp();  // (keeps the selects behind a branch)
                // keys past `last_key` are invisible
                const uint32_t hidden = __float_as_uint(scale_log2 >= 0.f ? -INFINITY : INFINITY);
#pragma unroll
                for (int e = 0; e < 128; ++e)
                    if (e > last_key) sc[e] = hidden;
            }
            // row extremum of the raw scores: the maximum of scale*log2(e)*score is that factor times the largest
            // (smallest, for a negative scale) raw score
            // (eight independent running extrema: one warp per scheduler has no other work to cover the latency of a
            // dependent chain)
            float ex[8];
            if (scale_log2 >= 0.f) {
#pragma unroll
                for (int u = 0; u < 8; ++u) ex[u] = -INFINITY;
#pragma unroll
                for (int e = 0; e < 64; ++e)  // two keys per step: a three-input maximum
                    ex[e & 7] = fmaxf(ex[e & 7], fmaxf(__uint_as_float(sc[e]), __uint_as_float(sc[e + 64])));
#pragma unroll
                for (int u = 4; u > 0; u >>= 1)
#pragma unroll
                    for (int w = 0; w < u; ++w) ex[w] = fmaxf(ex[w], ex[w + u]);
            } else {
#pragma unroll
                for (int u = 0; u < 8; ++u) ex[u] = INFINITY;
#pragma unroll
                for (int e = 0; e < 64; ++e)
                    ex[e & 7] = fminf(ex[e & 7], fminf(__uint_as_float(sc[e]), __uint_as_float(sc[e + 64])));
#pragma unroll
                for (int u = 4; u > 0; u >>= 1)
#pragma unroll
                    for (int w = 0; w < u; ++w) ex[w] = fminf(ex[w], ex[w + u]);
            }
            const float row_max = ex[0] * scale_log2;
            if (j <= 0) {
                m_used = row_max;  // a chain's first key tile has a visible key, so this is finite for finite inputs
                l = 0.f;
            } else {
                const bool raise = (row_max - m_used) > kFwdRescaleLog2;
                if (__any_sync(0xffffffffu, raise)) {
                    // O must hold every earlier product before it is rescaled
                    if (!(ok = mbar_wait_warp(&sm.bar_o_done[t], (j - 1) & 1, nullptr, 0, abort_flag, p.status, kWaitFwdO))) break;
                    tc_fence_after_sync();
                    const float alpha = raise ? fast_exp2(m_used - row_max) : 1.f;
#pragma unroll
                    for (int c = 0; c < D / 16; ++c) {  // narrow pieces: the score row holds most registers
                        uint32_t r[16];
                        tmem_ld16(tO + c * 16, r);
                        tmem_wait_ld();
#pragma unroll
                        for (int e = 0; e < 16; ++e) r[e] = __float_as_uint(__uint_as_float(r[e]) * alpha);
                        tmem_st16(tO + c * 16, r);
                    }
                    l *= alpha;
                    if (raise) m_used = row_max;
                }
            }
            // P = exp2(score - m_used) as fp16
            // (a chain may begin with a tile whose scores are all -inf, keys hidden by -inf in K; such a tile gets zeros here, as
            // it does where a tile with a finite maximum came before it)
            const float neg_m = fminf(-m_used, FLT_MAX);
            const uint64_t scale2 = f32x2(scale_log2, scale_log2), neg_m2 = f32x2(neg_m, neg_m);
            uint64_t rs[2] = {0ull, 0ull};  // independent partial row sums, two each
            auto exponentials = [&](int e0, int e1) {
#pragma unroll
                for (int e = e0; e < e1; e += 2) {
                    float2 x = f32x2_parts(f32x2_fma(f32x2(__uint_as_float(sc[e]), __uint_as_float(sc[e + 1])), scale2, neg_m2));
                    x.x = fast_exp2(x.x);
                    x.y = fast_exp2(x.y);
                    rs[(e >> 1) & 1] = f32x2_add(rs[(e >> 1) & 1], f32x2(x.x, x.y));
                    sc[e] = __float_as_uint(x.x);
                    sc[e + 1] = __float_as_uint(x.y);
                }
            };
            auto store_half = [&](int half) {
#pragma unroll
                for (int c = 2 * half; c < 2 * half + 2; ++c) {
                    uint32_t out[16];
#pragma unroll
                    for (int e = 0; e < 32; e += 2)
                        out[e / 2] = pack2<kBf16>(__uint_as_float(sc[c * 32 + e]), __uint_as_float(sc[c * 32 + e + 1]));
                    tmem_st16(tP + c * 16, out);
                }
            };
            // The two warps of a scheduler take turns at the exponential unit, in the order of the score products, so that one
            // chain's exponentials run beside the other's loads, maxima and hand-offs; the turn passes on a little before the
            // last ones (after 112 of 128 keys; 96 measures the same), which covers the hand-off.  Not with split keys: there a turn,
            // which also holds the packing and storing of the first half, is longer than what it hides.  us, turns / none (heads, S, D;
            // causal unless noted): 20, 2048, 128 32.3 / 31.5; 4, 8000, 128 66.5 / 63.8; 4, 4000, 64 unmasked 29.5 / 28.9; pairs: 128 / 16 of 4 096, 128
            // 521 / 532; 128 of 333, 64 15.0 / 15.2; 40, 777, 64 15.0 / 15.4; but 64 of 1531, 64 unmasked 66.9 / 65.1; 32, 4096, 64 106.1 / 103.6.
            // (Before the first store the products with the previous P must have read it, too.)
            constexpr bool kTurns = !kSplitKeys;
            if constexpr (kTurns) {
                const int m = j + (t == 0 ? min(j, j_last1 + 1) : min(j, j_last0) + 1);
                if (m > 0 && j >= 0 && !(ok = mbar_wait_warp(&sm.bar_exp[quad], (m - 1) & 1, j > 0 ? &sm.bar_o_done[t] : nullptr, (j - 1) & 1,
                                                             abort_flag, p.status, both_codes(kWaitFwdTurn, kWaitFwdO)))) break;
            } else if (j > 0 && !(ok = mbar_wait_warp(&sm.bar_o_done[t], (j - 1) & 1, nullptr, 0, abort_flag, p.status, kWaitFwdO))) {
                break;
            }
            tc_fence_after_sync();
            exponentials(0, 64);
            store_half(0);
            exponentials(64, 112);
            if constexpr (kTurns) {
                __syncwarp();
                if (lane == 0 && j >= 0) mbar_arrive(&sm.bar_exp[quad]);
            }
            // a half's probabilities are in place: their products may start
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0 && j >= 0) mbar_arrive(&sm.bar_p_half[t]);
            exponentials(112, 128);
            store_half(1);
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0 && j >= 0) mbar_arrive(&sm.bar_p_ready[t]);
            const float2 rs0 = f32x2_parts(rs[0]), rs1 = f32x2_parts(rs[1]);
            l += (rs0.x + rs0.y) + (rs1.x + rs1.y);
        }

        if (ok && j_last >= 0) {
            ok = mbar_wait_warp(&sm.bar_o_done[t], j_last & 1, nullptr, 0, abort_flag, p.status, kWaitFwdO);
        }
        if constexpr (kSplitKeys) {
            if (t == 1) {  // the other chain's warps put the two halves together
                sm.merge[row] = make_float2(m_used, l);  // (no odd key tile: -inf and 0)
                mbar_arrive(&sm.bar_merge);
            } else if (ok) {
                ok = mbar_wait(&sm.bar_merge, 0, abort_flag, p.status, kWaitFwdMerge) &&
                     (j_last1 < 0 || mbar_wait(&sm.bar_o_done[1], j_last1 & 1, abort_flag, p.status, kWaitFwdO));
                ok = __all_sync(0xffffffffu, ok);
            }
        }
        if (ok && j_last >= 0 && !(kSplitKeys && t == 1)) {
            tc_fence_after_sync();
            float w0 = 1.f, w1 = 0.f;  // weights of this chain's O and of the other's
            if constexpr (kSplitKeys) {
                const float2 o = sm.merge[row];
                const float m = fmaxf(m_used, o.x);
                w0 = fast_exp2(m_used - m);
                w1 = fast_exp2(o.x - m);
                l = l * w0 + o.y * w1;
                m_used = m;
            }
            const float inv_l = 1.f / l;
            w0 *= inv_l;
            w1 *= inv_l;
            const int s_row = i * kFwdTileRows + row;  // rows past S belong to nobody
            const long long q_row = static_cast<long long>(bh) * p.S + s_row;  // LSE is contiguous
            // The query tile has been used for the last time: a warp lays its 32 rows of O out in its place as a tile load
            // would, and a tile store takes them from there (rows past S are not written).  (Stored from the registers, each
            // thread its own row 16 bytes at a time, a pair of tiles took 3 300 cycles, now 2 300.)
            uint8_t *stage = sm.q[kSplitKeys ? 0 : t];
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {  // (run once, from a cold instruction cache: a loop is shorter)
                uint32_t r[32];
                tmem_ld32(tO + c * 32, r);
                uint32_t r1[32];
                if (kSplitKeys && j_last1 >= 0) tmem_ld32(tO + D + c * 32, r1);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 32; ++e) {
                    float x = __uint_as_float(r[e]) * w0;
                    if (kSplitKeys && j_last1 >= 0) x = fmaf(__uint_as_float(r1[e]), w1, x);
                    r[e] = __float_as_uint(x);
                }
#pragma unroll
                for (int v8 = 0; v8 < 4; ++v8) {
                    uint4 o;
                    o.x = pack2<kBf16>(__uint_as_float(r[8 * v8 + 0]), __uint_as_float(r[8 * v8 + 1]));
                    o.y = pack2<kBf16>(__uint_as_float(r[8 * v8 + 2]), __uint_as_float(r[8 * v8 + 3]));
                    o.z = pack2<kBf16>(__uint_as_float(r[8 * v8 + 4]), __uint_as_float(r[8 * v8 + 5]));
                    o.w = pack2<kBf16>(__uint_as_float(r[8 * v8 + 6]), __uint_as_float(r[8 * v8 + 7]));
                    *reinterpret_cast<uint4 *>(stage + (c >> 1) * kFwdBoxBytes + swz128_offset(row, (c & 1) * 32 + v8 * 8)) = o;
                }
            }
            fence_proxy_async_smem();
            grid_dependency_wait();
            __syncwarp();
            if (lane == 0 && i * kFwdTileRows + quad * 32 < p.S) {
#pragma unroll
                for (int x = 0; x < kBoxes; ++x)
                    tma_store_4d(&map_o, stage + x * kFwdBoxBytes + quad * 4096, x * 64, i * kFwdTileRows + quad * 32, h, b);
                bulk_commit_group();
            }
            // (split keys: the weight of one half, an approximate exponential, adds 1e-7 to LSE's error; two roundings fewer
            // here take off more)
            if (s_row < p.S) p.lse[q_row] = kSplitKeys ? fmaf(m_used, kFwdLn2, logf(l)) : (m_used + log2f(l)) * kFwdLn2;
            bulk_wait_group_read<0>();  // (shared memory stays until the stores have read it)
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

constexpr int kFwdSms = 148;  // (of a B200: the estimates below are fitted to it)

// Whether a CTA takes one query tile with its key tiles in two chains instead of two query tiles: by the estimated
// makespan in steps of both chains (about 1.6 us), with kFill for a CTA's start, fill and drain, kMerge for putting two
// softmaxes together, and a margin.  Fitted to 400 shapes near the line, both ways measured in graphs: there 0.10 % behind the
// faster one on average and 6 % at worst, on 300 others 0.04 % and 6 %.  (The constants
// of the kernel whose softmax warps began with a pass on nothing, 1.9, 0.6, 0.91 and 0.95: 2.0 % and 19 %; 0.8 % and 17 %.)
// us, pairs of tiles / split keys (heads, S; D = 128 under the causal mask unless noted): 8, 300 8.7 / 7.5; 20, 384 9.1 / 7.9; 32, 400
// 11.0 / 8.2; 32, 949 18.2 / 17.5; 31, 1455 unmasked 49.3 / 44.1; on the other side 32, 589 12.3 / 12.5; 40, 512 11.6 / 12.4; 33, 2326
// 58.6 / 61.1; 40, 400 11.0 / 12.3; 60, 1949 unmasked 125 / 130; 48, 5607 unmasked 693 / 744.
static bool splits_keys(int B, int Hq, int S, int causal) {
    constexpr int kSms = kFwdSms;
    constexpr double kFill = 2.2, kMerge = 0.2;
    const double heads = static_cast<double>(B) * Hq;
    const int n = (S + kFwdTileRows - 1) / kFwdTileRows, pairs = (n + 1) / 2;
    if (n < 2) return false;
    // walk(q): steps of a head's q-th heaviest CTA
    auto span = [&](int per_head, double head_steps, double fill, auto walk) {
        const double ctas = heads * per_head, longest = walk(0) + fill;
        if (!causal) return ceil(ctas / kSms) * longest;  // walks of one length: whole rounds
        double t = (heads * head_steps + fill * ctas) / kSms;
        if (t < longest) t = longest;
        if (ctas > kSms) {  // heavy CTAs first: one SM gets the last of the first round and the first of the second, or lighter ones
            const double two = walk(static_cast<int>((kSms - 1) / heads)) + walk(static_cast<int>(kSms / heads)) + 2. * fill;
            if (t < two) t = two;
        }
        return t;
    };
    // causal: a pair's walk is its later tile's, and a tile's chains have half its keys each
    const double pair_steps = static_cast<double>(pairs) * (pairs + 1) - (n & 1 ? 1 : 0);
    const double half = (n + 1) / 2, even = n / 2;
    const double split_steps = half * (half + 1) / 2 + even * (even + 1) / 2;
    const double split = span(n, split_steps, kFill + kMerge, [&](int q) { return static_cast<double>(causal ? (n - q + 1) / 2 : (n + 1) / 2); });
    const double whole = span(pairs, pair_steps, kFill, [&](int q) { return static_cast<double>(causal && q > 0 ? 2 * (pairs - q) : n); });
    return split < (causal ? 0.88 : 0.96) * whole;
}

// The kernel of a call: how its CTAs split the work, and the form of the issuing warp's walk (figures beside the walk): one copy
// at D = 64, and for one or two CTAs of up to 24 products per SM.  Measured both ways on 190 shapes at D = 128, from 2 to 64
// products and 8 to 1 232 CTAs: one copy is the faster one up to 8 products (1-7 %), on up to 24 under the causal mask with more
// CTAs than SMs (1-7 % up to 12, -3 to 2 % above), equal at 11 and 12 with fewer CTAs, and 1-3 % behind from 16 on without a mask; from
// 32 on it is 2-8 % behind.  The line is within 3 % of the faster one.
struct FwdPlan {
    bool split_keys, one_copy;
    int grid;
};
static FwdPlan fwd_plan(int B, int Hq, int S, int D, int causal) {
    const bool split = splits_keys(B, Hq, S, causal);
    const int n_tiles = (S + kFwdTileRows - 1) / kFwdTileRows;
    const int grid = B * Hq * (split ? n_tiles : (n_tiles + 1) / 2);
    return {split, D == 64 || (grid <= 2 * kFwdSms && n_tiles * (split ? 1 : 2) <= 24), grid};
}

template <int D, bool kBf16>
static int launch_fwd(const lt_half *Q, const lt_half *K, const lt_half *V, lt_half *O, float *LSE,
                      const lt_attn_layout &lay, int B, int Hq, int Hkv, int S, int causal, float scale,
                      void *workspace, cudaStream_t stream) {
    CUtensorMap mq, mk, mv, mo;
    int rc;
    if ((rc = make_bhsd_map(&mq, Q, B, Hq, S, D, lay.q, 128, kBf16)) != LT_OK) return rc;
    if ((rc = make_bhsd_map(&mk, K, B, Hkv, S, D, lay.k, 128, kBf16)) != LT_OK) return rc;
    if ((rc = make_bhsd_map(&mv, V, B, Hkv, S, D, lay.v, 128, kBf16)) != LT_OK) return rc;
    if ((rc = make_bhsd_map(&mo, O, B, Hq, S, D, lay.o, 32, kBf16)) != LT_OK) return rc;
    FwdParams prm;
    prm.lse = LSE;
    prm.status = reinterpret_cast<unsigned int *>(workspace);
    prm.B = B; prm.Hq = Hq; prm.Hkv = Hkv; prm.S = S; prm.causal = causal ? 1 : 0;
    prm.scale = scale;
    // at least 120 KB, so that one CTA (which takes all 512 tensor-memory columns) lives on an SM
    const size_t smem = std::max<size_t>(sizeof(FwdSmem<D>) + 1024, 120 * 1024);
    const FwdPlan plan = fwd_plan(B, Hq, S, D, causal);
    auto kernel = plan.split_keys ? fwd_kernel<D, kBf16, true, true> : fwd_kernel<D, kBf16, false, true>;
    if constexpr (D == 128)
        if (!plan.one_copy) kernel = plan.split_keys ? fwd_kernel<D, kBf16, true, false> : fwd_kernel<D, kBf16, false, false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return record_cuda_error("cudaFuncSetAttribute(fwd)", e);
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(plan.grid);
    cfg.blockDim = dim3(kFwdThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &pdl;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, mq, mk, mv, mo, prm);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return record_cuda_error("fwd_kernel launch", e);
    return LT_OK;
}

// Internal streams and events of the host-buffer entry point, created on first use per device.
constexpr int kHostMaxChunks = 6, kHostMaxDevices = 64;
struct HostPipe {
    bool ready = false;
    cudaStream_t s_in = nullptr, s_out = nullptr;
    cudaEvent_t ev_start = nullptr, ev_out = nullptr, ev_in[kHostMaxChunks] = {}, ev_do[kHostMaxChunks] = {}, ev_fwd[kHostMaxChunks] = {},
                ev_comp[kHostMaxChunks] = {};
};
static HostPipe g_host_pipe[kHostMaxDevices];
static std::mutex g_host_pipe_mu;

}  // namespace lt

extern "C" {

size_t lt_attn_fwd_workspace_bytes(int B, int Hq, int Hkv, int S, int D) {
    if (lt::check_shape(B, Hq, Hkv, S, D, 1.0f) != LT_OK) return 0;
    return lt::kStatusBytes;
}

int lt_attn_fwd_num_launches(void) { return 1; }

int lt_dbg_fwd_plan(int B, int Hq, int S, int D, int causal, int *split_keys, int *one_copy) {
    const int rc = lt::check_shape(B, Hq, Hq, S, D, 1.0f);
    if (rc != LT_OK) return rc;
    if (!split_keys || !one_copy) return LT_ERR_INVALID_ARG;
    const lt::FwdPlan plan = lt::fwd_plan(B, Hq, S, D, causal);
    *split_keys = plan.split_keys ? 1 : 0;
    *one_copy = plan.one_copy ? 1 : 0;
    return LT_OK;
}

int lt_attn_fwd(const lt_half *Q, const lt_half *K, const lt_half *V, lt_half *O, float *LSE, int B, int Hq, int Hkv,
                int S, int D, int causal, float scale, void *workspace, size_t workspace_bytes, lt_stream_t stream) {
    return lt_attn_fwd_strided(Q, K, V, O, LSE, nullptr, B, Hq, Hkv, S, D, causal, scale, workspace, workspace_bytes,
                               stream);
}

static int fwd_entry(const lt_half *Q, const lt_half *K, const lt_half *V, lt_half *O, float *LSE,
                     const lt_attn_layout *layout, int B, int Hq, int Hkv, int S, int D, int causal, float scale,
                     void *workspace, size_t workspace_bytes, lt_stream_t stream, bool bf16) {
    using namespace lt;
    if (!Q || !K || !V || !O || !LSE) return LT_ERR_INVALID_ARG;
    int rc = check_shape(B, Hq, Hkv, S, D, scale);
    if (rc != LT_OK) return rc;
    lt_attn_layout lay = contiguous_layout(Hq, Hkv, S, D);
    if (layout) {
        // the forward reads q, k, v, o only; the other entries may be left unset
        lay.q = layout->q; lay.k = layout->k; lay.v = layout->v; lay.o = layout->o;
        if ((rc = check_layout(lay, D)) != LT_OK) return rc;
    }
    const void *ptrs[] = {Q, K, V, O};
    for (const void *ptr : ptrs)
        if (!aligned16(ptr)) return LT_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(LSE) & 3u) != 0) return LT_ERR_UNSUPPORTED;  // fp32, read and written one at a time
    if (!workspace || !aligned256(workspace) || workspace_bytes < lt_attn_fwd_workspace_bytes(B, Hq, Hkv, S, D))
        return LT_ERR_WORKSPACE;
    if ((rc = check_device()) != LT_OK) return rc;
    if (bf16) {
        if (D == 64) return launch_fwd<64, true>(Q, K, V, O, LSE, lay, B, Hq, Hkv, S, causal, scale, workspace, stream);
        return launch_fwd<128, true>(Q, K, V, O, LSE, lay, B, Hq, Hkv, S, causal, scale, workspace, stream);
    }
    if (D == 64) return launch_fwd<64, false>(Q, K, V, O, LSE, lay, B, Hq, Hkv, S, causal, scale, workspace, stream);
    return launch_fwd<128, false>(Q, K, V, O, LSE, lay, B, Hq, Hkv, S, causal, scale, workspace, stream);
}

int lt_attn_fwd_strided(const lt_half *Q, const lt_half *K, const lt_half *V, lt_half *O, float *LSE,
                        const lt_attn_layout *layout, int B, int Hq, int Hkv, int S, int D, int causal, float scale,
                        void *workspace, size_t workspace_bytes, lt_stream_t stream) {
    return fwd_entry(Q, K, V, O, LSE, layout, B, Hq, Hkv, S, D, causal, scale, workspace, workspace_bytes, stream,
                     false);
}

int lt_attn_fwd_bf16(const lt_bf16 *Q, const lt_bf16 *K, const lt_bf16 *V, lt_bf16 *O, float *LSE,
                     const lt_attn_layout *layout, int B, int Hq, int Hkv, int S, int D, int causal, float scale,
                     void *workspace, size_t workspace_bytes, lt_stream_t stream) {
    return fwd_entry(Q, K, V, O, LSE, layout, B, Hq, Hkv, S, D, causal, scale, workspace, workspace_bytes, stream,
                     true);
}

// the arena with `workspace_bytes` for the backward
static size_t host_arena_bytes(int B, int Hq, int Hkv, int S, int D, size_t workspace_bytes) {
    const size_t nq = lt::round256(static_cast<size_t>(B) * Hq * S * D * 2);
    const size_t nk = lt::round256(static_cast<size_t>(B) * Hkv * S * D * 2);
    const size_t nl = lt::round256(static_cast<size_t>(B) * Hq * S * 4);
    // Q, dO, O, dQ | K, V, dK, dV | LSE | forward status block | backward workspace
    return 4 * nq + 4 * nk + nl + lt::kStatusBytes + workspace_bytes;
}

size_t lt_attn_host_arena_bytes(int B, int Hq, int Hkv, int S, int D) {
    const size_t wb = lt_attn_bwd_workspace_bytes(B, Hq, Hkv, S, D);
    return wb == 0 ? 0 : host_arena_bytes(B, Hq, Hkv, S, D, wb);
}

int lt_attn_fwd_bwd_host(const lt_half *Q, const lt_half *K, const lt_half *V, const lt_half *dO, lt_half *O,
                         float *LSE, lt_half *dQ, lt_half *dK, lt_half *dV, int B, int Hq, int Hkv, int S, int D,
                         int causal, float scale, void *arena, size_t arena_bytes, lt_stream_t stream) {
    using namespace lt;
    if (!Q || !K || !V || !dO || !dQ || !dK || !dV) return LT_ERR_INVALID_ARG;
    int rc = check_shape(B, Hq, Hkv, S, D, scale);
    if (rc != LT_OK) return rc;
    const size_t need = host_arena_bytes(B, Hq, Hkv, S, D, bwd_least_bytes(B, Hq, S, D));
    if (!arena || !aligned256(arena) || arena_bytes < need) return LT_ERR_WORKSPACE;
    const size_t bq = static_cast<size_t>(B) * Hq * S * D * 2, bk = static_cast<size_t>(B) * Hkv * S * D * 2;
    const size_t bl = static_cast<size_t>(B) * Hq * S * 4;
    const size_t nq = round256(bq), nk = round256(bk), nl = round256(bl);
    uint8_t *a = static_cast<uint8_t *>(arena);
    lt_half *d_Q = reinterpret_cast<lt_half *>(a);
    lt_half *d_dO = reinterpret_cast<lt_half *>(a + nq);
    lt_half *d_O = reinterpret_cast<lt_half *>(a + 2 * nq);
    lt_half *d_dQ = reinterpret_cast<lt_half *>(a + 3 * nq);
    uint8_t *kbase = a + 4 * nq;
    lt_half *d_K = reinterpret_cast<lt_half *>(kbase);
    lt_half *d_V = reinterpret_cast<lt_half *>(kbase + nk);
    lt_half *d_dK = reinterpret_cast<lt_half *>(kbase + 2 * nk);
    lt_half *d_dV = reinterpret_cast<lt_half *>(kbase + 3 * nk);
    float *d_lse = reinterpret_cast<float *>(kbase + 4 * nk);
    void *fwd_ws = kbase + 4 * nk + nl;
    void *ws = kbase + 4 * nk + nl + kStatusBytes;
    const size_t ws_bytes = arena_bytes - (4 * nq + 4 * nk + nl + kStatusBytes);

    // ---- chunks of (batch, kv head) units: the host-to-device copy of one chunk, the kernels of the
    // previous one and the device-to-host copy of the one before run at the same time (two copy engines
    // and the SMs), on two internal streams beside the caller's.  A chunk is a contiguous slice of every
    // tensor and a problem of its own with B = 1.
    // A chunk's forward starts when its Q, K, V are there (dO follows), and its O and LSE go back while its backward runs.
    const int G = Hq / Hkv;
    const int n_units = B * Hkv;
    const long long n_tiles = padded_rows(S) / 128;
    const long long unit_iters = static_cast<long long>(G) * (causal ? n_tiles * (n_tiles + 1) / 2 : n_tiles * n_tiles);
    // The copies in one direction take as long as those in the other, and the copies back can only begin when the first
    // chunk has come in and been worked on: the smaller that chunk, the better, but every copy beside others in the other
    // direction costs about 15 us on top of its bytes.  Four chunks, the last ones smaller, or six of about equal size.
    // Measured with O returned on 75 shapes (four / six, ratio of the times, and ms for some): one query head per key/value head and 22
    // units or more 0.96-1.08, median 1.02 (24 heads of 4 096 2.78 / 2.57; 32 of 3 000 2.83 / 2.73; 40 of 2 048 2.28 / 2.18; 64 of 2 048 3.58 /
    // 3.32; 8 x 8 heads of 2 048 unmasked 3.58 / 3.35); 20 units 0.98-1.00; fewer, for which six chunks get uneven, 0.93-1.08; grouped
    // queries 0.88-0.98 (40 / 8 heads of 4 096 2.80 / 2.86; 40 / 20 3.48 / 3.62; 64 / 8 of 2 048 2.11 / 2.25).
    int bounds[kHostMaxChunks + 1];
    int n_chunks = 1;
    bounds[0] = 0;
    bounds[1] = n_units;
    if (unit_iters * n_units >= 3000 && n_units > 1) {  // otherwise not worth the extra streams
        constexpr int kFew[4] = {30, 60, 85, 100}, kMany[6] = {17, 34, 51, 68, 85, 100};  // cumulative shares, %
        const bool many = G == 1 && n_units >= 20;
        const int *percent = many ? kMany : kFew;
        const int np = many ? 6 : 4;
        n_chunks = 0;
        for (int c = 0; c < np; ++c) {
            const int end = c == np - 1 ? n_units : (n_units * percent[c] + 50) / 100;
            if (end <= bounds[n_chunks]) continue;  // fewer units than chunks
            bounds[++n_chunks] = end;
        }
    }

    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return record_cuda_error("cudaGetDevice", e);
    if (dev < 0 || dev >= kHostMaxDevices) n_chunks = 1;
    std::lock_guard<std::mutex> lock(g_host_pipe_mu);
    HostPipe *pipe = nullptr;
    if (n_chunks > 1) {
        pipe = &g_host_pipe[dev];
        if (!pipe->ready) {
            bool ok = cudaStreamCreateWithFlags(&pipe->s_in, cudaStreamNonBlocking) == cudaSuccess &&
                      cudaStreamCreateWithFlags(&pipe->s_out, cudaStreamNonBlocking) == cudaSuccess &&
                      cudaEventCreateWithFlags(&pipe->ev_start, cudaEventDisableTiming) == cudaSuccess &&
                      cudaEventCreateWithFlags(&pipe->ev_out, cudaEventDisableTiming) == cudaSuccess;
            for (int c = 0; c < kHostMaxChunks && ok; ++c)
                ok = cudaEventCreateWithFlags(&pipe->ev_in[c], cudaEventDisableTiming) == cudaSuccess &&
                     cudaEventCreateWithFlags(&pipe->ev_do[c], cudaEventDisableTiming) == cudaSuccess &&
                     cudaEventCreateWithFlags(&pipe->ev_fwd[c], cudaEventDisableTiming) == cudaSuccess &&
                     cudaEventCreateWithFlags(&pipe->ev_comp[c], cudaEventDisableTiming) == cudaSuccess;
            if (!ok) return record_cuda_error("stream/event creation for the host pipeline", cudaGetLastError());
            pipe->ready = true;
        }
    }
    cudaStream_t s_in = pipe ? pipe->s_in : stream, s_out = pipe ? pipe->s_out : stream;
#define LT_CUDA(call, what)                      \
    if ((e = (call)) != cudaSuccess) return record_cuda_error(what, e)
    if (pipe) {
        // nothing of this call may start before the work already queued on the caller's stream
        LT_CUDA(cudaEventRecord(pipe->ev_start, stream), "cudaEventRecord");
        LT_CUDA(cudaStreamWaitEvent(s_in, pipe->ev_start, 0), "cudaStreamWaitEvent");
        LT_CUDA(cudaStreamWaitEvent(s_out, pipe->ev_start, 0), "cudaStreamWaitEvent");
    }
    for (int c = 0; c < n_chunks; ++c) {
        const int u0 = bounds[c], u1 = bounds[c + 1];
        const int hkv = u1 - u0, hq = hkv * G;
        const size_t oq = static_cast<size_t>(u0) * G * S * D, ok_ = static_cast<size_t>(u0) * S * D;  // elements
        const size_t ol = static_cast<size_t>(u0) * G * S;
        const size_t cq = static_cast<size_t>(hq) * S * D * 2, ck = static_cast<size_t>(hkv) * S * D * 2;
        const size_t cl = static_cast<size_t>(hq) * S * 4;
        LT_CUDA(cudaMemcpyAsync(d_Q + oq, Q + oq, cq, cudaMemcpyHostToDevice, s_in), "cudaMemcpyAsync");
        LT_CUDA(cudaMemcpyAsync(d_K + ok_, K + ok_, ck, cudaMemcpyHostToDevice, s_in), "cudaMemcpyAsync");
        LT_CUDA(cudaMemcpyAsync(d_V + ok_, V + ok_, ck, cudaMemcpyHostToDevice, s_in), "cudaMemcpyAsync");
        if (pipe) {
            LT_CUDA(cudaEventRecord(pipe->ev_in[c], s_in), "cudaEventRecord");
            LT_CUDA(cudaStreamWaitEvent(stream, pipe->ev_in[c], 0), "cudaStreamWaitEvent");
        }
        LT_CUDA(cudaMemcpyAsync(d_dO + oq, dO + oq, cq, cudaMemcpyHostToDevice, s_in), "cudaMemcpyAsync");
        if (pipe) LT_CUDA(cudaEventRecord(pipe->ev_do[c], s_in), "cudaEventRecord");
        rc = lt_attn_fwd(d_Q + oq, d_K + ok_, d_V + ok_, d_O + oq, d_lse + ol, 1, hq, hkv, S, D, causal, scale, fwd_ws,
                         kStatusBytes, stream);
        if (rc != LT_OK) return rc;
        if (pipe) {
            LT_CUDA(cudaEventRecord(pipe->ev_fwd[c], stream), "cudaEventRecord");
            LT_CUDA(cudaStreamWaitEvent(stream, pipe->ev_do[c], 0), "cudaStreamWaitEvent");
            LT_CUDA(cudaStreamWaitEvent(s_out, pipe->ev_fwd[c], 0), "cudaStreamWaitEvent");
        }
        if (O) {
            // One query head per key/value head: not in the middle of dO's copy in.  The 7B layer then took 3.49 or 3.69 ms, depending
            // on how the copies of the two directions came to lie beside one another, which a few us of the kernels decide; behind
            // it 3.45.  Other heads, S, ms at once / behind dO: 32, 2048 1.90 / 1.83; 34, 2600 2.56 / 2.37; 40, 4096 4.48 / 4.36; 20, 4096
            // 2.31 / 2.32.  With grouped queries dO is a third of a chunk's bytes and more, and too much time passes: 24/12, 8 x 700 2.79 /
            // 2.84; 40/8, 4096 2.77 / 2.84; 64/8, 2048 2.09 / 2.19.
            if (pipe && G == 1) LT_CUDA(cudaStreamWaitEvent(s_out, pipe->ev_do[c], 0), "cudaStreamWaitEvent");
            LT_CUDA(cudaMemcpyAsync(O + oq, d_O + oq, cq, cudaMemcpyDeviceToHost, s_out), "cudaMemcpyAsync");
        }
        if (LSE) LT_CUDA(cudaMemcpyAsync(LSE + ol, d_lse + ol, cl, cudaMemcpyDeviceToHost, s_out), "cudaMemcpyAsync");
        rc = lt_attn_bwd(d_Q + oq, d_K + ok_, d_V + ok_, d_O + oq, d_dO + oq, d_lse + ol, d_dQ + oq, d_dK + ok_,
                         d_dV + ok_, 1, hq, hkv, S, D, causal, scale, ws, ws_bytes, stream);
        if (rc != LT_OK) return rc;
        if (pipe) {
            LT_CUDA(cudaEventRecord(pipe->ev_comp[c], stream), "cudaEventRecord");
            LT_CUDA(cudaStreamWaitEvent(s_out, pipe->ev_comp[c], 0), "cudaStreamWaitEvent");
        }
        LT_CUDA(cudaMemcpyAsync(dQ + oq, d_dQ + oq, cq, cudaMemcpyDeviceToHost, s_out), "cudaMemcpyAsync");
        LT_CUDA(cudaMemcpyAsync(dK + ok_, d_dK + ok_, ck, cudaMemcpyDeviceToHost, s_out), "cudaMemcpyAsync");
        LT_CUDA(cudaMemcpyAsync(dV + ok_, d_dV + ok_, ck, cudaMemcpyDeviceToHost, s_out), "cudaMemcpyAsync");
    }
    if (pipe) {
        // the caller's stream is done when the last copy back is
        LT_CUDA(cudaEventRecord(pipe->ev_out, s_out), "cudaEventRecord");
        LT_CUDA(cudaStreamWaitEvent(stream, pipe->ev_out, 0), "cudaStreamWaitEvent");
    }
#undef LT_CUDA
    return LT_OK;
}

}  // extern "C"
