// Attention backward (Algorithm 1 of the paper, Section 4.1) for sm_100a.
//
// Three kernels per call:
//   bwd_preprocess_kernel : delta = rowsum(dO * O); writes -delta and -LSE/scale as fp16
//                           (hi, lo) pairs, zeroes the fp32 dQ accumulator, records (one slot per block)
//                           max |delta|, max ||dO_row||^2 and max ||V_row||^2 (together they bound |dS|)
//   bwd_main_kernel       : per (batch, kv head, key tile j): loop over the group's
//                           query heads and the visible query tiles i, recompute
//                           P^T from LSE, and run the five tile contractions on
//                           tcgen05 tensor cores with tensor-memory accumulators
//   bwd_finalize_kernel   : dQ fp32 accumulator -> fp16
// and, where key tiles are split over several CTAs, before the last one
//   bwd_shares_kernel     : fp32 shares of dK and dV -> fp16
// (Sequences of one tile: one or two launches, see one_tile_launches.)
//
// Loop order differs from Algorithm 1 (which is query-outer and reduces dK/dV partials
// across workers): here a CTA owns one key/value tile, keeps dK_j and dV_j resident in
// tensor memory for the whole loop, and the cross-CTA reduction falls on dQ instead.
//
// The main kernel is persistent (one CTA per SM claims work items, heavy ones first, from a counter)
// and warp specialised: 16 warps in four warpgroups, so that each group can resize its share of the
// register file (the control group hands most of its registers to the other three):
//   warp 0       TMA producer (one thread): K_j, V_j once; then a two-stage ring of Q_i and a
//                single-buffered dO_i; the warp also owns the tensor-memory allocation
//   warp 1       tensor-core issuer (one thread); warps 2-3 only fill up the control group
//   warps 4-11   softmax / dS warps: warps 4-7 take query columns 0-63 of a tile pair,
//                warps 8-11 columns 64-127; each thread owns one key row
//   warps 12-15  dQ reduction (tensor memory -> shared memory -> bulk add.f32 into the fp32
//                accumulator: linear 8 KB pieces at D = 128, swizzled boxes through a tensor map at
//                D = 64) and the per-item dK/dV epilogue
// Transposed scores are used (S^T = K Q^T, dP^T = V dO^T) so that P^T, written back to
// tensor memory as fp16, is directly the A operand of dV += P^T dO; dS^T is written both to
// tensor memory (A operand of dK += dS^T Q) and to shared memory (operand of the dQ product).
// The row terms -LSE_i/scale and -delta_i are added inside the S^T and dP^T products by one
// extra 16-element contraction step whose operands are (256, 1, 0...) and the (hi, lo, 0...)
// split of the term, so the softmax warps never touch LSE or delta.
//
// Instantiations of the main kernel: fp16 or bf16 operands; a variant that splits a key tile's tile
// pairs over several work items (see BwdDeal); one for sequences of one tile; and a
// variant that loads the probability tiles a forward pass saved (Section 4.1's own forward state,
// written by lt_attn_save_p) instead of recomputing them.
#include <math.h>
#include <mutex>
#include <stddef.h>
#include <stdio.h>
#include <type_traits>

#include "lt_common.cuh"
#include "lt_host.h"

namespace lt {

constexpr int kTileRows = 128;             // rows of a query tile and of a key/value tile
constexpr int kBoxBytesBwd = 128 * 128;    // one swizzled tile of 128 rows x 64 fp16
constexpr float kLog2e = 1.4426950408889634f;

// wait codes recorded in the status block when a bounded wait gives up
enum {
    kWaitKV = 201, kWaitStageEmpty = 202, kWaitStageFull = 203, kWaitSFull = 204, kWaitPReady = 205,
    kWaitDpFull = 206, kWaitDsReady = 207, kWaitDsFree = 208, kWaitDqFull = 209, kWaitDqEmpty = 210,
    kWaitDkvFull = 211, kWaitDoFull = 212, kWaitDoEmpty = 213, kWaitAccFree = 214,
    kWaitItem = 200, kBadSmemAlign = 220
};

// ----------------------------------------------------------------------------- preprocess
// One half-warp (D = 128) or quarter-warp (D = 64) per row, 16-byte loads of dO and O; each
// warp works on kPreUnroll groups of rows at a time so that enough loads are in flight to
// keep HBM busy.
constexpr int kPreUnroll = 4;
// Rows a block takes per trip, and the largest grid: three resident blocks on each of 148 multiprocessors.  The maxima a
// block found go, as one 8-byte slot, into the -LSE/scale row that starts its first trip (elements 4-6 of that operand
// row meet zero multipliers in the main kernel, so any finite 16-bit pattern is inert there): no memory has to be
// cleared before this kernel, and nothing is reduced with atomics.  The main kernel's CTAs combine the slots.
// Measured against a cleared status block and atomic maxima (one more operation on the stream): 16.2 -> 11.9 us for the
// smallest backward, replayed from a graph.
constexpr int kPreThreads = 256, kPreMaxBlocks = 444;
template <int D>
__host__ __device__ constexpr int pre_rows_per_block() { return (kPreThreads / 32) * (32 / (D / 8)) * kPreUnroll; }
template <int D>
__host__ __device__ constexpr int pre_blocks(long long n_rows) {
    const long long want = (n_rows + pre_rows_per_block<D>() - 1) / pre_rows_per_block<D>();
    return static_cast<int>(want < kPreMaxBlocks ? want : kPreMaxBlocks);
}
// A non-negative fp32 maximum as 16 bits: its upper half rounded up, so that it stays a bound; 0x7B00 (a finite
// pattern in fp16 and bf16) stands for anything above 6e35, infinities and NaNs included.
constexpr unsigned int kMaxSlotInf = 0x7B00u;
__device__ __forceinline__ unsigned int max_slot_bits(unsigned int fp32_bits) {
    return min((fp32_bits + 0xFFFFu) >> 16, kMaxSlotInf);
}

// What the preprocess pass reads and writes.
struct PreParams {
    const __half *dO, *O, *V;
    const float *lse;  // NULL in the saved-P variant
    uint4 *delta_ext, *lse_ext;
    float *dq_acc;  // zeroed; NULL when no accumulator is used
    int S, S_pad, Hq, Hkv;
    lt_tensor_strides do_st, o_st, v_st;
    int plain, v_plain;  // contiguous tensors and no padding: a row's index is its place
    float inv_scale;
};

// Rows [row_lo, row_hi) of the padded row space (every head rounded up to S_pad rows, the indexing of delta_ext, lse_ext
// and dq_acc; padding rows get zeros everywhere), spread over `n_warps` warps of which this is number `warp`.
template <int D, bool kBf16>
__device__ __forceinline__ void pre_rows(const PreParams &p, long long row_lo, long long row_hi, long long warp,
                                         long long n_warps, float &max_abs_delta, float &max_norm2) {
    constexpr int kLanesPerRow = D / 8;
    constexpr int kRowsPerWarp = 32 / kLanesPerRow;
    constexpr int kRowsPerTrip = kRowsPerWarp * kPreUnroll;
    const int lane = threadIdx.x & 31;
    const int sub = lane % kLanesPerRow;
    for (long long row0 = row_lo + warp * kRowsPerTrip; row0 < row_hi; row0 += n_warps * kRowsPerTrip) {
        uint4 a[kPreUnroll], b[kPreUnroll];
        float l[kPreUnroll];
#pragma unroll
        for (int u = 0; u < kPreUnroll; ++u) {
            const long long row = row0 + u * kRowsPerWarp + lane / kLanesPerRow;
            a[u] = b[u] = make_uint4(0u, 0u, 0u, 0u);
            l[u] = 0.f;
            // rows of dO, O and LSE behind padded row `row` (`plain`: all three are row `row` itself)
            long long src_do = row * D, src_o = row * D, src_lse = row;
            bool valid = row < row_hi;
            if (!p.plain && valid) {
                const int bh = static_cast<int>(row / p.S_pad);
                const int s_in = static_cast<int>(row - static_cast<long long>(bh) * p.S_pad);
                const int bb = bh / p.Hq, hh = bh - bb * p.Hq;
                valid = s_in < p.S;
                src_do = bb * p.do_st.batch + hh * p.do_st.head + s_in * p.do_st.row;
                src_o = bb * p.o_st.batch + hh * p.o_st.head + s_in * p.o_st.row;
                src_lse = static_cast<long long>(bh) * p.S + s_in;
            }
            if (valid) {
                a[u] = __ldcs(reinterpret_cast<const uint4 *>(p.dO + src_do) + sub);
                b[u] = __ldcs(reinterpret_cast<const uint4 *>(p.O + src_o) + sub);
                if (sub == 0 && p.lse) l[u] = __ldg(p.lse + src_lse);  // (no LSE in the saved-P variant)
            }
            if (p.dq_acc && row < row_hi) {
                // the zero fill does not depend on the loads: issue it while they are in flight
                float4 *z = reinterpret_cast<float4 *>(p.dq_acc + row * D) + sub * 2;
                z[0] = make_float4(0.f, 0.f, 0.f, 0.f);
                z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
#pragma unroll
        for (int u = 0; u < kPreUnroll; ++u) {
            const long long row = row0 + u * kRowsPerWarp + lane / kLanesPerRow;
            const uint32_t *ah = reinterpret_cast<const uint32_t *>(&a[u]);
            const uint32_t *bh = reinterpret_cast<const uint32_t *>(&b[u]);
            float acc = 0.f, n2 = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 x = unpack2<kBf16>(ah[e]);
                const float2 y = unpack2<kBf16>(bh[e]);
                acc = fmaf(x.x, y.x, acc);
                acc = fmaf(x.y, y.y, acc);
                n2 = fmaf(x.x, x.x, n2);
                n2 = fmaf(x.y, x.y, n2);
            }
#pragma unroll
            for (int off = kLanesPerRow / 2; off > 0; off >>= 1) {
                acc += __shfl_xor_sync(0xffffffffu, acc, off);
                n2 += __shfl_xor_sync(0xffffffffu, n2, off);
            }
            if (row < row_hi) {
                if (sub == 0) {
                    // operand rows of the main kernel's extra contraction step: 256*hi + lo = value
                    p.delta_ext[row] = split_ext<kBf16>(-acc);
                    p.lse_ext[row] = split_ext<kBf16>(-l[u] * p.inv_scale);
                }
                max_abs_delta = fmaxf(max_abs_delta, fabsf(acc));
                max_norm2 = fmaxf(max_norm2, n2);
            }
        }
    }
}

// Largest squared norm of V's rows [row_lo, row_hi) (rows of the logical [B,Hkv,S]): with the two maxima above it bounds
// |dS|, from which the main kernel picks the power of two that dS carries into fp16.  (Kept as a bit pattern:
// non-negative floats order like them, with inf above every finite value and NaN above inf, so non-finite inputs
// saturate the bound.)
template <int D, bool kBf16>
__device__ __forceinline__ void pre_v_rows(const PreParams &p, long long row_lo, long long row_hi, long long warp,
                                           long long n_warps, unsigned int &max_v2) {
    constexpr int kLanesPerRow = D / 8;
    constexpr int kRowsPerWarp = 32 / kLanesPerRow;
    constexpr int kRowsPerTrip = kRowsPerWarp * kPreUnroll;
    const int lane = threadIdx.x & 31;
    const int sub = lane % kLanesPerRow;
    for (long long row0 = row_lo + warp * kRowsPerTrip; row0 < row_hi; row0 += n_warps * kRowsPerTrip) {
        uint4 a[kPreUnroll];
#pragma unroll
        for (int u = 0; u < kPreUnroll; ++u) {
            const long long row = row0 + u * kRowsPerWarp + lane / kLanesPerRow;
            a[u] = make_uint4(0u, 0u, 0u, 0u);
            if (row < row_hi) {
                long long src = row * D;
                if (!p.v_plain) {
                    const int bg = static_cast<int>(row / p.S);
                    const int s_in = static_cast<int>(row - static_cast<long long>(bg) * p.S);
                    const int bb = bg / p.Hkv, gg = bg - bb * p.Hkv;
                    src = bb * p.v_st.batch + gg * p.v_st.head + s_in * p.v_st.row;
                }
                a[u] = __ldg(reinterpret_cast<const uint4 *>(p.V + src) + sub);  // (the main kernel reads V again)
            }
        }
#pragma unroll
        for (int u = 0; u < kPreUnroll; ++u) {
            const uint32_t *ah = reinterpret_cast<const uint32_t *>(&a[u]);
            float n2 = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float2 x = unpack2<kBf16>(ah[e]);
                n2 = fmaf(x.x, x.x, n2);
                n2 = fmaf(x.y, x.y, n2);
            }
#pragma unroll
            for (int off = kLanesPerRow / 2; off > 0; off >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, off);
            max_v2 = max(max_v2, __float_as_uint(n2) & 0x7fffffffu);
        }
    }
}

template <int D, bool kBf16>
__global__ void __launch_bounds__(kPreThreads, 3)  // three blocks per multiprocessor keep enough loads in flight
bwd_preprocess_kernel(const PreParams p, long long n_rows, long long v_rows, unsigned int *status) {
    grid_dependency_wait();    // launched under the tail of its predecessor, which may write O or read the workspace
    grid_launch_dependents();  // the main kernel sets itself up while this kernel's last blocks run
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        status[kStatusWordTimeout] = 0u;
        status[kStatusWordItemCounter] = 0u;
    }
    const int lane = threadIdx.x & 31;
    const long long warp_global = (static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
    const long long n_warps = (static_cast<long long>(gridDim.x) * blockDim.x) >> 5;
    float max_abs_delta = 0.f, max_norm2 = 0.f;
    unsigned int max_v2 = 0u;
    pre_rows<D, kBf16>(p, 0, n_rows, warp_global, n_warps, max_abs_delta, max_norm2);
    // (V from the other end of the grid, whose warps had the fewer rows above)
    pre_v_rows<D, kBf16>(p, 0, v_rows, n_warps - 1 - warp_global, n_warps, max_v2);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        max_abs_delta = fmaxf(max_abs_delta, __shfl_xor_sync(0xffffffffu, max_abs_delta, off));
        max_norm2 = fmaxf(max_norm2, __shfl_xor_sync(0xffffffffu, max_norm2, off));
        max_v2 = max(max_v2, __shfl_xor_sync(0xffffffffu, max_v2, off));
    }
    __shared__ unsigned int block_max[3][kPreThreads / 32];
    if (lane == 0) {
        block_max[0][threadIdx.x >> 5] = __float_as_uint(max_abs_delta) & 0x7fffffffu;
        block_max[1][threadIdx.x >> 5] = __float_as_uint(max_norm2) & 0x7fffffffu;
        block_max[2][threadIdx.x >> 5] = max_v2;
    }
    __syncthreads();  // (also orders the slot after this block's own store of the row it lies in)
    if (threadIdx.x == 0) {
        unsigned int m[3] = {0u, 0u, 0u};
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int w = 0; w < kPreThreads / 32; ++w) m[k] = max(m[k], block_max[k][w]);
        uint2 *slot = reinterpret_cast<uint2 *>(p.lse_ext + static_cast<long long>(blockIdx.x) * pre_rows_per_block<D>()) + 1;
        *slot = make_uint2(max_slot_bits(m[0]) | (max_slot_bits(m[1]) << 16), max_slot_bits(m[2]));
    }
}

// ----------------------------------------------------------------------------- finalize
template <bool kBf16>
__global__ void __launch_bounds__(256)
bwd_finalize_kernel(const float *__restrict__ dq_acc, __half *__restrict__ dQ, long long n_vec8, int vec_per_head,
                    int vec_per_padded_head, int vec_per_row, int Hq, lt_tensor_strides dq_st, int plain) {
    // n_vec8 groups of eight output elements, numbered over the logical [B,Hq,S,D]; the accumulator
    // is indexed in the padded row space (`plain`: contiguous dQ and no padding, so both are group v)
    grid_dependency_wait();  // launched while its predecessor drains: the main kernel's reductions must have landed
    const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
    for (long long v = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; v < n_vec8; v += stride) {
        long long src = v, dst = v * 8;
        if (!plain) {
            const int bh = static_cast<int>(v / vec_per_head);
            const int rem = static_cast<int>(v - static_cast<long long>(bh) * vec_per_head);
            const int s_in = rem / vec_per_row, c = rem - s_in * vec_per_row;
            const int bb = bh / Hq, hh = bh - bb * Hq;
            src = static_cast<long long>(bh) * vec_per_padded_head + rem;
            dst = bb * dq_st.batch + hh * dq_st.head + s_in * dq_st.row + c * 8;
        }
        const float4 a = __ldcs(reinterpret_cast<const float4 *>(dq_acc) + 2 * src);
        const float4 b = __ldcs(reinterpret_cast<const float4 *>(dq_acc) + 2 * src + 1);
        uint4 o;
        o.x = pack2<kBf16>(a.x, a.y);
        o.y = pack2<kBf16>(a.z, a.w);
        o.z = pack2<kBf16>(b.x, b.y);
        o.w = pack2<kBf16>(b.z, b.w);
        *reinterpret_cast<uint4 *>(dQ + dst) = o;
    }
}

// Two ways to spread the tile pairs of one key tile over several CTAs.  Each leaves fp32 shares of dK_j and dV_j in the
// workspace, which bwd_shares_kernel adds in the order of the pairs (the same result from run to run).
// Dealt out (ctas > 0), where the SMs would get only a few, or a few heavy, key tiles: the CTAs get consecutive stretches of
// equal cost of one walk over all (unit, key tile, pair)s, where a unit is a (batch, kv head) with its group of query heads,
// and a key tile costs its pairs plus kTileCost for filling the pipeline and storing dK_j and dV_j.  A CTA leaves at most
// two shares: the end of its first key tile and the beginning of its last.
// In halves (halves = 1): every key tile is two work items, claimed from the counter like whole ones.
constexpr int kTileCost = 2;  // (measured with 2, 4, 6, 8: 2 is the best or within 1 % of it on 16 shapes)
struct BwdDeal {
    int ctas, halves;  // both 0: key tiles are whole
    int n_units, G, n_tiles, causal;

    __host__ __device__ __forceinline__ bool any() const { return ctas > 0 || halves; }
    __host__ __device__ __forceinline__ int pairs(int j) const { return G * (causal ? n_tiles - j : n_tiles); }
    // cost of a unit's key tiles before tile j
    __host__ __device__ __forceinline__ int tile_start(int j) const {
        return j * kTileCost + G * (causal ? j * n_tiles - j * (j - 1) / 2 : j * n_tiles);
    }
    // where CTA c's stretch begins
    __host__ __device__ __forceinline__ int stretch(int c) const {
        const int cost = n_units * tile_start(n_tiles), each = cost / ctas;
        return each * c + (cost - each * ctas) * c / ctas;
    }
    // a stretch boundary x behind a key tile's start -> pairs of the tile before it
    __host__ __device__ __forceinline__ int cut(int x, int n) const {
        x -= kTileCost;
        return x < 0 ? 0 : x > n ? n : x;
    }
    // key tile of a unit that holds cost x
    __host__ __device__ __forceinline__ int tile_at(int x) const {
        int lo = 0, hi = n_tiles - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tile_start(mid) <= x) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    }
    // A share is a block of 2 x 128 x D floats: dK, then dV, each [D/4][128 rows][4], so that a warp stores or reads 512
    // consecutive bytes.  In halves they are numbered by key tile and half; dealt out, 2 c (the end of CTA c's first key
    // tile) and 2 c + 1 (the beginning of its last), or, where that takes fewer, c + key tile, which grows along the walk.
    __host__ __device__ __forceinline__ int tiles() const { return n_units * n_tiles; }
    __host__ __device__ __forceinline__ bool few_tiles() const { return tiles() <= ctas; }
    __host__ __device__ __forceinline__ int share(int c, int tile, bool begins) const {
        return few_tiles() ? c + tile : 2 * c + begins;
    }
    __host__ __device__ __forceinline__ int n_shares() const {
        return halves ? 2 * tiles() : few_tiles() ? ctas + tiles() - 1 : 2 * ctas;
    }
};

// dK_j and dV_j of the key tiles that were dealt out to several CTAs: the fp32 shares, added in the order of the walk,
// as 16-bit outputs.  Block (c, 32 columns of dK or dV) has the tile that CTA c's stretch ends in, if it began there
// or before; it does nothing where the stretch ends with a tile or another CTA's does the beginning.  In halves: key tile c.
// The dQ conversion behind it is launched early and waits for all of it: that wait is also the one for the main kernel's
// reductions.  Reading the accumulator under this kernel, on the strength of this kernel's own wait, saved 1-1.8 us per
// call (16 query heads on 4, 777 rows, D = 64: 24.4 against 26.2), but nothing promises a grid what another one waited for.
template <int D, bool kBf16>
__global__ void __launch_bounds__(256)
bwd_shares_kernel(const float4 *__restrict__ shares, __half *__restrict__ dK, __half *__restrict__ dV, const BwdDeal deal,
                  int Hkv, int S, lt_tensor_strides dk_st, lt_tensor_strides dv_st) {
    const int c = blockIdx.x, second = blockIdx.y & 1;
    int parts = 0, unit, j = 0, first_share = 0;
    if (deal.halves) {
        unit = c / deal.n_tiles;
        j = c - unit * deal.n_tiles;
        first_share = 2 * c;
        parts = 2;
    } else {
        const int unit_cost = deal.tile_start(deal.n_tiles), end = deal.stretch(c + 1);
        unit = end / unit_cost;
        if (unit < deal.n_units) {
            j = deal.tile_at(end - unit * unit_cost);
            first_share = deal.share(c, unit * deal.n_tiles + j, true);
            const int start = unit * unit_cost + deal.tile_start(j), n = deal.pairs(j);
            int upto = deal.cut(end - start, n);
            if (upto > 0 && upto < n && deal.cut(deal.stretch(c) - start, n) == 0)
                for (parts = 1; upto < n; ++parts) upto = deal.cut(deal.stretch(c + parts + 1) - start, n);
        }
    }
    grid_launch_dependents();
    grid_dependency_wait();  // launched while the main kernel drains: its shares must have landed
    if (parts == 0) return;
    constexpr int kShareVec = 128 * D / 4;  // float4s of dK or dV in a share
    const int row = threadIdx.x & 127;
    const int v8 = (blockIdx.y >> 1) * 4 + (threadIdx.x >> 7);
    const float4 *src = shares + second * kShareVec + (2 * v8) * 128 + row;
    const float4 *next = src + static_cast<long long>(first_share) * 2 * kShareVec;
    float4 a[2][2];
#pragma unroll
    for (int x = 0; x < 4; ++x) a[x >> 1][x & 1] = __ldcs(next + ((x >> 1) * 4 + (x & 1)) * 128);
    next += 2 * kShareVec;  // the second share follows the first, further ones are one or two apart
    const int apart = (deal.few_tiles() ? 2 : 4) * kShareVec;
#pragma unroll 4
    for (int k = 1; k < parts; ++k, next += apart) {
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const float4 y = __ldcs(next + ((x >> 1) * 4 + (x & 1)) * 128);
            float4 &t = a[x >> 1][x & 1];
            t.x += y.x; t.y += y.y; t.z += y.z; t.w += y.w;
        }
    }
    const int b = unit / Hkv, g = unit - b * Hkv, s_row = j * 128 + row;
    const lt_tensor_strides &st = second ? dv_st : dk_st;
    __half *dst = (second ? dV : dK) + b * st.batch + g * st.head + s_row * st.row + v8 * 8;
    if (s_row >= S) return;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
        uint4 o;
        o.x = pack2<kBf16>(a[x][0].x, a[x][0].y);
        o.y = pack2<kBf16>(a[x][0].z, a[x][0].w);
        o.z = pack2<kBf16>(a[x][1].x, a[x][1].y);
        o.w = pack2<kBf16>(a[x][1].z, a[x][1].w);
        *reinterpret_cast<uint4 *>(dst + x * 16) = o;
    }
}

// ----------------------------------------------------------------------------- optional cycle trace
// Built only with -DLT_BWD_TRACE (development aid): per-role cycle totals, summed over all CTAs.
// Slot = 16 * role + (wait code - 200); slot 16 * role + 15 = the role's whole loop.
enum { kRoleProducer = 0, kRoleMma = 1, kRoleCompute = 2, kRoleReduce = 3 };
#ifdef LT_BWD_TRACE
__device__ unsigned long long g_bwd_trace[80];
struct Trace {
    unsigned int acc[16];
    unsigned int t0;
    __device__ __forceinline__ void start() {
        t0 = static_cast<unsigned int>(clock());
#pragma unroll
        for (int i = 0; i < 16; ++i) acc[i] = 0;
    }
    __device__ __forceinline__ void flush(int role) {
        acc[15] = static_cast<unsigned int>(clock()) - t0;
        if ((threadIdx.x & 31) == 0) {
#pragma unroll
            for (int i = 0; i < 16; ++i)
                if (acc[i]) atomicAdd(&g_bwd_trace[16 * role + i], static_cast<unsigned long long>(acc[i]));
        }
    }
};
#define LT_TRACE_BEGIN() Trace trace_; trace_.start()
#define LT_TRACE_MARK(var) const unsigned int var = static_cast<unsigned int>(clock())
#define LT_TRACE_SINCE(slot, var) trace_.acc[slot] += static_cast<unsigned int>(clock()) - var
#define LT_TRACE_END(role) trace_.flush(role)
#define LT_WAIT(bar, parity, code) traced_wait(trace_, bar, parity, abort_flag, p.status, code)
__device__ __forceinline__ bool traced_wait(Trace &tr, uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                            unsigned int *status, int code) {
    const unsigned int t0 = static_cast<unsigned int>(clock());
    const bool r = mbar_wait(bar, parity, abort_flag, status, code);
    tr.acc[code - 200] += static_cast<unsigned int>(clock()) - t0;
    return r;
}
#define LT_WAIT_BOTH(bar_a, parity_a, bar_b, parity_b, code) \
    traced_wait_warp(trace_, bar_a, parity_a, bar_b, parity_b, abort_flag, p.status, code)
// (two barriers one after the other, so that each gets the cycles that it took)
__device__ __forceinline__ bool traced_wait_warp(Trace &tr, uint64_t *bar_a, uint32_t parity_a, uint64_t *bar_b, uint32_t parity_b,
                                                 volatile int *abort_flag, unsigned int *status, int code) {
    const unsigned int t0 = static_cast<unsigned int>(clock());
    bool r = mbar_wait_warp(bar_a, parity_a, nullptr, 0, abort_flag, status, code);
    const unsigned int t1 = static_cast<unsigned int>(clock());
    tr.acc[(code >= 1000 ? code / 1000 : code) - 200] += t1 - t0;
    if (r && bar_b) {
        r = mbar_wait_warp(bar_b, parity_b, nullptr, 0, abort_flag, status, code);
        tr.acc[code % 1000 - 200] += static_cast<unsigned int>(clock()) - t1;
    }
    return r;
}
#else
#define LT_TRACE_BEGIN()
#define LT_TRACE_MARK(var)
#define LT_TRACE_SINCE(slot, var)
#define LT_TRACE_END(role)
#define LT_WAIT(bar, parity, code) mbar_wait(bar, parity, abort_flag, p.status, code)
#define LT_WAIT_BOTH(bar_a, parity_a, bar_b, parity_b, code) mbar_wait_warp(bar_a, parity_a, bar_b, parity_b, abort_flag, p.status, code)
#endif
// the same wait by a whole warp, on one or two barriers (the second one may be NULL), with a warp-uniform outcome
#define LT_WAIT_ALL(bar, parity, code) LT_WAIT_BOTH(bar, parity, nullptr, 0, code)

// Built only with -DLT_BWD_TIMELINE=<cta> (development aid): clock stamps of that CTA's first 256 iterations.
#ifdef LT_BWD_TIMELINE
__device__ long long g_bwd_timeline[20 * 256];  // [event][iteration]; events are listed in paper_2606_10415_b200/timeline.py
#define LT_TL(cond, ev, iter)                                                                        \
    do {                                                                                             \
        if ((cond) && blockIdx.x == LT_BWD_TIMELINE && (iter) < 256) g_bwd_timeline[(ev) * 256 + (iter)] = clock64(); \
    } while (0)
#else
#define LT_TL(cond, ev, iter) do {} while (0)
#endif

// ----------------------------------------------------------------------------- main kernel
constexpr int kQStages = 2;   // Q_i ring; dO_i is single-buffered (it is dead once dV has been issued)
constexpr int kBwdThreads = 512;  // 16 warps; 128 registers per thread at launch
constexpr int kComputeWarp0 = 4, kNumComputeWarps = 8;
constexpr int kReduceWarp0 = 12, kNumReduceWarps = 4;
// registers per thread once the warpgroups have resized their shares (the SM has 64 K)
constexpr int kRegsAtLaunch = 65536 / kBwdThreads;
constexpr int kRegsControl = 56, kRegsCompute = 160, kRegsReduce = 136;
static_assert(128 * kRegsControl + kNumComputeWarps * 32 * kRegsCompute + kNumReduceWarps * 32 * kRegsReduce <= 65536,
              "register shares exceed the register file");
constexpr int kDqStageBufs = 3, kDqStageRows = 16;
constexpr int kExtBytes = 2048;            // 128 rows x 16 bytes: one operand of the extra contraction step
constexpr float kPScaleLog2Max = 14.f;     // P is kept as P * 2^c with c <= 14 so that fp16(P') <= 16384
constexpr int kBarReduceWarps = 1, kBarScale = 2;  // named barrier ids
constexpr int kItemRing = 4;  // roles are never more than two items apart
constexpr double kL2BatchBytes = 80.0e6;  // working set of one batch of work items (L2 holds 126 MB)

// A CTA's way through its stretch (in shared memory: the producer has few registers).
struct BwdWalk {
    int unit, j, start, begin, end;  // the next key tile and its place in the walk, the stretch

    __device__ __forceinline__ void reset(const BwdDeal &d) {
        const int unit_cost = d.tile_start(d.n_tiles);
        begin = d.stretch(blockIdx.x);
        end = d.stretch(blockIdx.x + 1);
        unit = begin / unit_cost;
        j = d.tile_at(begin - unit * unit_cost);
        start = unit * unit_cost + d.tile_start(j);
    }
    __device__ __forceinline__ int4 next(const BwdDeal &d) {
        while (start < end) {
            const int n = d.pairs(j), tile = unit * d.n_tiles + j;
            const int from = d.cut(begin - start, n), to = d.cut(end - start, n);
            start += kTileCost + n;
            if (++j == d.n_tiles) j = 0, ++unit;
            if (to > from) return make_int4(tile, from, to, from == 0 && to == n ? -1 : d.share(blockIdx.x, tile, from == 0));
        }
        return make_int4(-1, 0, 0, 0);
    }
};
template <int D>
struct BwdSmem {
    static constexpr int kBoxes = D / 64;
    static constexpr int kTile = kBoxes * kBoxBytesBwd;
    uint8_t k[kTile];
    uint8_t v[kTile];
    uint8_t q[kQStages][kTile];
    uint8_t d_o[kTile];
    uint8_t ds[2 * kBoxBytesBwd];      // dS^T: rows = key index, 128 query columns in two swizzled tiles
    // operands of the extra contraction step that subtracts LSE/scale from S and delta from dP
    uint8_t ext_ones[kExtBytes];       // rows (256, 1, 0...): goes with K_j and with V_j
    uint8_t ext_q[kQStages][kExtBytes];// rows (hi, lo, 0...) of -LSE/scale for the stage's query tile
    uint8_t ext_do[kExtBytes];         // rows (hi, lo, 0...) of -delta
    uint8_t ext_zero[kExtBytes];       // contraction elements 8-15 of all of the above
    // staging of the dQ partial for bulk reduction into global memory (D = 128 only):
    // each buffer holds 16 accumulator rows (16 query rows x 128 floats)
    // (D = 64: two buffers of a whole partial, 128 query rows x 64 floats, each as two swizzled boxes of 32 columns)
    float dq_stage[D == 128 ? kDqStageBufs : 2][D == 128 ? kDqStageRows * 128 : kTileRows * 64];
    // per work item: K/V landed; dK/dV accumulators complete; accumulators read out
    uint64_t bar_kv, bar_dkv_full, bar_acc_free;
    // work items are claimed from a global counter by the producer and published to the other roles
    uint64_t bar_item[kItemRing];
    int4 item_ring[kItemRing];  // (x alone where key tiles are whole)
    // per (query head, query tile) iteration
    uint64_t bar_q_full[kQStages], bar_q_empty[kQStages], bar_do_full, bar_do_empty;
    uint64_t bar_s_full, bar_p_ready, bar_dp_full, bar_ds_ready, bar_ds_free, bar_dq_full, bar_dq_empty;
    BwdWalk walk;
    int4 first_item;
    uint32_t tmem_base;
    int abort_flag;
    unsigned int call_max[3];  // the call's maxima (slot bits of max |delta|, max ||dO_row||^2, max ||V_row||^2)
};

static_assert(sizeof(BwdSmem<128>) <= 232448, "main kernel shared memory exceeds the 227 KB per-block limit");

// What the one-tile variant needs besides BwdParams: the preprocess pass's operands and the dQ output.
struct BwdOneTileParams {
    PreParams pre;
    __half *dQ;
    lt_tensor_strides dq_st;
    int own_pre;  // run that pass in the main kernel
};

struct BwdParams {
    const uint4 *lse_ext;    // per query row: fp16 (hi, lo, 0 x 6) with 256*hi + lo = -LSE / scale
    const uint4 *delta_ext;  // per query row: fp16 (hi, lo, 0 x 6) with 256*hi + lo = -delta
    float *dq_acc;
    __half *dK;
    __half *dV;
    unsigned int *status;
    int B, Hq, Hkv, S, S_pad, causal;  // S_pad: S rounded up to whole 128-row tiles
    int units_per_batch;  // (batch, kv head) units per L2-sized batch of work items
    BwdDeal deal;         // of the variant that splits key tiles
    float4 *shares;
    float scale;
    lt_tensor_strides dk_st, dv_st;  // element strides of dK and dV
};

// One work item = key tile j of (batch b, kv head g): the flattened (query head of the group, query tile) loop, or a
// stretch of it.
struct BwdItem {
    int j, b, g, i_first, tiles_per_head, n_iter;
    int n_first;  // first iteration of the flattened loop this item covers
    int share;    // where its dK_j and dV_j go: a share, or (-1) the outputs
};
// Items are numbered batch of (batch, kv head) units by batch; inside a batch key tile by key tile (heavy tiles
// first), all units of the batch per key tile.  A batch is sized so that everything its items touch (K, V, the
// group's Q and dO, the fp32 dQ rows) stays in L2 while the CTAs work through it; with one batch this is the plain
// heavy-first order.
__device__ __forceinline__ void bwd_item_place(const BwdParams &p, int item, int &j, int &bg) {
    const int n_tiles = (p.S + kTileRows - 1) / kTileRows;  // the last tile may be ragged
    const int batch = item / (p.units_per_batch * n_tiles);
    const int first_unit = batch * p.units_per_batch;
    const int units = min(p.units_per_batch, p.B * p.Hkv - first_unit);
    const int within = item - first_unit * n_tiles;
    j = within / units;
    bg = first_unit + within - j * units;
}
// half `item & 1` of item `item >> 1`, as the producer publishes parts of key tiles: {unit * key tiles + j, first pair, end, share}
__device__ __forceinline__ int4 bwd_half_item(const BwdParams &p, int item) {
    int j, bg;
    bwd_item_place(p, item >> 1, j, bg);
    const int n = p.deal.pairs(j), tile = bg * p.deal.n_tiles + j, mid = (n + 1) >> 1, half = item & 1;
    return make_int4(tile, half ? mid : 0, half ? n : mid, 2 * tile + half);
}
template <bool kSplit>
__device__ __forceinline__ BwdItem bwd_item(const BwdParams &p, const int4 &rec) {
    BwdItem w;
    const int n_tiles = (p.S + kTileRows - 1) / kTileRows;
    int bg;
    if constexpr (kSplit) {
        bg = rec.x / n_tiles;
        w.j = rec.x - bg * n_tiles;
    } else {
        bwd_item_place(p, rec.x, w.j, bg);
    }
    w.b = bg / p.Hkv;
    w.g = bg - w.b * p.Hkv;
    w.i_first = p.causal ? w.j : 0;
    w.tiles_per_head = n_tiles - w.i_first;
    w.n_first = kSplit ? rec.y : 0;
    w.n_iter = kSplit ? rec.z - rec.y : (p.Hq / p.Hkv) * w.tiles_per_head;
    w.share = kSplit ? rec.w : -1;
    return w;
}
// Iteration n of an item -> its query tile: batch, query head, first row inside the head, and the tile's first row in the padded row space of the workspace arrays
// (every head rounded up to whole tiles, so tiles never straddle heads).
struct BwdQTile {
    int b, h, s0;
    long long padded_row0;
};
__device__ __forceinline__ BwdQTile bwd_q_tile(const BwdParams &p, const BwdItem &w, int n) {
    n += w.n_first;
    const int hh = n / w.tiles_per_head;
    const int i = w.i_first + (n - hh * w.tiles_per_head);
    BwdQTile q;
    q.b = w.b;
    q.h = w.g * (p.Hq / p.Hkv) + hh;
    q.s0 = i * kTileRows;
    q.padded_row0 = (static_cast<long long>(w.b) * p.Hq + q.h) * p.S_pad + q.s0;
    return q;
}

// The saved P^T tile (128 keys x 128 queries, fp16, 32 KB) of key tile w.j and query tile qt.
__device__ __forceinline__ const __half *saved_p_tile(const BwdParams &p, const BwdItem &w, const BwdQTile &qt) {
    const long long n_tiles = p.S_pad / kTileRows;
    const long long tile = ((static_cast<long long>(qt.b) * p.Hq + qt.h) * n_tiles + w.j) * n_tiles + qt.s0 / kTileRows;
    return reinterpret_cast<const __half *>(p.lse_ext) + tile * (kTileRows * kTileRows);
}

// The exponent c of the power of two that P carries (P' = P * 2^c, c <= 14), and with it dS, so that
// dS' uses fp16's normal range without overflow when it is rounded: chosen from a bound on
// |dS| <= |dP| + |delta| <= max ||dO_row|| * max ||V_row|| + max |delta| over the whole call (the
// three maxima come from the preprocess kernel, one slot per block of it).  dV and dQ / dK undo the factor
// exactly in their epilogues.  Run once per CTA by the softmax and reduction warps together.
// slots_used = false: the maxima are in call_max already.
template <int D>
__device__ __forceinline__ int bwd_p_scale_log2(const BwdParams &p, unsigned int *call_max, bool slots_used) {
    constexpr int kThreads = (kNumComputeWarps + kNumReduceWarps) * 32;
    const long long n_rows = static_cast<long long>(p.B) * p.Hq * p.S_pad;
    // (the -LSE/scale rows follow the -delta rows; the saved-P variant's lse_ext points elsewhere)
    const uint2 *slots = reinterpret_cast<const uint2 *>(p.delta_ext + n_rows) + 1;
    const int n = slots_used ? pre_blocks<D>(n_rows) : 0;
    unsigned int m[3] = {0u, 0u, 0u};
#pragma unroll
    for (int u = 0; u < (kPreMaxBlocks + kThreads - 1) / kThreads; ++u) {
        const int k = static_cast<int>(threadIdx.x) - kComputeWarp0 * 32 + u * kThreads;
        if (k < n) {
            const uint2 v = __ldcg(slots + static_cast<long long>(k) * (pre_rows_per_block<D>() * 2));
            m[0] = max(m[0], v.x & 0xFFFFu);
            m[1] = max(m[1], v.x >> 16);
            m[2] = max(m[2], v.y);
        }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        m[k] = __reduce_max_sync(0xffffffffu, m[k]);
        if ((threadIdx.x & 31) == 0 && m[k]) atomicMax(call_max + k, m[k]);
    }
    named_barrier_sync(kBarScale, kThreads);
    const unsigned int delta = call_max[0], do2 = call_max[1], v2 = call_max[2];
    if (max(max(delta, do2), v2) >= kMaxSlotInf) return -14;  // inf/NaN inputs: outputs are non-finite anyway
    const float bound = sqrtf(__uint_as_float(do2 << 16)) * sqrtf(__uint_as_float(v2 << 16)) + __uint_as_float(delta << 16);
    if (!(bound < 3.0e38f)) return -14;
    if (!(bound > 1e-30f)) return static_cast<int>(kPScaleLog2Max);  // all-zero dO: any factor works
    return min(static_cast<int>(kPScaleLog2Max), max(-14, ilogbf(32768.f / bound)));
}

// kSavedP: the variant that loads the probability tiles a forward pass saved (lt_attn_save_p's store)
// instead of recomputing them.  It issues no S product; the producer asks for each P^T tile to be
// brought into L2 one iteration ahead and every softmax thread reads its own 128 bytes of the tile
// straight into registers.  BwdParams::lse_ext, which this variant does not need, carries the
// store's address (the parameter block keeps its size).
//
// kOneTile: the variant for sequences of one tile (S <= 128).  A query tile then has one partial, so dQ leaves the
// reduction warps rounded, without accumulator, zero fill and conversion kernel; and where a CTA has few heads to
// go through (own_pre) it runs the preprocess pass over its own units' rows itself and picks its own factor 2^c, so that
// the call is one launch.  Work items are dealt out by block number.  one_tile_launches() says when and what it measured.
template <int D, bool kBf16, bool kSplit, bool kSavedP = false, bool kOneTile = false>
__global__ void __launch_bounds__(kBwdThreads, 1)
bwd_main_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_do,
                const BwdParams p, const __grid_constant__ CUtensorMap map_dq, const __grid_constant__ CUtensorMap map_dk,
                const __grid_constant__ CUtensorMap map_dv, const BwdOneTileParams one) {
    // map_dq (D = 64 only): the fp32 dQ accumulator as rows of 64 floats, boxes of 128 rows x 32 columns
    // map_dk, map_dv (whole key tiles only): the outputs, boxes of 32 rows x 64 columns
    using Smem = BwdSmem<D>;
    constexpr int kBoxes = D / 64;
    constexpr uint32_t kTileBytes = kBoxes * kBoxBytesBwd;
    constexpr uint32_t kTmemCols = 512;
    constexpr uint32_t kColS = 0, kColdP = 128, kColdV = 256, kColdK = 384;

    extern __shared__ __align__(1024) uint8_t smem_raw[];
    Smem &sm = *reinterpret_cast<Smem *>(smem_raw);
#ifdef LT_BWD_TRACE
    const long long trace_cta_t0 = clock64();
#endif
    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int n_items = p.B * p.Hkv * (p.S_pad / kTileRows) * (kSplit ? 2 : 1);  // (split: in halves)

    // the swizzled tiles need 1024-byte alignment; the shared window is expected to give it
    const bool smem_ok = (smem_u32(smem_raw) & 1023u) == 0u;
    if (tid == 0) {
        sm.abort_flag = smem_ok ? 0 : 1;
        sm.call_max[0] = sm.call_max[1] = sm.call_max[2] = 0u;
        mbar_init(&sm.bar_kv, 1);
        mbar_init(&sm.bar_dkv_full, 1);
        mbar_init(&sm.bar_acc_free, kNumReduceWarps);
        for (int r = 0; r < kItemRing; ++r) mbar_init(&sm.bar_item[r], 1);
        for (int s = 0; s < kQStages; ++s) {
            mbar_init(&sm.bar_q_full[s], 1);
            mbar_init(&sm.bar_q_empty[s], 1);
        }
        mbar_init(&sm.bar_do_full, 1);
        mbar_init(&sm.bar_do_empty, 1);
        mbar_init(&sm.bar_s_full, 1);
        mbar_init(&sm.bar_p_ready, kNumComputeWarps);
        mbar_init(&sm.bar_dp_full, 1);
        mbar_init(&sm.bar_ds_ready, kNumComputeWarps);
        mbar_init(&sm.bar_ds_free, 1);
        mbar_init(&sm.bar_dq_full, 1);
        mbar_init(&sm.bar_dq_empty, kNumReduceWarps);
        mbar_fence_init();
        tma_prefetch_desc(&map_q);
        tma_prefetch_desc(&map_k);
        tma_prefetch_desc(&map_v);
        tma_prefetch_desc(&map_do);
    }
    if (warp == 0) {
        tmem_alloc(&sm.tmem_base, kTmemCols);
        tmem_relinquish();
    }
    if (warp == 1) {
        // constant operands of the extra contraction step
        const uint2 mult = ext_multipliers<kBf16>();
        for (int r = lane; r < kTileRows; r += 32) {
            reinterpret_cast<uint4 *>(sm.ext_ones)[r] = make_uint4(mult.x, mult.y, 0u, 0u);
            reinterpret_cast<uint4 *>(sm.ext_zero)[r] = make_uint4(0u, 0u, 0u, 0u);
        }
        fence_proxy_async_smem();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    // The first work item of a CTA is its block number, and its first tiles are fetched while the preprocess kernel is
    // still running: they are the caller's tensors, complete before that kernel let this one start (it does so after
    // its own wait for its predecessor).  Saves the claim (800 cycles) and the tile latency (1 800) of every call.
    // (A call of one launch has no such predecessor, and fetches after its wait.)
    // (There, where a CTA's only pair is its own unit's, the row operands of the extra contraction steps go straight to shared
    // memory instead of to the workspace and back: 8.4 -> 8.0 us for the smallest call, 11.9 -> 11.3 for 16 heads of 64 rows, D = 128.)
    bool own_rows = false;
    if constexpr (kOneTile) {
        if (one.own_pre) grid_dependency_wait();
        own_rows = one.own_pre && p.Hq == p.Hkv && p.B * p.Hkv == static_cast<int>(gridDim.x);
    }
    const uint32_t ext_tx = own_rows ? 0u : kExtBytes;
    if (warp == 0 && lane == 0 && smem_ok) {
        int4 rec = make_int4(static_cast<int>(blockIdx.x), 0, 0, 0);
        if constexpr (kSplit) {
            if (p.deal.halves) {
                rec = bwd_half_item(p, static_cast<int>(blockIdx.x));
            } else {
                sm.walk.reset(p.deal);
                rec = sm.walk.next(p.deal);
            }
            sm.first_item = rec;
        }
        if (!kSplit || rec.x >= 0) {
            const BwdItem w = bwd_item<kSplit>(p, rec);
            const BwdQTile qt = bwd_q_tile(p, w, 0);
            mbar_arrive_expect_tx(&sm.bar_q_full[0], kSavedP ? kTileBytes : kTileBytes + ext_tx);
            mbar_arrive_expect_tx(&sm.bar_kv, 2 * kTileBytes);
            mbar_arrive_expect_tx(&sm.bar_do_full, kTileBytes + ext_tx);
#pragma unroll
            for (int x = 0; x < kBoxes; ++x) {
                tma_load_4d(sm.q[0] + x * kBoxBytesBwd, &map_q, &sm.bar_q_full[0], x * 64, qt.s0, qt.h, qt.b);
                tma_load_4d(sm.k + x * kBoxBytesBwd, &map_k, &sm.bar_kv, x * 64, w.j * kTileRows, w.g, w.b);
                tma_load_4d(sm.d_o + x * kBoxBytesBwd, &map_do, &sm.bar_do_full, x * 64, qt.s0, qt.h, qt.b);
                tma_load_4d(sm.v + x * kBoxBytesBwd, &map_v, &sm.bar_kv, x * 64, w.j * kTileRows, w.g, w.b);
            }
        }
    }
    // everything above ran while the preprocess kernel was finishing; its results (row operands, zeroed
    // accumulator, running maxima, item counter) are read only from here on
    grid_dependency_wait();
    if constexpr (kOneTile) {
        if (one.own_pre) {
            if (blockIdx.x == 0 && tid == 0) p.status[kStatusWordTimeout] = 0u;  // (a wait gives up after a second at the earliest)
            float max_abs_delta = 0.f, max_norm2 = 0.f;
            unsigned int max_v2 = 0u;
            __syncwarp();
            PreParams pre = one.pre;
            if (own_rows) {  // rows blockIdx.x * 128 and on
                pre.delta_ext = reinterpret_cast<uint4 *>(sm.ext_do) - static_cast<long long>(blockIdx.x) * kTileRows;
                pre.lse_ext = reinterpret_cast<uint4 *>(sm.ext_q[0]) - static_cast<long long>(blockIdx.x) * kTileRows;
            }
            for (int un = blockIdx.x; un < p.B * p.Hkv; un += gridDim.x) {
                const long long rows = static_cast<long long>(p.Hq / p.Hkv) * p.S_pad;  // the group's heads are neighbours
                pre_rows<D, kBf16>(pre, un * rows, (un + 1) * rows, warp, kBwdThreads / 32, max_abs_delta, max_norm2);
                pre_v_rows<D, kBf16>(one.pre, static_cast<long long>(un) * p.S, static_cast<long long>(un + 1) * p.S,
                                     kBwdThreads / 32 - 1 - warp, kBwdThreads / 32, max_v2);
            }
            const unsigned int m[3] = {__float_as_uint(max_abs_delta) & 0x7fffffffu, __float_as_uint(max_norm2) & 0x7fffffffu, max_v2};
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const unsigned int v = __reduce_max_sync(0xffffffffu, m[k]);
                if (lane == 0 && v) atomicMax(sm.call_max + k, max_slot_bits(v));
            }
            // the operand rows written above are read by bulk copies of this CTA
            asm volatile("fence.proxy.async;" ::: "memory");
            __syncthreads();
        }
    }
    if (!smem_ok && tid == 0) atomicCAS(p.status + kStatusWordTimeout, 0u, static_cast<unsigned int>(kBadSmemAlign));
    const uint32_t tmem = sm.tmem_base;
    volatile int *abort_flag = &sm.abort_flag;
#ifdef LT_BWD_TRACE
    const long long trace_prologue_end = clock64();
    int trace_iters = 0;
#endif

    // Every role walks the same list of work items and keeps its own running iteration count
    // `it` (over all items): each per-iteration barrier completes once per iteration, so its
    // phase parity is a function of `it`; the per-item barriers use the item count `ic`.
    if (warp < kComputeWarp0) {
        // ================================================================= control group
        warpgroup_regs_set<kRegsControl, kRegsAtLaunch>();
        if (warp == 0) {
            // ================================================================= TMA producer
            if (lane == 0 && smem_ok) {
                LT_TRACE_BEGIN();
                bool ok = true;
                int it = 0, ic = 0;
                int last_q = -1, last_do = -1, kv_loads = 0;  // for the cleanup after an abandoned wait
                // claim the next unclaimed item (heavy ones have the low numbers; the grid's first ones are the CTAs'
                // first items) and publish it to the other roles; -1 tells everybody that the list is exhausted
                auto claim = [&](int slot_ic) -> int4 {
                    int4 rec = make_int4(-1, 0, 0, 0);
                    if (kSplit && slot_ic == 0) {
                        rec = sm.first_item;
                    } else if (kSplit && !p.deal.halves) {
                        rec = sm.walk.next(p.deal);
                    } else {
                        unsigned int v = blockIdx.x;
                        if constexpr (kOneTile) v += slot_ic * gridDim.x;
                        else if (slot_ic > 0) v = atomicAdd(p.status + kStatusWordItemCounter, 1u) + gridDim.x;
                        if (v < static_cast<unsigned int>(n_items)) {
                            rec.x = static_cast<int>(v);
                            if constexpr (kSplit) rec = bwd_half_item(p, rec.x);
                        }
                    }
                    if constexpr (kSplit) sm.item_ring[slot_ic % kItemRing] = rec;
                    else sm.item_ring[slot_ic % kItemRing].x = rec.x;
                    mbar_arrive(&sm.bar_item[slot_ic % kItemRing]);
                    return rec;
                };
                int4 item = claim(0);
                while (item.x >= 0 && ok) {
                    const BwdItem w = bwd_item<kSplit>(p, item);
                    int4 next_item = make_int4(-1, 0, 0, 0);
                    for (int n = 0; n < w.n_iter && ok; ++n, ++it) {
                        const int s = it & 1, k = it >> 1;
                        const BwdQTile qt = bwd_q_tile(p, w, n);
                        if (k >= 1 && !(ok = LT_WAIT(&sm.bar_q_empty[s], (k - 1) & 1, kWaitStageEmpty))) break;
                        if (it > 0) {  // (the tiles of the first pair are on their way)
                            mbar_arrive_expect_tx(&sm.bar_q_full[s], kSavedP ? kTileBytes : kTileBytes + kExtBytes);
#pragma unroll
                            for (int x = 0; x < kBoxes; ++x)
                                tma_load_4d(sm.q[s] + x * kBoxBytesBwd, &map_q, &sm.bar_q_full[s], x * 64, qt.s0, qt.h, qt.b);
                        }
                        if constexpr (kSavedP)
                            bulk_prefetch_l2(saved_p_tile(p, w, qt), kTileRows * kTileRows * 2);
                        else if (!own_rows)
                            bulk_load_1d(sm.ext_q[s], p.lse_ext + qt.padded_row0, kExtBytes, &sm.bar_q_full[s]);
                        last_q = it;
                        if (it >= 1 && !(ok = LT_WAIT(&sm.bar_do_empty, (it - 1) & 1, kWaitDoEmpty))) break;
                        if (it > 0) {
                            mbar_arrive_expect_tx(&sm.bar_do_full, kTileBytes + kExtBytes);
#pragma unroll
                            for (int x = 0; x < kBoxes; ++x)
                                tma_load_4d(sm.d_o + x * kBoxBytesBwd, &map_do, &sm.bar_do_full, x * 64, qt.s0, qt.h, qt.b);
                        }
                        if (!own_rows) bulk_load_1d(sm.ext_do, p.delta_ext + qt.padded_row0, kExtBytes, &sm.bar_do_full);
                        last_do = it;
                        if (n == 0) {
                            // K_j and V_j follow the first query tile: they may only be overwritten once every
                            // product of the previous item has completed
                            if (ic >= 1) {
                                if (!(ok = LT_WAIT(&sm.bar_dkv_full, (ic - 1) & 1, kWaitDkvFull))) break;
                                mbar_arrive_expect_tx(&sm.bar_kv, 2 * kTileBytes);
#pragma unroll
                                for (int x = 0; x < kBoxes; ++x) {
                                    tma_load_4d(sm.k + x * kBoxBytesBwd, &map_k, &sm.bar_kv, x * 64, w.j * kTileRows, w.g, w.b);
                                    tma_load_4d(sm.v + x * kBoxBytesBwd, &map_v, &sm.bar_kv, x * 64, w.j * kTileRows, w.g, w.b);
                                }
                            }
                            ++kv_loads;
                        }
                        if (n == w.n_iter - 1) {
                            // with the last query tile of this item on its way, claim the next item and ask for
                            // its K/V tiles to be brought into L2 while this item finishes
                            next_item = claim(ic + 1);
                            if (next_item.x >= 0) {
                                const BwdItem wn = bwd_item<kSplit>(p, next_item);
#pragma unroll
                                for (int x = 0; x < kBoxes; ++x) {
                                    tma_prefetch_l2_4d(&map_k, x * 64, wn.j * kTileRows, wn.g, wn.b);
                                    tma_prefetch_l2_4d(&map_v, x * 64, wn.j * kTileRows, wn.g, wn.b);
                                }
                            }
                        }
                    }
                    item = next_item;
                    ++ic;
                }
                LT_TRACE_END(kRoleProducer);
                if (*abort_flag) {
                    // abandoned: give this CTA's own copies a bounded time to land before shared memory is released
                    if (kv_loads > 0)
                        for (int t = 0; t < (1 << 16) && !mbar_try_wait(&sm.bar_kv, (kv_loads - 1) & 1); ++t) {}
                    for (int n = max(0, last_q - 1); n <= last_q; ++n)
                        for (int t = 0; t < (1 << 16) && !mbar_try_wait(&sm.bar_q_full[n & 1], (n >> 1) & 1); ++t) {}
                    if (last_do >= 0)
                        for (int t = 0; t < (1 << 16) && !mbar_try_wait(&sm.bar_do_full, last_do & 1); ++t) {}
                }
            }
            __syncwarp();
        } else if (warp == 1) {
            // ================================================================= tensor-core issuer
            // The whole warp walks the loop, so that loop counters, wait results (voted) and descriptor arithmetic are
            // warp-uniform; one elected lane issues the products and commits.
            if (smem_ok) {
                const bool leader = elect_one();
                LT_TRACE_BEGIN();
                // Every operand descriptor is a compile-time constant (built from the operand's offset inside
                // the shared window) plus the window's base in the address field (bits 0-13, units of 16
                // bytes; shared memory stays below 256 KB, so the sum never carries out of the field).  The
                // issuing thread spends one 64-bit add per descriptor, so the tensor pipe, not this thread,
                // sets the pace.  The base is re-read through window_base() once per tile pair: otherwise the
                // compiler keeps all ~80 sums of an iteration in registers across the loop, and the control
                // group could not hand most of its registers to the other warpgroups.
                const uint32_t base16 = smem_u32(smem_raw) >> 4;
                auto window_base = [&]() -> uint64_t {
                    uint32_t v;
                    asm volatile("mov.u32 %0, %1;" : "=r"(v) : "r"(base16));
                    return static_cast<uint64_t>(v);
                };
                constexpr uint32_t oK = offsetof(Smem, k), oV = offsetof(Smem, v), oQ = offsetof(Smem, q);
                constexpr uint32_t oDo = offsetof(Smem, d_o), oDs = offsetof(Smem, ds), oZero = offsetof(Smem, ext_zero);
                constexpr uint32_t oOnes = offsetof(Smem, ext_ones), oExtQ = offsetof(Smem, ext_q), oExtDo = offsetof(Smem, ext_do);
                constexpr uint64_t dK_k = desc_kmajor(oK), dV_k = desc_kmajor(oV);
                constexpr uint64_t dK_mn = desc_mnmajor(oK, kBoxBytesBwd);
                constexpr uint64_t ddS_mn = desc_mnmajor(oDs, kBoxBytesBwd);
                constexpr uint64_t ddO_k = desc_kmajor(oDo), ddO_mn = desc_mnmajor(oDo, kBoxBytesBwd);
                constexpr uint64_t dQ_k0 = desc_kmajor(oQ), dQ_mn0 = desc_mnmajor(oQ, kBoxBytesBwd);
                constexpr uint64_t kQStageStep = static_cast<uint64_t>(Smem::kTile) >> 4;  // next Q stage
                constexpr uint64_t desc_ones = desc_kmajor_noswz(oOnes, oZero - oOnes, 128);
                constexpr uint64_t desc_ext_do = desc_kmajor_noswz(oExtDo, oZero - oExtDo, 128);
                constexpr uint64_t desc_ext_q0 = desc_kmajor_noswz(oExtQ, oZero - oExtQ, 128);
                constexpr uint64_t desc_ext_q1 = desc_kmajor_noswz(oExtQ + kExtBytes, oZero - oExtQ - kExtBytes, 128);
                // address-field increments of contraction step kk: within a contraction-contiguous tile
                // (32 bytes per step, next 64-column tile after four steps) and within a row-contracted
                // tile (16 rows of 128 bytes per step)
                constexpr auto koff = [](int kk) -> uint64_t { return static_cast<uint64_t>((kk >> 2) * (kBoxBytesBwd >> 4) + (kk & 3) * 2); };
                constexpr auto roff = [](int kk) -> uint64_t { return static_cast<uint64_t>(kk * (2048 >> 4)); };
                constexpr uint32_t idesc_s = make_idesc(128, 128, false, false, kBf16);
                constexpr uint32_t idesc_dv = make_idesc(128, D, false, true, kBf16);
                constexpr uint32_t idesc_dq = make_idesc(128, D == 128 ? 128 : D, true, true, kBf16);
                auto issue_s = [&](int t) {  // S^T = K_j Q_i^T - LSE_i / scale, for running iteration t
                    if (!leader) return;
                    const uint64_t wb = window_base();
                    const uint64_t dQ_k = wb + (t & 1) * kQStageStep;
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk)
                        umma_ss(tmem + kColS, wb + (dK_k + koff(kk)), dQ_k + (dQ_k0 + koff(kk)), idesc_s, kk > 0);
                    umma_ss(tmem + kColS, wb + desc_ones, wb + ((t & 1) ? desc_ext_q1 : desc_ext_q0), idesc_s, 1);
                    umma_commit(&sm.bar_s_full);
                };
                bool ok = true;
                int it = 0, ic = 0;
                for (;; ++ic) {
                    if (!(ok = LT_WAIT_ALL(&sm.bar_item[ic % kItemRing], (ic / kItemRing) & 1, kWaitItem))) break;
                    const int4 item = sm.item_ring[ic % kItemRing];
                    if (item.x < 0) break;
                    const BwdItem w = bwd_item<kSplit>(p, item);
                    if (!(ok = LT_WAIT_BOTH(&sm.bar_kv, ic & 1, &sm.bar_q_full[it & 1], (it >> 1) & 1,
                                            both_codes(kWaitKV, kWaitStageFull)))) break;
                    tc_fence_after_sync();
                    LT_TL(leader, 14, it);
                    if constexpr (!kSavedP) issue_s(it);
                    for (int n = 0; n < w.n_iter && ok; ++n, ++it) {
                        const int s = it & 1;
                        const uint64_t wb = window_base();
                        const uint64_t dQ_mn = wb + s * kQStageStep;
                        // dP^T = V_j dO_i^T - delta_i   (its columns held the previous dQ partial until the
                        //                                reduce warps drained it)
                        auto issue_dp = [&]() {
                            if (!leader) return;
#pragma unroll
                            for (int kk = 0; kk < D / 16; ++kk)
                                umma_ss(tmem + kColdP, wb + (dV_k + koff(kk)), wb + (ddO_k + koff(kk)), idesc_s, kk > 0);
                            umma_ss(tmem + kColdP, wb + desc_ones, wb + desc_ext_do, idesc_s, 1);
#ifdef LT_BWD_GIVEUP_TEST
                            // test build only: the hand-off of running iteration LT_BWD_GIVEUP_TEST is dropped, so
                            // the waits downstream of it run out and the kernel has to leave through its give-up path
                            if (it != LT_BWD_GIVEUP_TEST)
#endif
                            umma_commit(&sm.bar_dp_full);
                        };
                        // dV_j += P'^T dO_i   (A = P'^T from tensor memory; query columns 0-63 sit at columns
                        //                      0-31, query columns 64-127 at columns 64-95 of the S region)
                        auto issue_dv = [&]() {
                            if (!leader) return;
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk)
                                umma_ts(tmem + kColdV, tmem + kColS + (kk >> 2) * 64 + (kk & 3) * 8, wb + (ddO_mn + roff(kk)),
                                        idesc_dv, (n > 0) | (kk > 0));
                        };
                        LT_TL(leader, 0, it);
                        // dO_i and the -delta rows have landed (both dP and dV read them), the dQ partial has been drained
                        if (!(ok = LT_WAIT_BOTH(&sm.bar_do_full, it & 1, it > 0 ? &sm.bar_dq_empty : nullptr, (it - 1) & 1,
                                                both_codes(kWaitDoFull, kWaitDqEmpty)))) break;
                        tc_fence_after_sync();
                        LT_TL(leader, 1, it);
                        issue_dp();
                        LT_TL(leader, 2, it);
                        // (the first product of an item overwrites accumulators the previous item's epilogue reads)
                        if (!(ok = LT_WAIT_BOTH(&sm.bar_p_ready, it & 1, n == 0 && ic > 0 ? &sm.bar_acc_free : nullptr, (ic - 1) & 1,
                                                both_codes(kWaitPReady, kWaitAccFree)))) break;
                        LT_TL(leader, 3, it);
                        tc_fence_after_sync();
                        issue_dv();
                        if (leader) umma_commit(&sm.bar_do_empty);
                        // the next S^T overwrites P'^T; the tensor pipe executes in issue order
                        if (n + 1 < w.n_iter) {
                            if (!(ok = LT_WAIT_ALL(&sm.bar_q_full[(it + 1) & 1], ((it + 1) >> 1) & 1, kWaitStageFull))) break;
                            if constexpr (!kSavedP) issue_s(it + 1);
                        }
                        LT_TL(leader, 4, it);
                        if (!(ok = LT_WAIT_ALL(&sm.bar_ds_ready, it & 1, kWaitDsReady))) break;
                        tc_fence_after_sync();
                        LT_TL(leader, 5, it);
                        // dK_j += dS'^T Q_i   (A = dS'^T from tensor memory, stored like P'^T: query columns
                        //                       0-63 at columns 0-31 and 64-127 at columns 64-95 of the dP region)
                        if (leader) {
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk)
                                umma_ts(tmem + kColdK, tmem + kColdP + (kk >> 2) * 64 + (kk & 3) * 8, dQ_mn + (dQ_mn0 + roff(kk)), idesc_dv,
                                        (n > 0) | (kk > 0));
                            umma_commit(&sm.bar_q_empty[s]);
                        }
                        // dQ_i partial (contraction over key rows); it overwrites the dP columns, which is safe
                        // after dK because the tensor pipe executes in issue order.  For D = 128 it is
                        // produced transposed, dQ^T = K_j^T dS^T (lanes = head dim, columns = query rows), so
                        // that the reduction moves whole accumulator rows; for D = 64 as dQ = dS K_j.
                        if (leader) {
#pragma unroll
                            for (int kk = 0; kk < 8; ++kk) {
                                if constexpr (D == 128)
                                    umma_ss(tmem + kColdP, wb + (dK_mn + roff(kk)), wb + (ddS_mn + roff(kk)), idesc_dq, kk > 0);
                                else
                                    umma_ss(tmem + kColdP, wb + (ddS_mn + roff(kk)), wb + (dK_mn + roff(kk)), idesc_dq, kk > 0);
                            }
                            umma_commit(&sm.bar_dq_full);
                            umma_commit(&sm.bar_ds_free);
                        }
                        LT_TL(leader, 6, it);
                    }
                    if (!ok) break;
                    if (leader) umma_commit(&sm.bar_dkv_full);
                }
                LT_TRACE_END(kRoleMma);
            }
            __syncwarp();
        }
    } else if (warp < kReduceWarp0) {
        // ================================================================= softmax / dS warps
        warpgroup_regs_set<kRegsCompute, kRegsAtLaunch>();
        const int quad = warp & 3;                           // tensor-memory lane quadrant
        const int half_sel = (warp - kComputeWarp0) >> 2;    // 0: query columns 0-63, 1: 64-127
        const int row = quad * 32 + lane;                    // key row inside the tile
        const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
        const uint32_t cbase = half_sel * 64;
        const float scale_log2 = p.scale * kLog2e;
        uint8_t *ds_tile = sm.ds + half_sel * kBoxBytesBwd;
        uint32_t pv[64];  // bits of this thread's 64 fp32 values of P' = P * 2^c for the current tile pair
        const float p_scale_log2 = static_cast<float>(bwd_p_scale_log2<D>(p, sm.call_max, !kOneTile || !one.own_pre));
        const uint64_t scale_log2_2 = f32x2(scale_log2, scale_log2), p_scale_log2_2 = f32x2(p_scale_log2, p_scale_log2);
        bool ok = smem_ok;
        int it = 0, ic = 0;
        LT_TRACE_BEGIN();

        // saved-P variant: this thread's 64 saved probabilities of the current tile pair (ph) and of the
        // next one (pn, in flight while dS of the current pair is formed), as packed fp16 pairs
        uint32_t ph[32], pn[32];
        auto load_saved_p = [&](const BwdItem &w, int n, uint32_t *dst) {
            // the store keeps a tile as sixteen blocks of eight query columns, each [128 keys][8 queries]:
            // the 32 lanes of a warp (consecutive key rows) read 512 contiguous bytes per load
            const uint4 *src = reinterpret_cast<const uint4 *>(saved_p_tile(p, w, bwd_q_tile(p, w, n))) + (cbase / 8) * kTileRows + row;
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const uint4 u = ld_nc_v4(src + v * kTileRows);
                dst[4 * v] = u.x; dst[4 * v + 1] = u.y; dst[4 * v + 2] = u.z; dst[4 * v + 3] = u.w;
            }
        };
        // P' of running iteration t; masked: some keys of the tile are hidden.  D = 64 has an instantiation of its own for
        // that: as selects behind a uniform flag the masks cost every tile 400 cycles of a pass that its tensor products
        // wait for.  D = 128 is not bound by these warps, and a second copy of the pass cost it 3 %.
        auto form_p = [&](const BwdItem &w, int t, bool diag, bool masked, auto masked_tag) -> bool {
            constexpr bool kMasked = decltype(masked_tag)::value;
            if constexpr (kSavedP) {
                // P'^T of the previous pair must have been read by its dV product before it is replaced
                if (t > 0 && !LT_WAIT_ALL(&sm.bar_do_empty, (t - 1) & 1, kWaitDoEmpty)) return false;
                tc_fence_after_sync();
                const uint32_t mult = pack_half2(exp2f(p_scale_log2), exp2f(p_scale_log2));  // 2^c <= 2^14
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t out[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) out[e] = hmul2_bits(ph[c * 16 + e], mult);
                    tmem_st16(tmem + lane_base + kColS + cbase + c * 16, out);
                }
                tmem_wait_st();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.bar_p_ready);
                return true;
            }
            if (!LT_WAIT_ALL(&sm.bar_s_full, t & 1, kWaitSFull)) return false;
            tc_fence_after_sync();
            LT_TL(tid == kComputeWarp0 * 32, 7, t);
            LT_TRACE_MARK(tp0);
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                // (one load at a time: asking for both halves before the first is used measured 2 % slower)
                uint32_t sv[32];
                tmem_ld32(tmem + lane_base + kColS + cbase + c * 32, sv);
                tmem_wait_ld();
                // P' = exp2(scale*log2e * (K.Q - LSE/scale) + c)
#pragma unroll
                for (int e = 0; e < 32; e += 2) {
                    const float2 x = f32x2_parts(f32x2_fma(f32x2(__uint_as_float(sv[e]), __uint_as_float(sv[e + 1])), scale_log2_2, p_scale_log2_2));
                    pv[c * 32 + e] = __float_as_uint(fast_exp2(x.x));
                    pv[c * 32 + e + 1] = __float_as_uint(fast_exp2(x.y));
                }
            }
            if (kMasked || (D == 128 && masked)) {
                // the key row is hidden from the query columns before it (causal diagonal), or it lies past the end of
                // the sequence (ragged last tile): its zero-filled K row has score 0, which LSE does not bound, so its P
                // is not a probability
                const int first = w.j * kTileRows + row >= p.S ? 64 : diag ? row - static_cast<int>(cbase) : 0;
#pragma unroll
                for (int e = 0; e < 64; ++e)
                    if (e < first) pv[e] = 0u;
            }
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                uint32_t out[16];
#pragma unroll
                for (int e = 0; e < 16; ++e)
                    out[e] = pack2<kBf16>(__uint_as_float(pv[c * 32 + 2 * e]), __uint_as_float(pv[c * 32 + 2 * e + 1]));
                // in place: these columns lie inside the 64 columns this thread has just read
                tmem_st16(tmem + lane_base + kColS + cbase + c * 16, out);
            }
            tmem_wait_st();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm.bar_p_ready);
            LT_TL(tid == kComputeWarp0 * 32, 8, t);
            LT_TRACE_SINCE(12, tp0);
            return true;
        };

        // tile: the query tile's index inside its head, counted from the first visible one
        auto compute_p = [&](const BwdItem &w, int t, int tile) -> bool {
            const bool diag = p.causal && tile == 0;
            const bool masked = !kSavedP && (diag || (w.j + 1) * kTileRows > p.S);
            if constexpr (D == 64 && !kSavedP)
                if (masked) return form_p(w, t, diag, true, std::true_type{});
            return form_p(w, t, diag, masked, std::false_type{});
        };

        int last_item = -1;
        for (;; ++ic) {
            if (!ok || !(ok = LT_WAIT_ALL(&sm.bar_item[ic % kItemRing], (ic / kItemRing) & 1, kWaitItem))) break;
            const int4 item = sm.item_ring[ic % kItemRing];
            if (item.x < 0) break;
            last_item = item.x;
            const BwdItem w = bwd_item<kSplit>(p, item);
            if constexpr (kSavedP) load_saved_p(w, 0, ph);
            int tile = kSplit ? w.n_first % w.tiles_per_head : 0;
            ok = compute_p(w, it, tile);
            for (int n = 0; n < w.n_iter && ok; ++n, ++it) {
                if constexpr (kSavedP)
                    if (n + 1 < w.n_iter) load_saved_p(w, n + 1, pn);
                // (the previous dS^T tile must have been consumed by the dQ product before it is overwritten)
                if (!(ok = LT_WAIT_BOTH(&sm.bar_dp_full, it & 1, it > 0 ? &sm.bar_ds_free : nullptr, (it - 1) & 1,
                                        both_codes(kWaitDpFull, kWaitDsFree)))) break;
                tc_fence_after_sync();
                LT_TL(tid == kComputeWarp0 * 32, 9, it);
                LT_TRACE_MARK(td0);
                const float saved_mult = kSavedP ? exp2f(p_scale_log2) : 0.f;
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    uint32_t dp[32];
                    tmem_ld32(tmem + lane_base + kColdP + cbase + c * 32, dp);
                    tmem_wait_ld();
                    // dS' = P' * (dP - delta); the subtraction happened inside the tensor-core product.
                    // The fp16 result goes to shared memory (32 query columns = four 16-byte chunks of row
                    // `row` in this half's tile; operand of the dQ product) and, in place, to tensor
                    // memory (operand of dK).
                    uint32_t o[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        if constexpr (kSavedP) {
                            const float2 f = unpack2<false>(ph[c * 16 + e]);
                            o[e] = pack2<kBf16>(f.x * saved_mult * __uint_as_float(dp[2 * e]),
                                                f.y * saved_mult * __uint_as_float(dp[2 * e + 1]));
                        } else {
                            const float2 x = f32x2_parts(f32x2_mul(f32x2(__uint_as_float(pv[c * 32 + 2 * e]), __uint_as_float(pv[c * 32 + 2 * e + 1])),
                                                                   f32x2(__uint_as_float(dp[2 * e]), __uint_as_float(dp[2 * e + 1]))));
                            o[e] = pack2<kBf16>(x.x, x.y);
                        }
                    }
#pragma unroll
                    for (int v4 = 0; v4 < 4; ++v4)
                        *reinterpret_cast<uint4 *>(ds_tile + swz128_offset(row, c * 32 + v4 * 8)) =
                            make_uint4(o[4 * v4], o[4 * v4 + 1], o[4 * v4 + 2], o[4 * v4 + 3]);
                    // these 16 columns lie inside the columns this thread has already read
                    tmem_st16(tmem + lane_base + kColdP + cbase + c * 16, o);
                }
                tmem_wait_st();
                LT_TRACE_SINCE(13, td0);
                fence_proxy_async_smem();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm.bar_ds_ready);
                LT_TL(tid == kComputeWarp0 * 32, 10, it);
                LT_TRACE_SINCE(14, td0);
                if constexpr (kSavedP) {
#pragma unroll
                    for (int e = 0; e < 32; ++e) ph[e] = pn[e];
                }
                if (++tile == w.tiles_per_head) tile = 0;
                if (n + 1 < w.n_iter) ok = compute_p(w, it + 1, tile);
            }

        }
        // dK_j and dV_j of the CTA's last item leave through these warps, which have nothing else left to do, while the reduction
        // warps bring the last dQ partial out.  They are laid out in place of K_j and V_j, as a tile load would, for tile stores.
        // (Behind that partial, by the reduction warps alone and from their registers, each thread its own row 16 bytes at a time,
        // they took 7 500 cycles from the last product: 45.0 -> 44.0 us for 32 heads of 1 024, 13.2 -> 12.3 for 16 of 64, D = 128.)
        // (Not where key tiles are split: 40/8 heads of 2 048 139.8 instead of 136.8 us.)
        if (!kSplit && ok && ic > 0 && (ok = LT_WAIT_ALL(&sm.bar_dkv_full, (ic - 1) & 1, kWaitDkvFull))) {
            tc_fence_after_sync();
            const BwdItem w = bwd_item<false>(p, make_int4(last_item, 0, 0, 0));
            const float inv_p_scale = exp2f(-p_scale_log2);
            const float mult = half_sel == 0 ? p.scale * inv_p_scale : inv_p_scale;  // half of the warps takes dK, the others dV
            const uint32_t acc = tmem + lane_base + (half_sel == 0 ? kColdK : kColdV);
            uint8_t *stage = half_sel == 0 ? sm.k : sm.v;
#pragma unroll 1
            for (int c = 0; c < D / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(acc + c * 32, r);
                tmem_wait_ld();
#pragma unroll
                for (int v8 = 0; v8 < 4; ++v8) {
                    uint32_t o[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        o[e] = pack2<kBf16>(__uint_as_float(r[8 * v8 + 2 * e]) * mult, __uint_as_float(r[8 * v8 + 2 * e + 1]) * mult);
                    *reinterpret_cast<uint4 *>(stage + (c >> 1) * kBoxBytesBwd + swz128_offset(row, (c & 1) * 32 + v8 * 8)) =
                        make_uint4(o[0], o[1], o[2], o[3]);
                }
            }
            const int row0 = w.j * kTileRows + quad * 32;
            if (row0 < p.S) {  // (rows past S are not written)
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    const CUtensorMap *map = half_sel == 0 ? &map_dk : &map_dv;
#pragma unroll
                    for (int x = 0; x < kBoxes; ++x)
                        tma_store_4d(map, stage + x * kBoxBytesBwd + quad * 4096, x * 64, row0, w.g, w.b);
                    bulk_commit_group();
                    bulk_wait_group_read<0>();  // (shared memory stays until the stores have read it)
                }
            }
        }
        LT_TRACE_END(kRoleCompute);
    } else {
        // ================================================================= dQ reduction warps
        warpgroup_regs_set<kRegsReduce, kRegsAtLaunch>();
        const int quad = warp & 3;
        // P carried the factor 2^c through dS into the accumulators; the epilogues take it out again (exact)
        const float inv_p_scale = exp2f(-static_cast<float>(bwd_p_scale_log2<D>(p, sm.call_max, !kOneTile || !one.own_pre)));
        const float dq_mult = p.scale * inv_p_scale;
        bool ok = smem_ok;
        int it = 0, ic = 0;
        uint32_t gq = 0;  // running number of the sixteen-row groups staged so far (D = 128)
        LT_TRACE_BEGIN();
        for (;; ++ic) {
            // the four reduction warps share named barriers (D = 128), so after every wait they vote
            // and leave together
            ok = ok && LT_WAIT_ALL(&sm.bar_item[ic % kItemRing], (ic / kItemRing) & 1, kWaitItem);
            ok = named_barrier_and(kBarReduceWarps, kNumReduceWarps * 32, ok);
            if (!ok) break;
            const int4 item = sm.item_ring[ic % kItemRing];
            if (item.x < 0) break;
            const BwdItem w = bwd_item<kSplit>(p, item);
            for (int n = 0; n < w.n_iter; ++n, ++it) {
                ok = LT_WAIT_ALL(&sm.bar_dq_full, it & 1, kWaitDqFull);
                // The four reduction warps share named barriers below, so they leave the loop together.  The
                // staging buffers form a ring that runs on across tile pairs (running group number gq): at
                // most the last two reductions of the previous pair are still reading their buffers here,
                // the buffer the first group of this pair goes to is free.
                if constexpr (D == 128)
                    if (warp == kReduceWarp0 && lane == 0) bulk_wait_group_read<2>();
                ok = named_barrier_and(kBarReduceWarps, kNumReduceWarps * 32, ok);
                if (!ok) break;
                tc_fence_after_sync();
                LT_TL(tid == kReduceWarp0 * 32, 11, it);
                LT_TRACE_MARK(tr0);
                float *dq_tile = p.dq_acc + bwd_q_tile(p, w, n).padded_row0 * D;
                if constexpr (D == 128) {
                    // dQ^T: this thread holds head-dim element d = 32*quad + lane of all 128 query rows.
                    // Sixteen query rows at a time are scaled, staged in shared memory exactly as they lie
                    // in the accumulator (16 rows x 128 floats, contiguous) and added to it by one bulk
                    // reduction; three staging buffers keep the copies in flight.
                    const int d_idx = quad * 32 + lane;
                    const uint32_t taddr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + kColdP;
                    const bool elected = (warp == kReduceWarp0) && (lane == 0);
                    auto store_rows = [&](int k, const uint32_t *r) {  // r: 16 values, query rows 16k .. 16k+15
                        float *buf = sm.dq_stage[(gq + k) % kDqStageBufs];
#pragma unroll
                        for (int e = 0; e < kDqStageRows; ++e) buf[e * 128 + d_idx] = __uint_as_float(r[e]) * dq_mult;
                    };
                    // one tile: the group's rows are final; eight threads per row round sixteen elements each
                    const BwdQTile qt = bwd_q_tile(p, w, n);
                    auto put_rows = [&](int k) {
                        const int rt = tid - kReduceWarp0 * 32, r_in = rt >> 3, c0 = (rt & 7) * 16;
                        const int s_row = qt.s0 + k * kDqStageRows + r_in;
                        if (s_row < p.S) {
                            const float4 *src = reinterpret_cast<const float4 *>(sm.dq_stage[(gq + k) % kDqStageBufs] + r_in * 128 + c0);
                            uint4 *dst = reinterpret_cast<uint4 *>(one.dQ + qt.b * one.dq_st.batch + qt.h * one.dq_st.head +
                                                                   s_row * one.dq_st.row + c0);
#pragma unroll
                            for (int v = 0; v < 2; ++v) {
                                const float4 x = src[2 * v], y = src[2 * v + 1];
                                dst[v] = make_uint4(pack2<kBf16>(x.x, x.y), pack2<kBf16>(x.z, x.w), pack2<kBf16>(y.x, y.y),
                                                    pack2<kBf16>(y.z, y.w));
                            }
                        }
                    };
                    auto add_rows = [&](int k) {
                        bulk_reduce_add_f32(dq_tile + k * kDqStageRows * 128, sm.dq_stage[(gq + k) % kDqStageBufs],
                                            kDqStageRows * 128 * sizeof(float));
                        bulk_commit_group();
                    };
                    // Seven eighths of the partial are read, one group of rows is parked in shared memory to make
                    // room for the last eighth, and the dP columns are released before any reduction of this
                    // pair is issued.
                    uint32_t r0a[16], r0b[16], r1[32], r2[32], r3[16];
                    tmem_ld16(taddr, r0a);
                    tmem_ld16(taddr + 16, r0b);
                    tmem_ld32(taddr + 32, r1);
                    tmem_ld32(taddr + 64, r2);
                    tmem_ld16(taddr + 96, r3);
                    tmem_wait_ld();
                    store_rows(0, r0a);
                    tmem_ld16(taddr + 112, r0a);
                    tmem_wait_ld();
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.bar_dq_empty);
                    LT_TL(tid == kReduceWarp0 * 32, 12, it);
                    LT_TRACE_SINCE(12, tr0);
                    fence_proxy_async_smem();
                    // the buffer where group 1 goes was read by the last reduction but one of the previous pair
                    if (elected) bulk_wait_group_read<1>();
                    named_barrier_sync(kBarReduceWarps, kNumReduceWarps * 32);
                    if constexpr (kOneTile) put_rows(0);
                    else if (elected) add_rows(0);
                    // groups 1..7 rotate through the three buffers: before group k is issued, the bulk
                    // reduction of group k-2 has finished reading, which frees the buffer of group k+1
                    auto stage_rows = [&](int k, const uint32_t *r) {
                        store_rows(k, r);
                        fence_proxy_async_smem();
                        if (elected) bulk_wait_group_read<1>();
                        named_barrier_sync(kBarReduceWarps, kNumReduceWarps * 32);
                        if constexpr (kOneTile) put_rows(k);
                        else if (elected) add_rows(k);
                    };
                    stage_rows(1, r0b);
                    stage_rows(2, r1);
                    stage_rows(3, r1 + 16);
                    stage_rows(4, r2);
                    stage_rows(5, r2 + 16);
                    stage_rows(6, r3);
                    stage_rows(7, r0a);
                    gq += 8;
                } else {
                    // D = 64: dQ partial with lanes = query rows.  A thread holds the 64 floats of one query row.
                    // The partial is scaled and staged in shared memory as two boxes of 128 rows x 32 floats with
                    // the 128-byte swizzle (rows 128 bytes apart: the swizzle spreads a warp's 16-byte stores over
                    // all banks), and two tiled reductions add the boxes to the accumulator; two staging buffers.
                    const int q_row = quad * 32 + lane;
                    const uint32_t taddr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + kColdP;
                    const bool elected = (warp == kReduceWarp0) && (lane == 0);
                    uint32_t r[2][32];
                    tmem_ld32(taddr, r[0]);
                    tmem_ld32(taddr + 32, r[1]);
                    tmem_wait_ld();
                    // the whole partial is in registers: the dP columns may be overwritten
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.bar_dq_empty);
                    LT_TRACE_SINCE(12, tr0);
                    if constexpr (kOneTile) {  // the rows are final
                        const BwdQTile qt = bwd_q_tile(p, w, n);
                        if (qt.s0 + q_row < p.S) {
                            uint4 *dst = reinterpret_cast<uint4 *>(one.dQ + qt.b * one.dq_st.batch + qt.h * one.dq_st.head +
                                                                   (qt.s0 + q_row) * one.dq_st.row);
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                const uint32_t *x = &r[c >> 2][(c & 3) * 8];
                                uint32_t o[4];
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    o[e] = pack2<kBf16>(__uint_as_float(x[2 * e]) * dq_mult, __uint_as_float(x[2 * e + 1]) * dq_mult);
                                dst[c] = make_uint4(o[0], o[1], o[2], o[3]);
                            }
                        }
                        continue;
                    }
                    // the buffer of this tile was last read by the reductions issued two tiles ago
                    if (elected) bulk_wait_group_read<1>();
                    named_barrier_sync(kBarReduceWarps, kNumReduceWarps * 32);
                    uint8_t *buf = reinterpret_cast<uint8_t *>(sm.dq_stage[it & 1]);
#pragma unroll
                    for (int bx = 0; bx < 2; ++bx)
#pragma unroll
                        for (int c = 0; c < 8; ++c)
                            *reinterpret_cast<float4 *>(buf + bx * (kTileRows * 128) + q_row * 128 + ((c ^ (q_row & 7)) << 4)) =
                                make_float4(__uint_as_float(r[bx][4 * c]) * dq_mult, __uint_as_float(r[bx][4 * c + 1]) * dq_mult,
                                            __uint_as_float(r[bx][4 * c + 2]) * dq_mult, __uint_as_float(r[bx][4 * c + 3]) * dq_mult);
                    fence_proxy_async_smem();
                    named_barrier_sync(kBarReduceWarps, kNumReduceWarps * 32);
                    if (elected) {
                        const int y = static_cast<int>(bwd_q_tile(p, w, n).padded_row0);
                        tma_reduce_add_2d(&map_dq, buf, 0, y);
                        tma_reduce_add_2d(&map_dq, buf + kTileRows * 128, 32, y);
                        bulk_commit_group();
                    }
                }
                LT_TL(tid == kReduceWarp0 * 32, 13, it);
                LT_TRACE_SINCE(13, tr0);
            }
            if (!ok) break;
            // item epilogue (these warps are idle while the pipeline of the next item fills; the last item's is the softmax warps'):
            // dK_j and dV_j leave tensor memory as fp16; thread = key row
            ok = LT_WAIT_BOTH(&sm.bar_dkv_full, ic & 1, kSplit ? nullptr : &sm.bar_item[(ic + 1) % kItemRing], ((ic + 1) / kItemRing) & 1,
                              kSplit ? kWaitDkvFull : both_codes(kWaitDkvFull, kWaitItem));
            ok = named_barrier_and(kBarReduceWarps, kNumReduceWarps * 32, ok);
            if (!ok) break;
            if (!kSplit && sm.item_ring[(ic + 1) % kItemRing].x < 0) continue;
            tc_fence_after_sync();
            {
                const int row = quad * 32 + lane;
                const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
#pragma unroll 1  // (runs once per item, out of a cold instruction cache: shorter is faster)
                for (int which = 0; which < 2; ++which) {
                    const float mult = which == 0 ? dq_mult : inv_p_scale;
                    const uint32_t col0 = which == 0 ? kColdK : kColdV;
                    const int s_row = w.j * kTileRows + row;  // rows past S are never stored
                    const lt_tensor_strides &st = which == 0 ? p.dk_st : p.dv_st;
                    __half *dst = (which == 0 ? p.dK : p.dV) + w.b * st.batch + w.g * st.head + s_row * st.row;
#pragma unroll 1
                    for (int c = 0; c < D / 32; ++c) {
                        uint32_t r[32];
                        tmem_ld32(tmem + lane_base + col0 + c * 32, r);
                        tmem_wait_ld();
                        if (which == 1 && c == D / 32 - 1) {
                            // both accumulators have been read: the next item may overwrite them
                            tc_fence_before_sync();
                            __syncwarp();
                            if (lane == 0) mbar_arrive(&sm.bar_acc_free);
                            LT_TL(tid == kReduceWarp0 * 32, 15, it);
                        }
                        if (kSplit && w.share >= 0) {
                            // (rows past S come from zero-filled key rows: finite, never read)
                            float4 *share = p.shares + (static_cast<long long>(w.share) * 2 + which) * (kTileRows * D / 4) + c * 8 * kTileRows + row;
#pragma unroll
                            for (int v4 = 0; v4 < 8; ++v4)
                                share[v4 * kTileRows] = make_float4(__uint_as_float(r[4 * v4 + 0]) * mult, __uint_as_float(r[4 * v4 + 1]) * mult,
                                                                    __uint_as_float(r[4 * v4 + 2]) * mult, __uint_as_float(r[4 * v4 + 3]) * mult);
                            continue;
                        }
#pragma unroll
                        for (int v8 = 0; v8 < 4; ++v8) {
                            uint4 o;
                            o.x = pack2<kBf16>(__uint_as_float(r[8 * v8 + 0]) * mult, __uint_as_float(r[8 * v8 + 1]) * mult);
                            o.y = pack2<kBf16>(__uint_as_float(r[8 * v8 + 2]) * mult, __uint_as_float(r[8 * v8 + 3]) * mult);
                            o.z = pack2<kBf16>(__uint_as_float(r[8 * v8 + 4]) * mult, __uint_as_float(r[8 * v8 + 5]) * mult);
                            o.w = pack2<kBf16>(__uint_as_float(r[8 * v8 + 6]) * mult, __uint_as_float(r[8 * v8 + 7]) * mult);
                            if (s_row < p.S) reinterpret_cast<uint4 *>(dst + c * 32)[v8] = o;
                        }
                    }
                }
            }
        }
        // shared memory must stay valid until the bulk reductions have read it (that they have been added is what the
        // end of the grid stands for)
        bulk_wait_group_read<0>();
        LT_TRACE_END(kRoleReduce);
#ifdef LT_BWD_TRACE
        trace_iters = it;
#endif
    }

#ifdef LT_BWD_TRACE
    const long long trace_teardown_begin = clock64();
#endif
    grid_launch_dependents();  // the dQ conversion kernel may be scheduled while the last CTAs finish
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kTmemCols);
#ifdef LT_BWD_TRACE
    if (tid == 0) {
        atomicAdd(&g_bwd_trace[64 + 3], static_cast<unsigned long long>(clock64() - trace_cta_t0));
        atomicAdd(&g_bwd_trace[64 + 1], 1ull);
        atomicAdd(&g_bwd_trace[64 + 0], static_cast<unsigned long long>(trace_prologue_end - trace_cta_t0));
        atomicAdd(&g_bwd_trace[64 + 4], static_cast<unsigned long long>(trace_teardown_begin - trace_prologue_end));
    }
    if (tid == kReduceWarp0 * 32) atomicAdd(&g_bwd_trace[64 + 2], static_cast<unsigned long long>(trace_iters));
#endif
}

#ifdef LT_BWD_TIMELINE
extern "C" int lt_dbg_bwd_timeline(long long *out) {  // out == NULL: clear the stamps
    if (!out) {
        void *sym = nullptr;
        if (cudaGetSymbolAddress(&sym, lt::g_bwd_timeline) != cudaSuccess) return LT_ERR_CUDA;
        return cudaMemset(sym, 0, sizeof(lt::g_bwd_timeline)) == cudaSuccess ? LT_OK : LT_ERR_CUDA;
    }
    return cudaMemcpyFromSymbol(out, lt::g_bwd_timeline, sizeof(lt::g_bwd_timeline)) == cudaSuccess ? LT_OK : LT_ERR_CUDA;
}
#endif
#ifdef LT_BWD_TRACE
extern "C" int lt_dbg_bwd_trace(unsigned long long *out, int reset) {
    if (out && cudaMemcpyFromSymbol(out, g_bwd_trace, sizeof(g_bwd_trace)) != cudaSuccess) return LT_ERR_CUDA;
    if (reset) {
        static unsigned long long zeros[80];
        if (cudaMemcpyToSymbol(g_bwd_trace, zeros, sizeof(zeros)) != cudaSuccess) return LT_ERR_CUDA;
    }
    return LT_OK;
}
#endif

// Multiprocessors of the current device (148 on a B200; that figure is also the answer when the query fails,
// so that the sizes derived from it never depend on an error path).
static int sm_count() {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        return 148;
    return sms;
}
// Whether and how key tiles are split (BwdDeal), with at most `room` bytes of shares.  Not at all: every key tile is one
// work item, claimed from a counter, its dK_j and dV_j accumulated in one CTA's tensor memory.
static size_t share_bytes(const BwdDeal &deal, int D) {
    return static_cast<size_t>(deal.any() ? deal.n_shares() : 0) * (2 * kTileRows * 4) * D;
}
static BwdDeal deal_pairs(int B, int Hq, int Hkv, int S, int D, int causal, size_t room = ~static_cast<size_t>(0)) {
    const int sms = sm_count();
    BwdDeal deal{0, 0, B * Hkv, Hq / Hkv, static_cast<int>(padded_rows(S) / kTileRows), causal ? 1 : 0};
    const double n_tiles = deal.n_tiles, G = deal.G, items = deal.n_units * n_tiles;
    const double pairs = B * G * Hkv * (causal ? 0.5 * n_tiles * (n_tiles + 1.) : n_tiles * n_tiles);
    const double cost = pairs + kTileCost * items;
    if (G * n_tiles < 2. || cost > 1.0e9) return deal;  // (nothing to split; costs are 32-bit numbers)
    // (small walks: stretches of two; a small workspace: as many as have room for their shares)
    int ctas = cost < 2. * sms ? static_cast<int>(cost / 2.) : sms;
    const size_t in_room = room / (static_cast<size_t>(2 * kTileRows * 4) * D), tiles = static_cast<size_t>(deal.tiles());
    const size_t most = in_room / 2 + 1 > tiles ? in_room + 1 - tiles : in_room / 2;  // (few_tiles() or not)
    if (most < static_cast<size_t>(ctas)) ctas = static_cast<int>(most);
    // Estimated makespans, in tile pairs (2-3 us each): whole key tiles, the longest one or the average work of an SM, in
    // whole rounds where all are equal; dealt out, the average plus what the parts cost: the shares stored and added (they
    // grow with the CTAs) by a kernel that the dQ conversion waits for, and a second pipeline filled in the CTAs whose stretch
    // crosses into another key tile.  Constants fitted to 240 short calls near the line, both ways in graphs: on those and on 240
    // others 0.2 % behind the faster one on average, 6 % at worst.  Measured, us per call, whole / dealt
    // out (batch, query / kv heads, S; D = 128 under the causal mask unless noted): 1, 40/8, 2048 244 / 149; 1, 40/8, 1024
    // 108 / 56; 1, 2/1, 3566 131 / 39; 1, 1/1, 4135, D = 64 60 / 26; 1, 2/2, 2999 unmasked 66 / 43; 8, 5/1, 2572, D = 64
    // unmasked 399 / 221; 1, 16/8, 208 22.0 / 19.1.  On the other side of the line: 1, 64/16, 2048 244 / 257; 1, 8/8, 4096
    // 105 / 127; 1, 32/32, 1024 45 / 61; 2, 8/8, 384 unmasked 19.0 / 22.6; near it: 8, 20/4, 512 81 / 78; 1, 8/8, 2048
    // 51 / 48; 1, 40/8, 4096 and 1, 32/8, 4096 equal.  One tile: 1, 32/8, 128 20.7 / 17.8; 8, 40/8, 128 32.0 / 35.6.
    double whole = cost / sms;
    if (whole < G * n_tiles + kTileCost) whole = G * n_tiles + kTileCost;
    if (!causal && whole < ceil(items / sms) * (G * n_tiles + kTileCost)) whole = ceil(items / sms) * (G * n_tiles + kTileCost);
    if (n_tiles == 1. && D == 64) whole -= 1.;  // (the one-tile variant has fewer launches)
    // Everything the items touch (K, V, Q, dO and the fp32 dQ rows), in L2s of 126 MB.  Dealt out, all units are walked at once,
    // whole key tiles batch by batch (launch_bwd), so the gain has to be the larger, the more there is.  380 shapes with
    // estimates of 0.6 and above, dealt against the faster of whole and halved key tiles: without that term the choice took
    // 2.0 % more than the faster one on average, up to 28 %, with it 0.7 %, up to 15 %.  us, dealt / whole, unmasked: 2, 64/16,
    // 1439 (1.8 L2s, estimate 0.92) 1.28 of the time; 8, 20/4, 3328 (4.8, 0.95) 1.26; 8, 32/4, 1472 (3.4, 0.90) 1244 / 1020; on the other
    // side 8, 8/2, 5009 (3.0, 0.88) 2355 / 2673; 4, 64/16, 1685, D = 64 (2.1, 0.89) 804 / 874; not told apart: 8, 32/4, 1472,
    // D = 64 (1.7, 0.90) 674 / 596.
    const double unit_bytes = static_cast<double>(padded_rows(S)) * D * (2.0 * 2 + G * (2.0 * 2 + 4));
    const double working_set = unit_bytes * deal.n_units / 126.0e6;
    if (ctas > 0) {
        const double crossings = items < ctas ? items / ctas : 1.;
        const double dealt = cost / ctas + 2.75 + 0.016 * ctas + 0.8 * crossings * crossings;
        if (dealt < (0.94 - 0.02 * working_set) * whole) {
            deal.ctas = ctas;
            return deal;
        }
    }
    if (G > 1. && items >= sms + sms / 2 && items < 4. * sms) {
        // Enough key tiles to fill the SMs, but too few to form L2-sized batches (a batch needs two items per SM) while the
        // working set is more than four times the L2: the accumulator rows of the heads in flight would be fetched and
        // written back again and again.  Halves make room for batches and even out the end of the walk; each costs a share
        // stored and added, and a pipeline filled.  What decides is how the GPU is driven: less DRAM traffic draws less power
        // (2, 64/8, 4096: 728 W against 852), which a long run gets back as clock and a single call does not.  us per call, whole
        // / halves, 0.6 s of calls on end (median of five in turn) and, in brackets, single calls on an idle GPU: 2, 64/8, 4096
        // 1760 / 1692 (1530 / 1499); 1, 64/8, 8192 3158 / 3010 (2779 / 2677); 4, 64/4, 2000 1136 / 1054 (983 / 904);
        // 4, 64/8, 2048 1033 / 1004 (895 / 903); 8, 64/8, 1024 658 / 663 (586 / 609).  Where both kinds of call alternate every
        // 3 ms and so share one clock, even grids of short key tiles lose: 986 / 1037 and 640 / 679 for the last two.
        if (working_set > 4.0) deal.halves = 1;
    }
    if (share_bytes(deal, D) > room) deal.halves = 0;
    return deal;
}

// Sequences of one tile: launches of a call in the one-tile variant, or 0 where the general path is the faster one.  With
// one launch a CTA's rows are read by that CTA alone, about 1 us per head; with two the preprocess kernel spreads them over
// the chip.  At D = 128 a partial that is rounded by the reduction warps themselves, not queued for the copy unit, holds up
// the next head, so only short walks through a group gain.  On 43 shapes the choice is 0.8 % behind the fastest one on
// average, 6 % at worst (8, 64/16, 128, D = 64: one launch 18.9, two, the choice, 19.9).  Measured, us of device time, general / two launches / one
// (batch, query / kv heads, S): D = 64: 1, 2/2, 128 11.2 / 9.4 / 8.8; 8, 16/16, 128 14.9 / 12.8 / 11.0; 2, 12/4, 128
// 14.6 / 13.2 / 13.9; 8, 40/8, 64 22.7 / 19.9 / 21.5.  D = 128: 4, 32/32, 128 20.6 / 18.7 / 16.5; 8, 32/16, 64
// 24.9 / 23.8 / 20.1; 8, 64/16, 128 40.8 / 37.8 / 36.2; 2, 8/4, 128 16.6 / 17.2 / 18.5; 1, 64/8, 128 29.8 / 35.5 / 47.4.
static int one_tile_launches(int B, int Hq, int Hkv, int S, int D) {
    if (S > kTileRows) return 0;
    const long long sms = sm_count(), units = static_cast<long long>(B) * Hkv, G = Hq / Hkv;
    const long long heads_per_cta = (units + sms - 1) / sms * G;
    if (D == 64) return heads_per_cta <= 2 ? 1 : 2;
    return heads_per_cta <= 4 && (G == 1 || units >= 96) ? 1 : 0;
}

template <int D, bool kBf16>
static int launch_bwd(const lt_half *Q, const lt_half *K, const lt_half *V, const lt_half *O, const lt_half *dO,
                      const float *LSE, lt_half *dQ, lt_half *dK, lt_half *dV, const lt_attn_layout &lay, int B,
                      int Hq, int Hkv, int S, int causal, float scale, void *workspace, size_t workspace_bytes, cudaStream_t stream,
                      cudaEvent_t ev_main_begin, cudaEvent_t ev_main_end, const lt_half *saved_p = nullptr) {
    // saved_p: the probability tiles of lt_attn_save_p; LSE is then not needed (fp16, whole groups only)
    const int S_pad = static_cast<int>(padded_rows(S));
    // fast addressing in the two streaming kernels when nothing is padded or strided
    auto is_contig = [&](const lt_tensor_strides &st, int H) {
        const lt_tensor_strides c = contiguous_strides(H, S, D);
        return st.batch == c.batch && st.head == c.head && st.row == c.row;
    };
    const int plain_pre = (S == S_pad && is_contig(lay.d_o, Hq) && is_contig(lay.o, Hq)) ? 1 : 0;
    const int plain_fin = (S == S_pad && is_contig(lay.dq, Hq)) ? 1 : 0;
    const long long n_rows = static_cast<long long>(B) * Hq * S_pad;  // padded row space of the workspace arrays
    uint8_t *ws = static_cast<uint8_t *>(workspace);
    unsigned int *status = reinterpret_cast<unsigned int *>(ws);
    const size_t ext_bytes = round256(static_cast<size_t>(n_rows) * 16);
    uint4 *delta_ext = reinterpret_cast<uint4 *>(ws + kStatusBytes);
    uint4 *lse_ext = reinterpret_cast<uint4 *>(ws + kStatusBytes + ext_bytes);
    float *dq_acc = reinterpret_cast<float *>(ws + kStatusBytes + 2 * ext_bytes);
    const size_t base_bytes = bwd_least_bytes(B, Hq, S, D);
    BwdDeal deal{};
    if (!saved_p) deal = deal_pairs(B, Hq, Hkv, S, D, causal, workspace_bytes - base_bytes);
    const bool split = deal.any();

    CUtensorMap mq, mk, mv, mdo, mdk, mdv;
    int rc;
    if ((rc = make_bhsd_map(&mq, Q, B, Hq, S, D, lay.q, 128, kBf16)) != LT_OK) return rc;
    if ((rc = make_bhsd_map(&mdo, dO, B, Hq, S, D, lay.d_o, 128, kBf16)) != LT_OK) return rc;
    if ((rc = make_bhsd_map(&mk, K, B, Hkv, S, D, lay.k, 128, kBf16)) != LT_OK) return rc;
    if ((rc = make_bhsd_map(&mv, V, B, Hkv, S, D, lay.v, 128, kBf16)) != LT_OK) return rc;
    mdk = mdv = mk;  // (split key tiles leave through shares and the reduction warps, never through these)
    if (!split && (rc = make_bhsd_map(&mdk, dK, B, Hkv, S, D, lay.dk, 32, kBf16)) != LT_OK) return rc;
    if (!split && (rc = make_bhsd_map(&mdv, dV, B, Hkv, S, D, lay.dv, 32, kBf16)) != LT_OK) return rc;

    // programmatic stream serialisation: each kernel may start before its predecessor has finished and
    // waits inside for it (grid_dependency_wait).  The conversion kernels do not let the next call's preprocess
    // kernel start early: with that, a call on the LLaMA-2-7B shape took 453 us in a loop instead of 434.
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    const int sms = sm_count();
    cudaError_t e = cudaSuccess;
    BwdOneTileParams one = {};
    one.pre.dO = reinterpret_cast<const __half *>(dO);
    one.pre.O = reinterpret_cast<const __half *>(O);
    one.pre.V = reinterpret_cast<const __half *>(V);
    one.pre.lse = LSE;
    one.pre.delta_ext = delta_ext;
    one.pre.lse_ext = lse_ext;
    one.pre.dq_acc = dq_acc;
    one.pre.S = S; one.pre.S_pad = S_pad; one.pre.Hq = Hq; one.pre.Hkv = Hkv;
    one.pre.do_st = lay.d_o; one.pre.o_st = lay.o; one.pre.v_st = lay.v;
    one.pre.plain = plain_pre;
    one.pre.v_plain = is_contig(lay.v, Hkv) ? 1 : 0;
    one.pre.inv_scale = 1.f / scale;
    one.dQ = reinterpret_cast<__half *>(dQ);
    one.dq_st = lay.dq;
    const int tile_launches = saved_p || split ? 0 : one_tile_launches(B, Hq, Hkv, S, D);
    const bool one_tile = tile_launches > 0;
    one.own_pre = tile_launches == 1 ? 1 : 0;
    if (one_tile) one.pre.dq_acc = nullptr;
    if (!one.own_pre) {
        cudaLaunchConfig_t cfg_pre = {};
        cfg_pre.gridDim = dim3(pre_blocks<D>(n_rows));
        cfg_pre.blockDim = dim3(kPreThreads);
        cfg_pre.stream = stream;
        cfg_pre.attrs = &pdl;
        cfg_pre.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg_pre, bwd_preprocess_kernel<D, kBf16>, one.pre, n_rows,
                               static_cast<long long>(B) * Hkv * S, status);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return record_cuda_error("bwd_preprocess_kernel launch", e);
    }

    BwdParams prm;
    prm.lse_ext = saved_p ? reinterpret_cast<const uint4 *>(saved_p) : lse_ext;
    prm.delta_ext = delta_ext;
    prm.dq_acc = dq_acc;
    prm.dK = reinterpret_cast<__half *>(dK);
    prm.dV = reinterpret_cast<__half *>(dV);
    prm.status = status;
    prm.B = B; prm.Hq = Hq; prm.Hkv = Hkv; prm.S = S; prm.S_pad = S_pad; prm.causal = causal ? 1 : 0;
    prm.scale = scale;
    prm.dk_st = lay.dk;
    prm.dv_st = lay.dv;
    {
        // bytes one (batch, kv head) unit keeps live: K, V, the group's Q, dO (fp16) and dQ rows (fp32)
        const int G = Hq / Hkv;
        const double unit_bytes = static_cast<double>(S_pad) * D * (2.0 * 2 + 2.0 * 2 * G + 4.0 * G);
        const int n_units = B * Hkv;
        int n_batches = static_cast<int>(unit_bytes * n_units / kL2BatchBytes) + 1;
        // CTAs flow from one batch into the next, but the last batch should still offer every SM two items
        const int max_batches = static_cast<int>(static_cast<long long>(n_units) * (S_pad / kTileRows) * (deal.halves ? 2 : 1) / (2 * sms));
        if (n_batches > max_batches) n_batches = max_batches;
        if (n_batches < 1) n_batches = 1;
        prm.units_per_batch = (n_units + n_batches - 1) / n_batches;
    }
    prm.deal = deal;
    prm.shares = reinterpret_cast<float4 *>(ws + base_bytes);
    const size_t smem = sizeof(BwdSmem<D>);
    auto main_kernel = split ? bwd_main_kernel<D, kBf16, true> : bwd_main_kernel<D, kBf16, false>;
    if constexpr (!kBf16)
        if (saved_p) main_kernel = bwd_main_kernel<D, false, false, true>;
    if (one_tile) main_kernel = bwd_main_kernel<D, kBf16, false, false, true>;
    e = cudaFuncSetAttribute(main_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return record_cuda_error("cudaFuncSetAttribute(bwd_main)", e);
    const int n_items = deal.ctas > 0 ? deal.ctas : B * Hkv * (S_pad / kTileRows) * (deal.halves ? 2 : 1);
    const int grid = n_items < sms ? n_items : sms;  // persistent: one CTA per SM walks the item list
    if (ev_main_begin && (e = cudaEventRecord(ev_main_begin, stream)) != cudaSuccess)
        return record_cuda_error("cudaEventRecord", e);
    cudaLaunchConfig_t cfg_main = {};
    cfg_main.gridDim = dim3(grid);
    cfg_main.blockDim = dim3(kBwdThreads);
    cfg_main.dynamicSmemBytes = smem;
    cfg_main.stream = stream;
    cfg_main.attrs = &pdl;
    cfg_main.numAttrs = 1;
    CUtensorMap mdq = mq;  // (D = 128 never touches it)
    if constexpr (D == 64)
        if ((rc = make_f32_tile_map(&mdq, dq_acc, static_cast<uint64_t>(n_rows), 64, 128)) != LT_OK) return rc;
    e = cudaLaunchKernelEx(&cfg_main, main_kernel, mq, mk, mv, mdo, prm, mdq, mdk, mdv, one);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return record_cuda_error("bwd_main_kernel launch", e);
    if (ev_main_end && (e = cudaEventRecord(ev_main_end, stream)) != cudaSuccess)
        return record_cuda_error("cudaEventRecord", e);

    if (one_tile) return LT_OK;  // dQ is written

    const long long n_vec8 = static_cast<long long>(B) * Hq * S * D / 8;
    const long long fwant = (n_vec8 + 255) / 256;
    const int fin_blocks = static_cast<int>(fwant < static_cast<long long>(sms) * 16 ? fwant : sms * 16);
    cudaLaunchConfig_t cfg_fin = {};
    cfg_fin.gridDim = dim3(fin_blocks);
    cfg_fin.blockDim = dim3(256);
    cfg_fin.stream = stream;
    cfg_fin.attrs = &pdl;
    cfg_fin.numAttrs = 1;
    if (split) {
        cfg_fin.gridDim = dim3(deal.halves ? deal.tiles() : deal.ctas, 2 * (D / 32));
        e = cudaLaunchKernelEx(&cfg_fin, bwd_shares_kernel<D, kBf16>, static_cast<const float4 *>(prm.shares),
                               reinterpret_cast<__half *>(dK), reinterpret_cast<__half *>(dV), deal, Hkv, S, lay.dk,
                               lay.dv);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return record_cuda_error("bwd_shares_kernel launch", e);
        cfg_fin.gridDim = dim3(fin_blocks);
    }
    e = cudaLaunchKernelEx(&cfg_fin, bwd_finalize_kernel<kBf16>, static_cast<const float *>(dq_acc),
                           reinterpret_cast<__half *>(dQ), n_vec8, S * (D / 8), S_pad * (D / 8), D / 8, Hq, lay.dq,
                           plain_fin);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return record_cuda_error("bwd_finalize_kernel launch", e);
    return LT_OK;
}

}  // namespace lt

namespace lt {
size_t bwd_least_bytes(int B, int Hq, int S, int D) {
    const size_t n_rows = static_cast<size_t>(B) * Hq * static_cast<size_t>(padded_rows(S));
    return kStatusBytes + 2 * round256(n_rows * 16) + round256(n_rows * D * 4);
}
}  // namespace lt

extern "C" {

size_t lt_attn_bwd_workspace_bytes(int B, int Hq, int Hkv, int S, int D) {
    if (lt::check_shape(B, Hq, Hkv, S, D, 1.0f) != LT_OK) return 0;
    size_t bytes = lt::bwd_least_bytes(B, Hq, S, D);
    // fp32 shares of dK and dV for shapes whose tile pairs are dealt out (under either mask)
    const size_t masked = lt::share_bytes(lt::deal_pairs(B, Hq, Hkv, S, D, 1), D);
    const size_t full = lt::share_bytes(lt::deal_pairs(B, Hq, Hkv, S, D, 0), D);
    bytes += masked > full ? masked : full;
    return bytes;
}

int lt_attn_bwd_num_launches(int B, int Hq, int Hkv, int S, int D, int causal) {
    if (lt::check_shape(B, Hq, Hkv, S, D, 1.0f) != LT_OK) return 0;
    // preprocess, main, dQ conversion; plus the sum of the shares of dK and dV where key tiles are split; sequences of one
    // tile need fewer (a workspace of the size lt_attn_bwd_workspace_bytes names)
    if (lt::deal_pairs(B, Hq, Hkv, S, D, causal).any()) return 4;
    const int tile_launches = lt::one_tile_launches(B, Hq, Hkv, S, D);
    return tile_launches > 0 ? tile_launches : 3;
}

static int bwd_entry(const lt_half *Q, const lt_half *K, const lt_half *V, const lt_half *O, const lt_half *dO,
                     const float *LSE, lt_half *dQ, lt_half *dK, lt_half *dV, const lt_attn_layout *layout, int B,
                     int Hq, int Hkv, int S, int D, int causal, float scale, void *workspace, size_t workspace_bytes,
                     lt_stream_t stream, lt_event_t main_begin, lt_event_t main_end, bool bf16 = false) {
    using namespace lt;
    if (!Q || !K || !V || !O || !dO || !LSE || !dQ || !dK || !dV) return LT_ERR_INVALID_ARG;
    int rc = check_shape(B, Hq, Hkv, S, D, scale);
    if (rc != LT_OK) return rc;
    const lt_attn_layout lay = layout ? *layout : contiguous_layout(Hq, Hkv, S, D);
    if (layout && (rc = check_layout(lay, D)) != LT_OK) return rc;
    const void *ptrs[] = {Q, K, V, O, dO, dQ, dK, dV};
    for (const void *ptr : ptrs)
        if (!aligned16(ptr)) return LT_ERR_UNSUPPORTED;
    if ((reinterpret_cast<uintptr_t>(LSE) & 3u) != 0) return LT_ERR_UNSUPPORTED;  // fp32, read one at a time
    if (!workspace || !aligned256(workspace) || workspace_bytes < bwd_least_bytes(B, Hq, S, D))
        return LT_ERR_WORKSPACE;
    if ((rc = check_device()) != LT_OK) return rc;
    if (bf16) {
        if (D == 64)
            return launch_bwd<64, true>(Q, K, V, O, dO, LSE, dQ, dK, dV, lay, B, Hq, Hkv, S, causal, scale, workspace,
                                        workspace_bytes, stream, main_begin, main_end);
        return launch_bwd<128, true>(Q, K, V, O, dO, LSE, dQ, dK, dV, lay, B, Hq, Hkv, S, causal, scale, workspace,
                                     workspace_bytes, stream, main_begin, main_end);
    }
    if (D == 64)
        return launch_bwd<64, false>(Q, K, V, O, dO, LSE, dQ, dK, dV, lay, B, Hq, Hkv, S, causal, scale, workspace,
                                     workspace_bytes, stream, main_begin, main_end);
    return launch_bwd<128, false>(Q, K, V, O, dO, LSE, dQ, dK, dV, lay, B, Hq, Hkv, S, causal, scale, workspace,
                                  workspace_bytes, stream, main_begin, main_end);
}

int lt_attn_bwd_saved_p(const lt_half *Q, const lt_half *K, const lt_half *V, const lt_half *O, const lt_half *dO,
                        const lt_half *P, lt_half *dQ, lt_half *dK, lt_half *dV, int B, int Hq, int Hkv, int S, int D,
                        int causal, float scale, void *workspace, size_t workspace_bytes, lt_stream_t stream) {
    using namespace lt;
    if (!Q || !K || !V || !O || !dO || !P || !dQ || !dK || !dV) return LT_ERR_INVALID_ARG;
    int rc = check_shape(B, Hq, Hkv, S, D, scale);
    if (rc != LT_OK) return rc;
    const void *ptrs[] = {Q, K, V, O, dO, dQ, dK, dV};
    for (const void *ptr : ptrs)
        if (!aligned16(ptr)) return LT_ERR_UNSUPPORTED;
    if (!aligned256(P)) return LT_ERR_UNSUPPORTED;
    if (!workspace || !aligned256(workspace) || workspace_bytes < bwd_least_bytes(B, Hq, S, D))
        return LT_ERR_WORKSPACE;
    if ((rc = check_device()) != LT_OK) return rc;
    const lt_attn_layout lay = contiguous_layout(Hq, Hkv, S, D);
    if (D == 64)
        return launch_bwd<64, false>(Q, K, V, O, dO, nullptr, dQ, dK, dV, lay, B, Hq, Hkv, S, causal, scale, workspace,
                                     workspace_bytes, static_cast<cudaStream_t>(stream), nullptr, nullptr, P);
    return launch_bwd<128, false>(Q, K, V, O, dO, nullptr, dQ, dK, dV, lay, B, Hq, Hkv, S, causal, scale, workspace,
                                  workspace_bytes, static_cast<cudaStream_t>(stream), nullptr, nullptr, P);
}

int lt_attn_bwd_profiled(const lt_half *Q, const lt_half *K, const lt_half *V, const lt_half *O, const lt_half *dO,
                         const float *LSE, lt_half *dQ, lt_half *dK, lt_half *dV, int B, int Hq, int Hkv, int S,
                         int D, int causal, float scale, void *workspace, size_t workspace_bytes,
                         lt_stream_t stream, lt_event_t main_begin, lt_event_t main_end) {
    return bwd_entry(Q, K, V, O, dO, LSE, dQ, dK, dV, nullptr, B, Hq, Hkv, S, D, causal, scale, workspace,
                     workspace_bytes, stream, main_begin, main_end);
}

int lt_attn_bwd_strided(const lt_half *Q, const lt_half *K, const lt_half *V, const lt_half *O, const lt_half *dO,
                        const float *LSE, lt_half *dQ, lt_half *dK, lt_half *dV, const lt_attn_layout *layout, int B,
                        int Hq, int Hkv, int S, int D, int causal, float scale, void *workspace,
                        size_t workspace_bytes, lt_stream_t stream) {
    return bwd_entry(Q, K, V, O, dO, LSE, dQ, dK, dV, layout, B, Hq, Hkv, S, D, causal, scale, workspace,
                     workspace_bytes, stream, nullptr, nullptr);
}

int lt_attn_bwd_bf16(const lt_bf16 *Q, const lt_bf16 *K, const lt_bf16 *V, const lt_bf16 *O, const lt_bf16 *dO,
                     const float *LSE, lt_bf16 *dQ, lt_bf16 *dK, lt_bf16 *dV, const lt_attn_layout *layout, int B,
                     int Hq, int Hkv, int S, int D, int causal, float scale, void *workspace,
                     size_t workspace_bytes, lt_stream_t stream) {
    return bwd_entry(Q, K, V, O, dO, LSE, dQ, dK, dV, layout, B, Hq, Hkv, S, D, causal, scale, workspace,
                     workspace_bytes, stream, nullptr, nullptr, true);
}

int lt_attn_bwd(const lt_half *Q, const lt_half *K, const lt_half *V, const lt_half *O, const lt_half *dO,
                const float *LSE, lt_half *dQ, lt_half *dK, lt_half *dV, int B, int Hq, int Hkv, int S, int D,
                int causal, float scale, void *workspace, size_t workspace_bytes, lt_stream_t stream) {
    return lt_attn_bwd_profiled(Q, K, V, O, dO, LSE, dQ, dK, dV, B, Hq, Hkv, S, D, causal, scale, workspace,
                                workspace_bytes, stream, nullptr, nullptr);
}

}  // extern "C"

// ----------------------------------------------------------------------------- backward without a caller workspace
// Scratch for lt_attn_bwd_noalloc: lives in the library image, so every GPU that loads the
// library carries these bytes until the process exits.  In host code the array's name is
// only a handle for the runtime; the address the kernels need is fetched once per device
// with cudaGetSymbolAddress.
namespace lt {
constexpr size_t kNoAllocScratchBytes = LT_ATTN_BWD_NOALLOC_MAX_SCRATCH_BYTES;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];
constexpr int kNoAllocMaxDevices = 64;
static void *g_noalloc_scratch_addr[kNoAllocMaxDevices];  // device address of the array, per device ordinal
static std::mutex g_noalloc_mutex;
}  // namespace lt

extern "C" {

int lt_attn_bwd_noalloc(const lt_half *Q, const lt_half *K, const lt_half *V, const lt_half *O, const lt_half *dO,
                        const float *LSE, lt_half *dQ, lt_half *dK, lt_half *dV, int B, int Hq, int Hkv, int S, int D,
                        int causal, float scale, lt_stream_t stream) {
    using namespace lt;
    if (!Q || !K || !V || !O || !dO || !LSE || !dQ || !dK || !dV) return LT_ERR_INVALID_ARG;
    int rc = check_shape(B, Hq, Hkv, S, D, scale);
    if (rc != LT_OK) return rc;
    const size_t need = bwd_least_bytes(B, Hq, S, D);
    if (need > kNoAllocScratchBytes) {
        char msg[160];
        snprintf(msg, sizeof(msg), "this shape needs %zu bytes of scratch but the built-in scratch holds %zu; "
                 "use lt_attn_bwd with a caller workspace", need, kNoAllocScratchBytes);
        set_last_error("lt_attn_bwd_noalloc", msg);
        return LT_ERR_WORKSPACE;
    }
    if ((rc = check_device()) != LT_OK) return rc;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return record_cuda_error("cudaGetDevice", e);
    if (dev < 0 || dev >= kNoAllocMaxDevices) {
        set_last_error("lt_attn_bwd_noalloc", "device ordinal out of range");
        return LT_ERR_UNSUPPORTED;
    }
    void *scratch = nullptr;
    {
        // first call on this device: look the array's device address up (no allocation happens)
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        if (!g_noalloc_scratch_addr[dev]) {
            void *addr = nullptr;
            e = cudaGetSymbolAddress(&addr, g_noalloc_scratch);
            if (e != cudaSuccess) return record_cuda_error("cudaGetSymbolAddress(scratch)", e);
            g_noalloc_scratch_addr[dev] = addr;
        }
        scratch = g_noalloc_scratch_addr[dev];
    }
    // every call clears the status words and zeroes the dQ accumulator itself where it uses them, so nothing left in the
    // scratch by an earlier call is read
    return lt_attn_bwd(Q, K, V, O, dO, LSE, dQ, dK, dV, B, Hq, Hkv, S, D, causal, scale, scratch, kNoAllocScratchBytes, stream);
}

int lt_attn_bwd_noalloc_check_status(lt_stream_t stream) {
    using namespace lt;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return record_cuda_error("cudaGetDevice", e);
    void *scratch = nullptr;
    if (dev >= 0 && dev < kNoAllocMaxDevices) {
        std::lock_guard<std::mutex> lock(g_noalloc_mutex);
        scratch = g_noalloc_scratch_addr[dev];
    }
    if (!scratch) return LT_OK;  // no lt_attn_bwd_noalloc call on this device yet: nothing to report
    return lt_attn_check_status(scratch, stream);
}

}  // extern "C"
