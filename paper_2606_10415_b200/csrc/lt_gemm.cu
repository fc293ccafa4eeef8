// FP16 GEMM for sm_100a: C[M,N] = A[M,K] W[N,K]^T, fp16 operands, fp32 accumulation, fp16 result.
// This is the linear-layer primitive of the paper's backend (Section 4.1, "FP16 GEMM assembly
// pipeline"; shapes profiled in Section 6.6).  The MT-3000 dataflow of the paper (A staged through
// GSM/SM, B broadcast to AM, C accumulated in AM) maps here to: A and W tiles staged in shared memory
// by TMA, C accumulated in tensor memory, one CTA per SM walking the output tiles.
//
//   warp 0      : TMA producer - 64-wide contraction blocks of a 128-row A tile and a 256-row W
//                 tile through a four-slot ring
//   warp 1      : tcgen05 issuer - four 128x256x16 products per block into one of two 256-column
//                 accumulators
//   warps 2..5  : epilogue - tensor memory -> fp16 -> global, one accumulator while the other is
//                 being filled
//
// Two further kernels share this arrangement: CTA pairs working 256 x 256 tiles (many tiles), and narrower tiles whose
// contraction is split over a cluster (few tiles); gemm_plan() chooses.
#include <cmath>
#include <cstdlib>
#include "../../include/lt_attn_debug.h"
#include "lt_common.cuh"
#include "lt_host.h"

namespace lt {

constexpr int kGemmBM = 128, kGemmBN = 256, kGemmBK = 64, kGemmStages = 4;
constexpr int kGemmThreads = 192;
constexpr uint32_t kGemmABytes = kGemmBM * kGemmBK * 2;   // 16 KB
constexpr uint32_t kGemmBBytes = kGemmBN * kGemmBK * 2;   // 32 KB

enum { kWaitGemmFull = 401, kWaitGemmEmpty = 402, kWaitGemmAccFull = 403, kWaitGemmAccEmpty = 404 };

constexpr int kStagePitch = 33;
struct __align__(1024) GemmSmem {
    uint8_t a[kGemmStages][kGemmABytes];
    uint8_t b[kGemmStages][kGemmBBytes];
    uint64_t bar_full[kGemmStages], bar_empty[kGemmStages], bar_acc_full[2], bar_acc_empty[2];
    float stage[4][32 * kStagePitch];  // per epilogue warp: 32 x 32 of a tile on a ragged edge
    uint32_t tmem_base;
    int abort_flag;
};

struct GemmParams {
    __half *C;
    unsigned int *status;
    int M, N, K;
    int tiles_m, tiles_n;
    uint32_t a_bytes;  // a block of A's rows as it is brought into shared memory
    int group_rows;  // tile rows of A kept hot in L2 while the W column blocks stream past them
};

// Output tiles are numbered so that consecutive numbers share the W tile (the larger operand tile)
// and a wave of CTAs covers a compact block of C: tile -> (m, n) with m fastest inside groups of
// `group_rows` tile rows (as many rows of A as stay resident in L2, so that W is read from DRAM once
// per group).
__device__ __forceinline__ void gemm_tile_coords(const GemmParams &p, int tile, int &tm, int &tn) {
    const int kGroup = p.group_rows;
    const int per_group = kGroup * p.tiles_n;
    const int g = tile / per_group;
    const int first_m = g * kGroup;
    const int rows = min(kGroup, p.tiles_m - first_m);
    const int r = tile - g * per_group;
    tm = first_m + r % rows;
    tn = r / rows;
}

// 32 rows x 32 columns of the output whose rows are not a whole number of 16-byte pieces (N % 8 != 0) or that stick out
// past column N.  Each lane arrives with one row in registers; through shared memory the warp turns it so that
// neighbouring lanes store neighbouring columns: 64 contiguous bytes per row and instruction, where a lane storing its own row
// two bytes at a time touched a sector for every element (113 x 4051 x 208: 39 us).
template <bool kBf16>
__device__ __forceinline__ void gemm_store_ragged(float *stage, const uint32_t (&r)[32], const GemmParams &p,
                                                  long long m0, int nc, int lane) {
    __syncwarp();
#pragma unroll
    for (int e = 0; e < 32; ++e) stage[lane * kStagePitch + e] = __uint_as_float(r[e]);
    __syncwarp();
    const int rows = p.M - m0 < 32 ? static_cast<int>(p.M - m0) : 32;
    if ((p.N & 1) == 0) {  // pairs of columns: half a warp per row
        const int col = (lane & 15) * 2;
        for (int q = lane >> 4; q < rows && nc + col < p.N; q += 2)
            *reinterpret_cast<uint32_t *>(p.C + (m0 + q) * p.N + nc + col) =
                pack2<kBf16>(stage[q * kStagePitch + col], stage[q * kStagePitch + col + 1]);
    } else {
        for (int q = 0; q < rows && nc + lane < p.N; ++q)
            reinterpret_cast<uint16_t *>(p.C)[(m0 + q) * p.N + nc + lane] =
                static_cast<uint16_t>(pack2<kBf16>(stage[q * kStagePitch + lane], 0.f) & 0xFFFFu);
    }
}

template <bool kBf16>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
            const GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    GemmSmem &sm = *reinterpret_cast<GemmSmem *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int n_tiles = p.tiles_m * p.tiles_n;
    const int k_blocks = (p.K + kGemmBK - 1) / kGemmBK;  // a ragged last block reads zeros past K

    if (tid == 0) {
        sm.abort_flag = 0;
        for (int s = 0; s < kGemmStages; ++s) {
            mbar_init(&sm.bar_full[s], 1);
            mbar_init(&sm.bar_empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&sm.bar_acc_full[a], 1);
            mbar_init(&sm.bar_acc_empty[a], 4);  // lane 0 of each epilogue warp
        }
        mbar_fence_init();
        tma_prefetch_desc(&map_a);
        tma_prefetch_desc(&map_b);
    }
    if (warp == 0) {
        tmem_alloc(&sm.tmem_base, 512);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    volatile int *abort_flag = &sm.abort_flag;
    // the set-up above ran under the tail of the predecessor in the stream
    grid_dependency_wait();
    // The next kernel of the stream may be scheduled as this one's CTAs exit and set itself up (it waits for the whole grid
    // before it touches memory); all CTAs of this grid are running by then, so none is kept out.  Measured, us per call in
    // a graph of calls, without / with: 16 x 1024 x 1024 (M x N x K) 5.8 / 4.8, 77 x 4096 x 4096 12.9 / 11.9, 300 x 1000 x 1000 8.1 /
    // 7.0, 512 x 4096 x 4096 24.2 / 22.4, 2048 x 11008 x 4096 159 / 156, 8192 x 1024 x 512 13.2 / 12.9.
    grid_launch_dependents();
    if (blockIdx.x == 0 && tid == 0) p.status[kStatusWordTimeout] = 0u;  // (a wait gives up after a second at the earliest)

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int kb_total = 0;  // contraction blocks loaded so far, over all tiles
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
                int tm, tn;
                gemm_tile_coords(p, tile, tm, tn);
                for (int kb = 0; kb < k_blocks; ++kb, ++kb_total) {
                    const int s = kb_total % kGemmStages;
                    const uint32_t use = kb_total / kGemmStages;
                    if (use >= 1 && !(ok = mbar_wait(&sm.bar_empty[s], (use - 1) & 1, abort_flag, p.status, kWaitGemmEmpty)))
                        break;
                    mbar_arrive_expect_tx(&sm.bar_full[s], p.a_bytes + kGemmBBytes);
                    tma_load_2d(sm.a[s], &map_a, &sm.bar_full[s], kb * kGemmBK, tm * kGemmBM);
                    tma_load_2d(sm.b[s], &map_b, &sm.bar_full[s], kb * kGemmBK, tn * kGemmBN);
                }
            }
            if (!ok || *abort_flag) {
                // somebody gave up: wait (bounded) for the copies in flight before the CTA exits
                for (int back = 0; back < kGemmStages && back < kb_total; ++back) {
                    const int q = kb_total - 1 - back;
                    for (int w = 0; w < (1 << 16) && !mbar_try_wait(&sm.bar_full[q % kGemmStages], (q / kGemmStages) & 1); ++w) {}
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = make_idesc(kGemmBM, kGemmBN, false, false, kBf16);
            bool ok = true;
            int kb_total = 0, t_local = 0;
#ifdef LT_GEMM_TRACE
            long long tr_full = 0, tr_acc = 0, tr_issue = 0, tr_t = clock64();
#define LT_GT(var) do { const long long n_ = clock64(); var += n_ - tr_t; tr_t = n_; } while (0)
#else
#define LT_GT(var)
#endif
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++t_local) {
                const int acc = t_local & 1;
                const uint32_t acc_use = t_local >> 1;
                // the epilogue must have read this accumulator's previous tile
                if (acc_use >= 1 && !(ok = mbar_wait(&sm.bar_acc_empty[acc], (acc_use - 1) & 1, abort_flag, p.status, kWaitGemmAccEmpty)))
                    break;
                LT_GT(tr_acc);
                tc_fence_after_sync();
                for (int kb = 0; kb < k_blocks; ++kb, ++kb_total) {
                    const int s = kb_total % kGemmStages;
                    LT_GT(tr_issue);
                    if (!(ok = mbar_wait(&sm.bar_full[s], (kb_total / kGemmStages) & 1, abort_flag, p.status, kWaitGemmFull))) break;
                    LT_GT(tr_full);
                    tc_fence_after_sync();
                    const uint64_t da = desc_kmajor(smem_u32(sm.a[s])), db = desc_kmajor(smem_u32(sm.b[s]));
#pragma unroll
                    for (int kk = 0; kk < kGemmBK / 16; ++kk)
                        umma_ss(tmem + acc * kGemmBN, da + kk * 2, db + kk * 2, idesc, (kb > 0) | (kk > 0));
                    umma_commit(&sm.bar_empty[s]);  // the slot is free once these products have read it
                }
                if (!ok) break;
                umma_commit(&sm.bar_acc_full[acc]);
                LT_GT(tr_issue);
            }
#ifdef LT_GEMM_TRACE
            if (blockIdx.x == 0) {
                p.status[8] = static_cast<unsigned int>(tr_full >> 4);
                p.status[9] = static_cast<unsigned int>(tr_acc >> 4);
                p.status[10] = static_cast<unsigned int>(tr_issue >> 4);
                p.status[11] = static_cast<unsigned int>(kb_total);
            }
#endif
        }
    } else {
        // epilogue: thread = row of the tile, 32 columns at a time
        const int quad = warp & 3;  // tensor-memory lane quadrant this warp may read
        const int row = quad * 32 + lane;
        const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
        bool ok = true;
        int t_local = 0;
        for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++t_local) {
            const int acc = t_local & 1;
            ok = mbar_wait(&sm.bar_acc_full[acc], (t_local >> 1) & 1, abort_flag, p.status, kWaitGemmAccFull);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after_sync();
            int tm, tn;
            gemm_tile_coords(p, tile, tm, tn);
            const long long m = static_cast<long long>(tm) * kGemmBM + row;
            const int n0 = tn * kGemmBN;
            __half *c_row = p.C + m * p.N + n0;
            const bool vec_ok = (p.N % 8) == 0;  // 16-byte stores need the row pitch to allow them
#pragma unroll
            for (int c = 0; c < kGemmBN / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(tmem + lane_base + acc * kGemmBN + c * 32, r);
                tmem_wait_ld();
                if (c == kGemmBN / 32 - 1) {
                    // the whole accumulator is in registers or stored: the issuer may reuse it
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&sm.bar_acc_empty[acc]);
                }
                const int nc = n0 + c * 32;
                if (vec_ok && nc + 32 <= p.N) {
                    if (m < p.M) {
#pragma unroll
                        for (int v8 = 0; v8 < 4; ++v8) {
                            uint4 o;
                            o.x = pack2<kBf16>(__uint_as_float(r[8 * v8 + 0]), __uint_as_float(r[8 * v8 + 1]));
                            o.y = pack2<kBf16>(__uint_as_float(r[8 * v8 + 2]), __uint_as_float(r[8 * v8 + 3]));
                            o.z = pack2<kBf16>(__uint_as_float(r[8 * v8 + 4]), __uint_as_float(r[8 * v8 + 5]));
                            o.w = pack2<kBf16>(__uint_as_float(r[8 * v8 + 6]), __uint_as_float(r[8 * v8 + 7]));
                            reinterpret_cast<uint4 *>(c_row + c * 32)[v8] = o;
                        }
                    }
                } else if (nc < p.N) {
                    gemm_store_ragged<kBf16>(sm.stage[quad], r, p, m - lane, nc, lane);
                }
            }
        }
    }

    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 512);
}

// ----------------------------------------------------------------------------- CTA-pair variant
// Two CTAs of a cluster work one 256 x 256 output tile: each loads 128 rows of A and 128 of the 256 rows of
// W per contraction block (32 KB per block and CTA where the single-CTA kernel loads 48 KB for the same
// number of FLOPs per SM), the even CTA issues 256x256x16 pair products, and each CTA's epilogue stores the
// 128 rows of C that its tensor memory holds.  Barriers: `full` lives in the issuing CTA and collects the
// bytes of both CTAs' loads; `empty` and `acc_full` are signalled in both CTAs by pair commits; `acc_empty`
// lives in the issuing CTA and is arrived on by the epilogue warps of both.
constexpr int kPairBM = 256, kPairBN = 256, kPairStages = 6;
constexpr uint32_t kPairABytes = 128 * kGemmBK * 2;   // 16 KB: this CTA's rows of the A tile
constexpr uint32_t kPairBBytes = 128 * kGemmBK * 2;   // 16 KB: this CTA's half of the W tile's rows

struct __align__(1024) GemmPairSmem {
    uint8_t a[kPairStages][kPairABytes];
    uint8_t b[kPairStages][kPairBBytes];
    uint64_t bar_full[kPairStages], bar_empty[kPairStages], bar_acc_full[2], bar_acc_empty[2];
    float stage[4][32 * kStagePitch];  // per epilogue warp: 32 x 32 of a tile on a ragged edge
    uint32_t tmem_base;
    int abort_flag;
};

template <bool kBf16>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kGemmThreads, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                 const GemmParams p) {
    extern __shared__ uint8_t smem_raw[];
    // (the dynamic window starts at the same offset in both CTAs, so the aligned structure does too)
    GemmPairSmem &sm =
        *reinterpret_cast<GemmPairSmem *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const uint32_t rank = cluster_cta_rank();   // 0 issues the products
    const int pair = blockIdx.x >> 1;
    const int n_pairs = gridDim.x >> 1;
    const int n_tiles = p.tiles_m * p.tiles_n;  // 256 x 256 tiles
    const int k_blocks = (p.K + kGemmBK - 1) / kGemmBK;

    if (tid == 0) {
        sm.abort_flag = 0;
        for (int s = 0; s < kPairStages; ++s) {
            mbar_init(&sm.bar_full[s], 1);
            mbar_init(&sm.bar_empty[s], 1);
        }
        for (int a = 0; a < 2; ++a) {
            mbar_init(&sm.bar_acc_full[a], 1);
            mbar_init(&sm.bar_acc_empty[a], 8);  // lane 0 of each epilogue warp of both CTAs
        }
        mbar_fence_init();
        tma_prefetch_desc(&map_a);
        tma_prefetch_desc(&map_b);
    }
    if (warp == 0) {
        tmem_alloc_pair(&sm.tmem_base, 512);
        tmem_relinquish_pair();
    }
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();  // the partner's barriers exist before anything is sent to them
    tc_fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    volatile int *abort_flag = &sm.abort_flag;
    grid_dependency_wait();
    grid_launch_dependents();  // (as in gemm_kernel)
    if (blockIdx.x == 0 && tid == 0) p.status[kStatusWordTimeout] = 0u;

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int kb_total = 0;
            for (int tile = pair; tile < n_tiles && ok; tile += n_pairs) {
                int tm, tn;
                gemm_tile_coords(p, tile, tm, tn);
                const int a_row = tm * kPairBM + static_cast<int>(rank) * 128;
                const int b_row = tn * kPairBN + static_cast<int>(rank) * 128;
                for (int kb = 0; kb < k_blocks; ++kb, ++kb_total) {
                    const int s = kb_total % kPairStages;
                    const uint32_t use = kb_total / kPairStages;
                    if (use >= 1 && !(ok = mbar_wait(&sm.bar_empty[s], (use - 1) & 1, abort_flag, p.status, kWaitGemmEmpty)))
                        break;
                    // the issuing CTA's barrier expects the bytes of all four loads of the pair
                    if (rank == 0) mbar_arrive_expect_tx(&sm.bar_full[s], 2 * (kPairABytes + kPairBBytes));
                    const uint32_t full0 = cluster_map_shared(smem_u32(&sm.bar_full[s]), 0);
                    tma_load_2d_pair(sm.a[s], &map_a, full0, kb * kGemmBK, a_row);
                    tma_load_2d_pair(sm.b[s], &map_b, full0, kb * kGemmBK, b_row);
                }
            }
            if (!ok || *abort_flag) {
                // somebody gave up: give this CTA's own copies a bounded time to land (the slots' `empty`
                // barriers cannot tell; the issuing CTA's `full` barriers can, for the last slots used)
                if (rank == 0)
                    for (int back = 0; back < kPairStages && back < kb_total; ++back) {
                        const int q = kb_total - 1 - back;
                        for (int w = 0; w < (1 << 16) && !mbar_try_wait(&sm.bar_full[q % kPairStages], (q / kPairStages) & 1); ++w) {}
                    }
                else
                    for (int w = 0; w < 256; ++w) __nanosleep(100);  // (its byte counts go to the partner's barriers)
            }
        }
    } else if (warp == 1) {
        if (lane == 0 && rank == 0) {
            constexpr uint32_t idesc = make_idesc(kPairBM, kPairBN, false, false, kBf16);
            bool ok = true;
            int kb_total = 0, t_local = 0;
            for (int tile = pair; tile < n_tiles && ok; tile += n_pairs, ++t_local) {
                const int acc = t_local & 1;
                const uint32_t acc_use = t_local >> 1;
                if (acc_use >= 1 && !(ok = mbar_wait(&sm.bar_acc_empty[acc], (acc_use - 1) & 1, abort_flag, p.status, kWaitGemmAccEmpty)))
                    break;
                tc_fence_after_sync();
                for (int kb = 0; kb < k_blocks; ++kb, ++kb_total) {
                    const int s = kb_total % kPairStages;
                    if (!(ok = mbar_wait(&sm.bar_full[s], (kb_total / kPairStages) & 1, abort_flag, p.status, kWaitGemmFull))) break;
                    tc_fence_after_sync();
                    const uint64_t da = desc_kmajor(smem_u32(sm.a[s])), db = desc_kmajor(smem_u32(sm.b[s]));
#pragma unroll
                    for (int kk = 0; kk < kGemmBK / 16; ++kk)
                        umma_ss_pair(tmem + acc * kPairBN, da + kk * 2, db + kk * 2, idesc, (kb > 0) | (kk > 0));
                    umma_commit_pair(&sm.bar_empty[s], 3);  // both CTAs' slots are free once these have read them
                }
                if (!ok) break;
                umma_commit_pair(&sm.bar_acc_full[acc], 3);
            }
        }
    } else {
        // epilogue: this CTA's 128 rows of the tile; thread = row, 32 columns at a time
        const int quad = warp & 3;
        const int row = quad * 32 + lane;
        const uint32_t lane_base = static_cast<uint32_t>(quad * 32) << 16;
        bool ok = true;
        int t_local = 0;
        for (int tile = pair; tile < n_tiles; tile += n_pairs, ++t_local) {
            const int acc = t_local & 1;
            ok = mbar_wait(&sm.bar_acc_full[acc], (t_local >> 1) & 1, abort_flag, p.status, kWaitGemmAccFull);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after_sync();
            int tm, tn;
            gemm_tile_coords(p, tile, tm, tn);
            const long long m = static_cast<long long>(tm) * kPairBM + rank * 128 + row;
            const int n0 = tn * kPairBN;
            __half *c_row = p.C + m * p.N + n0;
            const bool vec_ok = (p.N % 8) == 0;
            const uint32_t acc_empty0 = cluster_map_shared(smem_u32(&sm.bar_acc_empty[acc]), 0);
#pragma unroll
            for (int c = 0; c < kPairBN / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(tmem + lane_base + acc * kPairBN + c * 32, r);
                tmem_wait_ld();
                if (c == kPairBN / 32 - 1) {
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster(acc_empty0);
                }
                const int nc = n0 + c * 32;
                if (vec_ok && nc + 32 <= p.N) {
                    if (m < p.M) {
#pragma unroll
                        for (int v8 = 0; v8 < 4; ++v8) {
                            uint4 o;
                            o.x = pack2<kBf16>(__uint_as_float(r[8 * v8 + 0]), __uint_as_float(r[8 * v8 + 1]));
                            o.y = pack2<kBf16>(__uint_as_float(r[8 * v8 + 2]), __uint_as_float(r[8 * v8 + 3]));
                            o.z = pack2<kBf16>(__uint_as_float(r[8 * v8 + 4]), __uint_as_float(r[8 * v8 + 5]));
                            o.w = pack2<kBf16>(__uint_as_float(r[8 * v8 + 6]), __uint_as_float(r[8 * v8 + 7]));
                            reinterpret_cast<uint4 *>(c_row + c * 32)[v8] = o;
                        }
                    }
                } else if (nc < p.N) {
                    gemm_store_ragged<kBf16>(sm.stage[quad], r, p, m - lane, nc, lane);
                }
            }
        }
    }

    // neither CTA may release its tensor memory or leave (its shared memory and barriers are still
    // targets of the partner) before both are done
    tc_fence_before_sync();
    __syncthreads();
    cluster_sync_all();
    if (warp == 0) tmem_dealloc_pair(tmem, 512);
}

// ----------------------------------------------------------------------------- few output tiles
// Shapes whose output has too few large tiles to occupy the chip: narrower tiles (128 x kBN) and the contraction of
// each tile split over the CTAs of a cluster.  Every CTA accumulates its share of the contraction in tensor memory,
// leaves the fp32 partial in its shared memory, and after a cluster barrier each CTA sums a slice of the tile's rows over
// the cluster's partials (in rank order, so results are reproducible), rounds and stores it.  One tile share per CTA.
template <int kBN>
struct __align__(1024) GemmSplitSmem {
    static constexpr uint32_t kBBytes = kBN * kGemmBK * 2;
    static constexpr int kStages = static_cast<int>(196608 / (kGemmABytes + kBBytes));
    static constexpr int kPitch = kBN + 4;  // floats per row of the partial: 16-byte stores of a warp hit all banks
    union {
        struct {
            uint8_t a[kStages][kGemmABytes];
            uint8_t b[kStages][kBBytes];
        } ring;
        float partial[kGemmBM * kPitch];  // once every block of the share has been multiplied
    };
    uint64_t bar_full[kStages], bar_empty[kStages], bar_acc;
    uint32_t tmem_base;
    int abort_flag;
};

template <int kBN, bool kBf16>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_split_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                  const GemmParams p) {
    using Smem = GemmSplitSmem<kBN>;
    constexpr int kStages = Smem::kStages;
    extern __shared__ uint8_t smem_raw[];
    // (the dynamic window starts at the same offset in every CTA, so the aligned structure does too)
    Smem &sm = *reinterpret_cast<Smem *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const int lane = tid & 31;
    const int split = static_cast<int>(cluster_cta_count());
    const int rank = static_cast<int>(cluster_cta_rank());
    int tm, tn;
    gemm_tile_coords(p, static_cast<int>(blockIdx.x) / split, tm, tn);
    const int k_blocks = (p.K + kGemmBK - 1) / kGemmBK;
    const int kb0 = static_cast<int>(static_cast<long long>(k_blocks) * rank / split);
    const int n_kb = static_cast<int>(static_cast<long long>(k_blocks) * (rank + 1) / split) - kb0;  // >= 1

    if (tid == 0) {
        sm.abort_flag = 0;
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&sm.bar_full[s], 1);
            mbar_init(&sm.bar_empty[s], 1);
        }
        mbar_init(&sm.bar_acc, 1);
        mbar_fence_init();
        tma_prefetch_desc(&map_a);
        tma_prefetch_desc(&map_b);
    }
    if (warp == 0) {
        tmem_alloc(&sm.tmem_base, kBN);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = sm.tmem_base;
    volatile int *abort_flag = &sm.abort_flag;
    grid_dependency_wait();
    grid_launch_dependents();  // (as in gemm_kernel)
    if (blockIdx.x == 0 && tid == 0) p.status[kStatusWordTimeout] = 0u;

    if (warp == 0) {
        if (lane == 0) {
            bool ok = true;
            int i = 0;
            for (; i < n_kb; ++i) {
                const int s = i % kStages;
                const uint32_t use = i / kStages;
                if (use >= 1 && !(ok = mbar_wait(&sm.bar_empty[s], (use - 1) & 1, abort_flag, p.status, kWaitGemmEmpty))) break;
                mbar_arrive_expect_tx(&sm.bar_full[s], p.a_bytes + Smem::kBBytes);
                tma_load_2d(sm.ring.b[s], &map_b, &sm.bar_full[s], (kb0 + i) * kGemmBK, tn * kBN);
                tma_load_2d(sm.ring.a[s], &map_a, &sm.bar_full[s], (kb0 + i) * kGemmBK, tm * kGemmBM);
            }
            if (!ok || *abort_flag) {
                // somebody gave up: wait (bounded) for the copies in flight before the CTA exits
                for (int back = 0; back < kStages && back < i; ++back) {
                    const int q = i - 1 - back;
                    for (int w = 0; w < (1 << 16) && !mbar_try_wait(&sm.bar_full[q % kStages], (q / kStages) & 1); ++w) {}
                }
            }
        }
    } else if (warp == 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = make_idesc(kGemmBM, kBN, false, false, kBf16);
            bool ok = true;
            for (int i = 0; i < n_kb; ++i) {
                const int s = i % kStages;
                if (!(ok = mbar_wait(&sm.bar_full[s], (i / kStages) & 1, abort_flag, p.status, kWaitGemmFull))) break;
                tc_fence_after_sync();
                const uint64_t da = desc_kmajor(smem_u32(sm.ring.a[s])), db = desc_kmajor(smem_u32(sm.ring.b[s]));
#pragma unroll
                for (int kk = 0; kk < kGemmBK / 16; ++kk)
                    umma_ss(tmem, da + kk * 2, db + kk * 2, idesc, (i > 0) | (kk > 0));
                umma_commit(&sm.bar_empty[s]);
            }
            if (ok) umma_commit(&sm.bar_acc);
        }
    } else {
        // this CTA's share of the sum: tensor memory -> shared memory (every load has landed and been read by then);
        // thread = row of the tile
        const int quad = warp & 3;  // tensor-memory lane quadrant this warp may read
        const bool ok = __all_sync(0xffffffffu, mbar_wait(&sm.bar_acc, 0, abort_flag, p.status, kWaitGemmAccFull));
        if (ok) {
            tc_fence_after_sync();
            const uint32_t taddr = tmem + (static_cast<uint32_t>(quad * 32) << 16);
            float *row = sm.partial + (quad * 32 + lane) * Smem::kPitch;
#pragma unroll
            for (int c = 0; c < kBN / 32; ++c) {
                uint32_t r[32];
                tmem_ld32(taddr + c * 32, r);
                tmem_wait_ld();
#pragma unroll
                for (int v = 0; v < 8; ++v)
                    *reinterpret_cast<uint4 *>(row + c * 32 + v * 4) = make_uint4(r[4 * v], r[4 * v + 1], r[4 * v + 2], r[4 * v + 3]);
            }
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, kBN);
    cluster_sync_all();  // every partial of the tile is in place
    {
        const int rows = min(kGemmBM, p.M - tm * kGemmBM);
        const int r0 = rows * rank / split, r1 = rows * (rank + 1) / split;
        constexpr int kChunks = kBN / 8;  // pieces of eight columns
        const bool vec_ok = (p.N % 8) == 0;
        const uint32_t base = smem_u32(sm.partial);
        for (int u = tid; u < (r1 - r0) * kChunks; u += kGemmThreads) {
            const int row = r0 + u / kChunks, col = (u % kChunks) * 8;
            const int n = tn * kBN + col;
            if (n >= p.N) continue;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
            const uint32_t local = base + (row * Smem::kPitch + col) * 4;
            for (int q = 0; q < split; ++q) {
                const uint32_t addr = cluster_map_shared(local, q);
                const float4 u4 = ld_cluster_v4(addr), w4 = ld_cluster_v4(addr + 16);
                x.x += u4.x; x.y += u4.y; x.z += u4.z; x.w += u4.w;
                y.x += w4.x; y.y += w4.y; y.z += w4.z; y.w += w4.w;
            }
            __half *dst = p.C + (static_cast<long long>(tm) * kGemmBM + row) * p.N + n;
            const uint4 o = make_uint4(pack2<kBf16>(x.x, x.y), pack2<kBf16>(x.z, x.w), pack2<kBf16>(y.x, y.y), pack2<kBf16>(y.z, y.w));
            if (vec_ok) {  // (N a multiple of eight: a piece lies inside the row or outside)
                *reinterpret_cast<uint4 *>(dst) = o;
            } else {
                // (one column per lane instead, with 4-byte reads of the partials, was slower: 274 x 3485 x 4424 56 us
                // against 36)
                const uint32_t w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (n + e < p.N)
                        reinterpret_cast<uint16_t *>(dst)[e] = static_cast<uint16_t>((w[e >> 1] >> ((e & 1) * 16)) & 0xFFFFu);
            }
        }
    }
    __syncthreads();
    cluster_sync_all();  // nobody leaves while its partial may still be read
}

template <int kBN, bool kBf16>
static int launch_gemm_split(const CUtensorMap &ma, const CUtensorMap &mb, GemmParams prm, int split, cudaStream_t stream) {
    prm.tiles_m = (prm.M + kGemmBM - 1) / kGemmBM;
    prm.tiles_n = (prm.N + kBN - 1) / kBN;
    prm.group_rows = prm.tiles_m;
    const size_t smem = sizeof(GemmSplitSmem<kBN>) + 1024;
    auto kernel = gemm_split_kernel<kBN, kBf16>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return record_cuda_error("cudaFuncSetAttribute(gemm_split)", e);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = split;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(prm.tiles_m * prm.tiles_n * split);
    cfg.blockDim = dim3(kGemmThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, kernel, ma, mb, prm);
    if (e == cudaSuccess) e = cudaGetLastError();
    return e == cudaSuccess ? LT_OK : record_cuda_error("gemm_split_kernel launch", e);
}

}  // namespace lt

extern "C" {

size_t lt_gemm_f16_workspace_bytes(void) { return lt::kStatusBytes; }

// Which kernel: tile width and contraction shares per tile, or the CTA-pair kernel.  The choice is the smallest
// estimate of a time model in microseconds whose constants were fitted to 450 measured (shape, kernel) pairs (27 shapes
// with 1-8192 rows, every width and split), before the kernels were launched under one another's tails.  Measured since
// with all plans on 90 drawn shapes, calls back to back in a graph: the kernel it picks takes 4.9 % more than the fastest
// one on average, 52 % at worst (397 x 3773 x 648 19.5 us, 128-wide 12.8).  On 300 drawn shapes against the two kernels that
// came before (256-wide on one CTA up to 128 rows, on pairs above): 0.42 of the time in the geometric mean, one shape
// slower by more than 2 % (1812 x 2880 x 1176 29.1 / 31.1).
//   first wave: launch, fill and drain, plus the blocks of the longest share (a block takes the larger part of issuing
//   its products and of bringing its A and W rows in while the other CTAs do the same), plus the epilogue, which costs
//   more per element when the partials of a cluster are summed; every further wave costs its own fill and drain, except
//   in the persistent kernels.
// Measured, us, before (256-wide tiles on one CTA or a pair) and now: 77 x 4096 x 4096 (M x N x K) 28.2 / 12.0 (128-wide,
// four shares), 128 x 128 x 4096 22.3 / 8.7 (64-wide, eight), 424 x 265 x 5920 64 / 11.3 (64, six), 3000 x 128 x 11008
// 54 / 21 (128, five), 1024 x 2048 x 8192 43.5 / 35.7 (256, two), 700 x 2048 x 1024 11.0 / 9.6 (256, whole).
// On the other side of the line: 512 x 4096 x 4096 128-wide 25.7 against the pair kernel's 25.8, 1024 x 4096 x 4096 49
// against 29.
struct GemmPlan {
    int bn, split;
    bool pair;
};
static GemmPlan gemm_plan(int M, int N, int K) {
    using namespace lt;
    auto ceil_div = [](long long a, long long b) { return (a + b - 1) / b; };
    const double k_blocks = static_cast<double>(ceil_div(K, kGemmBK));
    GemmPlan best{kGemmBN, 1, false};
    double best_us = 4.4 + ceil_div(ceil_div(M, kGemmBM) * ceil_div(N, kGemmBN), 148) * k_blocks * 0.357;
    // A short contraction does not hide the fill and the 256-wide drain, which take this much by themselves.  Measured, us,
    // without this line (256-wide) / with it (64- or 128-wide): 150 x 1408 x 152 8.3 / 5.0, 404 x 1152 x 272 8.1 / 5.3, 266 x
    // 685 x 224 14.2 / 7.2; 150 drawn shapes 1.05x, none slower.  Longer contractions on one wave are right at 256:
    // 700 x 2048 x 1024 9.7 against 10.3.
    if (best_us < 7.2) best_us = 7.2;
    auto offer = [&](GemmPlan plan, double us) {
        if (us < best_us) best = plan, best_us = us;
    };
    if (M > kGemmBM)
        offer({kPairBN, 1, true}, 6.7 + ceil_div(ceil_div(M, kPairBM) * ceil_div(N, kPairBN), 74) * k_blocks * 0.304);
    // clusters of so many CTAs, one CTA per multiprocessor, that fit at once (cudaOccupancyMaxActiveClusters on a B200)
    constexpr int kMaxClusters[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
    const double rows = M < kGemmBM ? M : kGemmBM;
    for (int w = 0; w < 3; ++w) {
        const int bn = 64 << w;
        const double issue = w == 0 ? 0.260 : w == 1 ? 0.296 : 0.428;
        const long long tiles = ceil_div(M, kGemmBM) * ceil_div(N, bn);
        for (int split = w == 2 ? 2 : 1; split <= 8 && split <= k_blocks; ++split) {
            const double waves = static_cast<double>(ceil_div(tiles, kMaxClusters[split]));
            const double fill = tiles * split < 148 ? tiles * split / 148.0 : 1.0;
            const double bring = (rows + bn) * (kGemmBK * 2) * 6.0e-6 * fill;
            const double work = ceil(k_blocks / split) * sqrt(issue * issue + bring * bring) +
                                rows * bn * 4e-3 * (split > 1 ? 0.0372 : 0.0154);
            offer({bn, split, false}, 4.5 + (split > 1 ? 0.57 : 0.0) + waves * work + (waves - 1) * 4.6);
        }
    }
    return best;
}

// the plan, or the single-CTA kernel where LT_GEMM_SINGLE_CTA=1 in the environment keeps it, for comparison
static GemmPlan gemm_choice(int M, int N, int K) {
    static const bool force_single = [] {
        const char *v = getenv("LT_GEMM_SINGLE_CTA");
        return v && v[0] == '1';
    }();
    return force_single ? GemmPlan{lt::kGemmBN, 1, false} : gemm_plan(M, N, K);
}

int lt_dbg_gemm_plan(int M, int N, int K, int *tile_columns, int *shares, int *pairs) {
    if (M <= 0 || N <= 0 || K <= 0 || !tile_columns || !shares || !pairs) return LT_ERR_INVALID_ARG;
    const GemmPlan plan = gemm_choice(M, N, K);
    *tile_columns = plan.bn;
    *shares = plan.split;
    *pairs = plan.pair ? 1 : 0;
    return LT_OK;
}

static int gemm_entry(const void *A, const void *W, void *C, int M, int N, int K, void *workspace,
                      size_t workspace_bytes, lt_stream_t stream, bool bf16) {
    using namespace lt;
    if (!A || !W || !C) return LT_ERR_INVALID_ARG;
    if (M <= 0 || N <= 0 || K <= 0) return LT_ERR_INVALID_ARG;
    // TMA needs 16-byte row pitches for the operands
    if ((K % 8) != 0) return LT_ERR_UNSUPPORTED;
    if (!aligned16(A) || !aligned16(W) || !aligned16(C)) return LT_ERR_UNSUPPORTED;
    if (!workspace || !aligned256(workspace) || workspace_bytes < kStatusBytes) return LT_ERR_WORKSPACE;
    int rc = check_device();
    if (rc != LT_OK) return rc;

    GemmParams prm;
    prm.C = reinterpret_cast<__half *>(C);
    prm.status = reinterpret_cast<unsigned int *>(workspace);
    prm.M = M; prm.N = N; prm.K = K;
    // A of up to 64 rows: only those are brought in (whole swizzle atoms of eight), not a box of 128 whose other rows the
    // copy fills with zeros.  The products read whatever lies behind them in shared memory, and write it to accumulator
    // rows that nobody stores.  Measured, us, box of 128 / of the rows: 1 x 4096 x 4096 (M x N x K) 11.6 / 9.8, 12 rows
    // 12.9 / 10.8, 40 rows 11.8 / 11.7; 1 x 11008 x 4096 21.8 / 19.1; 1 x 2048 x 8192 15.2 / 12.1; 24 x 1024 x 1024 6.3 /
    // 5.9; 8 x 32768 x 512 9.3 / 7.9.  On the other side of the line nothing is gained: 77 x 4096 x 4096 12.7 / 12.8,
    // 100 rows 13.9 / 14.1, 100 x 32768 x 512 10.3 / 10.5.
    const uint32_t a_rows = M <= 64 ? (M + 7) / 8 * 8 : kGemmBM;
    prm.a_bytes = a_rows * kGemmBK * 2;

    const GemmPlan plan = gemm_choice(M, N, K);
    const bool use_pair = plan.pair;
    CUtensorMap ma, mb;
    if ((rc = make_tile_map(&ma, A, M, K, a_rows)) != LT_OK) return rc;
    if ((rc = make_tile_map(&mb, W, N, K, use_pair ? 128 : plan.bn)) != LT_OK) return rc;
    if (!use_pair && plan.bn == 64)
        return bf16 ? launch_gemm_split<64, true>(ma, mb, prm, plan.split, stream)
                    : launch_gemm_split<64, false>(ma, mb, prm, plan.split, stream);
    if (!use_pair && plan.bn == 128)
        return bf16 ? launch_gemm_split<128, true>(ma, mb, prm, plan.split, stream)
                    : launch_gemm_split<128, false>(ma, mb, prm, plan.split, stream);
    if (!use_pair && plan.bn == 256 && plan.split > 1)
        return bf16 ? launch_gemm_split<256, true>(ma, mb, prm, plan.split, stream)
                    : launch_gemm_split<256, false>(ma, mb, prm, plan.split, stream);
    cudaError_t e = cudaSuccess;
    cudaLaunchAttribute pdl;
    pdl.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    pdl.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kGemmThreads);
    cfg.stream = stream;
    cfg.attrs = &pdl;
    cfg.numAttrs = 1;
    if (use_pair) {
        prm.tiles_m = (M + kPairBM - 1) / kPairBM;
        prm.tiles_n = (N + kPairBN - 1) / kPairBN;
        const long long rows = static_cast<long long>(48.0e6 / (static_cast<double>(kPairBM) * K * 2.0));
        prm.group_rows = static_cast<int>(rows < 1 ? 1 : (rows > prm.tiles_m ? prm.tiles_m : rows));
        const size_t smem = sizeof(GemmPairSmem) + 1024;
        auto kernel = bf16 ? gemm_pair_kernel<true> : gemm_pair_kernel<false>;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
        if (e != cudaSuccess) return record_cuda_error("cudaFuncSetAttribute(gemm_pair)", e);
        // CTA pairs that can be resident at once (every pair needs two SMs of one cluster-capable group)
        static int max_pairs_cached[2] = {0, 0};
        int &max_pairs = max_pairs_cached[bf16 ? 1 : 0];
        if (max_pairs == 0) {
            cudaLaunchConfig_t one = {};
            one.gridDim = dim3(2);
            one.blockDim = dim3(kGemmThreads);
            one.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = 2;
            attr.val.clusterDim.y = 1;
            attr.val.clusterDim.z = 1;
            one.attrs = &attr;
            one.numAttrs = 1;
            int n = 0;
            e = cudaOccupancyMaxActiveClusters(&n, kernel, &one);
            if (e != cudaSuccess || n < 1) return record_cuda_error("cudaOccupancyMaxActiveClusters", e);
            max_pairs = n;
        }
        const long long n_tiles = static_cast<long long>(prm.tiles_m) * prm.tiles_n;
        const int pairs = static_cast<int>(n_tiles < max_pairs ? n_tiles : max_pairs);
        cfg.gridDim = dim3(2 * pairs);
        cfg.dynamicSmemBytes = smem;
        e = cudaLaunchKernelEx(&cfg, kernel, ma, mb, prm);
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e != cudaSuccess) return record_cuda_error("gemm_pair_kernel launch", e);
        return LT_OK;
    }

    prm.tiles_m = (M + kGemmBM - 1) / kGemmBM;
    prm.tiles_n = (N + kGemmBN - 1) / kGemmBN;
    {
        // about 48 MB of A rows per group (L2 holds 126 MB; the rest is for the W blocks in flight and C)
        const long long rows = static_cast<long long>(48.0e6 / (static_cast<double>(kGemmBM) * K * 2.0));
        prm.group_rows = static_cast<int>(rows < 1 ? 1 : (rows > prm.tiles_m ? prm.tiles_m : rows));
    }
    const size_t smem = sizeof(GemmSmem) + 1024;
    auto kernel = bf16 ? gemm_kernel<true> : gemm_kernel<false>;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return record_cuda_error("cudaFuncSetAttribute(gemm)", e);
    int sms = 148;
    {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    const long long n_tiles = static_cast<long long>(prm.tiles_m) * prm.tiles_n;
    const int grid = static_cast<int>(n_tiles < sms ? n_tiles : sms);
    cfg.gridDim = dim3(grid);
    cfg.dynamicSmemBytes = smem;
    e = cudaLaunchKernelEx(&cfg, kernel, ma, mb, prm);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return record_cuda_error("gemm_kernel launch", e);
    return LT_OK;
}

int lt_gemm_f16(const lt_half *A, const lt_half *W, lt_half *C, int M, int N, int K, void *workspace,
                size_t workspace_bytes, lt_stream_t stream) {
    return gemm_entry(A, W, C, M, N, K, workspace, workspace_bytes, stream, false);
}

int lt_gemm_bf16(const lt_bf16 *A, const lt_bf16 *W, lt_bf16 *C, int M, int N, int K, void *workspace,
                 size_t workspace_bytes, lt_stream_t stream) {
    return gemm_entry(A, W, C, M, N, K, workspace, workspace_bytes, stream, true);
}

}  // extern "C"
