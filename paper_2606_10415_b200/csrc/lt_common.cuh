// Shared device-side building blocks for the sm_100a attention kernels:
// mbarrier waits with an iteration/time limit, TMA tile loads, tcgen05 (UMMA) issue,
// tensor-memory allocation and access, and the operand descriptors.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace lt {

// ----------------------------------------------------------------------------- status block
// First 256 bytes of every workspace.  Word 0: 0 = ok, otherwise the code of the wait
// that gave up.  Word 3: work-item counter (backward).  The other words are not used.
constexpr int kStatusBytes = 256;
constexpr int kStatusWordTimeout = 0;
constexpr int kStatusWordItemCounter = 3;  // next unclaimed work item of the backward main kernel

// A wait gives up after this many clock cycles (about one second; the build of the give-up test
// shortens it).
#ifndef LT_WAIT_LIMIT_CYCLES
#define LT_WAIT_LIMIT_CYCLES 2000000000LL
#endif
constexpr long long kWaitLimitCycles = LT_WAIT_LIMIT_CYCLES;

// ----------------------------------------------------------------------------- small helpers
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "elect.sync _|p, 0xffffffff;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(pred));
    return pred != 0;
}

// ----------------------------------------------------------------------------- mbarrier
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait.  Returns false when the wait was abandoned: either this thread ran out
// of time (it then raises *abort_flag and records `code` in the status block) or another
// thread already raised the flag.  Callers leave their loops and go to the common
// teardown when they see false.
// (Every wait is expanded in place, a few dozen of them in a kernel whose loops together about fill the instruction cache:
// hence the low halves of the clock, and the hint that moves the waiting out of the way.)
static_assert(kWaitLimitCycles < 4000000000LL, "the limit is compared with a 32-bit difference");
__device__ __forceinline__ uint32_t clock_low() {
    uint32_t t;
    asm volatile("mov.u32 %0, %%clock;" : "=r"(t));
    return t;
}
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, volatile int *abort_flag,
                                          unsigned int *status, int code) {
    if (__builtin_expect(mbar_try_wait(bar, parity), 1)) return true;
    const uint32_t t0 = clock_low();
    uint32_t spins = 0;
    while (!mbar_try_wait(bar, parity)) {
        if ((++spins & 63u) == 0u) {
            if (*abort_flag) return false;
            if (clock_low() - t0 > static_cast<uint32_t>(kWaitLimitCycles)) {
                *abort_flag = 1;
                atomicCAS(status + kStatusWordTimeout, 0u, static_cast<unsigned int>(code));
                return false;
            }
        }
    }
    return true;
}

// The code of a wait on two barriers names both.  (Finding out which of them is late, when the time is over, costs the loops
// around the waits registers and instruction cache: the forward 4 % at D = 128, the backward on split key tiles 1 %.)
constexpr int both_codes(int code_a, int code_b) { return code_a * 1000 + code_b; }

// The same wait by a whole warp on one or two barriers, with a warp-uniform outcome.  The first test of both is voted on
// directly: a barrier that has completed costs no divergent branch, and two of them one round trip.  (In a loop that issues
// products, mbar_wait with its outcome voted afterwards took 170-240 cycles for a completed barrier, and there are several per
// tile.)
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar_a, uint32_t parity_a, uint64_t *bar_b, uint32_t parity_b,
                                               volatile int *abort_flag, unsigned int *status, int code) {
    auto done = [&]() {
        const bool a = mbar_try_wait(bar_a, parity_a), b = !bar_b || mbar_try_wait(bar_b, parity_b);
        return __all_sync(0xffffffffu, a && b) != 0;
    };
    if (__builtin_expect(done(), 1)) return true;
    const uint32_t t0 = clock_low();
    uint32_t spins = 0;
    while (!done()) {
        if ((++spins & 63u) == 0u) {
            const bool late = clock_low() - t0 > static_cast<uint32_t>(kWaitLimitCycles);
            if (late) {
                *abort_flag = 1;
                atomicCAS(status + kStatusWordTimeout, 0u, static_cast<unsigned int>(code));
            }
            if (__any_sync(0xffffffffu, late || *abort_flag)) return false;
        }
    }
    return true;
}

// ----------------------------------------------------------------------------- dependent launches
// A kernel launched with programmatic stream serialisation may start while the previous kernel of
// the stream is still running; it must not touch that kernel's results before grid_dependency_wait().
// The previous kernel lets it start early with grid_launch_dependents() (which takes effect once every
// CTA of that kernel has executed it or exited).  Without the launch attribute both are no-ops.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ----------------------------------------------------------------------------- register budget
// The registers of a CTA are split evenly between its warps at launch.  A warpgroup (four
// consecutive warps, the first a multiple of four) can hand registers back or take more; every
// warp of the group must execute the same instruction, and an increase waits until other groups
// have released enough.  N: registers per thread afterwards, a multiple of 8 in [24, 256].
// kFrom is the count the group holds before the call: handing registers back and taking more are two
// different instructions, and asking for "more" with a smaller count (or the reverse) is undefined.
template <int N, int kFrom>
__device__ __forceinline__ void warpgroup_regs_set() {
    static_assert(N % 8 == 0 && N >= 24 && N <= 256, "register count must be a multiple of 8 in [24, 256]");
    if constexpr (N < kFrom) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
    else if constexpr (N > kFrom) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// ----------------------------------------------------------------------------- fences
__device__ __forceinline__ void fence_proxy_async_smem() {
    // generic-proxy writes to shared memory become visible to the async proxy (TMA, UMMA)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before_sync() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after_sync() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// ----------------------------------------------------------------------------- TMA
__device__ __forceinline__ void tma_prefetch_desc(const CUtensorMap *map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// 2-D tile load global -> shared; completion is counted in bytes on `bar`.
// x = innermost (element) coordinate, must be a multiple of 8 for fp16; y = row.
__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}

// The same on a 4-D view [batch][head][row][element] (w = batch, z = head, y = row inside the head), and the request to
// bring such a tile into L2 ahead of the load that will use it.  Rows past the end of a head read as zeros, so a ragged last
// tile needs no special load, and layouts whose heads are interleaved inside a row are just other strides.
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, uint64_t *bar, int x, int y, int z,
                                            int w) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(w)
        : "memory");
}
__device__ __forceinline__ void tma_prefetch_l2_4d(const CUtensorMap *map, int x, int y, int z, int w) {
    asm volatile("cp.async.bulk.prefetch.tensor.4d.L2.global.tile [%0, {%1, %2, %3, %4}];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(z), "r"(w)
                 : "memory");
}

// The tile store shared -> global on such a view: x a multiple of 8 elements, no coordinate negative; rows past the end of a head are
// not written.  Completion is tracked in bulk groups.
__device__ __forceinline__ void tma_store_4d(const CUtensorMap *map, const void *src, int x, int y, int z, int w) {
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4, %5}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z), "r"(w)
                 : "memory");
}

// 1-D bulk copy global -> shared (both 16-byte aligned, size a multiple of 16 bytes);
// completion is counted in bytes on `bar`.
__device__ __forceinline__ void bulk_load_1d(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// 1-D bulk reduction shared -> global: adds `bytes` of fp32 from shared memory into global
// memory (both 16-byte aligned, size a multiple of 16).  Completion is tracked per thread
// in bulk groups: commit, then wait until at most N groups are still reading shared memory
// (wait_read) or until everything has been written (wait_all).
__device__ __forceinline__ void bulk_reduce_add_f32(float *dst_gmem, const void *src_smem, uint32_t bytes) {
    asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(
                     reinterpret_cast<uint64_t>(dst_gmem)),
                 "r"(smem_u32(src_smem)), "r"(bytes)
                 : "memory");
}
// 2-D tiled reduction shared -> global through a tensor map: adds the box at (x, y) (x = innermost element
// coordinate, x * element size a multiple of 16 bytes; both coordinates non-negative) of fp32 values from shared
// memory, laid out with the map's swizzle, into global memory.  Completion is tracked in bulk groups like above.
__device__ __forceinline__ void tma_reduce_add_2d(const CUtensorMap *map, const void *src_smem, int x, int y) {
    asm volatile("cp.reduce.async.bulk.tensor.2d.global.shared::cta.add.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(smem_u32(src_smem)), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_group_read() {
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_group_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void named_barrier_sync(int id, int threads) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Named barrier over `threads` threads that also ANDs a predicate across them.
__device__ __forceinline__ bool named_barrier_and(int id, int threads, bool pred) {
    uint32_t out;
    asm volatile(
        "{\n"
        ".reg .pred p, q;\n"
        "setp.ne.u32 q, %1, 0;\n"
        "bar.red.and.pred p, %2, %3, q;\n"
        "selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(out)
        : "r"(static_cast<uint32_t>(pred)), "r"(id), "r"(threads)
        : "memory");
    return out != 0;
}

// ----------------------------------------------------------------------------- tensor memory
__device__ __forceinline__ void tmem_alloc(uint32_t *dst_smem, uint32_t ncols) {  // one full warp
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {  // same warp that allocated
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// ----------------------------------------------------------------------------- CTA pairs (cta_group::2)
// Two CTAs of a cluster (ranks 2k and 2k+1) can run one tensor-core product together: each supplies 128
// rows of A and half of the rows of B from its own shared memory (same offsets in both) and receives its
// 128 rows of D in its own tensor memory.  The CTA with the even rank issues; barriers that both must see
// are signalled with a commit that arrives in both CTAs, and a CTA reaches its partner's barrier through
// the partner's address in the cluster's shared window.
__device__ __forceinline__ uint32_t cluster_cta_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_cta_count() {  // CTAs of this cluster
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(r));
    return r;
}
// 16 bytes of another CTA's shared memory (`cluster_addr` from cluster_map_shared)
__device__ __forceinline__ float4 ld_cluster_v4(uint32_t cluster_addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(cluster_addr) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync_all() {  // every thread of every CTA of the cluster
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// address of this CTA's shared-memory location `local` as seen in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_map_shared(uint32_t local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// tile load for a pair product: data lands in this CTA's shared memory, the byte count is credited to the
// barrier at cluster address `bar_cluster_addr` (the issuing CTA's)
__device__ __forceinline__ void tma_load_2d_pair(void *dst, const CUtensorMap *map, uint32_t bar_cluster_addr, int x,
                                                 int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(map)), "r"(bar_cluster_addr), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t *dst_smem, uint32_t ncols) {  // one full warp in each CTA
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// D[tmem of both CTAs] (+)= A * B over the pair: M = 256 (128 rows per CTA), B's N rows split between them
__device__ __forceinline__ void umma_ss_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// when all pair products issued so far have completed, arrive once on the barrier at this shared-memory
// offset in every CTA of `cta_mask` (bit r = rank r of the cluster)
__device__ __forceinline__ void umma_commit_pair(uint64_t *bar, uint16_t cta_mask) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"(cta_mask)
        : "memory");
}

// ----------------------------------------------------------------------------- UMMA descriptors
// Shared-memory operand descriptor for tiles stored as rows of 128 bytes (64 fp16) with
// the 128-byte swizzle a TMA tile load produces; every tile starts on a 1024-byte boundary.
//   contraction-contiguous ("K-major") operand : rows are M (or N); 8-row groups are
//       1024 bytes apart (stride field); the leading field is not used by the hardware.
//   row-index-contracted ("MN-major") operand   : rows are the contraction index; the 64
//       M/N elements of a row are contiguous; the next 64 M/N elements live in the next
//       tile (`mn_atom_stride` bytes away, leading field); 8-row groups are 1024 bytes apart.
// The address field (bits 0-13, units of 16 bytes) is linear in the address: a descriptor built for an
// offset inside the shared window plus (window base >> 4) is the descriptor of base + offset, as long as
// the window ends below 256 KB (the sum then never carries out of the field).
constexpr uint64_t kDescFixed = (1ull << 46) /* descriptor version for sm_100 */ | (2ull << 61) /* 128B swizzle */;

__host__ __device__ constexpr uint64_t desc_kmajor(uint32_t smem_addr) {
    return kDescFixed | (static_cast<uint64_t>(1) << 16) | (static_cast<uint64_t>(1024 >> 4) << 32) |
           static_cast<uint64_t>((smem_addr & 0x3FFFF) >> 4);
}
__host__ __device__ constexpr uint64_t desc_mnmajor(uint32_t smem_addr, uint32_t mn_atom_stride) {
    return kDescFixed | (static_cast<uint64_t>((mn_atom_stride >> 4) & 0x3FFF) << 16) |
           (static_cast<uint64_t>(1024 >> 4) << 32) | static_cast<uint64_t>((smem_addr & 0x3FFFF) >> 4);
}

// Unswizzled contraction-contiguous operand for one 16-element contraction step: rows of
// 16 bytes (8 fp16) grouped in blocks of 8 rows (128 contiguous bytes); `sbo` bytes between
// 8-row blocks, `lbo` bytes from the block holding elements 0-7 to the one holding 8-15.
__host__ __device__ constexpr uint64_t desc_kmajor_noswz(uint32_t smem_addr, uint32_t lbo, uint32_t sbo) {
    return (1ull << 46) | (static_cast<uint64_t>((lbo >> 4) & 0x3FFF) << 16) |
           (static_cast<uint64_t>((sbo >> 4) & 0x3FFF) << 32) | static_cast<uint64_t>((smem_addr & 0x3FFFF) >> 4);
}

// Two fp32 values rounded to a pair of 16-bit floats (fp16, or bf16 when kBf16), first value in
// the low half, and back.
template <bool kBf16>
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    if constexpr (kBf16) {
        __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t *>(&h);
    } else {
        __half2 h = __floats2half2_rn(lo, hi);
        return *reinterpret_cast<uint32_t *>(&h);
    }
}
template <bool kBf16>
__device__ __forceinline__ float2 unpack2(uint32_t w) {
    if constexpr (kBf16) return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w));
    else return __half22float2(*reinterpret_cast<const __half2 *>(&w));
}

// A per-row fp32 value x is added inside a tensor-core product by one extra contraction step whose
// other operand holds the multipliers kExtMult = (256, 1, 1/256, 0, ...).  The row stored for x holds
// 16-bit floats (hi, mid, lo, 0, ...) with 256*hi + mid + lo/256 = x: two terms for fp16 (about 22
// significant bits, lo = 0), three for bf16 (24 bits).  Returned as the 16-byte row.
template <bool kBf16>
__device__ __forceinline__ uint4 split_ext(float x) {
    if constexpr (kBf16) {
        const __nv_bfloat16 hi = __float2bfloat16_rn(x * (1.f / 256.f));
        const float r1 = x - 256.f * __bfloat162float(hi);
        const __nv_bfloat16 mid = __float2bfloat16_rn(r1);
        const __nv_bfloat16 lo = __float2bfloat16_rn((r1 - __bfloat162float(mid)) * 256.f);
        return make_uint4(static_cast<uint32_t>(__bfloat16_as_ushort(hi)) |
                              (static_cast<uint32_t>(__bfloat16_as_ushort(mid)) << 16),
                          static_cast<uint32_t>(__bfloat16_as_ushort(lo)), 0u, 0u);
    } else {
        const __half hi = __float2half_rn(x * (1.f / 256.f));
        const __half mid = __float2half_rn(x - 256.f * __half2float(hi));
        return make_uint4(static_cast<uint32_t>(__half_as_ushort(hi)) | (static_cast<uint32_t>(__half_as_ushort(mid)) << 16),
                          0u, 0u, 0u);
    }
}
// the first two words of the multiplier row (256, 1 | 1/256, 0)
template <bool kBf16>
__device__ __forceinline__ uint2 ext_multipliers() {
    return make_uint2(pack2<kBf16>(256.f, 1.f), pack2<kBf16>(1.f / 256.f, 0.f));
}

// Instruction descriptor, kind::f16: fp16 (or bf16) A and B, fp32 accumulator, dense.
constexpr uint32_t make_idesc(int M, int N, bool a_mn_major, bool b_mn_major, bool bf16 = false) {
    return (1u << 4)                                   // accumulator format: f32
           | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10)   // A, B format: f16 = 0, bf16 = 1
           | (static_cast<uint32_t>(a_mn_major) << 15) | (static_cast<uint32_t>(b_mn_major) << 16) |
           (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}

// D[tmem] (+)= A[smem] * B[smem]; issued by one thread.
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]; A holds M lanes x K fp16 packed two per 32-bit column.
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
    asm volatile(
        "{\n"
        ".reg .pred p;\n"
        "setp.ne.b32 p, %4, 0;\n"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
        "}\n" ::"r"(d_tmem),
        "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive on `bar` once every UMMA issued so far by this thread has completed.
__device__ __forceinline__ void umma_commit(uint64_t *bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// ----------------------------------------------------------------------------- tensor memory access
// 32 lanes x 32-bit, N consecutive columns: thread t of warp w reads lane 32*(w%4)+t.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
// 16 lanes x 256 bits per repetition, 8 repetitions along the columns (64 fp32 columns):
// thread t of the warp receives, for repetition k, registers r[4k..4k+3] =
//   { (lane t/4, col 8k + 2(t%4)), (t/4, 8k + 2(t%4) + 1), (t/4 + 8, same two columns) }
// where "lane" counts from the lane given in the address.  Four neighbouring threads
// therefore hold 32 contiguous bytes of one row.
__device__ __forceinline__ void tmem_ld_16x256b_x8(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
// The store with the same arrangement (the registers of tmem_ld_16x256b_x8 written back).
__device__ __forceinline__ void tmem_st_16x256b_x8(uint32_t taddr, const uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]),
        "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]),
        "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
        : "memory");
}
// 16 lanes x 128 bits per repetition, 8 repetitions along the columns (32 columns): for repetition k
// thread t supplies r[2k] = (lane t/4, col 4k + t%4) and r[2k+1] = (lane t/4 + 8, same column).  This is
// where the 16-bit pairs packed from the registers of tmem_ld_16x256b_x8 belong.
__device__ __forceinline__ void tmem_st_16x128b_x8(uint32_t taddr, const uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.st.sync.aligned.16x128b.x8.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
        : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ----------------------------------------------------------------------------- numerics helpers
// two fp32 operations in one instruction, each rounded like the single one
__device__ __forceinline__ uint64_t f32x2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float2 f32x2_parts(uint64_t v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ uint64_t f32x2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t f32x2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f32x2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ float fast_exp2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ void red_add_v4(float *addr, float a, float b, float c, float d) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d)
                 : "memory");
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) { return pack2<false>(lo, hi); }
// product of two packed fp16 pairs, element by element
__device__ __forceinline__ uint32_t hmul2_bits(uint32_t a, uint32_t b) {
    uint32_t d;
    asm("mul.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
    return d;
}
// 16-byte read-only global load that does not allocate in L1 (data read once)
__device__ __forceinline__ uint4 ld_nc_v4(const uint4 *ptr) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(ptr));
    return v;
}
// ask for `bytes` (a multiple of 16) of global memory at a 16-byte aligned address to be brought into L2
__device__ __forceinline__ void bulk_prefetch_l2(const void *gptr, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(gptr), "r"(bytes) : "memory");
}

// Byte offset of element (row, col) inside one swizzled tile of 64 fp16 columns
// (rows of 128 bytes, 16-byte chunks XORed with row % 8), the layout TMA's 128B swizzle
// writes and the UMMA descriptors above read.
__device__ __forceinline__ uint32_t swz128_offset(uint32_t row, uint32_t col /* 0..63 */) {
    return row * 128u + ((((col >> 3) ^ (row & 7u)) << 4) | ((col & 7u) << 1));
}

}  // namespace lt
