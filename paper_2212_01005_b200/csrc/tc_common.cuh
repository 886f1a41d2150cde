// sm_100a building blocks for the fused kernels: mbarriers with bounded waits,
// TMA tile loads, tensor-memory allocation, tcgen05 MMA issue / commit / loads
// and the shared-memory matrix descriptors they consume.
//
// Hang safety: every wait is bounded by a wall-clock deadline read from
// %globaltimer. When a wait gives up it records a code in the handle's status
// word and raises a CTA-wide abort flag that makes all later waits return at
// once; the kernel then runs to its end (results undefined), frees its tensor
// memory and exits, so the context stays usable.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace ago {
namespace tc {

constexpr unsigned long long kWaitBudgetNs = 1000000000ull;  // 1 s per wait

// The handle's device status block (four 32-bit words; kernels get a pointer to word 0, or null):
//   [0] code of the first wait site that gave up (0: none)       -- written by kernels, read and cleared by the host
//   [1] wait budget in microseconds (0: the default above)        -- written by the host only
//   [2] test hook: the site code whose producer skips ONE signal  -- written by the host only (0: none)
// Words 1 and 2 exist so that a test can make a bounded wait run out on a tiny problem without faulting, trapping
// or hanging anything: the skipped signal is an mbarrier arrival, the waiter gives up after the budget, the kernel
// runs to its end and frees its tensor memory.
constexpr int kStatusWords = 4;
__device__ __forceinline__ bool skip_signal_for_test(const unsigned int* status, uint32_t code) {
  return status != nullptr && __ldg(status + 2) == code;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// ---- mbarrier -------------------------------------------------------------------

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// The same with a suspend-time hint: the hardware parks the thread until the phase completes or
// about `hint_ns` have passed, so a waiting warp takes no issue slots from the warps that have work.
__device__ __forceinline__ bool mbar_try_wait_parked(uint64_t* bar, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}

// Bounded wait. `abort_flag` is a CTA-shared word, `status` the handle's device
// status word, `code` identifies the wait site. Returns false when it gave up.
static __device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag,
                                            unsigned int* status, uint32_t code) {
  const unsigned long long t0 = globaltimer_ns();
  const unsigned int budget_us = status ? *(volatile const unsigned int*)(status + 1) : 0u;
  const unsigned long long budget = budget_us ? (unsigned long long)budget_us * 1000ull : kWaitBudgetNs;
  while (true) {
    for (int i = 0; i < 16; ++i)
      if (mbar_try_wait_parked(bar, parity, 20000u)) return true;
    if (*abort_flag) return false;
    if (globaltimer_ns() - t0 > budget) {
      *abort_flag = 1u;
      if (status) atomicCAS(status, 0u, code);
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag,
                                          unsigned int* status, uint32_t code) {
  if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow(bar, parity, abort_flag, status, code);
}

// The same bounded wait for the single-thread roles (TMA producer, MMA issuer) of a pipelined main loop: it polls
// with the plain try_wait (which itself blocks for a short, implementation-defined time) instead of parking with a
// long suspend hint, so the role reacts to the completion at once; one polling thread costs few issue slots.
static __device__ __noinline__ bool mbar_wait_poll_slow(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag,
                                                        unsigned int* status, uint32_t code) {
  const unsigned long long t0 = globaltimer_ns();
  const unsigned int budget_us = status ? *(volatile const unsigned int*)(status + 1) : 0u;
  const unsigned long long budget = budget_us ? (unsigned long long)budget_us * 1000ull : kWaitBudgetNs;
  while (true) {
    for (int i = 0; i < 256; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (globaltimer_ns() - t0 > budget) {
      *abort_flag = 1u;
      if (status) atomicCAS(status, 0u, code);
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait_poll(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag,
                                               unsigned int* status, uint32_t code) {
#pragma unroll 1
  for (int i = 0; i < 64; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return mbar_wait_poll_slow(bar, parity, abort_flag, status, code);
}

// Barrier among a subset of the CTA's warps (id 1..15; `threads` a multiple of 32).
__device__ __forceinline__ void named_barrier_sync(uint32_t id, uint32_t threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// ---- programmatic dependent launch -----------------------------------------------------------------
// The fused kernels are launched with programmatic stream serialization: a grid may be scheduled while the
// previous grid of the stream is still running, so that its launch latency and its set-up (barriers, tensor
// memory, index arithmetic) overlap that grid's tail. grid_dependency_wait() returns once the previous grid has
// completed and its memory is visible -- every thread calls it before its first access to device memory.
// (Without the launch attribute both are no-ops.)
// One thread's grid_launch_dependents() counts for its CTA. A CTA that takes tensor memory calls it only once it has its columns:
// from the warp that allocated them, or behind a __syncthreads() after the allocation. The allocation blocks until columns are
// free, without a limit; a CTA of the next grid that shares the SM could otherwise take them first and then wait for this grid.
// (The allocating warp alone, predicated: up to 1 % of a small kernel's time, the first of sixteen warps is earlier by that. Behind a
// barrier of its own 3 % and behind the staging's 5 %, the inverted-residual block of 14 x 14 pixels.)
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_dependents_if(bool yes) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %0, 0;\n\t@q griddepcontrol.launch_dependents;\n\t}" ::"r"((uint32_t)yes) : "memory");
}

// ---- proxies and fences ---------------------------------------------------------------

// Make generic-proxy shared-memory writes visible to the async proxy (TMA, tcgen05.mma).
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tcgen05_fence_before_sync() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tcgen05_fence_after_sync() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// x / d for x, d < 65536 with recip = 2^32 / d + 1 computed on the host (fast_div_recip); d == 1 has no 32-bit
// reciprocal and is passed through.
__device__ __forceinline__ uint32_t fast_div(uint32_t x, uint32_t d, uint32_t recip) { return d == 1u ? x : __umulhi(x, recip); }
inline uint32_t fast_div_recip(int d) { return (uint32_t)((1ull << 32) / (uint64_t)d + 1ull); }

// ---- thread-block clusters: distributed shared memory, remote barriers ---------------------------

// Shared-memory address of `local_saddr` (a shared::cta address of this CTA's layout) in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_map(uint32_t local_saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_saddr), "r"(rank));
  return r;
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The two halves of a cluster barrier (all threads) that publishes nothing: where barriers are made visible by fence_mbar_init and
// data by the copies' own completion, the arrival can be relaxed. A release at cluster scope takes 1200 cycles, more behind
// outstanding stores.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_meet() { cluster_arrive(); cluster_wait(); }
// One arrival on the mbarrier at cluster address `remote_bar` that also announces `bytes` of pending copy traffic.
__device__ __forceinline__ void mbar_remote_arrive_expect_tx(uint32_t remote_bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.release.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(remote_bar), "r"(bytes) : "memory");
}
// Bulk copy of `bytes` (a multiple of 16; both addresses 16-byte aligned) from this CTA's shared memory to the
// cluster address `remote_dst`; completion is counted in bytes on the mbarrier at cluster address `remote_bar`.
__device__ __forceinline__ void bulk_copy_to_cluster(uint32_t remote_dst, uint32_t local_src, uint32_t bytes, uint32_t remote_bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(remote_dst), "r"(local_src), "r"(bytes), "r"(remote_bar) : "memory");
}

// ---- per-thread asynchronous copies (global -> shared, 16 bytes, zero-filled beyond src_bytes) ----------

__device__ __forceinline__ void cp_async_16(uint32_t dst_saddr, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_saddr), "l"(src), "r"(src_bytes) : "memory");
}
// ... through L1: for what the CTAs of an SM all read (whole 128-byte lines are requested, once per SM)
__device__ __forceinline__ void cp_async_16_l1(uint32_t dst_saddr, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst_saddr), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// all of this thread's commit groups but the most recent one are complete
__device__ __forceinline__ void cp_async_wait_but_one() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// ---- TMA (cp.async.bulk.tensor), every load into the issuing CTA only ---------------------

__device__ __forceinline__ void tma_prefetch_desc(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}
__device__ __forceinline__ void tma_load_2d(void* dst, const void* tmap, uint64_t* bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(void* dst, const void* tmap, uint64_t* bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
// The same from a converged warp, on its elected lane (see "MMA issue from a converged warp").
__device__ __forceinline__ void tma_load_2d_elected(uint32_t dst_saddr, const void* tmap, uint32_t bar_saddr, int c0, int c1, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n\t}"
      ::"r"(dst_saddr), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar_saddr), "r"(c0), "r"(c1), "r"(elected)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_elected(uint32_t dst_saddr, const void* tmap, uint32_t bar_saddr, int c0, int c1, int c2, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %6, 0;\n\t"
      "@q cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];\n\t}"
      ::"r"(dst_saddr), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar_saddr), "r"(c0), "r"(c1), "r"(c2), "r"(elected)
      : "memory");
}
// Store of a shared-memory tile into a 3-D tensor (the part of the box outside the tensor is clipped). The copy belongs to
// the issuing thread's bulk group: that thread commits the group and waits for it (for its reads of shared memory before the
// tile is overwritten, for all of it before the CTA exits).
__device__ __forceinline__ void tma_store_3d(const void* tmap, const void* src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// all of this thread's bulk groups but the most recent one have read their shared-memory source
__device__ __forceinline__ void bulk_wait_group_read_but_one() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_group_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_group_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void tma_load_4d(void* dst, const void* tmap, uint64_t* bar, int c0, int c1, int c2,
                                            int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(smem_u32(dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2),
      "r"(c3)
      : "memory");
}

// ---- tensor memory ---------------------------------------------------------------------------

// One full warp allocates `ncols` (power of two, 32..512) columns; the base
// address lands in *dst_smem.
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// ---- descriptors --------------------------------------------------------------------------------

enum SwizzleMode : uint32_t { SW_NONE = 0, SW_128B = 2, SW_64B = 4, SW_32B = 6 };

// Shared-memory matrix descriptor. Addresses and offsets are encoded in 16-byte
// units. For K-major swizzled operands LBO is unused (one swizzle row holds the
// whole K extent of a block) and SBO is the distance between 8-row groups.
__device__ __forceinline__ uint64_t make_smem_desc(uint32_t saddr, uint32_t lbo_bytes, uint32_t sbo_bytes,
                                                   uint32_t swizzle) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version of this architecture
  d |= (uint64_t)swizzle << 61;
  return d;
}

// Instruction descriptor, kind::f16: bf16 x bf16 -> fp32, dense, no negation.
// a_mn_major / b_mn_major: 0 = K-major operand, 1 = MN-major operand.
__host__ __device__ constexpr uint32_t make_idesc_bf16(uint32_t M, uint32_t N, uint32_t a_mn_major = 0,
                                                       uint32_t b_mn_major = 0) {
  return (1u << 4)                 // accumulator format: fp32
         | (1u << 7)               // A format: bf16
         | (1u << 10)              // B format: bf16
         | (a_mn_major << 15) | (b_mn_major << 16) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// ---- MMA issue from a converged warp --------------------------------------------------------------
// Writing the issue as `if (lane == 0) { ... tcgen05.mma ... }` makes the operands lane-dependent values behind a divergent
// branch; next to warps with dense arithmetic such an issuing thread got one MMA out every 170-550 cycles (measured, 28
// FMA-bound neighbours). The same loop run by the whole warp, converged, with the MMA predicated on a lane elected once
// and the descriptors ready as 64-bit values, issues one every 50-60 cycles. All lanes execute these helpers; `elected`
// is elect_one() of the calling warp, taken while it is converged (the same lane then issues the MMAs and the commit).
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.u32 %0, 1, 0, q;\n\t}" : "=r"(r));
  return r;
}
template <bool ACC>
__device__ __forceinline__ void umma_bf16_elected(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %4, 0;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(elected), "n"(ACC ? 1 : 0)
      : "memory");
}
// accumulate flag known only at run time
__device__ __forceinline__ void umma_bf16_elected_acc(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t elected,
                                                      uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %4, 0;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(elected), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void umma_commit_cluster_elected(uint32_t bar_cluster_addr, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(bar_cluster_addr), "r"(elected)
      : "memory");
}
__device__ __forceinline__ void umma_commit_elected(uint64_t* bar, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(smem_u32(bar)), "r"(elected)
      : "memory");
}

// ---- paired CTAs (cta_group::2): one MMA spans the two CTAs of a cluster of two -------------------------------
// The CTA with the even cluster rank (the leader) issues every MMA; an M = 256 product takes rows 0..127 of A and of
// the accumulator from the leader and rows 128..255 from its peer, and each CTA holds one half (N / 2 columns) of B
// at the same shared-memory offsets. Each CTA fetches its own operands with its own TMA loads (no multicast); the
// loads of both CTAs complete on the leader's barrier.

// TMA load whose completion is counted on a barrier that may live in the peer CTA (`bar_cluster_addr` is a
// shared::cluster address, see cluster_map); the data lands in the issuing CTA. From a converged warp, on its elected lane (see
// "MMA issue from a converged warp"), and a box of a 3-D tensor.
__device__ __forceinline__ void tma_load_2d_pair_elected(uint32_t dst_saddr, const void* tmap, uint32_t bar_cluster_addr, int c0, int c1, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n\t}"
      ::"r"(dst_saddr), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar_cluster_addr), "r"(c0), "r"(c1), "r"(elected)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair_elected(uint32_t dst_saddr, const void* tmap, uint32_t bar_cluster_addr, int c0, int c1, int c2,
                                                         uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %6, 0;\n\t"
      "@q cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];\n\t}"
      ::"r"(dst_saddr), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(bar_cluster_addr), "r"(c0), "r"(c1), "r"(c2), "r"(elected)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx_elected(uint32_t bar_saddr, uint32_t bytes, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %2, 0;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}"
      ::"r"(bar_saddr), "r"(bytes), "r"(elected) : "memory");
}
// Plain arrival on a barrier given by its cluster address (this CTA's or the peer's).
__device__ __forceinline__ void mbar_remote_arrive(uint32_t bar_cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster_addr) : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// For a converged warp of the leader CTA: every lane executes, the lane chosen once by elect_one() issues.
// D[tmem of both CTAs] (+)= A * B across the pair.
__device__ __forceinline__ void umma_bf16_pair_elected(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t elected,
                                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 q, %4, 0;\n\t"
      "setp.ne.b32 p, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(elected), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at that cluster address once all MMAs issued so far by this thread have completed in both CTAs.
__device__ __forceinline__ void umma_commit_pair_elected(uint32_t bar_cluster_addr, uint32_t elected) {
  asm volatile(
      "{\n\t.reg .pred q;\n\t"
      "setp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
      ::"r"(bar_cluster_addr), "r"(elected) : "memory");
}
// TMA store of a 2-D tile (clipped at the tensor's edges); bulk-group completion as tma_store_3d.
__device__ __forceinline__ void tma_store_2d(const void* tmap, const void* src, int c0, int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(src)), "r"(c0), "r"(c1)
               : "memory");
}

// ---- tensor memory -> registers ------------------------------------------------------------------
// Warp w may touch TMEM lanes 32*(w%4) .. 32*(w%4)+31; thread t of the warp
// reads lane 32*(w%4)+t, N consecutive 32-bit columns.

__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_x32(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// The same wait, naming the 16 registers of an outstanding load as in/out operands: no use of them can be moved above
// the wait, and a later load into the same registers cannot be moved above their last use.
__device__ __forceinline__ void tmem_ld_wait_on(uint32_t (&v)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]),
                 "+r"(v[9]), "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
               :
               : "memory");
}

// ---- small helpers ---------------------------------------------------------------------------------

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// Eight words to 32 bytes of device memory (32-byte aligned): one sector.
__device__ __forceinline__ void store_global_32(void* dst, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" :: "l"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]),
               "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]) : "memory");
}
// 32 bytes of read-only device memory (32-byte aligned): one sector.
__device__ __forceinline__ void load_global_32(const void* src, uint32_t (&w)[8]) {
  asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]) : "l"(src));
}
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// 16-byte shared-memory accesses by 32-bit shared address (immediate byte offset for the load).
template <int OFF = 0>
__device__ __forceinline__ float4 lds128f(uint32_t saddr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4+%5];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(saddr), "n"(OFF));
  return v;
}
__device__ __forceinline__ void sts128(uint32_t saddr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(saddr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Byte offset of 16-byte chunk `chunk` of row `row` in a K-major tile whose rows
// are `row_bytes` (32, 64 or 128) long and swizzled with the matching mode: the
// chunk index is XORed with address bits [7, 7+log2(row_bytes/16)).
__device__ __forceinline__ uint32_t swz_offset(uint32_t row, uint32_t chunk, uint32_t row_bytes) {
  const uint32_t lin = row * row_bytes + chunk * 16u;
  const uint32_t mask = (row_bytes >> 4) - 1u;
  return lin ^ (((lin >> 7) & mask) << 4);
}

}  // namespace tc
}  // namespace ago
