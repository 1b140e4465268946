// tc_ptx.cuh -- inline-PTX wrappers for the tcgen05 kernels (sm_103a): mbarriers with
// bounded waits, TMA, tcgen05 MMA / commit / TMEM loads, CTA-pair (cluster) forms.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "common.cuh"

#ifndef AQD_WAIT_HINT_NS
#define AQD_WAIT_HINT_NS 0
#endif

namespace aqd {
namespace tc {

constexpr uint64_t kTimeoutNs = 1000000000ull;  // 1 s per wait

// ---------------------------------------------------------------- PTX wrappers

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  uint64_t st;
  asm volatile("mbarrier.arrive.shared::cta.b64 %0, [%1];" : "=l"(st) : "r"(bar) : "memory");
  (void)st;
}
// An arrival that hands TMEM over (after tcgen05.wait::ld and tcgen05.fence::before_thread_sync):
// no memory of this thread is published by it, so it need not wait for its earlier stores, as
// the default release does.
__device__ __forceinline__ void mbar_arrive_relaxed(uint32_t bar) {
  uint64_t st;
  asm volatile("mbarrier.arrive.relaxed.cta.shared::cta.b64 %0, [%1];" : "=l"(st) : "r"(bar) : "memory");
  (void)st;
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  uint64_t st;
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 %0, [%1], %2;"
               : "=l"(st) : "r"(bar), "r"(bytes) : "memory");
  (void)st;
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// try_wait that lets the hardware suspend the thread (up to `ns`) until the phase
// completes, instead of returning at once: waiting warps then take no issue slots
__device__ __forceinline__ bool mbar_try_sleep(uint32_t bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity), "r"(ns) : "memory");
  return ok != 0;
}

// Non-blocking test of a phase. The MMA-issuing thread polls with this: measured on
// sm_103a, a try_wait in a thread with tcgen05.mma in flight costs ~165 cycles even when
// the phase has completed, a test_wait ~13.
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
static __device__ __noinline__ bool mbar_poll_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  // a few cheap tests first (short waits), then the suspending try_wait so a long wait
  // does not take issue slots from the other warps of this SM sub-partition
  for (int i = 0; i < 8; ++i)
    if (mbar_test(bar, parity)) return true;
  const uint64_t deadline = globaltimer() + kTimeoutNs;
  for (uint32_t spin = 1;; ++spin) {
    if (mbar_try(bar, parity)) return true;
    if ((spin & 15) == 0) {
      if (*abort_flag) return false;
      if (globaltimer() > deadline) return false;
    }
  }
}
__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_test(bar, parity) || mbar_poll_slow(bar, parity, abort_flag);
}

// Bounded wait: false if the deadline (kLimitNs after the call) passed or another role
// aborted. The kernels use the 1 s limit; the wait self-test instantiates a short one.
template <uint64_t kLimitNs = kTimeoutNs>
__device__ __forceinline__ bool mbar_wait_loop(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  const uint64_t deadline = globaltimer() + kLimitNs;
  for (uint32_t spin = 1;; ++spin) {
    if (AQD_WAIT_HINT_NS > 0 ? mbar_try_sleep(bar, parity, AQD_WAIT_HINT_NS) : mbar_try(bar, parity)) return true;
    if ((spin & 63) == 0) {
      if (*abort_flag) return false;
      if (globaltimer() > deadline) return false;
    }
  }
}
template <uint64_t kLimitNs = kTimeoutNs>
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait_loop<kLimitNs>(bar, parity, abort_flag);
}

template <uint64_t kLimitNs = kTimeoutNs>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_try(bar, parity) || mbar_wait_slow<kLimitNs>(bar, parity, abort_flag);
}
// The same without a call, where the caller has no registers to keep across one.
__device__ __forceinline__ bool mbar_wait_inline(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_try(bar, parity) || mbar_wait_loop<kTimeoutNs>(bar, parity, abort_flag);
}

__device__ __forceinline__ void fail(volatile int* abort_flag, uint32_t* status) {
  *abort_flag = 1;
  atomicCAS(status, 0u, (uint32_t)kStatusTimeout);
}

// One lane of a converged warp, by elect.sync: the compiler then knows that a single thread runs
// the branch and issues its tensor-core and TMA instructions directly; under "lane == 0" it
// wraps each in a loop over the active lanes (measured: 4 MMAs and their commit 650 cycles
// against under 512, a TMA box about 650 cycles of its issuing thread).
__device__ __forceinline__ bool elect_one() {
  uint32_t one;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "elect.sync _|p, 0xffffffff;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(one));
  return one != 0;
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// orders this thread's generic-proxy view of global memory with its async-proxy (TMA)
// accesses: after a store that TMA reads elsewhere, and after the acquire that makes other
// threads' stores visible, before this thread's TMA loads of them
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
__device__ __forceinline__ uint32_t ld_relaxed_gpu(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// with a preceding relaxed load that observed a release, forms the acquire side of the pattern
__device__ __forceinline__ void fence_acq_rel_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
__device__ __forceinline__ void red_release_gpu_add(uint32_t* p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Bounded wait until c[i] >= target for every i in [0, n): the counters are read together
// (relaxed loads, no ordering among them) until all are reached, then one fence.acq_rel
// makes the writes released before them visible to this thread. False if the deadline passed
// or another role aborted.
static __device__ __noinline__ bool counters_wait(const uint32_t* c, int n, uint32_t target, volatile int* abort_flag) {
  uint64_t deadline = 0;
  for (uint32_t spin = 0;; ++spin) {
    bool all = true;
    for (int i = 0; i < n; ++i) all &= ld_relaxed_gpu(c + i) >= target;
    if (all) break;
    if (spin == 0) deadline = globaltimer() + kTimeoutNs;
    __nanosleep(64);
    if ((spin & 15) == 15) {
      if (*abort_flag) return false;
      if (globaltimer() > deadline) return false;
    }
  }
  fence_acq_rel_gpu();
  return true;
}
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Whether a set of epilogue warps does the work of a loop's tile lt: sets of warps take tiles in turn
// (sets is a power of two), and all of them meet at the named barriers of some tiles, which have no limit.
// So a set whose wait ran out (ok is false) stays in the loop to its end and meets the others at those
// barriers, without waiting or storing; if it left, a set that had run ahead would wait there for ever.
__device__ __forceinline__ bool takes_tile(bool ok, uint32_t lt, int sets, int set) {
  return ok && (int)(lt & (uint32_t)(sets - 1)) == set;
}
__device__ __forceinline__ void named_bar(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
// named barrier that also returns the AND of `pred` over the participating threads
__device__ __forceinline__ int named_bar_and(int id, int n, int pred) {
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %3, 0;\n\t"
      "bar.red.and.pred q, %1, %2, p;\n\t"
      "selp.b32 %0, 1, 0, q;\n\t}"
      : "=r"(r) : "r"(id), "r"(n), "r"(pred) : "memory");
  return r;
}
__device__ __forceinline__ int32_t add_sat(int32_t a, int32_t b) {
  int32_t r;
  asm("add.sat.s32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

template <int kBytes>
__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, bool ok) {
  const uint32_t n = ok ? kBytes : 0;  // 0 source bytes = zero fill
  if constexpr (kBytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
  else if constexpr (kBytes == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar) : "memory");
}

// Programmatic dependent launch: wait for the previous kernel in the stream to finish (and
// its writes to be visible); allow the next kernel's CTAs to be scheduled.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// SW128 K-major shared-memory matrix descriptor (tcgen05 format): start address >> 4,
// leading byte offset 16 (unused for swizzled K-major), stride byte offset 1024 between
// 8-row groups, descriptor version 1, swizzle mode 2 = 128B.
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// SW64 K-major descriptor (operand rows of 64 bytes): stride byte offset 512 between
// 8-row groups, swizzle mode 4 = 64B.
__device__ __forceinline__ uint64_t sdesc_sw64(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;
  d |= (uint64_t)(512 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)4 << 61;
  return d;
}
// descriptor for K chunks of kBK bytes (128: SW128, 64: SW64)
template <int kBK>
__device__ __forceinline__ uint64_t sdesc_k(uint32_t saddr) {
  static_assert(kBK == 128 || kBK == 64, "K chunks of 64 or 128 bytes");
  if constexpr (kBK == 128) return sdesc_sw128(saddr);
  else return sdesc_sw64(saddr);
}

// Instruction descriptor, kind::f8f6f4 (A=B=E4M3) or kind::f16 (A=B=F16, the same type
// code 0): D=F32, both K-major, N>>3, M>>4. M=256 exists only for cta_group::2.
constexpr int kMmaM = 128;
__device__ __forceinline__ uint32_t idesc_e4m3(int n, int m = kMmaM) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

// Instruction descriptor, kind::mxf4nvf4 (block-scaled): A = B = E2M1 (format code 1),
// scale factors UE8M0 (bit 23), both K-major, N>>3, M>>4, scale-factor ids 0, dense K = 64.
__device__ __forceinline__ uint32_t idesc_fp4(int n, int m = kMmaM) {
  return (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | (1u << 23) | ((uint32_t)(m >> 4) << 24);
}
// D (+)= A B with E2M1 operands (K = 64 per instruction, 32 bytes of each operand row) and
// one UE8M0 scale per 32 K elements, read from TMEM at sfa / sfb (scale_vec::2X)
__device__ __forceinline__ void mma_fp4(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t sfa,
                                        uint32_t sfb, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::mxf4nvf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%4], [%5], p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(sfa), "r"(sfb), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_fp4_pair(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t sfa,
                                             uint32_t sfb, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %6, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::mxf4nvf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%4], [%5], p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(sfa), "r"(sfb), "r"(acc) : "memory");
}
// 16 TMEM columns of this warp's lanes, every word v
__device__ __forceinline__ void tmem_st16_fill(uint32_t taddr, uint32_t v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};"
      ::"r"(taddr), "r"(v) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void mma_e4m3(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
// F16 operands (K = 16 per instruction, 32 bytes of each operand row); the instruction descriptor is
// idesc_e4m3's (F16 has the same type code)
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_f16_pair(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(bar) : "memory");
}

// ---- 2-SM (CTA pair) forms. In a cluster of two CTAs, the even CTA issues
// tcgen05.mma.cta_group::2 with M = 256: each CTA holds its 128 rows of A and half of the
// N rows of B in shared memory at the same offsets, and receives its 128 rows x N columns
// of D in its own TMEM.
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cluster address of shared-memory offset `saddr` in CTA `rank` of this cluster
__device__ __forceinline__ uint32_t mapa_shared(uint32_t saddr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
  return r;
}
// (relaxed: a TMEM hand-over, as mbar_arrive_relaxed)
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
__device__ __forceinline__ void mma_e4m3_pair(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
// arrive on the barrier at this shared-memory offset in both CTAs of the pair, once the
// MMAs issued so far have completed
__device__ __forceinline__ void mma_commit_pair_both(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
      ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(bar) : "memory");
}
// TMA load into this CTA's shared memory that signals a barrier in either CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y,
                                                 uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar_cluster) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// Makes every later use of r depend on this point: right after tmem_wait_ld, so that no read of a register
// that a TMEM load writes moves above the wait.
__device__ __forceinline__ void reg_fence8(uint32_t (&r)[8]) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]));
}
__device__ __forceinline__ void reg_fence16(uint32_t (&r)[16]) {
  asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
               "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]),
               "+r"(r[14]), "+r"(r[15]));
}

}  // namespace tc
}  // namespace aqd
