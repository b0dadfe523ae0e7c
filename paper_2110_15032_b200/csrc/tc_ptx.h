// What the tensor-core kernels share: mbarriers with bounded waits, cluster addresses, tiled copies, tensor
// memory and matrix descriptors.  Device symbols are one copy per translation unit.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include "sbp_internal.h"

namespace sbp {

constexpr unsigned long long kWaitLimitNs = 2000000000ull;

namespace {
__device__ int g_tc_timeout_flag = 0;      // set by a wait that ran out

inline sbp_status read_and_clear_timeout_flag(bool* timed_out) {
  int flag = 0, zero = 0;
  SBP_CUDA_TRY(cudaMemcpyFromSymbol(&flag, g_tc_timeout_flag, sizeof(int)));
  if (flag) SBP_CUDA_TRY(cudaMemcpyToSymbol(g_tc_timeout_flag, &zero, sizeof(int)));
  *timed_out = flag != 0;
  return SBP_OK;
}
}  // namespace

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

// One try_wait with a suspend-time hint: the thread sleeps in hardware until the phase completes
// or the hint (in ns) runs out, instead of spinning and taking issue slots and power from the
// tensor pipe (measured: +8 % MatMul throughput against a bare polling loop).
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 0x10000;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}

// Bounded wait.  Returns false (and raises the abort flag) when the limit expires.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int* abort_flag) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = now_ns();
  for (;;) {
    if (mbar_try(bar, parity)) return true;
    if (*abort_flag) return false;
    if (now_ns() - t0 > kWaitLimitNs) {
      *abort_flag = 1;
      atomicExch(&g_tc_timeout_flag, 1);
      return false;
    }
  }
}

// The same wait made by a whole converged warp; the answer is the same in all of its lanes.
__device__ __forceinline__ bool mbar_wait_warp(unsigned bar, unsigned parity, volatile int* abort_flag) {
  if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag)) != 0;
}

// One lane of a converged warp, the same one every time.
__device__ __forceinline__ bool elect_one() {
  unsigned p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Address of the same shared-memory object in CTA `rank` of this cluster.
__device__ __forceinline__ unsigned map_to_cta(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// Arrive on an mbarrier that may live in the partner CTA (cluster-space address).  The arrive
// carries the default (CTA-scope) release: what it hands over is tensor memory whose reads have
// completed (tcgen05.wait::ld, then tcgen05.fence::before_thread_sync), not data in memory, and a
// cluster-scope release here cost every epilogue warp some thousand clocks per tile (fused
// classifier forward 0.472 -> 0.450 ms, backward 0.577 -> 0.533 ms).
__device__ __forceinline__ void mbar_arrive_cluster(unsigned cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

__device__ __forceinline__ unsigned cluster_ctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// TMA load into this CTA's shared memory; the byte count is credited to `bar`, which may be the
// partner CTA's barrier (pair form of the instruction; no multicast).
__device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, unsigned src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(map), "r"(x),
               "r"(y), "r"(src)
               : "memory");
}

// One MMA of a single CTA.
__device__ __forceinline__ void umma_bf16_cta(unsigned d_tmem, unsigned long long a_desc, unsigned long long b_desc, unsigned idesc,
                                              unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrives on this CTA's barrier once every tcgen05 operation issued so far by this thread is done.
__device__ __forceinline__ void umma_commit_cta(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// One MMA across the CTA pair: D[256 x 256] (+)= A[256 x 16] * B[16 x 256].
__device__ __forceinline__ void umma_bf16(unsigned d_tmem, unsigned long long a_desc, unsigned long long b_desc,
                                          unsigned idesc, unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrives on the barrier at this offset in BOTH CTAs of the pair once every tcgen05 operation
// issued so far by this thread is done.  (mask: the pair's two CTAs inside the cluster.)
__device__ __forceinline__ void umma_commit_pair(unsigned bar, unsigned short mask = 3) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"(mask)
               : "memory");
}

__device__ __forceinline__ void tmem_ld8(unsigned taddr, float* v) {
  unsigned* r = reinterpret_cast<unsigned*>(v);
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}

__device__ __forceinline__ void tmem_ld32(unsigned taddr, float* v) {
  unsigned* r = reinterpret_cast<unsigned*>(v);
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}

// Shared-memory matrix descriptor (lbo / sbo in bytes): bits 0-13 start address
// >> 4, bits 16-29 lbo >> 4, bits 32-45 sbo >> 4, bit 46 the descriptor version of this architecture,
// bits 61-63 the swizzle: 2 = 128 bytes, 4 = 64 bytes.  It is handled in two parts: what never changes (the high
// word, and the leading-dimension field of the low word) and the start-address field, so that the
// MMA-issuing thread builds a descriptor with one add and one register pair.
__host__ __device__ constexpr unsigned desc_lo_fixed(unsigned lbo) { return (lbo >> 4) << 16; }
__host__ __device__ constexpr unsigned desc_hi_fixed(unsigned sbo, unsigned swizzle = 2) { return (sbo >> 4) | (1u << 14) | (swizzle << 29); }
__device__ __forceinline__ unsigned long long desc_pack(unsigned lo, unsigned hi) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}

}  // namespace sbp
