// cluster_copy.cuh -- bulk copies between the CTAs of a cluster, counted on the
// receiver's mbarrier, with bounded waits (panel_lu_reg.cu, panel_qr_reg.cu).
//
// A wait that gives up (limit clocks, about 2 s by default) leaves its column
// with whatever the buffer holds; the thread then neither waits nor sends any
// more, and tells the cluster.  Before the cluster leaves, all of it then waits
// a bounded time for what is still on its way: nothing arrives in the memory
// of a CTA that has left.
#pragma once
#include "ca_internal.cuh"

namespace cagb {

constexpr long long kPanelWait = 4000000000ll;  // about 2 s of SM clock

// Host state of the test hook: the limit of the waits and whether a cluster's
// last CTA sends nothing.
long long panel_wait_limit();
int panel_withhold();

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// bytes of this CTA's shared memory to CTA `rank`'s, counted on its barrier
__device__ __forceinline__ void bulk_to(const void *dst, const void *src, unsigned bytes, const void *bar, int rank) {
  asm volatile(
      "{\n\t.reg .b32 d, m;\n\t"
      "mapa.shared::cluster.u32 d, %0, %4;\n\t"
      "mapa.shared::cluster.u32 m, %2, %4;\n\t"
      "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [d], [%1], %3, [m];\n\t}\n" ::"r"(
          smem_addr(dst)),
      "r"(smem_addr(src)), "r"(smem_addr(bar)), "r"(bytes), "r"(rank)
      : "memory");
}
__device__ __forceinline__ void bar_expect(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_try(unsigned addr, unsigned parity) {  // waits a while by itself
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(done)
      : "r"(addr), "r"(parity)
      : "memory");
  return done != 0;
}
// false when the phase did not complete within the limit
__device__ __forceinline__ bool bar_wait(unsigned long long *bar, unsigned parity, long long limit) {
  const unsigned addr = smem_addr(bar);
  const long long t0 = clock64();
  while (true) {
    if (bar_try(addr, parity)) return true;
    if (clock64() - t0 > limit) return false;
  }
}

// After the last column: if a thread of this CTA gave up, every CTA of the
// cluster is told (flag: a word of shared memory, zero before the first
// exchange), and the host.  Every thread calls it, outside the column loops;
// inline, because a call costs the 254-register TSQR node 2 % of its time.
__device__ __forceinline__ void tell_gave_up(cg::cluster_group &cl, bool dead, int *flag, int *status) {
  if (!__syncthreads_or(dead)) return;
  for (int r = threadIdx.x; r < (int)cl.num_blocks(); r += blockDim.x) atomicExch(cl.map_shared_rank(flag, r), 1);
  if (dead && status) atomicOr(status, CA_STATUS_PANEL_TIMEOUT);
}

// After the cluster barrier that follows the last exchange: whether any thread
// of the cluster gave up.  If so nobody sends any more, and what was sent
// before has landed when this returns; every CTA then passes one more cluster
// barrier before it leaves.
__device__ __forceinline__ bool cluster_gave_up(const int *flag) {
  if (*(volatile const int *)flag == 0) return false;
  const long long t0 = clock64();  // a copy takes about a thousand clocks
  while (clock64() - t0 < 100000) {
  }
  return true;
}

}  // namespace cagb
