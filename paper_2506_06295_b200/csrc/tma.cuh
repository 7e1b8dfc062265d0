// mbarrier / TMA device helpers and the host-side tensor-map cache (sm_100a).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace dllm {

// Every device-side wait gives up after this many nanoseconds of %globaltimer (2 s unless a test shortens it).
// One copy per translation unit; DLLM_WAIT_LIMIT_HOOK(stem) defines the host function that sets it on the
// current device.
constexpr unsigned long long WAIT_LIMIT_DEFAULT_NS = 2000000000ull;
static __device__ unsigned long long g_wait_limit_ns = WAIT_LIMIT_DEFAULT_NS;
#define DLLM_WAIT_LIMIT_HOOK(stem)                                                                      \
  namespace dllm {                                                                                      \
  cudaError_t set_wait_limit_##stem(unsigned long long ns) {                                            \
    const unsigned long long v = ns ? ns : WAIT_LIMIT_DEFAULT_NS;                                       \
    return cudaMemcpyToSymbol(g_wait_limit_ns, &v, sizeof v);                                           \
  }                                                                                                     \
  }

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t gtime() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrival on a barrier of another CTA of the cluster (shared::cluster address, see cluster_addr).
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait.  Returns false if the barrier did not flip within the limit or
// another role of the CTA already gave up (abort_flag lives in shared memory).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = gtime();
  uint32_t it = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++it & 63u) == 0u) {
      if (*abort_flag) return false;
      if (gtime() - t0 > g_wait_limit_ns) {
        *abort_flag = 1;
        return false;
      }
    }
  }
  return true;
}
// One lane of a converged warp.  Code that issues TMA copies and tcgen05 instructions runs in all 32 lanes and guards
// each group of instructions with this: behind `lane == 0` the compiler cannot tell that one thread is active and
// moves every operand through a per-lane sequence (four MMAs and a commit took 330 cycles of the issuing thread
// against 150 behind elect, and that thread was what bounded the GEMM main loops: 600 against 460 cycles per k-block
// of a 256 x 128 tile).
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}
// Whether the phase has completed, without waiting; the whole warp, which gets one answer.
__device__ __forceinline__ bool mbar_peek_warp(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return __all_sync(0xffffffffu, ok != 0);
}
// mbar_wait by a converged warp, which gets one answer.  `ready`: an earlier mbar_peek_warp of this phase said so.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               bool ready = false) {
  if (ready || __all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const uint64_t t0 = gtime();
  uint32_t it = 0;
  while (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) {
    if ((++it & 63u) == 0u) {
      bool stop = *abort_flag != 0;
      if (!stop && gtime() - t0 > g_wait_limit_ns) {
        *abort_flag = 1;
        stop = true;
      }
      if (__any_sync(0xffffffffu, stop)) return false;
    }
  }
  return true;
}
// Lets copies that may still be in flight land before shared memory is released.
__device__ __forceinline__ void drain_delay() {
  const uint64_t t0 = gtime();
  while (gtime() - t0 < 200000ull) {
  }
}
__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* tm) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tm)) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
// Tile load by one CTA of a pair (cta_group::2): the data lands in this CTA's shared memory, the bytes are
// counted on `bar_cluster`, a shared::cluster address that may name the other CTA's barrier (see cluster_addr).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, uint32_t bar_cluster, int c0,
                                                 int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar_cluster), "r"(c0), "r"(c1)
      : "memory");
}
// Tile loads marked evict-first in L2 where ONCE: the weights of a product with one activation tile are read once per
// step, and a layer's 436 MB of them push out what every launch needs again (activations, caches, partial sums).  Without
// the mark the plain instruction is used (an explicit evict-normal policy measured 1 % slower), chosen at compile time (a
// branch in the copying loop cost the 768-row step 2 %).
__device__ __forceinline__ uint64_t evict_first_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
template <bool ONCE>
__device__ __forceinline__ void tma_load_2d_weights(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1) {
  if constexpr (ONCE)
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4}], "
        "[%2], %5;" ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar), "r"(c0), "r"(c1), "l"(evict_first_policy())
        : "memory");
  else
    tma_load_2d(dst, tm, bar, c0, c1);
}
template <bool ONCE>
__device__ __forceinline__ void tma_load_2d_pair_weights(uint32_t dst, const CUtensorMap* tm, uint32_t bar_cluster, int c0,
                                                         int c1) {
  if constexpr (ONCE)
    asm volatile(
        "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, "
        "{%3, %4}], [%2], %5;" ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar_cluster), "r"(c0), "r"(c1),
        "l"(evict_first_policy())
        : "memory");
  else
    tma_load_2d_pair(dst, tm, bar_cluster, c0, c1);
}
// Untiled bulk copy global -> shared: both addresses 16-byte aligned, bytes a multiple of 16; completes on `bar`.
__device__ __forceinline__ void bulk_load_1d(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the location that has shared::cta address `addr` in the CTA of rank `rank`
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// every thread of every CTA of the cluster
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// Host: bf16 tensor maps with a 64-element (128-byte) inner box and 128-byte
// swizzle, cached by (base, shape, box).  2-D: [rows, cols] row-major, box
// box_rows x 64.  3-D: [batch, rows, cols], box 1 x box_rows x 64.
bool get_tensor_map_2d(const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, CUtensorMap* out);
bool get_tensor_map_3d(const void* base, uint64_t batch, uint64_t rows, uint64_t cols, uint32_t box_rows,
                       CUtensorMap* out);

}  // namespace dllm
