// The persistent CTA-pair GEMM (tcgen05, cta_group::2), with the epilogue as a parameter.
//
// FORM: what happens to a finished tile (a kernel argument), W = BN / GROUPS of its columns by each of GROUPS groups of 128
// epilogue threads.  ex_bytes<W>() of staging and Shared<W> static shared memory per group; ahead() runs before the
// accumulator is waited for, drain() behind it (tl = 0..127 = TMEM lane; a group meets on its named barrier).  One kernel
// instance holds one form's code: an epilogue runs once per launch from a cold instruction cache, and a form's unused
// neighbours in the same body cost more than their branches.
// An epilogue is bound by the latency of its own instructions: one group puts one warp on each scheduler, which waits for
// every result it needs next.  Two groups halve the staged forms: SwiGLU of 256 rows 5.8 -> 3.9 us, placed and rotated rows
// 16 -> about 6 (with fewer instructions per row, see gemm_rows.cu).  Slabs take 2.8 us either way (their stores) and keep
// one group, whose 192 small threads leave room for the next kernel's CTAs.
#pragma once
#include <algorithm>

#include "internal.h"
#include "tma.cuh"
#include "umma.cuh"

namespace dllm {

namespace {

constexpr int TILE_W = 128;  // weight rows per CTA (UMMA M)
constexpr int TILE_K = 64;   // k per stage: 64 bf16 = one 128-byte swizzle row
constexpr int UMMA_K = 16;
constexpr uint32_t W_STAGE_BYTES = TILE_W * TILE_K * 2;
constexpr int MAX_STAGES = 12;
constexpr int RASTER = 16;     // activation tiles per group of the launch-order remap

// A group of 128 epilogue threads meets on named barrier 1 or 2 (numbers in the code: a barrier named by a register would
// reserve all sixteen).
__device__ __forceinline__ void group_sync(int bar) {
  if (bar == 1)
    asm volatile("bar.sync 1, 128;" ::: "memory");
  else
    asm volatile("bar.sync 2, 128;" ::: "memory");
}
template <int BAR>
__device__ __forceinline__ bool group_all_on(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, %2, 128, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(BAR)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ bool group_all(int bar, bool v) { return bar == 1 ? group_all_on<1>(v) : group_all_on<2>(v); }

// ---------------------------------------------------------------- persistent CTA-pair kernel
// The product for more than 128 activation rows, with cta_group::2: two CTAs of a cluster work on one tile of 256
// weight rows x BN activation rows.  Each stages its own 128 weight rows and HALF of the activation tile, one thread of
// the first CTA issues MMAs that read both CTAs' shared memory, and each CTA ends with its own 128 x BN accumulator in
// its own TMEM.  What bounds such a product is the L2 -> SM fabric (about 12 TB/s over all SMs on B200): a 128 x 256 tile
// of one CTA moves 48 KB per k-block of 512 tensor cycles, the pair's share of 256 x 256 moves 32 KB.
// One pair per two SMs walks through units p, p + pairs, ... (a unit = a tile, or a tile's share of the k range) with
// fixed roles: warp 0 requests operands without a gap between units, warp 1 issues the MMAs into one of TWO accumulators
// in tensor memory, and the other warps drain one accumulator while the other fills.  The k loop of a tile is the one-tile
// kernel's: results are bit-identical to it.  With a split k range every split writes its own slab.  Loads carry no
// multicast: every byte is requested by the CTA that stages it.
// (In the replayed response refresh of 256 rows of a 4096-wide model, us from the release to the first stage / accumulators
// complete / rows written: Q / K / V, placed and rotated, 1.9 / 23.9 / 30.0; O in four splits 2.5 / 8.7 / 11.8; gate / up with
// SwiGLU, two rounds, 3.1 / 27.8-51.6 / 31.5-55.2; down in four 1.9 / 19.8 / 22.8.)
template <typename FORM>
constexpr int PAIR_THREADS = 64 + 128 * FORM::GROUPS;
template <int BN, typename FORM>
struct PairLayout {
  static constexpr uint32_t A_HALF_BYTES = (BN / 2) * TILE_K * 2;
  static constexpr uint32_t STAGE_BYTES = W_STAGE_BYTES + A_HALF_BYTES;
  static constexpr int W = BN / FORM::GROUPS;
  // staging of the forms that go through shared memory, all groups'
  static constexpr uint32_t EX_GROUP = FORM::template ex_bytes<W>(), EX_BYTES = FORM::GROUPS * EX_GROUP;
  static constexpr uint32_t total(int stages, bool staged) {
    return (uint32_t)stages * STAGE_BYTES + (staged ? EX_BYTES : 0) + 1024;
  }
  static constexpr int most(bool staged) {
    const int shared = FORM::GROUPS * (int)sizeof(typename FORM::template Shared<W>);
    const int fit = (227 * 1024 - 1024 - 512 - shared - (staged ? (int)EX_BYTES : 0)) / (int)STAGE_BYTES;
    return fit < MAX_STAGES ? fit : MAX_STAGES;
  }
};

// Unit u of the walk over m_tiles x n_pairs tiles x splits -> (activation tile, weight pair, split).  Splits are
// outermost; inside, groups of RASTER activation tiles with the weight pairs inside a group, so that pairs that
// run together share operands in L2.
__device__ __forceinline__ void pair_unit(int u, int m_tiles, int n_pairs, int& mt, int& np, int& z) {
  const int tiles = m_tiles * n_pairs;
  z = u / tiles;
  const int t = u - z * tiles, per = RASTER * n_pairs, grp = t / per, within = t - grp * per;
  const int wide = min(RASTER, m_tiles - grp * RASTER);
  np = within / wide;
  mt = grp * RASTER + within - np * wide;
}

template <int BN, bool ONCE, typename FORM>
__global__ void __launch_bounds__(PAIR_THREADS<FORM>, 2)
    gemm_bf16_pair_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmA,
                          float* __restrict__ part, int M, int N, int num_kb, int kb_per_split, size_t split_stride,
                          int m_tiles, int n_pairs, int units, int STAGES, const __grid_constant__ FORM form,
                          int* __restrict__ status) {
  using PL = PairLayout<BN, FORM>;
  // column distance of the two accumulators: an allocation is a power of two, so 192-row tiles sit 256 apart
  constexpr uint32_t ACC = BN > 128 ? 256 : BN > 64 ? 128 : BN > 32 ? 64 : 32;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES];   // used in the pair's first CTA: bytes of both CTAs
  __shared__ __align__(8) uint64_t empty_bar[MAX_STAGES];  // in each CTA: its stage may be refilled
  __shared__ __align__(8) uint64_t acc_full[2];            // in each CTA: accumulator complete
  __shared__ __align__(8) uint64_t acc_empty[2];           // used in the first CTA: both CTAs' epilogues have read it
  __shared__ typename FORM::template Shared<PL::W> fs[FORM::GROUPS];
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
  const uint32_t tiles_s = (smem_u32(smem_raw) + 1023u) & ~1023u;
  float* ex = reinterpret_cast<float*>(smem_raw + (tiles_s - smem_u32(smem_raw)) + (size_t)STAGES * PL::STAGE_BYTES);
  // k-blocks of split z: [z * kb_per_split, kb_end(z)), never empty by construction of the plan
  auto kb_end = [&](int z) { return min(num_kb, (z + 1) * kb_per_split); };

  if (warp == 0 && elect_one()) {
    abort_flag = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full_bar[s]), 1);
      mbar_init(smem_u32(&empty_bar[s]), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(smem_u32(&acc_full[a]), 1);
      mbar_init(smem_u32(&acc_empty[a]), 2 * 4 * FORM::GROUPS);  // one arrival per epilogue warp of both CTAs
    }
    mbar_fence_init();
    prefetch_tensormap(&tmW);
    prefetch_tensormap(&tmA);
  }
  if (warp == 1) {  // the same warp of both CTAs: two accumulators of BN fp32 columns x 128 lanes in each CTA's TMEM
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"(2u * ACC)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before either signals the other's
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = tmem_base_slot;
  volatile int* abortp = &abort_flag;

  int pre = 0;  // stages whose weight tile was requested before the dependency wait
  if (warp == 0 && pair < units) {
    int mt, np, z;
    pair_unit(pair, m_tiles, n_pairs, mt, np, z);
    const int kb0 = z * kb_per_split;
    pre = min(STAGES, kb_end(z) - kb0);  // weights are written by no kernel: stream them ahead of the dependency
    if (elect_one())
      for (int i = 0; i < pre; ++i) {
        if (leader) mbar_expect_tx(smem_u32(&full_bar[i]), 2 * PL::STAGE_BYTES);
        tma_load_2d_pair_weights<ONCE>(tiles_s + i * PL::STAGE_BYTES, &tmW, cluster_addr(smem_u32(&full_bar[i]), 0),
                              (kb0 + i) * TILE_K, (2 * np + rank) * TILE_W);
      }
    __syncwarp();
  }
  pdl_wait();     // the activation rows and the output buffer belong to the preceding kernels
  pdl_trigger();
  bool ok = true;

  if (warp == 0) {
    // ---------------- TMA producer (both CTAs) ----------------
    int s = 0, issued = 0;
    uint32_t ph = 0;
    for (int u = pair; u < units && ok; u += pairs) {
      int mt, np, z;
      pair_unit(u, m_tiles, n_pairs, mt, np, z);
      const int n0 = (2 * np + rank) * TILE_W, m0 = mt * BN + rank * (BN / 2);
      const int kb1 = kb_end(z);
      for (int kb = z * kb_per_split; kb < kb1; ++kb, ++issued) {
        if (issued >= pre && !mbar_wait_warp(smem_u32(&empty_bar[s]), ph ^ 1u, abortp)) {
          if (status && lane == 0) atomicCAS(status, ST_OK, ST_TIMEOUT_TMA);
          ok = false;
          break;
        }
        if (elect_one()) {
          const uint32_t fb = cluster_addr(smem_u32(&full_bar[s]), 0);
          const uint32_t dst = tiles_s + s * PL::STAGE_BYTES;
          if (issued >= pre) {
            if (leader) mbar_expect_tx(smem_u32(&full_bar[s]), 2 * PL::STAGE_BYTES);
            tma_load_2d_pair_weights<ONCE>(dst, &tmW, fb, kb * TILE_K, n0);
          }
          tma_load_2d_pair(dst + W_STAGE_BYTES, &tmA, fb, kb * TILE_K, m0);
        }
        __syncwarp();
        if (++s == STAGES) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (first CTA of the pair) ----------------
    if (leader) {
      constexpr uint32_t idesc = make_idesc(2 * TILE_W, BN);
      int s = 0, j = 0;
      uint32_t ph = 0;
      bool ready = false;
      for (int u = pair; u < units && ok; u += pairs, ++j) {
        const int a = j & 1;
        const int z = u / (m_tiles * n_pairs), kb0 = z * kb_per_split, kb1 = kb_end(z);
        // the epilogues of the unit that used this accumulator two units ago have read it
        if (!mbar_wait_warp(smem_u32(&acc_empty[a]), ((uint32_t)(j >> 1) & 1u) ^ 1u, abortp)) {
          if (status && lane == 0) atomicCAS(status, ST_OK, ST_TIMEOUT_MMA);
          ok = false;
          break;
        }
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait_warp(smem_u32(&full_bar[s]), ph, abortp, ready)) {
            if (status && lane == 0) atomicCAS(status, ST_OK, ST_TIMEOUT_MMA);
            ok = false;
            break;
          }
          if (j == 0 && kb == kb0 && lane == 0) timeline_mark(1);   // first stage complete
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sW = tiles_s + s * PL::STAGE_BYTES, empty = smem_u32(&empty_bar[s]);
          if (++s == STAGES) {
            s = 0;
            ph ^= 1u;
          }
          ready = mbar_peek_warp(smem_u32(&full_bar[s]), ph);  // answered while the MMAs below are issued
          if (elect_one()) {
            const uint64_t dW = make_smem_desc(sW);
            const uint64_t dA = make_smem_desc(sW + W_STAGE_BYTES);
#pragma unroll
            for (int k = 0; k < TILE_K / UMMA_K; ++k)
              umma_bf16_pair(tmem_d + (uint32_t)a * ACC, dW + (uint64_t)(2 * k), dA + (uint64_t)(2 * k), idesc,
                             (kb > kb0 || k > 0) ? 1u : 0u);
            umma_commit_pair(empty);  // both CTAs may refill the stage once these MMAs have read it
            if (kb == kb1 - 1) umma_commit_pair(smem_u32(&acc_full[a]));
          }
          __syncwarp();
        }
      }
    }
  } else {
    // ---------------- epilogue warps of both CTAs: own 128 weight rows, TMEM lanes 32 * (warp % 4) .. + 31; warps 2-5 the
    // first W activation rows, warps 6-9 (where there are two groups) the others ----
    constexpr int W = PL::W;
    const int tl = (warp & 3) * 32 + lane, group = FORM::GROUPS == 1 ? 0 : (warp - 2) >> 2, bar = 1 + group;
    int j = 0;
    for (int u = pair; u < units; u += pairs, ++j) {
      const int a = j & 1;
      int mt, np, z;
      pair_unit(u, m_tiles, n_pairs, mt, np, z);
      const int m0 = mt * BN + group * W;
      form.template ahead<W>(fs[group], tl, m0, M);
      bool have = mbar_wait(smem_u32(&acc_full[a]), (uint32_t)(j >> 1) & 1u, abortp);
      // the 128 threads of the group agree (the TMEM loads are warp-collective and the staged forms exchange data)
      have = group_all(bar, have);
      if (!have) {
        if (tl == 0 && status) atomicCAS(status, ST_OK, ST_TIMEOUT_EPI);
        ok = false;
        break;
      }
      if (tl == 0 && group == 0) timeline_mark(3);                   // accumulator complete
      const int nt = 2 * np + rank;
      if (nt * TILE_W < N)  // the second CTA of the last pair has no rows when the weight tiles are odd in number
        form.template drain<W>(fs[group], tmem_d + (uint32_t)(a * ACC + group * W),
                               ex + group * (PL::EX_GROUP / 4), tl, bar, m0, nt * TILE_W, nt, M, N,
                               part + (size_t)z * split_stride);
      if (tl == 0 && group == 0) timeline_mark(4);                         // this thread's part of the epilogue written
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(cluster_addr(smem_u32(&acc_empty[a]), 0));
    }
  }
  ok = __syncthreads_and(ok);
  if (!ok) drain_delay();  // gave up: let copies in flight land before shared memory is released
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync();  // neither CTA leaves, nor is TMEM freed, while the other may still use this one's memory
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(2u * ACC) : "memory");
  }
}

template <int BN, bool ONCE, typename FORM>
cudaError_t launch_pair_form(const Launch& L, const CUtensorMap& tmW, const CUtensorMap& tmA, float* part, int M, int N,
                        int num_kb, const GemmPlan& plan, const FORM& form, bool staged) {
  using PL = PairLayout<BN, FORM>;
  static DeviceOnce once;
  cudaError_t e0 = once.run([] {
    return cudaFuncSetAttribute(gemm_bf16_pair_kernel<BN, ONCE, FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                227 * 1024 - 512 - FORM::GROUPS * (int)sizeof(typename FORM::template Shared<BN / FORM::GROUPS>));
  });
  if (e0 != cudaSuccess) return e0;
  const int most = PL::most(staged), stages = plan.stages < 2 ? 2 : plan.stages > most ? most : plan.stages;
  const int m_tiles = (M + BN - 1) / BN, n_pairs = (N + 2 * TILE_W - 1) / (2 * TILE_W);
  const int units = m_tiles * n_pairs * plan.S_max;
  const int pairs = std::min(units, sm_count() / 2);
  cudaError_t e = launch_k_cluster(L, gemm_bf16_pair_kernel<BN, ONCE, FORM>, dim3(2 * pairs), dim3(PAIR_THREADS<FORM>),
                                   PL::total(stages, staged), dim3(2, 1, 1), tmW, tmA, part, M, N, num_kb, plan.upc,
                                   (size_t)M * N, m_tiles, n_pairs, units, stages, form, L.d_status);
  L.count();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

}  // namespace dllm
