// bf16 GEMM for sm_100a:  part[z][M][N] (fp32) = A[M, Kz] * W[N, Kz]^T
//
// Every projection of the cached step (V for all response rows; Q/K, O and the
// SwiGLU matrices for the gathered active rows; the LM head) is
// "few activation rows x a large weight matrix".  With M between 3 and a few
// hundred rows the product is bound by streaming W from HBM once, so the kernel
// is laid out around the weight stream:
//
//   * the WEIGHT tile (128 rows of W, 64 k) is the M-side operand of
//     tcgen05.mma (UMMA M = 128) and the ACTIVATION tile (BN = 32..256 rows of
//     A, 64 k) is the N-side operand, so small row counts cost no padding of
//     the 128-row dimension and the accumulator D[128 weight rows][BN act rows]
//     sits in BN TMEM columns;
//   * both tiles arrive by TMA (128-byte swizzle) into a ring of shared-memory
//     stages guarded by full/empty mbarriers; one thread issues the copies,
//     one thread issues the MMAs, tcgen05.commit releases a stage;
//   * TMEM lane = output column n, so for a fixed activation row the 32 lanes
//     of a warp store 32 consecutive floats: the epilogue writes row-major
//     [M, N] coalesced straight from tcgen05.ld registers;
//   * split-K over blockIdx.z puts >= 148 CTAs on the weight stream when N/128
//     is small; every split writes its own slab and the consumer kernel adds
//     the slabs in order (no atomics, bit-reproducible);
//   * weight tiles are requested before griddepcontrol.wait: with programmatic
//     dependent launch the ring fills while the kernel that produces the
//     activation rows is still running; the activation tile of a stage follows
//     after the wait and the stage's barrier completes when both have landed;
//   * rows of A beyond M and k beyond K are zero-filled by TMA.
//
// Every wait on an mbarrier is bounded (2 s of %globaltimer); on expiry the
// CTA records a code in the status word, skips its epilogue, lets copies in
// flight land, frees its TMEM and returns.
#include <algorithm>
#include <mutex>
#include <unordered_map>

#include "../../include/dllm.h"
#include "internal.h"
#include "tma.cuh"
#include "umma.cuh"
#include "gemm_pair.cuh"

namespace dllm {

namespace {

// Test hook for the bounded waits: while non-zero, the TMA producer of CTA (0, 0, 0) of every launch of the
// one-CTA kernel leaves out the activation tile of its first k-block, so that stage's barrier never completes
// and the CTA's waits run into their limit (it then records a status code and returns; nothing faults).
static __device__ int g_debug_skip_act_load = 0;


template <int BN>
struct SmemLayout {
  static constexpr uint32_t A_STAGE_BYTES = BN * TILE_K * 2;
  static constexpr uint32_t STAGE_BYTES = W_STAGE_BYTES + A_STAGE_BYTES;
  static constexpr uint32_t total(int stages) { return (uint32_t)stages * STAGE_BYTES + 1024; }  // + slack to align the base to 1024
};

// Epilogue of W columns of a tile by a group of 128 threads: the accumulator, TMEM lanes = 128 weight rows from n0 (tile
// number tile_y), columns = W activation rows from m0, goes to the fp32 slab (coalesced: lane = output column), through
// the SwiGLU combination (act_out) or into estimate records (m_ffn < 0).  `ex`: PlainStage<W>::BYTES of shared memory that
// nothing else uses meanwhile.  tl = 0..127 identifies the thread: it works on TMEM lane tl, so its warp must be the one
// allowed to touch lanes 32 * (tl / 32) .. + 31 (warp index % 4 == tl / 32).  The group meets on named barrier `bar` (1 or 2).
// Two groups share a tile, half of its columns each: one group of four warps spends most of the epilogue waiting for
// tensor memory and for its stores to issue.
template <int W>
struct PlainStage {
  static constexpr int CH = W < 32 ? W : 32;   // activation rows staged at a time
  static constexpr int EXS = 132;              // floats per staged row: 16-byte aligned, rows 4 banks apart
  static constexpr uint32_t BYTES = CH * EXS * 4;
};
// CH columns of tensor memory on their way into registers; landed: they are there; then they go to staging.  The loops below
// wait for what they have requested in the same trip: between a load and its wait nothing may read or move the registers, and
// the compiler may move what a loop carries round its edge.
template <int CH>
__device__ __forceinline__ void tmem_fetch(uint32_t taddr, uint32_t (&r)[CH / 16][16]) {
#pragma unroll
  for (int i = 0; i < CH / 16; ++i) tmem_ld16(taddr + 16u * i, r[i]);
}
template <int CH>
__device__ __forceinline__ void tmem_landed(uint32_t (&r)[CH / 16][16]) {
#pragma unroll
  for (int i = 0; i < CH / 16; ++i) tmem_ld16_wait(r[i]);
}
template <int CH, int EXS>
__device__ __forceinline__ void tmem_stage(const uint32_t (&r)[CH / 16][16], float* ex, int tl) {
#pragma unroll
  for (int i = 0; i < CH / 16; ++i)
#pragma unroll
    for (int j = 0; j < 16; ++j) ex[(16 * i + j) * EXS + tl] = __uint_as_float(r[i][j]);
}
enum PlainKind { SLABS, SWIGLU, ESTIMATE };
template <int W, PlainKind KIND>
__device__ __forceinline__ void gemm_epilogue(uint32_t tmem_d, float* ex, int tl, int bar, int m0, int n0, int tile_y, int M,
                                              int N, float* __restrict__ slab, __nv_bfloat16* __restrict__ act_out,
                                              int m_ffn) {
  const int lane = tl & 31;
  const uint32_t tmem_w = tmem_d + ((uint32_t)(tl >> 5) << 21);
  constexpr int CH = PlainStage<W>::CH, EXS = PlainStage<W>::EXS;
  auto sync = [&] { group_sync(bar); };
  if (m0 >= M) return;  // uniform across the group
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if constexpr (KIND == ESTIMATE) {
    // Estimate epilogue of the LM head (no split-K, act_out == nullptr, m_ffn = -1 - mask id): instead of 128
    // logits per row the CTA writes one record per activation row, {max, sum exp(v - max), argmax, -} over its
    // 128 vocabulary columns (Eq. 4; the mask id and columns past N are skipped); a merge over the tiles
    // follows.  Staged like the SwiGLU epilogue; four threads share a row, 32 columns each (the same sums in every tile
    // width).
    const int mask_id = -1 - m_ffn, n_tiles = (N + TILE_W - 1) / TILE_W;
    float4* rec = reinterpret_cast<float4*>(slab);
    const int rr = tl >> 2, part = tl & 3;
    uint32_t r[CH / 16][16];
    tmem_fetch<CH>(tmem_w, r);
    tmem_landed<CH>(r);
#pragma unroll 1
    for (int c0 = 0; c0 < W && m0 + c0 < M; c0 += CH) {
      tmem_stage<CH, EXS>(r, ex, tl);
      sync();
      tmem_fetch<CH>(tmem_w + (uint32_t)min(c0 + CH, W - CH), r);   // the next rows (again the last ones in the last trip)
      MaxSum t{-INFINITY, 0.f, 0x7fffffff};
      if (rr < CH) {
        // two passes over the thread's 32 columns: maximum and its first index, then the exponentials as four
        // independent sums (one serial chain of dependent exponentials would dominate the epilogue)
        const float* row = ex + rr * EXS + part * 32;
        const int nb = n0 + part * 32;
#pragma unroll 4
        for (int j = 0; j < 32; j += 4) {
          const float4 v = *reinterpret_cast<const float4*>(row + j);
          const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int n = nb + j + q;
            if (n < N && n != mask_id && e[q] > t.m) {
              t.m = e[q];
              t.a = n;
            }
          }
        }
        if (t.m > -INFINITY) {
          float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
          for (int j = 0; j < 32; j += 4) {
            const float4 v = *reinterpret_cast<const float4*>(row + j);
            const float e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int n = nb + j + q;
              s4[q] += (n < N && n != mask_id) ? expf(e[q] - t.m) : 0.f;
            }
          }
          t.s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
        }
      }
#pragma unroll
      for (int x = 1; x <= 2; x <<= 1) {
        MaxSum o;
        o.m = __shfl_xor_sync(0xffffffffu, t.m, x);
        o.s = __shfl_xor_sync(0xffffffffu, t.s, x);
        o.a = __shfl_xor_sync(0xffffffffu, t.a, x);
        t = merge(t, o);
      }
      const int m = m0 + c0 + rr;
      if (rr < CH && part == 0 && m < M)
        rec[(size_t)m * n_tiles + tile_y] = make_float4(t.m, t.s, __int_as_float(t.a), 0.f);
      tmem_landed<CH>(r);
      sync();
    }
  } else if constexpr (KIND == SWIGLU) {
    // SwiGLU epilogue (no split-K): the tile's 128 weight rows are 64 gate rows followed by the 64 up rows
    // of the same FFN columns, so TMEM lanes 0..63 hold gate and 64..127 hold up.  The accumulator goes
    // through shared memory (every MMA has completed) CH activation rows at a time, transposed to
    // [row][weight row], the next ones on their way out of tensor memory meanwhile, and comes back as silu(gate) * up in
    // bf16, 8 bytes per thread.
    const int q = tl & 15, rsub = tl >> 4;  // 4 FFN columns, 8 rows per pass
    const int col = tile_y * 64 + 4 * q;
    uint32_t r[CH / 16][16];
    tmem_fetch<CH>(tmem_w, r);
    tmem_landed<CH>(r);
#pragma unroll 1
    for (int c0 = 0; c0 < W && m0 + c0 < M; c0 += CH) {
      tmem_stage<CH, EXS>(r, ex, tl);
      sync();
      tmem_fetch<CH>(tmem_w + (uint32_t)min(c0 + CH, W - CH), r);   // the next rows (again the last ones in the last trip)
#pragma unroll 2
      for (int rr = rsub; rr < CH; rr += 8) {
        const int m = m0 + c0 + rr;
        const float4 gt = *reinterpret_cast<const float4*>(ex + rr * EXS + 4 * q);
        const float4 up = *reinterpret_cast<const float4*>(ex + rr * EXS + 64 + 4 * q);
        if (m < M && col < m_ffn) {
          // silu(g) * u with the fast exponential and division (relative error ~1e-6, far below the bf16 rounding
          // of the result)
          const __nv_bfloat162 lo = __floats2bfloat162_rn(__fdividef(gt.x, 1.f + __expf(-gt.x)) * up.x,
                                                          __fdividef(gt.y, 1.f + __expf(-gt.y)) * up.y);
          const __nv_bfloat162 hi = __floats2bfloat162_rn(__fdividef(gt.z, 1.f + __expf(-gt.z)) * up.z,
                                                          __fdividef(gt.w, 1.f + __expf(-gt.w)) * up.w);
          uint2 pk;
          pk.x = *reinterpret_cast<const uint32_t*>(&lo);
          pk.y = *reinterpret_cast<const uint32_t*>(&hi);
          *reinterpret_cast<uint2*>(act_out + (size_t)m * m_ffn + col) = pk;
        }
      }
      tmem_landed<CH>(r);
      sync();
    }
  } else {
    const int n = n0 + (tl >> 5) * 32 + lane;
    float* out = slab + n;
    // (16 columns per trip and little code: an epilogue runs once per launch from a cold instruction cache, and 64 columns
    // unrolled took 0.5 to 1.5 us longer per projection)
#pragma unroll 1
    for (int c0 = 0; c0 < W; c0 += 16) {
      if (m0 + c0 >= M) break;  // uniform across the group
      uint32_t r[16];
      tmem_ld16(tmem_w + (uint32_t)c0, r);
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (n < N) {
        float* row = out + (size_t)(m0 + c0) * N;
        if (m0 + c0 + 16 <= M) {
#pragma unroll
          for (int j = 0; j < 16; ++j) row[(size_t)j * N] = __uint_as_float(r[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (m0 + c0 + j < M) row[(size_t)j * N] = __uint_as_float(r[j]);
        }
      }
    }
  }
}

// One-tile kernel: warp 0 requests operands, warp 1 issues the MMAs, and all eight drain the accumulator, two per quarter
// of the TMEM lanes with half of the activation rows each.
constexpr int ONE_THREADS = 256;
template <int BN, bool ONCE>
__global__ void __launch_bounds__(ONE_THREADS) gemm_bf16_tcgen05_kernel(const __grid_constant__ CUtensorMap tmW,
                                                                const __grid_constant__ CUtensorMap tmA,
                                                                float* __restrict__ part, int M, int N, int num_kb,
                                                                int kb_per_split, size_t split_stride, int STAGES,
                                                                __nv_bfloat16* __restrict__ act_out, int m_ffn, int turned,
                                                                int* __restrict__ status) {
  using SL = SmemLayout<BN>;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t empty_bar[MAX_STAGES];
  __shared__ __align__(8) uint64_t accum_bar;
  __shared__ uint32_t tmem_base_slot;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Tile of this CTA.  With many activation tiles, CTAs that run together (consecutive in x-major launch order)
  // take RASTER activation tiles times a few weight tiles, so that their operands stay in L2 while the other
  // dimension is swept; otherwise every sweep over the weight tiles would re-read all activations from HBM.
  int mt = blockIdx.x, nt = blockIdx.y;
  if (gridDim.x > RASTER) {
    const int lin = blockIdx.x + gridDim.x * blockIdx.y, per = RASTER * gridDim.y;
    const int grp = lin / per, within = lin - grp * per;
    const int wide = min(RASTER, (int)gridDim.x - grp * RASTER);
    nt = within / wide;
    mt = grp * RASTER + within - nt * wide;
  }
  const int m0 = mt * BN;       // activation rows
  const int n0 = nt * TILE_W;   // weight rows = output columns
  const int kb0 = blockIdx.z * kb_per_split;
  const int kb1 = min(num_kb, kb0 + kb_per_split);
  const int nkb = kb1 - kb0;            // >= 1 by construction of the plan
  const int turn = turned && ((nt >> 1) & 1) ? nkb / 2 : 0;   // see launch_gemm_bf16
  auto k_block = [&](int i) {           // the i-th k-block of the walk
    const int j = i + turn;
    return kb0 + (j < nkb ? j : j - nkb);
  };

  const uint32_t tiles = (smem_u32(smem_raw) + 1023u) & ~1023u;

  const int pre = min(STAGES, nkb);  // stages whose weight tile is requested before the dependency wait
  int dbg_skip = 0;
  if (warp == 0) {
    dbg_skip = g_debug_skip_act_load;  // read here, long before it is used: not on the path behind the dependency wait
    if (elect_one()) {
      abort_flag = 0;
      for (int s = 0; s < STAGES; ++s) {
        mbar_init(smem_u32(&full_bar[s]), 1);
        mbar_init(smem_u32(&empty_bar[s]), 1);
      }
      mbar_init(smem_u32(&accum_bar), 1);
      mbar_fence_init();
      prefetch_tensormap(&tmW);
      prefetch_tensormap(&tmA);
      for (int i = 0; i < pre; ++i) {  // weights are written by no kernel: stream them ahead of the dependency
        const uint32_t fb = smem_u32(&full_bar[i]);
        mbar_expect_tx(fb, SL::STAGE_BYTES);
        tma_load_2d_weights<ONCE>(tiles + i * SL::STAGE_BYTES, &tmW, fb, k_block(i) * TILE_K, n0);
      }
    }
    __syncwarp();
  }
  if (warp == 1) {  // TMEM: BN fp32 columns x 128 lanes
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_slot)),
                 "r"((uint32_t)BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_d = tmem_base_slot;
  volatile int* abortp = &abort_flag;
  pdl_wait();     // the activation rows and the slab buffer belong to the preceding kernels
  pdl_trigger();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    int s = 0;
    uint32_t ph = 0;
    for (int i = 0; i < nkb; ++i) {
      const uint32_t fb = smem_u32(&full_bar[s]);
      const uint32_t dstW = tiles + s * SL::STAGE_BYTES;
      const int kc = k_block(i) * TILE_K;
      const bool skip = i == 0 && dbg_skip != 0 && (blockIdx.x | blockIdx.y | blockIdx.z) == 0;
      if (i >= pre && !mbar_wait_warp(smem_u32(&empty_bar[s]), ph ^ 1u, abortp)) {
        if (status && lane == 0) atomicCAS(status, ST_OK, ST_TIMEOUT_TMA);
        break;
      }
      if (elect_one()) {
        if (i >= pre) {
          mbar_expect_tx(fb, SL::STAGE_BYTES);
          tma_load_2d_weights<ONCE>(dstW, &tmW, fb, kc, n0);
        }
        if (!skip) tma_load_2d(dstW + W_STAGE_BYTES, &tmA, fb, kc, m0);
      }
      __syncwarp();
      if (++s == STAGES) {
        s = 0;
        ph ^= 1u;
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    constexpr uint32_t idesc = make_idesc(TILE_W, BN);
    bool ok = true, ready = false;
    int s = 0;
    uint32_t ph = 0;
    for (int i = 0; i < nkb && ok; ++i) {
      if (!mbar_wait_warp(smem_u32(&full_bar[s]), ph, abortp, ready)) {
        if (status && lane == 0) atomicCAS(status, ST_OK, ST_TIMEOUT_MMA);
        ok = false;
        break;
      }
      if (lane == 0) {
        if (i == 0) timeline_mark(1);                    // first stage complete: activations have arrived
        else if (i == STAGES) timeline_mark(2);          // first stage whose weights were not requested ahead of the wait
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t sW = tiles + s * SL::STAGE_BYTES, empty = smem_u32(&empty_bar[s]);
      if (++s == STAGES) {
        s = 0;
        ph ^= 1u;
      }
      ready = mbar_peek_warp(smem_u32(&full_bar[s]), ph);  // answered while the MMAs below are issued
      if (elect_one()) {
        const uint64_t dW = make_smem_desc(sW);
        const uint64_t dA = make_smem_desc(sW + W_STAGE_BYTES);
#pragma unroll
        for (int k = 0; k < TILE_K / UMMA_K; ++k) {
          // advance 32 bytes (16 bf16) along K inside the swizzle row: +2 in 16-byte units
          umma_bf16(tmem_d, dW + (uint64_t)(2 * k), dA + (uint64_t)(2 * k), idesc, (i > 0 || k > 0) ? 1u : 0u);
        }
        umma_commit(empty);  // stage reusable once these MMAs have read it
        if (i == nkb - 1) umma_commit(smem_u32(&accum_bar));
      }
      __syncwarp();
    }
  }
  __syncwarp();

  // ---------------- epilogue: TMEM -> registers -> global (all eight warps) ----------------
  const bool have = mbar_wait(smem_u32(&accum_bar), 0u, abortp);
  if (!have && threadIdx.x == 0 && status) atomicCAS(status, ST_OK, ST_TIMEOUT_EPI);
  if (threadIdx.x == 0) timeline_mark(3);              // accumulator complete
  // the whole warp must agree before the warp-collective TMEM loads
  bool warp_ok = __all_sync(0xffffffffu, have);
  if (act_out || m_ffn < 0) warp_ok = __syncthreads_and(warp_ok);  // these epilogues exchange data between warps
  if (warp_ok) {
    constexpr int W = BN / 2;
    const int half = (int)threadIdx.x >> 7;
    float* ex = reinterpret_cast<float*>(smem_raw + (tiles - smem_u32(smem_raw)) + half * PlainStage<W>::BYTES);  // the drained ring
    const uint32_t tmem_h = tmem_d + (uint32_t)(half * W);
    const int tl = (int)threadIdx.x & 127, bar = 1 + half, m0h = m0 + half * W;
    if (m_ffn < 0)
      gemm_epilogue<W, ESTIMATE>(tmem_h, ex, tl, bar, m0h, n0, nt, M, N, part, act_out, m_ffn);
    else if (act_out)
      gemm_epilogue<W, SWIGLU>(tmem_h, ex, tl, bar, m0h, n0, nt, M, N, part, act_out, m_ffn);
    else
      gemm_epilogue<W, SLABS>(tmem_h, ex, tl, bar, m0h, n0, nt, M, N, part + (size_t)blockIdx.z * split_stride, act_out, m_ffn);
    if (threadIdx.x == 0) timeline_mark(4);            // this thread's part of the epilogue written
  } else {
    drain_delay();  // gave up: let copies in flight land before shared memory is released
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"((uint32_t)BN) : "memory");
  }
}

// The pair kernel's plain forms.  Slabs leave at the rate of the stores with one group of epilogue warps already (2.8 us for
// 256 rows either way); the staged ones take two.
template <PlainKind KIND>
struct PlainForm {
  __nv_bfloat16* act_out;
  int m_ffn;
  static constexpr int GROUPS = KIND == SLABS ? 1 : 2;
  template <int W>
  static constexpr uint32_t ex_bytes() { return KIND == SLABS ? 0 : PlainStage<W>::BYTES; }
  template <int W>
  struct Shared {};
  template <int W>
  __device__ __forceinline__ void ahead(Shared<W>&, int, int, int) const {}
  template <int W>
  __device__ __forceinline__ void drain(Shared<W>&, uint32_t tmem_d, float* ex, int tl, int bar, int m0, int n0, int tile_y,
                                        int M, int N, float* slab) const {
    gemm_epilogue<W, KIND>(tmem_d, ex, tl, bar, m0, n0, tile_y, M, N, slab, act_out, m_ffn);
  }
};

// ---------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

struct MapKey {
  const void* base;
  uint64_t batch, rows, cols;
  uint32_t box_rows;
  int device;  // a map is encoded in the context of the device that was current
  bool operator==(const MapKey& o) const {
    return base == o.base && batch == o.batch && rows == o.rows && cols == o.cols && box_rows == o.box_rows &&
           device == o.device;
  }
};
struct MapKeyHash {
  size_t operator()(const MapKey& k) const {
    size_t h = std::hash<const void*>()(k.base);
    h ^= std::hash<uint64_t>()(k.rows * 1315423911ull + k.cols + k.batch * 2654435761ull) + 0x9e3779b97f4a7c15ull +
         (h << 6) + (h >> 2);
    return h ^ (k.box_rows * 2654435761u) ^ ((size_t)k.device << 56);
  }
};

bool get_map(const MapKey& key, CUtensorMap* out) {
  static std::unordered_map<MapKey, CUtensorMap, MapKeyHash> cache;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(key);
  if (it != cache.end()) {
    *out = it->second;
    return true;
  }
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) return false;
  const bool three = key.batch > 0;
  cuuint64_t dims[3] = {key.cols, key.rows, three ? key.batch : 1};
  cuuint64_t strides[2] = {key.cols * 2, key.rows * key.cols * 2};
  cuuint32_t box[3] = {(cuuint32_t)TILE_K, key.box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUtensorMap tm;
  CUresult r = enc(&tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, three ? 3 : 2, const_cast<void*>(key.base), dims, strides,
                   box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  if (cache.size() > 8192) cache.clear();
  cache.emplace(key, tm);
  *out = tm;
  return true;
}

// Most stages whose ring fits the 227 KB of shared memory one CTA may use.
constexpr int max_stages(int bn) {
  const int fit = (227 * 1024 - 1024 - 256) / (int)(W_STAGE_BYTES + bn * TILE_K * 2);
  return fit < MAX_STAGES ? fit : MAX_STAGES;
}

template <int BN, bool ONCE>
cudaError_t launch_one(const Launch& L, const CUtensorMap& tmW, const CUtensorMap& tmA, float* part, int M, int N,
                       int num_kb, const GemmPlan& plan, void* act_out, int m_ffn, bool turned) {
  using SL = SmemLayout<BN>;
  static DeviceOnce once;
  cudaError_t e0 = once.run([] {
    return cudaFuncSetAttribute(gemm_bf16_tcgen05_kernel<BN, ONCE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)SL::total(max_stages(BN)));
  });
  if (e0 != cudaSuccess) return e0;
  const int stages = plan.stages < 2 ? 2 : plan.stages > max_stages(BN) ? max_stages(BN) : plan.stages;
  dim3 grid((M + BN - 1) / BN, (N + TILE_W - 1) / TILE_W, plan.S_max);
  cudaError_t e = launch_k(L, gemm_bf16_tcgen05_kernel<BN, ONCE>, grid, dim3(ONE_THREADS), SL::total(stages), tmW, tmA, part, M, N,
                           num_kb, plan.upc, (size_t)M * N, stages, (__nv_bfloat16*)act_out, m_ffn, (int)turned, L.d_status);
  L.count();
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int BN, bool ONCE>
cudaError_t launch_pair(const Launch& L, const CUtensorMap& tmW, const CUtensorMap& tmA, float* part, int M, int N,
                        int num_kb, const GemmPlan& plan, void* act_out, int m_ffn, bool) {
  auto go = [&](auto form, bool staged) {
    return launch_pair_form<BN, ONCE>(L, tmW, tmA, part, M, N, num_kb, plan, form, staged);
  };
  __nv_bfloat16* const act = (__nv_bfloat16*)act_out;
  return m_ffn < 0 ? go(PlainForm<ESTIMATE>{act, m_ffn}, true)
         : act     ? go(PlainForm<SWIGLU>{act, m_ffn}, true)
                   : go(PlainForm<SLABS>{act, m_ffn}, false);
}

}  // namespace

static int current_device() {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess ? dev : -1;
}
bool get_tensor_map_2d(const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows, CUtensorMap* out) {
  return get_map(MapKey{base, 0, rows, cols, box_rows, current_device()}, out);
}
bool get_tensor_map_3d(const void* base, uint64_t batch, uint64_t rows, uint64_t cols, uint32_t box_rows,
                       CUtensorMap* out) {
  return get_map(MapKey{base, batch, rows, cols, box_rows, current_device()}, out);
}

int sm_count() {
  static std::atomic<int> per_device[64];  // zero-initialised: not yet asked
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;  // no device visible (host-only size queries): a B200's count
  const bool tracked = dev >= 0 && dev < 64;
  if (tracked && (v = per_device[dev].load(std::memory_order_relaxed)) > 0) return v;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) return 148;
  if (tracked) per_device[dev].store(v, std::memory_order_relaxed);
  return v;
}

// tuning / test override of the kernel choice: 0 automatic, 1 the pair kernel for unsplit plans with 256-row tiles too,
// -1 the one-tile kernel (see dllm_debug_gemm_plan)
int g_gemm_force_persistent = 0;

int gemm_plan_mode() { return g_gemm_force_persistent; }

Partials make_partials(const float* p, int M, int N, const GemmPlan& plan) {
  return Partials{p, (size_t)M * N, plan.S_max, N};  // every element has S_max slabs
}

// Activation tile and split of the persistent pair kernel, by what bounds it: the pairs work in rounds of whole
// units, a k-block of a unit takes the larger of the issue / tensor time of its tile (0.33 / 0.27 / 0.25 us for 256 /
// 192 / 128 rows) and its bytes' share of the L2 -> SM fabric (12 TB/s over all SMs: 0.40 / 0.35 / 0.30 us when every
// SM is busy), and a split adds slabs that are written and read once more (10 TB/s); epilogues are not in it (2.8 us for
// slabs, 3.9 for SwiGLU, about 6 for rotated and placed rows of a 256-row tile).  Measured with it, B200, us
// (before -> now): 768 x 4096 x 12288 77 -> 63, 768 x 24576 x 4096 120 -> 110, 4096 x 24576 x 4096 614 -> 583, 4096 x
// 4096 x 12288 362 -> 306, 24576 x 4096 x 4096 711 -> 646, 256 x 126464 x 4096 258 -> 221.
static double plan_pair(int M, int N, int K, int max_split, int exact_split, int* bn, int* splits) {
  const int pairs = sm_count() / 2, num_kb = (K + TILE_K - 1) / TILE_K;
  const long n_pairs = (N + 2 * TILE_W - 1) / (2 * TILE_W);
  double best = -1.0;
  for (int BN : {256, 192, 128}) {
    const long tiles = n_pairs * ((M + BN - 1) / BN);
    const double issue = BN == 256 ? 0.33 : BN == 192 ? 0.27 : 0.25, bytes = (TILE_W + BN / 2) * TILE_K * 2.0;
    const int S0 = exact_split > 0 ? exact_split : 1;
    for (int S = S0; S == S0 || (exact_split == 0 && S <= max_split && S * tiles <= pairs && S <= num_kb / 4); ++S) {
      const long units = tiles * S, rounds = (units + pairs - 1) / pairs;
      const double ctas = 2.0 * (units < pairs ? units : pairs), fabric = bytes * ctas / 12.0e6;
      const double us = (double)rounds * ((num_kb + S - 1) / S) * (issue > fabric ? issue : fabric) +
                        (S > 1 ? S * (double)M * N * 8.0 / 10.0e6 : 0.0);
      if (best < 0.0 || us < best) {
        best = us;
        *bn = BN;
        *splits = S;
      }
    }
  }
  return best;
}

double gemm_pair_us(int M, int N, int K) {
  int bn, splits;
  return plan_pair(M, N, K, 16, 0, &bn, &splits);
}

// Tile shape, ring depth and split-K factor, from sweeps on B200.  Up to 128 activation rows the product is bound by
// streaming W: one CTA per weight tile, k ranges split until at least one CTA per SM (two with 128-row tiles) streams
// weights.  Above that the activation tile's trips through the L2 -> SM fabric bound it: CTA pairs.
GemmPlan plan_gemm_bf16(int M, int N, int K, int force_split, int force_stages, int force_bn, int force_pair,
                        int force_persistent) {
  GemmPlan p;
  const int sms = sm_count();
  const long n_tiles = (N + TILE_W - 1) / TILE_W;
  const int exact = force_split < 0 ? -force_split : 0;
  if (exact) force_split = 0;
  if (force_persistent == 0) force_persistent = g_gemm_force_persistent;
  p.num_kb = (K + TILE_K - 1) / TILE_K;
  p.BN = M <= 32 ? 32 : M <= 64 ? 64 : M <= 256 ? 128 : 256;
  p.pair = 0;
  int S = 0;
  // Pairs, for weight matrices of 2 M elements or more: up to 128 rows they would take 0.99-1.25 of the one-tile kernel's
  // time (B200, isolated, ten projections of 65 / 96 / 128 rows; only the LM head's 126464 x 4096 0.95-0.97).  Smaller
  // weights are over before a cluster launch pays at few rows (144..256 rows: 5.9-9.4 us against 6.9-10.9 on pairs); pairs
  // take them where the 256-row tiles need a second wave (8192 x 2560 x 448 35.6 -> 30.1 us, 12288 x 512 x 3584 53 -> 38)
  // or where one wave of them would be split for many rows, whose slabs cost more (1024 x 1792 x 1024 19.1 -> 9.5,
  // 4096 x 512 x 3584 30 -> 22; at 444 rows 11.3 against 11.5).
  const bool many_rows = ((M + 255) / 256) * n_tiles > sms || (M >= 768 && K >= 1024);
  if (force_pair == 0 && force_bn == 0 && force_split <= 1 && M > 128 && ((long)N * K >= 1L << 21 || many_rows)) {
    p.wide = true;
    plan_pair(M, N, K, force_split == 1 ? 1 : 16, exact, &p.BN, &S);
    p.pair = force_persistent >= 0;
    if (!p.pair && p.BN == 192) p.BN = 128;   // the one-tile kernel on the same splits: the same sums, the same slabs
  } else if (force_pair == 0 && force_bn == 0 && force_split == 0 && M > 64 && M <= 128 && n_tiles * ((M + 63) / 64) <= sms) {
    // 65..128 rows against few weight tiles (the product will be split): two 64-row tiles per weight tile put
    // twice the CTAs on the weight stream (128 x 4096 x 4096: 14.9 against 17.8 us, 128 x 4096 x 3584: 10.0
    // against 11.8 us; with many weight tiles the 128-row tile stays: every weight tile crosses the fabric once)
    p.BN = 64;
  } else if (force_pair == 0 && force_bn == 0 && force_split <= 1 && M > 128 && M <= 1024) {
    // a small weight: the tile halved where that still is one wave of CTAs, so more and shorter ones (448-wide bf16 model,
    // two layers: response refresh of 144 rows 93.2 -> 79.0 us, of 576 rows 126.2 -> 104.0, of 360 rows 118 -> 95)
    const int half = M <= 256 ? 64 : 128;
    if (n_tiles * ((M + half - 1) / half) <= sms) p.BN = half;
  }
  if (force_bn == 32 || force_bn == 64 || force_bn == 128 || force_bn == 192 || force_bn == 256) p.BN = force_bn;
  if (force_pair > 0 || force_bn == 192 || (p.BN == 256 && force_persistent > 0 && force_split <= 1)) p.pair = p.BN >= 64;
  p.stages = force_stages > 0 ? force_stages : p.pair ? MAX_STAGES : (p.BN == 128 ? 3 : 4);
  p.m_tiles = (M + p.BN - 1) / p.BN;
  const long tiles = (long)p.m_tiles * n_tiles;
  if (S == 0) {
    // every split adds a slab the consumer has to read: with few activation rows
    // one wave of CTAs is enough, with 128-row tiles two CTAs per SM pay off
    // (two CTAs per SM also for 64-row tiles when there are two or more of them per weight tile)
    const bool two_per_sm = !p.pair && (p.BN == 128 || (p.BN == 64 && p.m_tiles > 1));
    S = two_per_sm ? (int)(2L * sms / tiles) : (int)((sms + tiles - 1) / tiles);  // all CTAs resident at once
    const int max_s = p.num_kb / 4 > 1 ? p.num_kb / 4 : 1;
    if (S > max_s) S = max_s;
    if (S < 1) S = 1;
  }
  if (exact || force_split > 0) S = std::min(exact ? exact : force_split, p.num_kb);
  // weight matrices that no L2 keeps until the next step (smaller ones may: a small model's layers stay there)
  p.w_stream = (long)N * K >= 8L << 20;
  p.upc = (p.num_kb + S - 1) / S;                 // k-blocks per split
  p.S_max = (p.num_kb + p.upc - 1) / p.upc;       // no empty split
  return p;
}

cudaError_t launch_gemm_bf16(const Launch& L, const void* A, const void* W, float* part, int M, int N, int K,
                             const GemmPlan& plan, const char** err, void* act_out, int m_ffn) {
  static const char* e_shape = "bf16 GEMM needs K % 8 == 0 and 16-byte aligned operands";
  static const char* e_map = "cuTensorMapEncodeTiled failed or is unavailable";
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (K <= 0 || (K & 7) || ((uintptr_t)A & 15) || ((uintptr_t)W & 15)) {
    if (err) *err = e_shape;
    return cudaErrorInvalidValue;
  }
  if (!act_out && m_ffn < 0 && (plan.S_max != 1 || ((uintptr_t)part & 15))) {
    if (err) *err = "the estimate epilogue needs an unsplit plan";
    return cudaErrorInvalidValue;
  }
  if (act_out && (plan.S_max != 1 || N != 2 * m_ffn || (m_ffn & 63) || ((uintptr_t)act_out & 7))) {
    if (err) *err = "the SwiGLU epilogue needs an unsplit plan and d_ffn % 64 == 0";
    return cudaErrorInvalidValue;
  }
  CUtensorMap tmW, tmA;
  if (!get_tensor_map_2d(W, (uint64_t)N, (uint64_t)K, TILE_W, &tmW) ||
      !get_tensor_map_2d(A, (uint64_t)M, (uint64_t)K, (uint32_t)(plan.pair ? plan.BN / 2 : plan.BN), &tmA)) {
    if (err) *err = e_map;
    return cudaErrorInvalidValue;
  }
  const int num_kb = (K + TILE_K - 1) / TILE_K;
  // evict-first weights where one activation tile reads them (128-row tiles of the one-CTA kernel gained nothing)
  const bool once = plan.w_stream && plan.m_tiles == 1;
  // Gate / up weights whose rows lie a multiple of 8 KB apart, streamed once by unsplit one-tile CTAs: all CTAs in step read
  // the same few address bits of every row, and every other pair of tiles half a row ahead spreads them.  B200, us per layer
  // of adaptive steps of 3 / 32 / 64 / 115 rows: 4096 wide, d_ffn 12288 102.1 / 105.9 / 116.4 / 126.9 -> 100.3 / 103.9 / 114.4 /
  // 124.8, d_ffn 14336 103.8 / 104.9 / 113.6 / 122.0 -> 99.1 / 102.6 / 111.2 / 120.2, d_ffn 16384 2 % faster; 8192 wide (16 KB
  // rows) even.  Not where the product is split or has other row lengths (O and down of the same models even, a down product of
  // 20480 long rows 1.5 % slower, gate / up of 7 KB rows 1.5 % slower), nor on CTA pairs (2 % slower); other turns and
  // four or eight starting points gave less.  Not for products whose sums are the same in every kind of step.
  const bool turned = act_out && !plan.pair && !plan.wide && plan.m_tiles == 1 && plan.BN <= 128 && plan.w_stream && K % 4096 == 0;
#define DLLM_LAUNCH(kind, bn, may)                                                                          \
  ((may) && once ? launch_##kind<bn, may>(L, tmW, tmA, part, M, N, num_kb, plan, act_out, m_ffn, turned)    \
                 : launch_##kind<bn, false>(L, tmW, tmA, part, M, N, num_kb, plan, act_out, m_ffn, turned))
  if (plan.pair) {
    switch (plan.BN) {
      case 64: return DLLM_LAUNCH(pair, 64, false);
      case 128: return DLLM_LAUNCH(pair, 128, false);
      case 192: return DLLM_LAUNCH(pair, 192, true);
      default: return DLLM_LAUNCH(pair, 256, true);
    }
  }
  switch (plan.BN) {
    case 32: return DLLM_LAUNCH(one, 32, true);
    case 64: return DLLM_LAUNCH(one, 64, true);
    case 128: return DLLM_LAUNCH(one, 128, false);
    default: return DLLM_LAUNCH(one, 256, false);
  }
#undef DLLM_LAUNCH
}

}  // namespace dllm

namespace dllm {
cudaError_t set_debug_skip_act_load(int enable) {
  const int v = enable != 0;
  return cudaMemcpyToSymbol(g_debug_skip_act_load, &v, sizeof v);
}
}  // namespace dllm

extern "C" dllm_status dllm_debug_gemm_plan(int persistent) {
  if (persistent < -1 || persistent > 1) {
    dllm::set_last_error("dllm_debug_gemm_plan: -1, 0 or 1");
    return DLLM_INVALID_ARG;
  }
  dllm::g_gemm_force_persistent = persistent;
  return DLLM_OK;
}

DLLM_TIMELINE_HOOKS(gemm_tcgen05)
DLLM_WAIT_LIMIT_HOOK(gemm_tcgen05)
