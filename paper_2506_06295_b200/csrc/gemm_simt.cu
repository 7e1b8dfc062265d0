// C[M,N] (fp32) = A[M,K] * W[N,K]^T on the plain fp32 ALUs.
//
// This is the GEMM of the fp32 mode (the tiny configuration asks for 1e-4 relative error, which TF32 tensor cores do
// not give) and the independent cross-check for the tensor-core kernels in tests.
//
// The fp32 models are small, so a product is bound by latency: a loop over the whole k range with two block barriers per
// 16 k took 12 us at K = 256 and 30 us at K = 688 for 50 MFLOP.  Here the eight warps of a CTA take DIFFERENT 32-wide
// k-chunks (warp w the chunks w, w + 8, ...) of a small output tile, each with a shared-memory buffer of its own and no
// barrier in the loop: K = 256 is one chunk per warp, all of whose loads are in flight together, and the weight half of
// the first chunk is requested ahead of the dependency wait.  The eight partial tiles are added in warp order at the end.
// An element's sum does not depend on the tile (same chunks, same order), so rows are bit-identical whatever the number
// of rows in the launch.
#include "internal.h"

namespace dllm {

namespace {

constexpr int SG_WARPS = 8, SG_K = 32, SG_LD = SG_K + 4;  // row stride in shared memory: 16-byte aligned, 4 banks apart

// four consecutive elements from column k of a row (zero past K); vec: the row allows one vector load
template <typename T>
__device__ __forceinline__ float4 load4(const T* row, bool in, int k, int K, bool vec) {
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!in || k >= K) return v;
  if (vec) {
    if constexpr (sizeof(T) == 4) {
      v = __ldcg(reinterpret_cast<const float4*>(row + k));
    } else {
      const uint2 u = __ldcg(reinterpret_cast<const uint2*>(row + k));
      v = make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xFFFF0000u), __uint_as_float(u.y << 16),
                      __uint_as_float(u.y & 0xFFFF0000u));
    }
  } else {
    float t[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (k + j < K) t[j] = to_f32<T>(row[k + j]);
    v = make_float4(t[0], t[1], t[2], t[3]);
  }
  return v;
}

// Tile of 4 TM rows x 8 TN columns; a lane holds TM x TN outputs (rows 4 i + lane / 8, columns 8 j + lane % 8).
template <typename T, int TM, int TN>
__global__ void __launch_bounds__(SG_WARPS * 32)
    gemm_simt_kernel(const T* __restrict__ A, const T* __restrict__ W, float* __restrict__ C, int M, int N, int K, bool vec) {
  constexpr int BM = 4 * TM, BN = 8 * TN;
  extern __shared__ __align__(16) float sg_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* As = sg_smem + warp * (BM + BN) * SG_LD;
  float* Ws = As + BM * SG_LD;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int lr = lane >> 3, lk = (lane & 7) * 4;            // loads: four rows per pass, 8 lanes x 4 k per row
  const int chunks = (K + SG_K - 1) / SG_K;
  // chunks of a warp whose operands are on their way at once: small tiles have the registers for three, and less arithmetic
  // per chunk than a load takes (K = 688 is three chunks of most warps: the tiny configuration's generation 516 -> 499 us)
  constexpr int DEPTH = TM * TN <= 4 ? 3 : 1;
  float4 ra[DEPTH][TM], rw[DEPTH][2 * TN];
  auto load_w = [&](int d, int c) {
#pragma unroll
    for (int i = 0; i < 2 * TN; ++i)
      rw[d][i] = load4(W + (size_t)(n0 + 4 * i + lr) * K, n0 + 4 * i + lr < N, c * SG_K + lk, K, vec);
  };
  auto load_a = [&](int d, int c) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
      ra[d][i] = load4(A + (size_t)(m0 + 4 * i + lr) * K, m0 + 4 * i + lr < M, c * SG_K + lk, K, vec);
  };
#pragma unroll
  for (int d = 0; d < DEPTH; ++d)
    if (warp + d * SG_WARPS < chunks) load_w(d, warp + d * SG_WARPS);   // weights are written by no kernel
  pdl_wait();
  pdl_trigger();
#pragma unroll
  for (int d = 0; d < DEPTH; ++d)
    if (warp + d * SG_WARPS < chunks) load_a(d, warp + d * SG_WARPS);
  float acc[TM][TN] = {};
  const int ly = lane >> 3, lx = lane & 7;
  for (int c0 = warp; c0 < chunks; c0 += DEPTH * SG_WARPS) {
#pragma unroll
    for (int d = 0; d < DEPTH; ++d) {
      const int c = c0 + d * SG_WARPS;
      if (c >= chunks) break;
      __syncwarp();
#pragma unroll
      for (int i = 0; i < TM; ++i) *reinterpret_cast<float4*>(As + (4 * i + lr) * SG_LD + lk) = ra[d][i];
#pragma unroll
      for (int i = 0; i < 2 * TN; ++i) *reinterpret_cast<float4*>(Ws + (4 * i + lr) * SG_LD + lk) = rw[d][i];
      __syncwarp();
      if (c + DEPTH * SG_WARPS < chunks) {                    // the warp's next chunk travels under this one's arithmetic
        load_w(d, c + DEPTH * SG_WARPS);
        load_a(d, c + DEPTH * SG_WARPS);
      }
#pragma unroll
      for (int k = 0; k < SG_K; k += 4) {
        float4 a[TM], w[TN];
#pragma unroll
        for (int i = 0; i < TM; ++i) a[i] = *reinterpret_cast<const float4*>(As + (4 * i + ly) * SG_LD + k);
#pragma unroll
        for (int j = 0; j < TN; ++j) w[j] = *reinterpret_cast<const float4*>(Ws + (8 * j + lx) * SG_LD + k);
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN; ++j) {
            acc[i][j] = fmaf(a[i].x, w[j].x, acc[i][j]);
            acc[i][j] = fmaf(a[i].y, w[j].y, acc[i][j]);
            acc[i][j] = fmaf(a[i].z, w[j].z, acc[i][j]);
            acc[i][j] = fmaf(a[i].w, w[j].w, acc[i][j]);
          }
      }
    }
  }
  // partial tiles through shared memory (every warp is done with the buffers), added in warp order
  static_assert(BM * BN <= (BM + BN) * SG_LD, "a warp's partial tile must fit its buffer");
  __syncwarp();
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) As[(4 * i + ly) * BN + 8 * j + lx] = acc[i][j];
  __syncthreads();
  for (int e = threadIdx.x; e < BM * BN; e += SG_WARPS * 32) {
    const int m = m0 + e / BN, n = n0 + e % BN;
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < SG_WARPS; ++w) s += sg_smem[w * (BM + BN) * SG_LD + e];
    if (m < M && n < N) C[(size_t)m * N + n] = s;
  }
}

template <typename T, int TM, int TN>
void launch_tile(const Launch& L, const void* A, const void* W, float* C, int M, int N, int K) {
  constexpr int BM = 4 * TM, BN = 8 * TN, SMEM = SG_WARPS * (BM + BN) * SG_LD * 4;
  static DeviceOnce once;
  if (once.run([] { return cudaFuncSetAttribute(gemm_simt_kernel<T, TM, TN>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM); }) !=
      cudaSuccess)
    return;  // the error stays for the caller's cudaGetLastError
  const bool vec = K % 4 == 0 && (((uintptr_t)A | (uintptr_t)W) & (4 * sizeof(T) - 1)) == 0;
  // a grid is at most 65535 high: millions of rows take several launches (a third grid dimension in the kernel's indices
  // cost the tiny configuration's generations up to 3 %)
  constexpr int MOST = 65535 * BM;
  for (long r = 0; r < M; r += MOST) {
    const int rows = (int)(M - r < MOST ? M - r : MOST);
    launch_k(L, gemm_simt_kernel<T, TM, TN>, dim3((N + BN - 1) / BN, (rows + BM - 1) / BM), dim3(SG_WARPS * 32), SMEM,
             (const T*)A + (size_t)r * K, (const T*)W, C + (size_t)r * N, rows, N, K, vec);
  }
}

}  // namespace

void launch_gemm_simt(const Launch& L, int dtype, const void* A, const void* W, float* C, int M, int N, int K) {
  if (M <= 0 || N <= 0) return;
  // 32 x 64 tiles (half the shared-memory reads per product) once they are two per SM, 16 x 32 below: more CTAs, and a
  // shorter chain in each
  const bool big = (long)((M + 31) / 32) * ((N + 63) / 64) >= 2L * sm_count();
  // 8 x 16 tiles where 16 x 32 ones would leave half of the SMs idle: a quarter of the arithmetic in each warp's chain (in the
  // replayed step of the tiny configuration, 8 rows: 256 x 256 2.8 -> 2.0 us, 1376 x 256 2.9 -> 2.0, 256 x 688 5.7 -> 3.9)
  const bool small = (long)((M + 15) / 16) * ((N + 31) / 32) * 2 <= sm_count();
  auto go = [&](auto t) {
    using T = decltype(t);
    if (big) launch_tile<T, 8, 8>(L, A, W, C, M, N, K);
    else if (small) launch_tile<T, 2, 2>(L, A, W, C, M, N, K);
    else launch_tile<T, 4, 4>(L, A, W, C, M, N, K);
  };
  if (dtype == 0) go(float{});
  else go(__nv_bfloat16{});
  L.count();
}

}  // namespace dllm

DLLM_TIMELINE_HOOKS(gemm_simt)
