// Projections of more than 128 rows that put their bf16 rows where they belong: into a cache tensor (V, AttnOut, FFNOut)
// or, for the stacked Q / K (/ V) product, rotated into the query buffer and the K cache (and the V cache).
//
// Without a split k range the fp32 result of a projection is final, and writing it for a row-wise kernel to round and
// scatter costs 8 bytes per element of traffic and a launch.  Here the pair kernel's epilogue rounds it to what the cache
// holds: the same bits.  The accumulator goes through shared memory 16 activation rows at a time, the next ones
// on their way out of tensor memory meanwhile; 16 threads per row take
// the columns 4 q .. 4 q + 3 and the same 64 further, which are pairs of the rotation (32 further within a block of 64
// columns for head_dim 64; a tile holds whole heads): 128 coalesced bytes per half warp.  Rows' places are worked out
// before the accumulator is complete, and a trip's rotation values are requested one trip ahead (fetched where they were
// used they came from L2 or memory eight times behind the main loop: 12 us for a 256-row tile).  LLaDA-8B shape, full step
// 11579 -> 11243 us with two groups of epilogue warps and the per-row arithmetic reduced to one multiply-add per pointer.
//
// VERIFY: V of all response rows of an adaptive step, compared (Eq. 6) with the rows it overwrites: a thread's eight columns,
// the sixteen threads of a row, one triple of sums per row and 128 columns for a small merge.  Without it the fp32 result
// went to memory and back for a kernel that read it beside the old rows (8192 rows of the LLaDA-8B shape: 54 us per layer).
#include <type_traits>

#include "gemm_pair.cuh"

namespace dllm {

namespace {

enum RowKind { PLACE, HEADS, VERIFY };
template <RowKind KIND>
struct RowForm {
  RowOut o;
  static constexpr bool QKV = KIND == HEADS;
  static constexpr int GROUPS = 2;
  // rows per trip; floats per staged row (no padding: a quarter warp's 16-byte reads lie in one row)
  static constexpr int CH = 16, EXS = 128;
  template <int W>
  static constexpr uint32_t ex_bytes() { return CH * EXS * 4; }
  // a row's place: {row of the query buffer, row of the K / V caches, position} or its address in the cache tensor
  using Place = typename std::conditional<QKV, int4, unsigned long long>::type;
  template <int W>
  struct Shared {
    Place row[W];
  };
  template <int W>
  __device__ __forceinline__ void ahead(Shared<W>& s, int tl, int m0, int M) const {
#pragma unroll 1
    for (int i = tl; i < W && m0 + i < M; i += 128) {
      const int c = o.act ? __ldcg(o.act + m0 + i) : o.base + m0 + i;
      if constexpr (QKV) {
        int b, pos;
        carried_to_pos(c, o.g, b, pos);
        const int at = b * o.g.n + pos;
        s.row[i] = make_int4(o.q_by_slot ? at : m0 + i, at, pos, 0);
      } else {
        s.row[i] = m0 + i < o.slab_rows ? reinterpret_cast<unsigned long long>(o.slab + (size_t)(m0 + i) * o.g.d)
                                        : reinterpret_cast<unsigned long long>(o.rows.row<__nv_bfloat16>(c, o.g));
      }
    }
  }
  static __device__ __forceinline__ uint2 pack(float4 f) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(f.x, f.y), b = __floats2bfloat162_rn(f.z, f.w);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
  }
  static __device__ __forceinline__ float4 lo4(float4 l, float4 h, float4 c, float4 t) {
    return make_float4(rope_lo(l.x, h.x, c.x, t.x), rope_lo(l.y, h.y, c.y, t.y), rope_lo(l.z, h.z, c.z, t.z),
                       rope_lo(l.w, h.w, c.w, t.w));
  }
  static __device__ __forceinline__ float4 hi4(float4 l, float4 h, float4 c, float4 t) {
    return make_float4(rope_hi(l.x, h.x, c.x, t.x), rope_hi(l.y, h.y, c.y, t.y), rope_hi(l.z, h.z, c.z, t.z),
                       rope_hi(l.w, h.w, c.w, t.w));
  }
  template <int W>
  __device__ __forceinline__ void drain(Shared<W>& s, uint32_t tmem_d, float* ex, int tl, int bar, int m0, int n0, int tile_y,
                                        int M, int N, float*) const {
    if (m0 >= M) return;   // uniform across the group
    const int rows = min(W, M - m0);
    const uint32_t tmem_w = tmem_d + ((uint32_t)(tl >> 5) << 21);
    const int q = tl & 15, rsub = tl >> 4;
    int lo = 4 * q, hi = 64 + 4 * q;
    if (QKV && o.hd == 64) {
      lo = (q >> 3) * 64 + (q & 7) * 4;
      hi = lo + 32;
    }
    // What depends on the thread's two column pieces alone is settled here; a trip's instructions per row are what an epilogue
    // spends its time on (one warp per scheduler and group, each waiting for its own last result).
    const int nlo = n0 + lo, nhi = n0 + hi;
    const bool rot = QKV && nlo < o.dq + o.dkv, vlo = nlo < N, vhi = nhi < N;
    // V rows before v_from are there already; the two pieces of a rotated pair lie in one head, others each in their own place
    const int lo_from = QKV && nlo >= o.dq + o.dkv ? o.v_from - m0 : 0, hi_from = QKV && nhi >= o.dq + o.dkv ? o.v_from - m0 : 0;
    auto column = [&](int n) {
      return n < o.dq ? o.q + n : n < o.dq + o.dkv ? o.k + (n - o.dq) : o.v + (n - o.dq - o.dkv);
    };
    __nv_bfloat16 *const blo = QKV ? column(nlo) : nullptr, *const bhi = QKV ? column(nhi) : nullptr;
    const bool qlo = nlo < o.dq, qhi = nhi < o.dq;
    const unsigned slo = qlo ? o.dq : o.dkv, shi = qhi ? o.dq : o.dkv;   // elements from row to row
    const float* const tab = QKV ? o.rope_tab + nlo % o.hd : nullptr;
    constexpr int U = CH / 8;
    float4 cs[U], sn[U];
    uint2 olo[U], ohi[U];   // V-verify: the rows' old values
    Place at[U];
    auto fetch = [&](int c0) {   // places and rotation values of this thread's rows c0 + rsub + 8 u (the last one past the end)
#pragma unroll
      for (int u = 0; u < U; ++u) {
        at[u] = s.row[min(c0 + rsub + 8 * u, rows - 1)];
        if constexpr (QKV) {
          if (rot) {
            const float* t = tab + (size_t)((unsigned)at[u].z * (unsigned)o.hd);
            cs[u] = *reinterpret_cast<const float4*>(t);
            sn[u] = *reinterpret_cast<const float4*>(t + (o.hd >> 1));
          }
        }
        if constexpr (KIND == VERIFY) {
          const __nv_bfloat16* p = reinterpret_cast<const __nv_bfloat16*>(at[u]);
          olo[u] = vlo ? __ldcg(reinterpret_cast<const uint2*>(p + nlo)) : make_uint2(0, 0);
          ohi[u] = vhi ? __ldcg(reinterpret_cast<const uint2*>(p + nhi)) : make_uint2(0, 0);
        }
      }
    };
    fetch(0);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    auto sync = [&] { group_sync(bar); };
    uint32_t r[CH];
    tmem_ld16(tmem_w, r);
    tmem_ld16_wait(r);
#pragma unroll 1
    for (int c0 = 0; c0 < rows; c0 += CH) {
#pragma unroll
      for (int j = 0; j < CH; ++j) ex[j * EXS + tl] = __uint_as_float(r[j]);
      sync();
      tmem_ld16(tmem_w + (uint32_t)min(c0 + CH, W - CH), r);   // the next trip's rows (again the last ones in the last)
      float4 a[U], b[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float* row = ex + (rsub + 8 * u) * EXS;
        a[u] = *reinterpret_cast<const float4*>(row + lo);
        b[u] = *reinterpret_cast<const float4*>(row + hi);
      }
      sync();                                                  // read: the staging is free for the next trip
      uint2 plo[U], phi[U];
      __nv_bfloat16 *dlo[U], *dhi[U];
      unsigned long long raw_at[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        plo[u] = pack(rot ? lo4(a[u], b[u], cs[u], sn[u]) : a[u]);
        phi[u] = pack(rot ? hi4(a[u], b[u], cs[u], sn[u]) : b[u]);
        if constexpr (QKV) {
          dlo[u] = blo + (unsigned long long)(unsigned)(qlo ? at[u].x : at[u].y) * slo;
          dhi[u] = bhi + (unsigned long long)(unsigned)(qhi ? at[u].x : at[u].y) * shi;
        } else {
          raw_at[u] = at[u];
          dlo[u] = reinterpret_cast<__nv_bfloat16*>(at[u]) + nlo;
          dhi[u] = reinterpret_cast<__nv_bfloat16*>(at[u]) + nhi;
        }
      }
      if constexpr (KIND == VERIFY) {
        // Eq. 6 on what the cache will hold: this thread's eight columns, then the row's sixteen threads
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t nw[4] = {plo[u].x, plo[u].y, phi[u].x, phi[u].y}, od[4] = {olo[u].x, olo[u].y, ohi[u].x, ohi[u].y};
          float dot = 0.f, na = 0.f, nb = 0.f;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const bool used = i < 4 ? vlo : vhi;
            const float x = used ? __uint_as_float(i & 1 ? nw[i >> 1] & 0xFFFF0000u : nw[i >> 1] << 16) : 0.f;
            const float y = __uint_as_float(i & 1 ? od[i >> 1] & 0xFFFF0000u : od[i >> 1] << 16);
            if (o.metric == 0) {
              dot += x * y;
              na += x * x;
              nb += y * y;
            } else {
              const float df = x - y;
              dot += df * df;
            }
          }
#pragma unroll
          for (int x = 8; x > 0; x >>= 1) {
            dot += __shfl_xor_sync(0xffffffffu, dot, x);
            na += __shfl_xor_sync(0xffffffffu, na, x);
            nb += __shfl_xor_sync(0xffffffffu, nb, x);
          }
          const int row = c0 + rsub + 8 * u;
          if (q == 0 && row < rows) o.verify[(size_t)(m0 + row) * ((N + TILE_W - 1) / TILE_W) + tile_y] = make_float4(dot, na, nb, 0.f);
        }
      }
      fetch(c0 + CH);
      const int stored = KIND == VERIFY && o.keep_rows ? 0 : rows;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int row = c0 + rsub + 8 * u;
        if constexpr (KIND == PLACE) {
          if (m0 + row < o.slab_rows) {   // (their columns 4 q .. and 64 further, as the others')
            float* const raw = reinterpret_cast<float*>(raw_at[u]);
            if (vlo && row < stored) *reinterpret_cast<float4*>(raw + nlo) = a[u];
            if (vhi && row < stored) *reinterpret_cast<float4*>(raw + nhi) = b[u];
            continue;
          }
        }
        if (vlo && row < stored && row >= lo_from) *reinterpret_cast<uint2*>(dlo[u]) = plo[u];
        if (vhi && row < stored && row >= hi_from) *reinterpret_cast<uint2*>(dhi[u]) = phi[u];
      }
      tmem_ld16_wait(r);   // in the trip that requested them: the compiler may move what it carries round the loop
    }
    sync();   // the rows' places are free
  }
};

}  // namespace

cudaError_t launch_gemm_rows(const Launch& L, const void* A, const void* W, int M, int N, int K, const GemmPlan& plan,
                             const RowOut& out, const char** err) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (K <= 0 || (K & 7) || (N & 3) || ((uintptr_t)A & 15) || ((uintptr_t)W & 15) || !plan.pair || plan.S_max != 1) {
    if (err) *err = "row epilogues need an unsplit pair plan, K % 8 == 0, N % 4 == 0 and 16-byte aligned operands";
    return cudaErrorInvalidValue;
  }
  CUtensorMap tmW, tmA;
  if (!get_tensor_map_2d(W, (uint64_t)N, (uint64_t)K, TILE_W, &tmW) ||
      !get_tensor_map_2d(A, (uint64_t)M, (uint64_t)K, (uint32_t)(plan.BN / 2), &tmA)) {
    if (err) *err = "cuTensorMapEncodeTiled failed or is unavailable";
    return cudaErrorInvalidValue;
  }
  const int num_kb = (K + TILE_K - 1) / TILE_K;
  const bool once = plan.w_stream && plan.m_tiles == 1;
  auto go = [&](auto form) {
    switch (plan.BN) {
      case 128: return launch_pair_form<128, false>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true);
      case 192: return once ? launch_pair_form<192, true>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true)
                            : launch_pair_form<192, false>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true);
      case 256: return once ? launch_pair_form<256, true>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true)
                            : launch_pair_form<256, false>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true);
      default: return cudaErrorInvalidValue;
    }
  };
  return out.qkv ? go(RowForm<HEADS>{out}) : out.verify ? go(RowForm<VERIFY>{out}) : go(RowForm<PLACE>{out});
}

}  // namespace dllm

DLLM_TIMELINE_HOOKS(gemm_rows)
DLLM_WAIT_LIMIT_HOOK(gemm_rows)
