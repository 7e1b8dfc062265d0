// Projections of more than 128 rows that put their bf16 rows where they belong: into a cache tensor (V, AttnOut, FFNOut)
// or, for the stacked Q / K (/ V) product, rotated into the query buffer and the K cache (and the V cache).
//
// Without a split k range the fp32 result of a projection is final, and writing it for a row-wise kernel to round and
// scatter costs 8 bytes per element of traffic and a launch.  Here the pair kernel's epilogue rounds it to what the cache
// holds: the same bits.  The accumulator goes through shared memory 16 activation rows at a time, the next
// ones on their way out of tensor memory meanwhile; 16 threads per row take
// the columns 4 q .. 4 q + 3 and the same 64 further, which are pairs of the rotation (32 further within a block of 64
// columns for head_dim 64; a tile holds whole heads): 128 coalesced bytes per half warp.  Rows' places are worked out
// before the accumulator is complete, and a trip's rotation values are requested one trip ahead (fetched where they were
// used they came from L2 or memory eight times behind the main loop: 12 us for a 256-row tile).
#include "gemm_pair.cuh"

namespace dllm {

namespace {

struct RowForm {
  RowOut o;
  static constexpr int CH = 16, EXS = 132;   // rows per trip; floats per staged row (16-byte aligned, rows 4 banks apart)
  static constexpr uint32_t EX_BYTES = 2 * CH * EXS * 4;
  template <int BN>
  struct Shared {
    int2 row[BN];   // cache rows: {address}; Q / K / V: {row of the K / V caches, position}
  };
  template <int BN>
  __device__ __forceinline__ void ahead(Shared<BN>& s, int tl, int m0, int M) const {
#pragma unroll 1
    for (int i = tl; i < BN && m0 + i < M; i += 128) {
      const int c = o.act ? __ldcg(o.act + m0 + i) : o.base + m0 + i;
      if (o.qkv) {
        int b, pos;
        carried_to_pos(c, o.g, b, pos);
        s.row[i] = make_int2(b * o.g.n + pos, pos);
      } else {
        const unsigned long long a = reinterpret_cast<unsigned long long>(o.rows.row<__nv_bfloat16>(c, o.g));
        s.row[i] = make_int2((int)(unsigned)a, (int)(unsigned)(a >> 32));
      }
    }
  }
  static __device__ __forceinline__ uint2 pack(float4 f) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(f.x, f.y), b = __floats2bfloat162_rn(f.z, f.w);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
  }
  template <int BN>
  __device__ __forceinline__ void drain(Shared<BN>& s, uint32_t tmem_d, float* ex, int tl, int m0, int n0, int, int M, int N,
                                        float*) const {
    const uint32_t tmem_w = tmem_d + ((uint32_t)(tl >> 5) << 21);
    const int q = tl & 15, rsub = tl >> 4;
    int lo = 4 * q, hi = 64 + 4 * q;
    if (o.qkv && o.hd == 64) {
      lo = (q >> 3) * 64 + (q & 7) * 4;
      hi = lo + 32;
    }
    const int nlo = n0 + lo, nhi = n0 + hi;
    const bool rot = o.qkv && nlo < o.dq + o.dkv, vlo = nlo < N, vhi = nhi < N;
    const int lo_from = o.qkv && nlo >= o.dq + o.dkv ? o.v_from : 0, hi_from = o.qkv && nhi >= o.dq + o.dkv ? o.v_from : 0;
    // the two pieces of a rotated pair lie in one head; otherwise each has a place of its own
    auto column = [&](int n) {
      return n < o.dq ? o.q + n : n < o.dq + o.dkv ? o.k + (n - o.dq) : o.v + (n - o.dq - o.dkv);
    };
    __nv_bfloat16 *blo = column(nlo), *bhi = column(nhi);
    constexpr int U = CH / 8;
    float4 cs[U], sn[U];
    auto fetch = [&](int c0) {   // rotation values of this thread's rows c0 + rsub + 8 u
      if (!rot) return;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int row = c0 + rsub + 8 * u;
        if (row < BN && m0 + row < M) {
          const float* tab = o.rope_tab + (size_t)s.row[row].y * o.hd + nlo % o.hd;
          cs[u] = *reinterpret_cast<const float4*>(tab);
          sn[u] = *reinterpret_cast<const float4*>(tab + (o.hd >> 1));
        }
      }
    };
    fetch(0);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    auto landed = [&](uint32_t (&r)[CH], float* stage) {   // the rows on their way out of tensor memory -> staging
      asm volatile("tcgen05.wait::ld.sync.aligned;"
                   : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
                     "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])::"memory");
#pragma unroll
      for (int j = 0; j < CH; ++j) stage[j * EXS + tl] = __uint_as_float(r[j]);
    };
    uint32_t r[CH];
    tmem_ld16(tmem_w, r);
    landed(r, ex);
    asm volatile("bar.sync 1, 128;" ::: "memory");
#pragma unroll 1
    for (int c0 = 0; c0 < BN && m0 + c0 < M; c0 += CH) {
      const float* cur = ex + (c0 & CH) / CH * (CH * EXS);
      tmem_ld16(tmem_w + (uint32_t)min(c0 + CH, BN - CH), r);   // the next trip's rows (again the last ones in the last)
      uint2 plo[U], phi[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float* row = cur + (rsub + 8 * u) * EXS;
        float4 a = *reinterpret_cast<const float4*>(row + lo), b = *reinterpret_cast<const float4*>(row + hi);
        if (rot) {
          const float4 l = a, h = b, c = cs[u], t = sn[u];
          a = make_float4(rope_lo(l.x, h.x, c.x, t.x), rope_lo(l.y, h.y, c.y, t.y), rope_lo(l.z, h.z, c.z, t.z),
                          rope_lo(l.w, h.w, c.w, t.w));
          b = make_float4(rope_hi(l.x, h.x, c.x, t.x), rope_hi(l.y, h.y, c.y, t.y), rope_hi(l.z, h.z, c.z, t.z),
                          rope_hi(l.w, h.w, c.w, t.w));
        }
        plo[u] = pack(a);
        phi[u] = pack(b);
      }
      fetch(c0 + CH);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int row = c0 + rsub + 8 * u;
        if (m0 + row >= M) break;
        const int2 ri = s.row[row];
        __nv_bfloat16 *dlo, *dhi;
        if (o.qkv) {
          const size_t at = (size_t)ri.x, ql = o.q_by_slot ? at : (size_t)(m0 + row);
          dlo = blo + (nlo < o.dq ? ql * o.dq : at * o.dkv);
          dhi = bhi + (nhi < o.dq ? ql * o.dq : at * o.dkv);
        } else {
          __nv_bfloat16* base =
              reinterpret_cast<__nv_bfloat16*>(((unsigned long long)(unsigned)ri.y << 32) | (unsigned)ri.x);
          dlo = base + nlo;
          dhi = base + nhi;
        }
        if (vlo && m0 + row >= lo_from) *reinterpret_cast<uint2*>(dlo) = plo[u];
        if (vhi && m0 + row >= hi_from) *reinterpret_cast<uint2*>(dhi) = phi[u];
      }
      landed(r, ex + ((c0 + CH) & CH) / CH * (CH * EXS));
      asm volatile("bar.sync 1, 128;" ::: "memory");     // staged; behind the last trip: the rows' places are free
    }
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
  const RowForm form{out};
  const bool once = plan.w_stream && plan.m_tiles == 1;
  switch (plan.BN) {
    case 128: return launch_pair_form<128, false>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true);
    case 192: return once ? launch_pair_form<192, true>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true)
                          : launch_pair_form<192, false>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true);
    case 256: return once ? launch_pair_form<256, true>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true)
                          : launch_pair_form<256, false>(L, tmW, tmA, nullptr, M, N, num_kb, plan, form, true);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace dllm

DLLM_TIMELINE_HOOKS(gemm_rows)
DLLM_WAIT_LIMIT_HOOK(gemm_rows)
