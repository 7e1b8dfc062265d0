// Flash-style attention on the 5th-generation tensor cores (tcgen05) for the
// steps with many active rows (response refresh, full steps, batched serving):
// non-causal attention of the active query rows over ALL n cached keys of
// their sequence (Sec. A.7), grouped KV heads packed along the row dimension.
//
// One CTA = TWO tiles of 128 "virtual rows" ((query, head-of-group) pairs) of
// one (sequence, KV head) x one split of the key range, key tiles of 64, eleven
// warps with fixed roles:
//   warp 10          TMA: K/V tiles into a six-stage ring (all that shared memory holds)
//   warp 8           issues the tcgen05.mma (warp 9 those of group 1 when the groups share a row tile)
//   warps 0-3, 4-7   the softmax group of row tile 0 resp. 1 (one row per thread)
// (a CTA of ONE row tile, two to an SM: warp 5 copies, warp 4 issues, warps 0-3 are its softmax group)
// Per key tile t and row tile i:
//   S_i = Q_i K^T     tcgen05.mma, M = 128 rows, N = 64 keys, contraction HD; Q_i is
//                     the A operand in tensor memory (written there once by its
//                     group), K in shared memory (K-major, 128-byte swizzle)
//   softmax           TMEM lane = row, so every thread of group i owns one row: it
//                     loads its 64 scores with tcgen05.ld, takes max / exp2 / sum
//                     locally (no shuffles) and writes P_i as bf16 pairs over the
//                     first 32 score columns: the A operand of the next product
//   O_i += P_i V      tcgen05.mma, M = 128 rows, N = HD, contraction 64 keys; V is
//                     used as stored ([key][hd], "MN-major" B operand); O_i
//                     accumulates in TMEM and is rescaled (tcgen05.ld / st) only
//                     when a row's maximum has grown by more than 2^8 since its
//                     reference was set
// One MMA warp issues O_i += P_i V of tile t and, right behind it, S_i of tile
// t+1, alternating between the row tiles: while one group is in its softmax the
// tensor pipe works for the other, and both row tiles read every K/V tile that
// arrives once.  A CTA with ONE live row tile (at most 128 rows per KV head, the
// odd last tile, or a plan of one-tile CTAs) and at least UA_KPAR_MIN_TILES key
// tiles gives both groups that tile's rows: group 0 takes the even key tiles of
// the CTA's range and group 1 the odd ones, each with its own MMA warp, running
// maximum, sum and output accumulator; the tiles' scores take three buffers in
// turn, and the two halves are merged through shared memory at the end (group
// 1's first).
// With many row tiles a CTA takes one of them with one softmax group, half of the ring and half of the tensor memory, and two
// CTAs share an SM.
// Key-range splits write unnormalised partials plus (max, sum) exactly like the
// mma.sync kernel, and the same merge kernel finishes them.  Every mbarrier wait
// is bounded.
#include <type_traits>

#include "attention_core.cuh"
#include "internal.h"
#include "tma.cuh"
#include "umma.cuh"

namespace dllm {

namespace {

constexpr int UA_ROWS = 128;   // virtual rows per row tile (UMMA M); a CTA works on two row tiles
constexpr int UA_TILES = 2;
constexpr int UA_KEYS = 64;    // keys per tile
// key tiles from which a CTA with one live row tile shares them between its two softmax groups: the exchange and merge of
// the two halves at the end cost 1.1 us, a shared tile takes 0.50 us instead of 0.93 (B200, 128 rows x 32 heads of 128, us
// not shared -> shared: 4 tiles 10.0 -> 9.3, 5 11.0 -> 9.9, 6 12.2 -> 10.7, 7 13.0 -> 11.1, 8 13.9 -> 11.6, 16 21.1 ->
// 15.4; heads of 64: 4 tiles 8.15 -> 7.3); the start takes three tiles at least
constexpr int UA_KPAR_MIN_TILES = 4;

// MN-major operand ([k][mn] rows of 64 mn-elements = 128 bytes, 128-byte swizzle,
// panels of 64 mn-elements): lbo = bytes between panels along MN, sbo = bytes
// between groups of 8 k-rows.
__device__ __forceinline__ uint64_t make_smem_desc_mn(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
        "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
        "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}


// Two fp32 operations in one instruction, each rounded as the scalar one.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tadd.rn.f32x2 rd, ra, rb;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// TILES = 2: one CTA per SM, two softmax groups; 1: two CTAs per SM, each with one row tile, one softmax group, one MMA and
// one TMA warp, half of the shared memory and of the tensor memory.
template <int HD, int TILES>
struct UaSmem {
  static constexpr int STAGES = TILES == 2 ? 6 : HD == 64 ? 6 : 3;              // K/V ring
  static constexpr int THREADS = TILES == 2 ? 352 : 192, MMA_WARP = 4 * TILES, TMA_WARP = TILES == 2 ? 10 : 5;
  static constexpr uint32_t KV_TILE = UA_KEYS * HD * 2;          // one K or V tile
  static constexpr uint32_t STAGE = 2 * KV_TILE;                 // K then V
  static constexpr uint32_t TOTAL = STAGES * STAGE + 1024;    // shared memory holds nothing but the K/V ring
  // Tensor memory, 128 lanes = the rows of a tile: Q_i as bf16 pairs (HD / 2 columns each), the scores S_i (64
  // fp32 columns each; the probabilities P_i overwrite the first 32 of them as bf16 pairs), the outputs O_i.
  // One row tile shared by the groups: one Q, three score buffers that the key tiles take in turn, O per group.
  static constexpr uint32_t Q_COL = 0, S_COL = TILES * (HD / 2), O_COL = TILES == 2 ? 64 + 3 * UA_KEYS : 64 + UA_KEYS;
  static constexpr uint32_t KPAR_S_COL = 64;
  static constexpr uint32_t TMEM_COLS = 256 * TILES;
  static_assert(S_COL + TILES * UA_KEYS <= O_COL, "scores and outputs must not overlap");
  static_assert(O_COL + TILES * HD <= TMEM_COLS, "tensor memory holds 512 columns, 256 for each of two CTAs");
};

template <int HD, int TILES>
__global__ void __launch_bounds__((UaSmem<HD, TILES>::THREADS), 3 - TILES)
    attn_umma_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                     const __nv_bfloat16* __restrict__ q,
                     __nv_bfloat16* __restrict__ o, float* __restrict__ o_part, float* __restrict__ ml_part, int a_seq,
                     int n, int H, int Hkv, int S, int keys_per_split, int row_tiles_per_cta, float scale_log2,
                     int* __restrict__ status) {
  using SM = UaSmem<HD, TILES>;
  constexpr int PANELS = HD / 64, UA_STAGES = SM::STAGES, UA_TMA_WARP = SM::TMA_WARP;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t kv_full[UA_STAGES], kv_empty[UA_STAGES];
  __shared__ __align__(8) uint64_t s_full[3], p_full[TILES], o_full[TILES], q_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t kv_s = base;
  volatile int* abortp = &abort_flag;

  const int G = H / Hkv;
  const int kh = blockIdx.y;
  const int b = blockIdx.z / S, split = blockIdx.z - b * S;
  // row_tiles_per_cta = 1: every CTA takes one 128-row tile only, which its softmax groups share where there are enough key
  // tiles (else the second idles)
  const int row0 = blockIdx.x * (row_tiles_per_cta * UA_ROWS);
  const int n_rows = a_seq * G;
  const int live = (row_tiles_per_cta > 1 && row0 + UA_ROWS < n_rows) ? 2 : 1;  // row tiles of this CTA that hold rows
  const int key_lo = split * keys_per_split;
  const int key_hi = min(n, key_lo + keys_per_split);
  const int n_tiles = (key_hi - key_lo + UA_KEYS - 1) / UA_KEYS;  // >= 1 by construction of the plan
  const int dq = H * HD;
  // one live row tile and enough key tiles: both softmax groups work on that tile's rows, group i on the key
  // tiles t with t % 2 == i
  const bool kpar = TILES == 2 && live == 1 && n_tiles >= UA_KPAR_MIN_TILES;

  if (tid == 0) {
    abort_flag = 0;
    for (int i = 0; i < UA_STAGES; ++i) {
      mbar_init(smem_u32(&kv_full[i]), 1);
      mbar_init(smem_u32(&kv_empty[i]), 1);
    }
    for (int i = 0; i < TILES; ++i) {
      mbar_init(smem_u32(&p_full[i]), UA_ROWS / 32);  // one arrival per warp of the tile's softmax group
      mbar_init(smem_u32(&o_full[i]), 1);
    }
    for (int i = 0; i < 3; ++i) mbar_init(smem_u32(&s_full[i]), 1);
    mbar_init(smem_u32(&q_bar), TILES * UA_ROWS / 32);  // one arrival per softmax warp
    mbar_fence_init();
    prefetch_tensormap(&tmK);
    prefetch_tensormap(&tmV);
  }
  if (warp == UA_TMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(SM::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  pdl_wait();  // Q, K and V come from the preceding kernels
  pdl_trigger();
  bool ok = true;

  if (warp == UA_TMA_WARP) {
    // ---------------- TMA producer: the K/V tiles of the key range ----------------
    for (int t = 0; t < n_tiles; ++t) {
      const int st = t % UA_STAGES;
      if (t >= UA_STAGES && !mbar_wait_warp(smem_u32(&kv_empty[st]), (uint32_t)(t / UA_STAGES - 1) & 1u, abortp)) {
        ok = false;
        break;
      }
      if (elect_one()) {
        const uint32_t fb = smem_u32(&kv_full[st]);
        mbar_expect_tx(fb, SM::STAGE);
        const uint32_t dst = kv_s + st * SM::STAGE;
        const int key0 = key_lo + t * UA_KEYS;
#pragma unroll
        for (int p = 0; p < PANELS; ++p) {
          tma_load_3d(dst + p * (UA_KEYS * 128), &tmK, fb, kh * HD + p * 64, key0, b);
          tma_load_3d(dst + SM::KV_TILE + p * (UA_KEYS * 128), &tmV, fb, kh * HD + p * 64, key0, b);
        }
      }
      __syncwarp();
    }
  } else if (warp >= SM::MMA_WARP) {
    // ---------------- MMA issuers: the first MMA warp, and the second for group 1 when the groups share a row tile ------
    // Per key tile t and row tile i:  S_i(t) = Q_i K(t)^T  ->  [softmax group i]  ->  O_i += P_i(t) V(t), and right
    // behind it S_i(t+1), so that the tensor pipe works on one row tile while the other is in its softmax.  Q_i
    // and P_i are A operands in tensor memory (P_i in the columns its scores came from), so shared memory is
    // read for K and V only.  A commit covers every MMA its thread issued before it, so when s_full[i] flips for tile t+1
    // the product O_i += P_i V of tile t has completed too: the group may then rescale O_i.  (With an issuing warp per row
    // tile the MMAs of both interleave and both groups wait longer: 305 -> 409 us at 4128 x 4128 x 32 heads.)
    constexpr uint32_t idesc_s = make_idesc(UA_ROWS, UA_KEYS);
    constexpr uint32_t idesc_o = make_idesc(UA_ROWS, HD) | (1u << 16);  // B operand (V) is MN-major
    auto issue_s = [&](uint32_t s_col, uint32_t q_col, int bar, int st) {
      if (elect_one()) {
        const uint64_t dk = make_smem_desc(kv_s + st * SM::STAGE);
#pragma unroll
        for (int ks = 0; ks < HD / 16; ++ks) {
          const uint32_t koff = (ks >> 2) * (UA_KEYS * 128) + (ks & 3) * 32;  // panel, then 32 bytes per k-step
          // A = 16 dimensions of Q_i from tensor memory (8 columns of bf16 pairs per k-step)
          umma_bf16_ta(tmem + s_col, tmem + q_col + (uint32_t)(ks * 8), dk + (uint64_t)(koff >> 4), idesc_s, ks > 0 ? 1u : 0u);
        }
        umma_commit(smem_u32(&s_full[bar]));
      }
      __syncwarp();
    };
    // O_i += P_i V: A = 16 keys of P_i from tensor memory; V: 16 key rows of 128 bytes
    auto issue_o = [&](int i, uint32_t s_col, int st, bool accumulate) {
      if (elect_one()) {
        const uint64_t dv = make_smem_desc_mn(kv_s + st * SM::STAGE + SM::KV_TILE, UA_KEYS * 128, 1024);
#pragma unroll
        for (int ks = 0; ks < UA_KEYS / 16; ++ks)
          umma_bf16_ta(tmem + SM::O_COL + (uint32_t)(i * HD), tmem + s_col + (uint32_t)(ks * 8),
                       dv + (uint64_t)((ks * 16 * 128) >> 4), idesc_o, (accumulate || ks > 0) ? 1u : 0u);
      }
      __syncwarp();
    };
    auto tile_ready = [&](int t) {
      const bool r = mbar_wait_warp(smem_u32(&kv_full[t % UA_STAGES]), (uint32_t)(t / UA_STAGES) & 1u, abortp);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      return r;
    };
    ok = mbar_wait_warp(smem_u32(&q_bar), 0u, abortp);
    if (kpar) {
      // Group i owns key tiles i, i + 2, ... and issuer i its MMAs.  Tile t has score buffer t % 3: S(0), S(1), S(2); then
      // per tile t O_i += P(t) V(t) and right behind it S(t + 3) over the same columns, so that a group finds its next
      // scores complete when it is through with a tile.
      // A buffer's tiles belong to the groups in turn, and a wait by parity passes early when the barrier is a whole phase
      // behind: a group may only wait for S(t) once S(t - 3), which it never waits for itself, is complete.  So issuer 0
      // alone issues the first three, in order (a commit covers what its thread issued before): group 1, through with tile
      // 1, knows S(0) complete when it waits for S(3), group 0 after tile 2 S(1).  S(2) precedes S(3) in issuer 0; from
      // tile 6 on S(t - 3) precedes the product of tile t - 4 in the same issuer, which the group has waited for.
      const int i = warp - SM::MMA_WARP;
      for (int t = 0; t < 3 && ok && i == 0; ++t) {
        ok = tile_ready(t);
        if (ok) issue_s(SM::KPAR_S_COL + (uint32_t)(t * UA_KEYS), SM::Q_COL, t, t);
      }
      int buf = i;
      for (int t = i, u = 0; t < n_tiles && ok; t += 2, ++u) {
        const uint32_t s_col = SM::KPAR_S_COL + (uint32_t)(buf * UA_KEYS);
        const int st = t % UA_STAGES;
        ok = mbar_wait_warp(smem_u32(&p_full[i]), (uint32_t)u & 1u, abortp);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        issue_o(i, s_col, st, u > 0);
        if (elect_one()) {
          umma_commit(smem_u32(&o_full[i]));     // the group may rescale O_i, or it is final
          umma_commit(smem_u32(&kv_empty[st]));  // only group i reads V(t), and S(t) completed before its softmax
        }
        __syncwarp();
        if (t + 3 < n_tiles) {
          ok = tile_ready(t + 3);
          if (!ok) break;
          issue_s(s_col, SM::Q_COL, buf, (t + 3) % UA_STAGES);
        }
        buf = buf == 0 ? 2 : buf - 1;   // (t + 2) % 3
      }
    } else if (warp == SM::MMA_WARP) {
      if (ok) ok = tile_ready(0);
      for (int i = 0; i < live && ok; ++i)
        issue_s(SM::S_COL + (uint32_t)(i * UA_KEYS), SM::Q_COL + (uint32_t)(i * (HD / 2)), i, 0);
      for (int t = 0; t < n_tiles && ok; ++t) {
        const int st = t % UA_STAGES;
        bool next_ready = t + 1 >= n_tiles;
        for (int i = 0; i < live && ok; ++i) {
          const uint32_t s_col = SM::S_COL + (uint32_t)(i * UA_KEYS);
          ok = mbar_wait_warp(smem_u32(&p_full[i]), (uint32_t)t & 1u, abortp);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          issue_o(i, s_col, st, t > 0);
          if (t + 1 < n_tiles) {
            if (!next_ready) {
              ok = tile_ready(t + 1);
              if (!ok) break;
              next_ready = true;
            }
            issue_s(s_col, SM::Q_COL + (uint32_t)(i * (HD / 2)), i, (t + 1) % UA_STAGES);
          } else {
            if (elect_one()) umma_commit(smem_u32(&o_full[i]));  // last tile: O_i is final when this fires
            __syncwarp();
          }
        }
        if (ok && elect_one()) umma_commit(smem_u32(&kv_empty[st]));  // the stage may be refilled once these MMAs have read it
        __syncwarp();
      }
    }
  } else {
    // ---------------- softmax groups: warps 0-3 own row tile 0, warps 4-7 row tile 1 ----------------
    const int i = warp >> 2;                                  // row tile
    const int row = (warp & 3) * 32 + lane;                   // row of the tile = TMEM lane
    const uint32_t row_lane = ((uint32_t)((warp & 3) * 32)) << 16;
    const uint32_t o_col = SM::O_COL + (uint32_t)(i * HD);
    const int gtid = tid & 127;
    {
      // Q to tensor memory as bf16 pairs, TMEM lane = row: every thread fetches its own row (zeros past the last one), all
      // loads in flight before the first use.  A group brings in the Q of its row tile, or its half of the one both work
      // on.  (Eight lanes per row and a turn through shared memory: 2 us longer per CTA when several follow on an SM.)
      const int vr = row0 + (kpar ? 0 : i * UA_ROWS) + row;
      const int p_lo = kpar ? (i * PANELS + 1) / 2 : 0, p_hi = kpar ? ((i + 1) * PANELS + 1) / 2 : i < live ? PANELS : 0;
      uint4 qv[HD / 8];
#pragma unroll
      for (int w = 0; w < HD / 8; ++w) qv[w] = make_uint4(0, 0, 0, 0);
      if (vr < n_rows) {
        const int qi = vr / G, g = vr - qi * G;
        const uint4* src = reinterpret_cast<const uint4*>(q + ((size_t)b * a_seq + qi) * dq + (kh * G + g) * HD);
#pragma unroll
        for (int w = 0; w < HD / 8; ++w)
          if (w / 8 >= p_lo && w / 8 < p_hi) qv[w] = __ldcg(src + w);
      }
#pragma unroll
      for (int p = 0; p < PANELS; ++p) {
        if (p < p_lo || p >= p_hi) continue;
        uint32_t r[32];
#pragma unroll
        for (int w = 0; w < 8; ++w) {
          r[4 * w] = qv[p * 8 + w].x;
          r[4 * w + 1] = qv[p * 8 + w].y;
          r[4 * w + 2] = qv[p * 8 + w].z;
          r[4 * w + 3] = qv[p * 8 + w].w;
        }
        tmem_st32(tmem + row_lane + SM::Q_COL + (uint32_t)((kpar ? 0 : i * (HD / 2)) + p * 32), r);  // waits for the store
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&q_bar));
    }
    if (gtid == 0 && i == 0) timeline_mark(1);  // Q in tensor memory

    constexpr float RESCALE_STEP = 8.f;  // log2 units a row's maximum may exceed its reference before O is rescaled
    // m_ref: the maximum the exponentials of this row refer to; it follows the true running maximum lazily (O in
    // TMEM is only rescaled when the maximum has grown by more than RESCALE_STEP, which keeps every exponential
    // below 2^8)
    float m_ref = -INFINITY, l_run = 0.f;
    // u counts this group's tiles; with KPAR they are the key tiles i, i + 2, ...  (one instance per mode: what the loop
    // spends on the other's bookkeeping shows in its time)
    auto softmax_tiles = [&](auto mode) {
      constexpr bool KPAR = decltype(mode)::value;
      constexpr int t_step = KPAR ? 2 : 1;
      const uint32_t s_first = tmem + row_lane + (KPAR ? SM::KPAR_S_COL : SM::S_COL);
      int buf = i;               // score buffer of the tile, and the parity of its barrier
      uint32_t par = 0;
      for (int t = KPAR ? i : 0, u = 0; t < n_tiles; t += t_step, ++u) {
        const uint32_t s_col = s_first + (uint32_t)(buf * UA_KEYS);
        ok = mbar_wait(smem_u32(&s_full[buf]), par, abortp);
        if (!ok) break;
        if (!KPAR) {
          par ^= 1u;
        } else if (buf == 0) {
          buf = 2;
        } else {
          --buf;
          par ^= 1u;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (gtid == 0 && i == 0) timeline_mark(2 + (u < 5 ? u : 5));  // scores of this group's tile u complete
        // ---- this thread's row of scores (raw: the scale is folded into the exponent's multiply-add)
        const int valid = key_hi - (key_lo + t * UA_KEYS);  // >= 1
        float sv[UA_KEYS];
        float mx;
        {
          uint32_t r0[32], r1[32];  // both loads in flight, one wait
          tmem_ld32(s_col, r0);
          tmem_ld32(s_col + 32u, r1);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            sv[j] = __uint_as_float(r0[j]);
            sv[32 + j] = __uint_as_float(r1[j]);
          }
          if (valid < UA_KEYS) {  // the ragged last tile of the sequence: keys past the end count for nothing
#pragma unroll
            for (int j = 0; j < UA_KEYS; ++j)
              if (j >= valid) sv[j] = -INFINITY;
          }
          float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};  // four chains instead of one of 64 steps
#pragma unroll
          for (int j = 0; j < UA_KEYS; ++j) mx4[j & 3] = fmaxf(mx4[j & 3], sv[j]);
          mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * scale_log2;  // scale_log2 > 0
        }
        // ---- lazy rescale of O (warp-uniform branch: the TMEM accesses are warp-collective)
        const bool grow = mx > m_ref + RESCALE_STEP;
        if (__any_sync(0xffffffffu, grow)) {
          const float corr = grow ? exp2f(m_ref - mx) : 1.f;  // first tile: exp2(-inf) = 0, O is not read (u == 0)
          if (grow) {
            m_ref = mx;
            l_run *= corr;
          }
          if (u > 0) {
            if (KPAR) {  // the group's previous product may still be running
              ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&o_full[i]), (uint32_t)(u - 1) & 1u, abortp));
              if (!ok) break;
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            }
#pragma unroll
            for (int c = 0; c < HD; c += 32) {
              uint32_t r[32];
              tmem_ld32(tmem + row_lane + o_col + (uint32_t)c, r);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) * corr);
              tmem_st32(tmem + row_lane + o_col + (uint32_t)c, r);
            }
          }
        }
        // ---- probabilities -> tensor memory as bf16 pairs (the A operand of O_i += P_i V), over the first 32 of
        // the columns this thread has just read its scores from
        // (multiply-adds and sums two keys at a time: the issue slots of the two groups' warps are what the exponentials
        // compete for)
        float2 p_sum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        const float ref = m_ref == -INFINITY ? 0.f : m_ref;  // no score above -inf so far: weights 0, not exp2(-inf + inf)
        const float2 scale2 = make_float2(scale_log2, scale_log2), ref2 = make_float2(-ref, -ref);
        uint32_t pk[UA_KEYS / 2];
#pragma unroll
        for (int c2 = 0; c2 < UA_KEYS / 2; ++c2) {
          const float2 e = fma2(make_float2(sv[2 * c2], sv[2 * c2 + 1]), scale2, ref2);
          const float2 pp = make_float2(fast_exp2(e.x), fast_exp2(e.y));
          p_sum[c2 & 1] = add2(p_sum[c2 & 1], pp);
          pk[c2] = pack_bf16(pp.x, pp.y);
        }
        l_run += (p_sum[0].x + p_sum[1].x) + (p_sum[0].y + p_sum[1].y);
        tmem_st32(s_col, pk);  // waits for the store
        if (KPAR && u > 0) {  // the other group's issuer may be ahead of this one's: not two arrivals that it has not seen
          ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&o_full[i]), (uint32_t)(u - 1) & 1u, abortp));
          if (!ok) break;
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&p_full[i]));
      }
    };
    if (i < live || kpar) {
      if (kpar) softmax_tiles(std::true_type{});
      else softmax_tiles(std::false_type{});
      // O_i is final: one commit after the last tile, or one per tile of the group
      if (ok) ok = mbar_wait(smem_u32(&o_full[i]), kpar ? (uint32_t)((n_tiles - i + 1) / 2 - 1) & 1u : 0u, abortp);
      ok = __all_sync(0xffffffffu, ok);  // the TMEM loads below are warp-collective
      // ---- one live row tile shared by the groups: group 1 hands its half (max, sum, unnormalised output) to
      // group 0 through the K/V ring, which nothing reads any more once both groups' last products are complete
      constexpr int XS = HD + 4;  // floats per exchanged row: 16-byte aligned, rows 4 banks apart
      float* xo = reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw)));
      float* xml = xo + UA_ROWS * XS;
      float w_self = 1.f, w_peer = 0.f;  // weights of this group's and the other group's half in the merged row
      bool peer = false, write_out = ok;
      if (kpar) {
        static_assert(TILES == 1 || (UA_ROWS * XS + 2 * UA_ROWS) * 4 <= UA_STAGES * SM::STAGE, "the exchange area must fit the ring");
        {  // both groups are past their last product (or gave up): all 256 threads agree
          uint32_t r;
          asm volatile(
              "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\tbar.red.and.pred p, 2, 256, q;\n\tselp.u32 %0, 1, 0, p;\n\t}"
              : "=r"(r)
              : "r"((uint32_t)ok)
              : "memory");
          ok = r != 0;
        }
        if (ok && i == 1) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int c = 0; c < HD; c += 32) {
            uint32_t r[32];
            tmem_ld32(tmem + row_lane + o_col + (uint32_t)c, r);
            tmem_ld_wait();
#pragma unroll
            for (int k = 0; k < 32; k += 4)
              *reinterpret_cast<uint4*>(xo + row * XS + c + k) = make_uint4(r[k], r[k + 1], r[k + 2], r[k + 3]);
          }
          xml[2 * row] = m_ref;
          xml[2 * row + 1] = l_run;
        }
        asm volatile("bar.sync 2, 256;" ::: "memory");
        write_out = ok && i == 0;  // group 0 writes the merged rows
        if (write_out) {
          const float m1 = xml[2 * row], l1 = xml[2 * row + 1];
          const float M = fmaxf(m_ref, m1);
          w_self = exp2f(m_ref - M);
          w_peer = exp2f(m1 - M);
          l_run = w_self * l_run + w_peer * l1;
          m_ref = M;
          peer = true;
        }
      }
      if (write_out) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (gtid == 0 && i == 0) timeline_mark(8);  // O complete
        const int vr = row0 + (kpar ? 0 : i * UA_ROWS) + row;
        const bool is_live = vr < n_rows;
        const int qi = is_live ? vr / G : 0, g = is_live ? vr - qi * G : 0;
        const size_t orow = ((size_t)b * a_seq + qi) * H + (kh * G + g);  // (row, head) index
        const float inv = 1.f / l_run;
        const size_t total = (size_t)gridDim.z / S * a_seq * H;
#pragma unroll
        for (int c = 0; c < HD; c += 32) {
          uint32_t r[32];
          tmem_ld32(tmem + row_lane + o_col + (uint32_t)c, r);  // warp-collective: every lane takes part
          tmem_ld_wait();
          if (!is_live) continue;
          if (peer) {
#pragma unroll
            for (int k = 0; k < 32; k += 4) {
              const float4 x = *reinterpret_cast<const float4*>(xo + row * XS + c + k);
              r[k] = __float_as_uint(w_self * __uint_as_float(r[k]) + w_peer * x.x);
              r[k + 1] = __float_as_uint(w_self * __uint_as_float(r[k + 1]) + w_peer * x.y);
              r[k + 2] = __float_as_uint(w_self * __uint_as_float(r[k + 2]) + w_peer * x.z);
              r[k + 3] = __float_as_uint(w_self * __uint_as_float(r[k + 3]) + w_peer * x.w);
            }
          }
          if (S == 1) {
            __nv_bfloat16* dst = o + orow * HD + c;
#pragma unroll
            for (int k = 0; k < 32; k += 8)
              *reinterpret_cast<uint4*>(dst + k) = make_uint4(
                  pack_bf16(__uint_as_float(r[k]) * inv, __uint_as_float(r[k + 1]) * inv),
                  pack_bf16(__uint_as_float(r[k + 2]) * inv, __uint_as_float(r[k + 3]) * inv),
                  pack_bf16(__uint_as_float(r[k + 4]) * inv, __uint_as_float(r[k + 5]) * inv),
                  pack_bf16(__uint_as_float(r[k + 6]) * inv, __uint_as_float(r[k + 7]) * inv));
          } else {
            float* dst = o_part + ((size_t)split * total + orow) * HD + c;
#pragma unroll
            for (int k = 0; k < 32; k += 4)
              *reinterpret_cast<uint4*>(dst + k) = make_uint4(r[k], r[k + 1], r[k + 2], r[k + 3]);
          }
        }
        if (is_live && S > 1) {
          float* ml = ml_part + ((size_t)split * total + orow) * 2;
          ml[0] = m_ref;
          ml[1] = l_run;
        }
      }
    }
  }
  // a wait that gave up anywhere in the CTA: record it once, let copies in flight land
  ok = __syncthreads_and(ok);
  if (!ok) {
    if (tid == 0 && status) atomicCAS(status, ST_OK, ST_TIMEOUT_ATTN_UMMA);
    drain_delay();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == UA_TMA_WARP) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(SM::TMEM_COLS) : "memory");
  }
}

template <int HD, int TILES>
cudaError_t launch_umma(const Launch& L, const CUtensorMap& tmK, const CUtensorMap& tmV, const void* q, void* o,
                        float* scratch, int B, int a_seq, int n, int H, int Hkv, int S, int keys_per_split,
                        int row_tiles_per_cta) {
  constexpr int SMEM = (int)UaSmem<HD, TILES>::TOTAL;
  static DeviceOnce once;
  cudaError_t e0 = once.run(
      [] { return cudaFuncSetAttribute(attn_umma_kernel<HD, TILES>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM); });
  if (e0 != cudaSuccess) return e0;
  const int G = H / Hkv;
  const size_t total = (size_t)B * a_seq * H;
  float* o_part = scratch;
  float* ml_part = scratch ? scratch + (size_t)S * total * HD : nullptr;
  const int rows_per_cta = row_tiles_per_cta * UA_ROWS;
  dim3 grid((a_seq * G + rows_per_cta - 1) / rows_per_cta, Hkv, B * S);
  const float scale_log2 = 1.4426950408889634f / sqrtf((float)HD);
  cudaError_t e = launch_k(L, attn_umma_kernel<HD, TILES>, grid, dim3(UaSmem<HD, TILES>::THREADS), SMEM, tmK, tmV, (const __nv_bfloat16*)q,
                           (__nv_bfloat16*)o, o_part, ml_part, a_seq, n, H, Hkv, S, keys_per_split, row_tiles_per_cta,
                           scale_log2, L.d_status);
  L.count();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Key-range splits for CTAs of two 128-row tiles, whole 64-key tiles per split, no more splits than the scratch
// holds.  A split shortens the key range a CTA walks through but adds a partial result per (row, head) pair that
// the merge has to write and read, and CTAs of one row tile are twice as many, so both are what a small cost model likes
// best (microseconds, fitted to sweeps on B200, one CTA per SM at a time: per CTA 10.6 us of fixed cost and 1.02 us per
// key tile with two row tiles, 8.6 and 0.44 us with one that the groups share, 8.6 and 0.9 us with one of fewer key tiles;
// for a merge 1.2 us plus 1040 bytes per pair and split at 10 TB/s).
AttnPlan plan_attention_umma(int B, int a_seq, int n, int H, int Hkv, size_t scratch_floats) {
  AttnPlan p;
  const int G = H / Hkv, sms = sm_count();
  const int key_tiles = (n + UA_KEYS - 1) / UA_KEYS;
  const size_t per_split = (size_t)B * a_seq * H * (128 + 2);
  const double pairs = (double)B * a_seq * H;
  int best_s = 1, best_rt = UA_TILES;
  double best_us = -1.0;
  for (int rt = UA_TILES; rt >= 1; --rt) {   // row tiles per CTA: two (the groups overlap), or one (twice the CTAs)
    if (g_attn_umma_row_tiles && rt != g_attn_umma_row_tiles) continue;
    const long ctas = (long)((a_seq * G + rt * UA_ROWS - 1) / (rt * UA_ROWS)) * Hkv * B;
    for (int S = 1; S <= key_tiles && S <= 16; ++S) {
      if (S > 1 && (size_t)S * per_split > scratch_floats) break;
      const int tps = (key_tiles + S - 1) / S;
      const double fixed_us = rt == 2 ? 10.6 : 8.6;
      const double tile_us = rt == 2 ? 1.02 : tps >= UA_KPAR_MIN_TILES ? 0.44 : 0.9;
      if (S > 1 && (key_tiles + tps - 1) / tps != S) continue;  // the same tiles per split as a smaller count
      const double waves = (double)((ctas * S + sms - 1) / sms);
      const double us = waves * (fixed_us + tps * tile_us) + (S > 1 ? 1.2 + S * pairs * 1040.0 / 10.0e6 : 0.0);
      if (best_us < 0.0 || us < best_us) {
        best_s = S;
        best_rt = rt;
        best_us = us;
      }
    }
  }
  int S = g_attn_force_splits > 0 ? g_attn_force_splits : best_s;
  if (S > key_tiles) S = key_tiles;
  if (S > 1 && (size_t)S * per_split > scratch_floats) S = (int)(scratch_floats / per_split);
  if (S < 1) S = 1;
  const int tiles_per_split = (key_tiles + S - 1) / S;
  p.keys_per_split = tiles_per_split * UA_KEYS;
  p.S = (key_tiles + tiles_per_split - 1) / tiles_per_split;
  p.scratch_floats = p.S > 1 ? (size_t)p.S * per_split : 0;
  p.row_tiles = a_seq * G <= UA_ROWS ? 1 : best_rt;
  // Three CTAs of one row tile per SM or more: two at a time, so that one's start and end (8 to 10 us of loads, merges and
  // stores) run beside the other's products.  B200, us, one CTA per SM -> two: 16 x 128 x 1536 x 32 heads 99 -> 86, 16 x 128 x
  // 768 69 -> 57, 8 x 300 x 700 75 -> 63, 4 x 1536 x 1536 209 -> 189, 4128 x 4128 301 -> 293; below, where a CTA's own chain is
  // what counts and two row tiles share each K / V tile: 1024 x 1024 30.5 -> 32.7, 4 x 128 x 1536 28 -> 34.
  const long tiles = (long)((a_seq * G + UA_ROWS - 1) / UA_ROWS) * Hkv * B;
  if (p.S == 1 && tiles >= 3L * sms && g_attn_umma_row_tiles == 0 && g_attn_force_splits == 0) {
    p.row_tiles = 1;
    p.two_per_sm = true;
  }
  return p;
}

cudaError_t launch_attention_umma(const Launch& L, const void* q, const void* Kc, const void* Vc, void* o, int B,
                                  int a_seq, int n, int H, int Hkv, int hd, float* scratch, size_t scratch_floats,
                                  int* S_out) {
  const AttnPlan p = plan_attention_umma(B, a_seq, n, H, Hkv, scratch ? scratch_floats : 0);
  CUtensorMap tmK, tmV;
  if (!get_tensor_map_3d(Kc, (uint64_t)B, (uint64_t)n, (uint64_t)Hkv * hd, 64, &tmK) ||
      !get_tensor_map_3d(Vc, (uint64_t)B, (uint64_t)n, (uint64_t)Hkv * hd, 64, &tmV))
    return cudaErrorInvalidValue;
  if (S_out) *S_out = p.S;
  auto go = [&](auto launch) { return launch(L, tmK, tmV, q, o, scratch, B, a_seq, n, H, Hkv, p.S, p.keys_per_split, p.row_tiles); };
  if (p.two_per_sm) return hd == 64 ? go(launch_umma<64, 1>) : go(launch_umma<128, 1>);
  return hd == 64 ? go(launch_umma<64, 2>) : go(launch_umma<128, 2>);
}

}  // namespace dllm

DLLM_TIMELINE_HOOKS(attention_umma)
DLLM_WAIT_LIMIT_HOOK(attention_umma)
