// attn_tc.cu — causal grouped-query attention on the tcgen05 tensor cores (head dimension HD 64 or
// 128, sequences of whole 64-token blocks), for the block window's attention: the forward
// (softmax(Q K^T / sqrt(d)) V per head over the keys up to the query's position, and the row's
// natural log-sum-exp for the backward), and the backward in two kernels (dQ per query tile,
// persistent over the forward's work items; dK and dV per key tile over the query heads
// sharing it), without atomics.
//
// A CTA of 8 elementwise warps (two warpgroups; warp w owns TMEM lanes 32 (w % 4)..), TMA warps and an
// MMA warp, one CTA per SM (512 TMEM columns).  A 128 x 128 tile costs the tensor cores 512 cycles a
// product and the elementwise warps about 600 issue slots a scheduler and, per warpgroup, some 2,500
// cycles of TMEM round trips and dependent steps; so each kernel keeps two independent pieces of
// elementwise work in flight and orders its MMAs so that they run beside them:
//
// Forward: persistent over (128-query tile, head, sequence) items, longest rows first.  Warpgroup c takes
// the item's key tiles c, c + 2, ... as an online softmax of its own, with its own score buffer,
// running maximum and output accumulator: S_j = Q K_j^T, P_j (bf16, over S_j) and O_c += P_j V_j.
// At the item's end the two halves of the row meet (maximum and sum through shared memory) and each
// warpgroup writes half of the columns.  The running maximum is raised lazily: only when a tile's
// maximum exceeds it by more than 8 (log2 units) is O rescaled (the thread's own TMEM row, after
// its chain's previous P V has completed), so P stays below 2^8 and most tiles leave O alone; O / l
// and the log-sum-exp are exact for whichever maximum was used.  Every wait is bounded.
//
// dQ: persistent over the same items; each warpgroup takes 64 of a tile's keys.  dP_{j+1} is issued when
// dS_j is ready, then dQ += dS_j K_j, then S_{j+2} into the buffer dS_j leaves.
//
// dK, dV: one CTA per (128-key tile, key/value head, sequence); each warpgroup takes 64 of a query tile's
// columns.  dV += P^T dO and the next S^T run while dS is formed, dK += dS^T Q and the next dP^T
// while the next P is.
//
// 4 x 2048 tokens, 32 query / 8 key-value heads of 128, one GB300 (with one elementwise warpgroup, products
// and softmax in turn, in parentheses): forward 154 us (187), dQ 222 (222), dK/dV 238 (341), against
// 71, 107 and 143 at the bf16 peak for the causal half.  The tiles on the diagonal are computed
// whole.  What bounds each: forward and dQ, the products with both operands in shared memory
// (930 - 1,100 cycles for 128 x 128 x 128, where 490 is the rate with one in TMEM; dQ has two per
// tile, forward one besides its softmax); dK/dV, the tensor cores (2,650 cycles a step of 2,050).
// 3 x 1088 tokens, 12 / 4 heads of 64: forward 22 us (mma.sync: 41), dQ 25 (47), dK/dV 41 (115).
//
// Tensor maps are 3-D (column, token of the sequence, sequence): a last tile of 64 tokens reads zeros
// past its sequence, never another sequence's rows.  As keys those lie after every real query, so
// the causal mask drops them; as queries they are not stored, and count as nothing in dK and dV.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "launch.h"
#include "ptx_sm100.cuh"

namespace catq {
namespace {

constexpr int kTq = 128;             // query rows per tile (MMA M, TMEM lanes)
constexpr int kTk = 128;             // keys per tile (MMA N of Q K^T, K of P V)
constexpr int kWarps = 8;            // elementwise warps
constexpr int kElem = 32 * kWarps;   // their threads
constexpr int kTmaWarp = 8, kMmaWarp = 9, kTma2Warp = 10;
constexpr int kThreadsTc = 10 * 32;  // elementwise, TMA, MMA
constexpr int kThreadsDq = 11 * 32;  // dQ: a second TMA warp
constexpr uint32_t kBox = 128 * 128;                 // one 64-column box of 128 rows, bytes
// Shared memory of a kernel, by head dimension: tiles of 128 rows (HD / 64 boxes), barriers, 1 KB of
// alignment slack; at least half an SM's, since the tensor memory allows one CTA per SM.
template <int HD>
struct Lay {
  static constexpr int kBoxes = HD / 64;
  static constexpr uint32_t kTile = kBoxes * kBox;
  // forward: Q, two K and two V tiles, the two halves' (maximum, sum) per row and item parity
  static constexpr uint32_t kOffQ = 0, kOffK = kTile, kOffV = 3 * kTile, kOffMl = 5 * kTile,
                            kOffBar = kOffMl + 2 * 2 * kTq * 8;
  static constexpr uint32_t kSmem = kOffBar + 256 + 1024 < 116 * 1024 ? 116 * 1024 : kOffBar + 256 + 1024;
  // dQ: Q, dO, three K and two V tiles
  static constexpr uint32_t kDqOffQ = 0, kDqOffDo = kTile, kDqOffK = 2 * kTile, kDqOffV = 5 * kTile,
                            kDqOffBar = 7 * kTile;
  static constexpr uint32_t kDqSmem = kDqOffBar + 256 + 1024 < 116 * 1024 ? 116 * 1024 : kDqOffBar + 256 + 1024;
  // dK, dV: a stage holds the query tile and its dO tile; two buffers of their rows' log-sum-exp and
  // delta beside them
  static constexpr uint32_t kKvOffK = 0, kKvOffV = kTile, kKvOffStage = 2 * kTile, kStageBytes = 2 * kTile;
  static constexpr uint32_t kKvOffRow = kKvOffStage + 2 * kStageBytes, kKvOffBar = kKvOffRow + 4 * kTq * 4;
  static constexpr uint32_t kKvSmem = kKvOffBar + 128 + 1024 < 116 * 1024 ? 116 * 1024 : kKvOffBar + 128 + 1024;
};
constexpr uint32_t kTmemCols = 512;
constexpr float kLazy = 8.0f;                        // rescale only past this rise (log2 units)
// A chain's maximum before it has seen a score above -inf: below every product of a score, and finite, so
// that scores of -inf weigh 2^(-inf - kNoMax) = 0 and not 2^(-inf + inf).
constexpr float kNoMax = -3e38f;

struct TcAttnArgs {
  uint16_t* out;
  float* lse;
  int32_t B, S, nh, nkv;
  float scale_log2;
  WaitCtl wc;
};

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// D[tmem] (+)= A[tmem] * B[smem] (A: M x K bf16 in TMEM, one row per lane, column j holding
// elements 2j and 2j + 1 of the row; B by its descriptor's lower half).
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 db;\n\tsetp.ne.b32 p, %4, 0;\n\tmov.b64 db, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], db, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "r"(b_lo), "r"(idesc), "r"(accumulate), "r"(kDescHi)
      : "memory");
}

__device__ __forceinline__ float fast_exp2(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// K-major SS products: D = A B^T over HD columns (A, B: 128 rows, HD / 64 boxes of 64 columns each).
template <int HD>
__device__ __forceinline__ void mma_kmajor(uint32_t d_tmem, uint32_t a_smem, uint32_t b_smem, uint32_t idesc) {
  const uint32_t ad = desc_lo(a_smem, 16), bd = desc_lo(b_smem, 16);
#pragma unroll
  for (int kk = 0; kk < HD / 16; ++kk) {
    const uint32_t off = ((kk >> 2) * kBox + (kk & 3) * 32) / 16;
    umma_lo<1>(d_tmem, ad + off, bd + off, idesc, kk > 0 ? 1u : 0u);
  }
}

// TS products: D (+)= A[tmem] B[smem] over 128 (A: 128 x 128 bf16 in TMEM, B: the 128-row
// tile read as K x N with N = HD contiguous).  A replaces 128 fp32 columns half by half: its elements
// 0 .. 63 lie in columns 0 .. 31, 64 .. 127 in columns 64 .. 95.
__device__ __forceinline__ void mma_ts_tile(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_smem, uint32_t idesc,
                                            bool accumulate) {
  const uint32_t bd = desc_lo(b_smem, kBox);
#pragma unroll
  for (int kk = 0; kk < 8; ++kk)
    umma_ts(d_tmem, a_tmem + (kk < 4 ? 8u * kk : 32u + 8u * kk), bd + kk * (2048 / 16), idesc,
            (accumulate || kk > 0) ? 1u : 0u);
}

// A warp's TMEM accesses are done: one arrival on its behalf.
__device__ __forceinline__ void warp_arrive(uint32_t bar, int lane) {
  tc_fence_before();
  __syncwarp();
  if (lane == 0) mbar_arrive_local(bar);
}

// 32 fp32 columns of one row per lane (a warp's 32 rows, `ld` elements apart from `row0` on, of which the
// first `rows` are real), times f, stored as bf16, transposed so that four lanes cover 64 contiguous
// bytes of a row: a store then writes 16 whole sectors where a lane per row touched 32 halves (an
// item's epilogue took 4,900 cycles).
__device__ __forceinline__ void store_cols32(uint16_t* row0, int64_t ld, int rows, const uint32_t (&o)[32], float f,
                                             int lane) {
  uint4 v[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    v[p].x = pack2(__uint_as_float(o[8 * p + 0]) * f, __uint_as_float(o[8 * p + 1]) * f);
    v[p].y = pack2(__uint_as_float(o[8 * p + 2]) * f, __uint_as_float(o[8 * p + 3]) * f);
    v[p].z = pack2(__uint_as_float(o[8 * p + 4]) * f, __uint_as_float(o[8 * p + 5]) * f);
    v[p].w = pack2(__uint_as_float(o[8 * p + 6]) * f, __uint_as_float(o[8 * p + 7]) * f);
  }
  transpose_quads(v, lane);
  // lane 4a + i holds chunk i of rows 4a .. 4a + 3
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int r = (lane & ~3) + j;
    if (r < rows) *reinterpret_cast<uint4*>(row0 + r * ld + 8 * (lane & 3)) = v[j];
  }
}

// Bounded wait for copies or MMAs still in flight when a launch gives up.
__device__ __forceinline__ void drain(uint32_t bar, uint32_t parity) {
  const uint64_t t0 = globaltimer_ns();
  while (!mbar_try_wait(bar, parity))
    if (globaltimer_ns() - t0 > 200000000ull) return;
}

// Work item -> (query tile, head, sequence), the longest rows first.
struct ItemOf {
  int nqt, nh, B;
  __device__ __forceinline__ void operator()(int it, int& qt, int& h, int& b) const {
    qt = nqt - 1 - it / (nh * B);
    const int rem = it % (nh * B);
    h = rem % nh;
    b = rem / nh;
  }
};

// The weights of one row's 128 scores (keys up to `last`) where its maximum m is 2^24 or more: there the
// fused product's unrounded part could exceed the exponent's range (the maximum is a rounded product), so
// the products are rounded first, like it.  A loop of few instructions, off the path of ordinary scores
// (which took 4 to 10 % longer with this in line).  P goes over the scores as there; returns its sum.
__device__ __forceinline__ float weigh_far(uint32_t sbuf, float scale_log2, float m, int last) {
  float sum = 0.0f;
#pragma unroll 1
  for (int k = 0; k < kTk / 8; ++k) {
    uint32_t s[8], pk[4];
    tmem_ld8(sbuf + 8u * k, s);
    tmem_ld_wait();
    float p[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float x = __fsub_rn(__fmul_rn(__uint_as_float(s[i]), scale_log2), m);
      p[i] = 8 * k + i > last ? 0.0f : fast_exp2(x);
      sum += p[i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) pk[i] = pack2(p[2 * i], p[2 * i + 1]);
    tmem_st4(sbuf + 64u * (k >> 3) + 4u * (k & 7), pk);
  }
  return sum;
}

template <int HD>
__global__ void __launch_bounds__(kThreadsTc, 1)
    attn_tc_fwd_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
                       const __grid_constant__ CUtensorMap tmv, const TcAttnArgs a) {
  using Y = Lay<HD>;
  constexpr uint32_t kTile = Y::kTile;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* const gbase = smem_raw + (base - raw);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + Y::kOffBar + 248);
  const uint32_t bar = base + Y::kOffBar;
  // per item: q_full, q_empty, o_free; per tile: k, v rings of 2; per chain: s_full, p_full, pv_done
  const uint32_t q_full = bar, q_empty = bar + 8, o_free = bar + 16, k_full0 = bar + 24, k_empty0 = bar + 40,
                 v_full0 = bar + 56, v_empty0 = bar + 72, s_full0 = bar + 120, p_full0 = bar + 136,
                 pv_done0 = bar + 152, final_bar = bar + 168;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nqt = (a.S + kTq - 1) / kTq;
  const int n_items = nqt * a.nh * a.B;
  const ItemOf item_of{nqt, a.nh, a.B};
  constexpr uint32_t kColS = 0, kColO = 256;  // S of chain c at 128 c, O of chain c at 256 + 128 c

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    mbar_init(o_free, kWarps);
    for (int i = 0; i < 2; ++i) {
      mbar_init(k_full0 + 8u * i, 1);
      mbar_init(k_empty0 + 8u * i, 1);
      mbar_init(v_full0 + 8u * i, 1);
      mbar_init(v_empty0 + 8u * i, 1);
    }
    for (int c = 0; c < 2; ++c) {
      mbar_init(s_full0 + 8u * c, 1);
      mbar_init(p_full0 + 8u * c, kWarps / 2);
      mbar_init(pv_done0 + 8u * c, 1);
    }
    mbar_init(final_bar, 1);
    fence_mbar_init_cluster();
  }
  if (warp == kMmaWarp) tmem_alloc<1>(smem_u32(tmem_slot), kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;

  if (warp == kTmaWarp) {
    if (lane == 0) {
      prefetch_tmap(&tmq);
      prefetch_tmap(&tmk);
      prefetch_tmap(&tmv);
      int g = 0, li = 0, q_loads = 0, k_loads = 0, v_loads = 0, s = 0;
      uint32_t ph = 1;
      for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x, ++li) {
        int qt, h, b;
        item_of(it, qt, h, b);
        const int hk = h / (a.nh / a.nkv);
        // the Q buffer is free once every score product of the previous item has completed
        if (li > 0 && !mbar_wait(q_empty, (li - 1) & 1, a.wc)) { ok = false; break; }
        ++q_loads;
        mbar_arrive_expect_tx(q_full, kTile);
        for (int hf = 0; hf < Y::kBoxes; ++hf)
          tma_load_3d(base + Y::kOffQ + hf * kBox, &tmq, q_full, h * HD + 64 * hf, qt * kTq, b);
        for (int j = 0; j <= qt; ++j, ++g) {
          if (!mbar_wait(k_empty0 + 8u * s, ph, a.wc)) { ok = false; break; }
          mbar_arrive_expect_tx(k_full0 + 8u * s, kTile);
          for (int hf = 0; hf < Y::kBoxes; ++hf)
            tma_load_3d(base + Y::kOffK + s * kTile + hf * kBox, &tmk, k_full0 + 8u * s, hk * HD + 64 * hf, j * kTk, b);
          ++k_loads;
          if (!mbar_wait(v_empty0 + 8u * s, ph, a.wc)) { ok = false; break; }
          mbar_arrive_expect_tx(v_full0 + 8u * s, kTile);
          for (int hf = 0; hf < Y::kBoxes; ++hf)
            tma_load_3d(base + Y::kOffV + s * kTile + hf * kBox, &tmv, v_full0 + 8u * s, hk * HD + 64 * hf, j * kTk, b);
          ++v_loads;
          if (++s == 2) { s = 0; ph ^= 1u; }
        }
      }
      // copies still in flight land before the CTA exits
      if (q_loads > 0) drain(q_full, (q_loads - 1) & 1);
      for (int t = max(0, k_loads - 2); t < k_loads; ++t) drain(k_full0 + 8u * (t & 1), (t >> 1) & 1);
      for (int t = max(0, v_loads - 2); t < v_loads; ++t) drain(v_full0 + 8u * (t & 1), (t >> 1) & 1);
    }
  } else if (warp == kMmaWarp) {
    // the whole warp walks the items, one elected lane issues (see elect_one)
    constexpr uint32_t idesc_s = idesc_bf16_f32(kTq, kTk, false, false);  // Q, K both K-major
    constexpr uint32_t idesc_o = idesc_bf16_f32(kTq, HD, false, true);    // V MN-major
    const bool issuer = elect_one();
    int ks = 0, vs = 0, li = 0;
    uint32_t kph = 0, vph = 0, pph[2] = {0u, 0u};
    // the item's next score product into its chain's buffer, which the chain's last P V has left
    auto issue_s = [&](int j, bool last) -> bool {
      if (!mbar_wait_warp(k_full0 + 8u * ks, kph, a.wc)) return false;
      tc_fence_after();
      if (issuer) {
        mma_kmajor<HD>(tmem + kColS + 128u * (j & 1), base + Y::kOffQ, base + Y::kOffK + ks * kTile, idesc_s);
        umma_commit<1>(s_full0 + 8u * (j & 1));
        umma_commit<1>(k_empty0 + 8u * ks);
        if (last) umma_commit<1>(q_empty);
      }
      if (++ks == 2) { ks = 0; kph ^= 1u; }
      return true;
    };
    for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x, ++li) {
      int qt, h, b;
      item_of(it, qt, h, b);
      const int n = qt + 1;
      if (!mbar_wait_warp(q_full, li & 1, a.wc) || !issue_s(0, n == 1) || (n > 1 && !issue_s(1, n == 2))) {
        ok = false;
        break;
      }
      for (int j = 0; ok && j < n; ++j) {
        const int c = j & 1;
        if (!mbar_wait_warp(v_full0 + 8u * vs, vph, a.wc) || !mbar_wait_warp(p_full0 + 8u * c, pph[c], a.wc)) {
          ok = false;
          break;
        }
        pph[c] ^= 1u;
        // the output accumulators are free once the previous item's epilogue has read them
        if (j == 0 && li > 0 && !mbar_wait_warp(o_free, (li - 1) & 1, a.wc)) { ok = false; break; }
        tc_fence_after();
        if (issuer) {
          mma_ts_tile(tmem + kColO + 128u * c, tmem + kColS + 128u * c, base + Y::kOffV + vs * kTile, idesc_o, j > 1);
          umma_commit<1>(pv_done0 + 8u * c);
          umma_commit<1>(v_empty0 + 8u * vs);
        }
        if (++vs == 2) { vs = 0; vph ^= 1u; }
        if (j + 2 < n && !issue_s(j + 2, j + 3 == n)) { ok = false; break; }
      }
    }
    // every MMA has completed before TMEM is released
    if (issuer) umma_commit<1>(final_bar);
    __syncwarp();
    drain(final_bar, 0);
  } else if (warp < kWarps) {
    // softmax and epilogue: query row r of each item's tile (TMEM lane r), key tiles c, c + 2, ...
    const int c = warp >> 2, r = (warp & 3) * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t sbuf = tmem + lane_off + kColS + 128u * c, orow = tmem + lane_off + kColO + 128u * c;
    float2* const ml = reinterpret_cast<float2*>(gbase + Y::kOffMl);  // [item parity][chain][row]
    uint32_t sph = 0;  // parity of the chain's next score product
    int done = 0;      // P V products of the chain so far
    int li = 0;
    for (int it = blockIdx.x; it < n_items; it += gridDim.x, ++li) {
      int qt, h, b;
      item_of(it, qt, h, b);
      const int n = qt + 1;
      float m = kNoMax, l = 0.0f;
      for (int j = c; j < n; j += 2) {
        if (!mbar_wait_warp(s_full0 + 8u * c, sph, a.wc)) { ok = false; break; }
        sph ^= 1u;
        tc_fence_after();
        // Half of the tile's 128 scores at a time: the registers hold 64 beside the products'.  Keys after
        // the row's query do not count in the diagonal tile.
        const bool diag = j == qt;
        uint32_t sr[2][32];
        auto load_half = [&](int hf) {
#pragma unroll
          for (int u = 0; u < 2; ++u) tmem_ld32(sbuf + 64u * hf + 32u * u, sr[u]);
          tmem_ld_wait();
          if (diag) {
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (64 * hf + 32 * u + i > r) sr[u][i] = __float_as_uint(-INFINITY);
          }
        };
        // the row maximum of the raw scores (scale > 0), in eight independent chains
        float mv[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) mv[i] = -INFINITY;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          load_half(hf);
#pragma unroll
          for (int u = 0; u < 2; ++u)
#pragma unroll
            for (int i = 0; i < 32; ++i) mv[i & 7] = fmaxf(mv[i & 7], __uint_as_float(sr[u][i]));
        }
#pragma unroll
        for (int w = 4; w > 0; w >>= 1)
#pragma unroll
          for (int i = 0; i < w; ++i) mv[i] = fmaxf(mv[i], mv[i + w]);
        const float mx = mv[0] * a.scale_log2;
        const bool raise = mx > m + kLazy;
        const float base = raise ? mx : m;
        const bool far = fabsf(base) >= 16777216.0f;  // (see weigh_far)
        if (__any_sync(0xffffffffu, far || (raise && j != c))) {
          // raise the maximum: past the item's first tile O's row (after the chain's previous P V) and l
          // scale by 2^(m - mx).  The warp goes together (tcgen05 loads and stores are the whole warp's):
          // rows that keep their maximum scale by 1.
          if (j != c) {
            const float f = raise ? fast_exp2(m - mx) : 1.0f;
            l *= f;
            if (!mbar_wait_warp(pv_done0 + 8u * c, (done - 1) & 1, a.wc)) { ok = false; break; }
            tc_fence_after();
#pragma unroll
            for (int u = 0; u < HD / 32; ++u) {
              uint32_t o[32];
              tmem_ld32(orow + 32u * u, o);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 32; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * f);
              tmem_st32(orow + 32u * u, o);
            }
          }
          if (__any_sync(0xffffffffu, far)) {
            m = base;
            l += weigh_far(sbuf, a.scale_log2, m, diag ? r : kTk);
            tmem_st_wait();
            warp_arrive(p_full0 + 8u * c, lane);
            ++done;
            continue;
          }
        }
        m = base;
        // P_j in bf16, each half over its own scores (the second half is still in registers)
        float ls[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) ls[i] = 0.0f;
#pragma unroll
        for (int hf = 1; hf >= 0; --hf) {
          if (hf == 0) load_half(0);
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            uint32_t pk[16];
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
              const float p0 = fast_exp2(fmaf(__uint_as_float(sr[u][i]), a.scale_log2, -m));
              const float p1 = fast_exp2(fmaf(__uint_as_float(sr[u][i + 1]), a.scale_log2, -m));
              ls[(i >> 1) & 7] += p0 + p1;
              pk[i / 2] = pack2(p0, p1);
            }
            tmem_st16(sbuf + 64u * hf + 16u * u, pk);
          }
        }
#pragma unroll
        for (int w = 4; w > 0; w >>= 1)
#pragma unroll
          for (int i = 0; i < w; ++i) ls[i] += ls[i + w];
        l += ls[0];
        tmem_st_wait();
        warp_arrive(p_full0 + 8u * c, lane);
        ++done;
      }
      // The chain's products have completed; the row's two halves meet.  (Threads whose wait gave up
      // come to the barrier too, and all leave together.)
      if (ok && c < n && !mbar_wait_warp(pv_done0 + 8u * c, (done - 1) & 1, a.wc)) ok = false;
      float2* const mine = ml + (li & 1) * 2 * kTq;
      mine[c * kTq + r] = make_float2(m, l);
      tc_fence_before();
      ok = bar_all(1, kElem, ok);
      if (!ok) break;
      tc_fence_after();
      const float2 e0 = mine[r], e1 = mine[kTq + r];  // chain 1 of a one-tile item: (kNoMax, 0)
      const float mm = fmaxf(e0.x, e1.x);
      const float f0 = fast_exp2(e0.x - mm), f1 = fast_exp2(e1.x - mm);
      const float lt = fmaf(e0.y, f0, e1.y * f1);
      const float w0 = f0 / lt, w1 = f1 / lt;
      const bool real = qt * kTq + r < a.S, two = n > 1;
      const int64_t ld = static_cast<int64_t>(a.nh) * HD;
      const int first = qt * kTq + (warp & 3) * 32;  // the warp's first query
      uint16_t* dst = a.out + (static_cast<int64_t>(b) * a.S + first) * ld + static_cast<int64_t>(h) * HD;
#pragma unroll
      for (int u = 0; u < HD / 64; ++u) {  // this warpgroup's half of the columns
        const int col = c * (HD / 2) + 32 * u;
        uint32_t o[32], q[32];
        tmem_ld32(tmem + lane_off + kColO + col, o);
        if (two) tmem_ld32(tmem + lane_off + kColO + 128u + col, q);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          float y = __uint_as_float(o[i]) * w0;
          if (two) y = fmaf(__uint_as_float(q[i]), w1, y);
          o[i] = __float_as_uint(y);
        }
        if (u + 1 == HD / 64) warp_arrive(o_free, lane);
        store_cols32(dst + col, ld, a.S - first, o, 1.0f, lane);
      }
      if (c == 0 && real)
        a.lse[(static_cast<int64_t>(b) * a.nh + h) * a.S + qt * kTq + r] = (mm + log2f(lt)) * 0.69314718055994531f;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc<1>(tmem, kTmemCols);
  }
}

// ---------------------------------------------------------------- backward
// With P = exp(scale S - lse) recomputed from the forward's log-sum-exp, dP = dO V^T and
// dS = P * (dP - delta) (delta = rowsum(dO * O), from attn_delta_kernel):
//   dQ = scale dS K,  dK = scale dS^T Q,  dV = P^T dO,
// in two kernels, so that every accumulator has one owner and no atomics are needed.

struct TcBwdArgs {
  uint16_t *dq, *dk, *dv;
  const float* lse;    // natural log-sum-exp per (sequence, head, row)
  const float* delta;  // rowsum(dO * O) per (sequence, head, row)
  int32_t B, S, nh, nkv;
  float scale_log2;
  float scale;
  WaitCtl wc;
};

constexpr float kLog2e = 1.4426950408889634f;

// dQ: persistent CTAs over (128-query tile, head, sequence) items, each over the key tiles up to the
// diagonal.  TMEM: S of tile t at 128 (t & 1) (dS over each warpgroup's own scores), dP [256, 384), dQ
// [384, 512).
template <int HD>
__global__ void __launch_bounds__(kThreadsDq, 1)
    attn_tc_dq_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmdo,
                      const __grid_constant__ CUtensorMap tmk, const __grid_constant__ CUtensorMap tmv,
                      const TcBwdArgs a) {
  using Y = Lay<HD>;
  constexpr uint32_t kTile = Y::kTile;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + (base - raw) + Y::kDqOffBar + 248);
  const uint32_t bar = base + Y::kDqOffBar;
  const uint32_t q_full = bar, q_empty = bar + 8, do_full = bar + 16, do_empty = bar + 24, k_full0 = bar + 32,
                 k_empty0 = bar + 56, v_full0 = bar + 80, v_empty0 = bar + 96, s_full0 = bar + 112, dp_full = bar + 128,
                 ds_full = bar + 136, item_done = bar + 144, dq_free = bar + 152, final_bar = bar + 160;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nqt = (a.S + kTq - 1) / kTq;
  const int n_items = nqt * a.nh * a.B;
  const ItemOf item_of{nqt, a.nh, a.B};
  constexpr uint32_t kColS = 0, kColP = 256, kColQ = 384;

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    mbar_init(do_full, 1);
    mbar_init(do_empty, 1);
    for (int i = 0; i < 3; ++i) {
      mbar_init(k_full0 + 8u * i, 1);
      mbar_init(k_empty0 + 8u * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(v_full0 + 8u * i, 1);
      mbar_init(v_empty0 + 8u * i, 1);
      mbar_init(s_full0 + 8u * i, 1);
    }
    mbar_init(dp_full, 1);
    mbar_init(ds_full, kWarps);
    mbar_init(item_done, 1);
    mbar_init(dq_free, kWarps);
    mbar_init(final_bar, 1);
    fence_mbar_init_cluster();
  }
  if (warp == kMmaWarp) tmem_alloc<1>(smem_u32(tmem_slot), kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;

  if (warp == kTmaWarp || warp == kTma2Warp) {
    // One warp copies Q and the K tiles (score products, dQ), the other dO and the V tiles (dP): neither
    // waits behind the other's buffers.
    if (lane == 0) {
      const bool first = warp == kTmaWarp;
      const CUtensorMap* const head_map = first ? &tmq : &tmdo;
      const CUtensorMap* const tile_map = first ? &tmk : &tmv;
      const uint32_t head_full = first ? q_full : do_full, head_empty = first ? q_empty : do_empty;
      const uint32_t full0 = first ? k_full0 : v_full0, empty0 = first ? k_empty0 : v_empty0;
      const uint32_t head_at = base + (first ? Y::kDqOffQ : Y::kDqOffDo);
      const uint32_t tile_at = base + (first ? Y::kDqOffK : Y::kDqOffV);
      const int ring = first ? 3 : 2;
      prefetch_tmap(head_map);
      prefetch_tmap(tile_map);
      int li = 0, heads = 0, loads = 0, s = 0;
      uint32_t ph = 1;
      for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x, ++li) {
        int qt, h, b;
        item_of(it, qt, h, b);
        const int hk = h / (a.nh / a.nkv);
        if (li > 0 && !mbar_wait(head_empty, (li - 1) & 1, a.wc)) { ok = false; break; }
        ++heads;
        mbar_arrive_expect_tx(head_full, kTile);
        for (int hf = 0; hf < Y::kBoxes; ++hf)
          tma_load_3d(head_at + hf * kBox, head_map, head_full, h * HD + 64 * hf, qt * kTq, b);
        for (int j = 0; j <= qt; ++j) {
          if (!mbar_wait(empty0 + 8u * s, ph, a.wc)) { ok = false; break; }
          mbar_arrive_expect_tx(full0 + 8u * s, kTile);
          for (int hf = 0; hf < Y::kBoxes; ++hf)
            tma_load_3d(tile_at + s * kTile + hf * kBox, tile_map, full0 + 8u * s, hk * HD + 64 * hf, j * kTk, b);
          ++loads;
          if (++s == ring) { s = 0; ph ^= 1u; }
        }
      }
      if (heads > 0) drain(head_full, (heads - 1) & 1);
      for (int t = max(0, loads - ring); t < loads; ++t) drain(full0 + 8u * (t % ring), (t / ring) & 1);
    }
  } else if (warp == kMmaWarp) {
    constexpr uint32_t idesc_s = idesc_bf16_f32(kTq, kTk, false, false);
    constexpr uint32_t idesc_q = idesc_bf16_f32(kTq, HD, false, true);
    const bool issuer = elect_one();
    // Three cursors over the CTA's stream of tiles: scores run two tiles ahead of dQ, dP one.
    struct Cursor {
      int it, li, j, n, t;  // item, its index, tile in it, its tiles, tile of the stream
    };
    auto enter = [&](Cursor& c) {
      c.j = 0;
      c.n = 0;
      if (c.it < n_items) c.n = nqt - c.it / (a.nh * a.B);
    };
    auto next = [&](Cursor& c) {
      ++c.t;
      if (++c.j < c.n) return;
      c.it += gridDim.x;
      ++c.li;
      enter(c);
    };
    Cursor sc{static_cast<int>(blockIdx.x), 0, 0, 0, 0};
    enter(sc);
    Cursor dc = sc, qc = sc;
    int sk = 0, qk = 0;  // K ring slots of the score and dQ cursors
    uint32_t skph = 0;
    auto issue_s = [&]() -> bool {  // the next score product, if there is one
      if (sc.it >= n_items) return true;
      if (sc.j == 0 && !mbar_wait_warp(q_full, sc.li & 1, a.wc)) return false;
      if (!mbar_wait_warp(k_full0 + 8u * sk, skph, a.wc)) return false;
      tc_fence_after();
      if (issuer) {
        mma_kmajor<HD>(tmem + kColS + 128u * (sc.t & 1), base + Y::kDqOffQ, base + Y::kDqOffK + sk * kTile, idesc_s);
        umma_commit<1>(s_full0 + 8u * (sc.t & 1));
        if (sc.j + 1 == sc.n) umma_commit<1>(q_empty);
      }
      if (++sk == 3) { sk = 0; skph ^= 1u; }
      next(sc);
      return true;
    };
    auto issue_dp = [&]() -> bool {  // the next dP = dO V^T
      if (dc.it >= n_items) return true;
      if (dc.j == 0 && !mbar_wait_warp(do_full, dc.li & 1, a.wc)) return false;
      if (!mbar_wait_warp(v_full0 + 8u * (dc.t & 1), (dc.t >> 1) & 1, a.wc)) return false;
      tc_fence_after();
      if (issuer) {
        mma_kmajor<HD>(tmem + kColP, base + Y::kDqOffDo, base + Y::kDqOffV + (dc.t & 1) * kTile, idesc_s);
        umma_commit<1>(dp_full);
        umma_commit<1>(v_empty0 + 8u * (dc.t & 1));
        if (dc.j + 1 == dc.n) umma_commit<1>(do_empty);
      }
      next(dc);
      return true;
    };
    if (!issue_s() || !issue_dp() || !issue_s()) ok = false;
    while (ok && qc.it < n_items) {
      if (!mbar_wait_warp(ds_full, qc.t & 1, a.wc)) { ok = false; break; }
      tc_fence_after();
      if (!issue_dp()) { ok = false; break; }  // (dP has been read: dS is ready)
      // the dQ accumulator is free once the previous item's epilogue has read it
      if (qc.j == 0 && qc.li > 0 && !mbar_wait_warp(dq_free, (qc.li - 1) & 1, a.wc)) { ok = false; break; }
      tc_fence_after();
      if (issuer) {
        mma_ts_tile(tmem + kColQ, tmem + kColS + 128u * (qc.t & 1), base + Y::kDqOffK + qk * kTile, idesc_q, qc.j > 0);
        umma_commit<1>(k_empty0 + 8u * qk);
        if (qc.j + 1 == qc.n) umma_commit<1>(item_done);
      }
      if (++qk == 3) qk = 0;
      next(qc);
      if (!issue_s()) { ok = false; break; }
    }
    if (issuer) umma_commit<1>(final_bar);
    __syncwarp();
    drain(final_bar, 0);
  } else {
    // query row r of the tile (TMEM lane r), keys 64 w .. 64 w + 63 of each key tile
    const int w = warp >> 2, r = (warp & 3) * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    int t = 0, li = 0;
    for (int it = blockIdx.x; ok && it < n_items; it += gridDim.x, ++li) {
      int qt, h, b;
      item_of(it, qt, h, b);
      const int n = qt + 1;
      const int64_t ridx = (static_cast<int64_t>(b) * a.nh + h) * a.S + qt * kTq + r;
      const bool real = qt * kTq + r < a.S;
      const float lse2 = real ? a.lse[ridx] * kLog2e : 0.0f, dl = real ? a.delta[ridx] : 0.0f;
      for (int j = 0; j < n; ++j, ++t) {
        const uint32_t scol = tmem + lane_off + kColS + 128u * (t & 1) + 64u * w;
        if (!mbar_wait_warp(s_full0 + 8u * (t & 1), (t >> 1) & 1, a.wc)) { ok = false; break; }
        tc_fence_after();
        uint32_t sv[2][32], pv[2][32];
#pragma unroll
        for (int u = 0; u < 2; ++u) tmem_ld32(scol + 32u * u, sv[u]);
        tmem_ld_wait();
        const bool diag = j == qt;
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            float p = fast_exp2(fmaf(__uint_as_float(sv[u][i]), a.scale_log2, -lse2));
            if (diag && 64 * w + 32 * u + i > r) p = 0.0f;
            sv[u][i] = __float_as_uint(p);
          }
        if (!mbar_wait_warp(dp_full, t & 1, a.wc)) { ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int u = 0; u < 2; ++u) tmem_ld32(tmem + lane_off + kColP + 64u * w + 32u * u, pv[u]);
        tmem_ld_wait();
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          uint32_t ds[16];
#pragma unroll
          for (int i = 0; i < 32; i += 2)
            ds[i / 2] = pack2(__uint_as_float(sv[u][i]) * (__uint_as_float(pv[u][i]) - dl),
                              __uint_as_float(sv[u][i + 1]) * (__uint_as_float(pv[u][i + 1]) - dl));
          tmem_st16(scol + 16u * u, ds);
        }
        tmem_st_wait();
        warp_arrive(ds_full, lane);
      }
      // every dQ product of the item has completed
      if (!ok || !mbar_wait_warp(item_done, li & 1, a.wc)) { ok = false; break; }
      tc_fence_after();
      const int64_t ld = static_cast<int64_t>(a.nh) * HD;
      const int first = qt * kTq + (warp & 3) * 32;  // the warp's first query
      uint16_t* dst = a.dq + (static_cast<int64_t>(b) * a.S + first) * ld + static_cast<int64_t>(h) * HD;
#pragma unroll
      for (int u = 0; u < HD / 64; ++u) {  // this warpgroup's half of the columns
        const int col = w * (HD / 2) + 32 * u;
        uint32_t o[32];
        tmem_ld32(tmem + lane_off + kColQ + col, o);
        tmem_ld_wait();
        if (u + 1 == HD / 64) warp_arrive(dq_free, lane);
        store_cols32(dst + col, ld, a.S - first, o, a.scale, lane);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc<1>(tmem, kTmemCols);
  }
}

// dK, dV: one CTA per (128-key tile, key/value head, sequence), over every query head of the
// group and the query tiles from the diagonal on, with the scores formed transposed (keys as
// TMEM lanes), so P^T and dS^T are the A operands of dV and dK straight from TMEM.
// TMEM: S^T [0, 128), dP^T [128, 256), dV [256, 384), dK [384, 512); P^T and dS^T (bf16) over each
// warpgroup's own scores and dP.
template <int HD>
__global__ void __launch_bounds__(kThreadsTc, 1)
    attn_tc_dkdv_kernel(const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmdo,
                        const __grid_constant__ CUtensorMap tmk, const __grid_constant__ CUtensorMap tmv,
                        const TcBwdArgs a) {
  using Y = Lay<HD>;
  constexpr uint32_t kTile = Y::kTile;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(gbase + Y::kKvOffBar + 96);
  const uint32_t bar = base + Y::kKvOffBar;
  const uint32_t kv_full = bar, st_full0 = bar + 8, st_empty0 = bar + 24, s_full = bar + 40, dp_full = bar + 48,
                 p_full = bar + 56, ds_full = bar + 64, final_bar = bar + 72;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nqt = (a.S + kTq - 1) / kTq;
  const int kt = static_cast<int>(blockIdx.x);  // key tile; the first ones have the most query tiles
  const int hk = blockIdx.y, b = blockIdx.z;
  const int rep = a.nh / a.nkv;
  const int nsteps = rep * (nqt - kt);  // query tiles kt .. nqt - 1 of each head of the group
  constexpr uint32_t kColS = 0, kColP = 128, kColV = 256, kColK = 384;
  struct Step {
    int h, i;  // query head, query tile
  };
  auto next = [&](Step& s) {
    if (++s.i == nqt) {
      s.i = kt;
      ++s.h;
    }
  };

  if (threadIdx.x == 0) {
    mbar_init(kv_full, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(st_full0 + 8u * i, 1);
      mbar_init(st_empty0 + 8u * i, 1);
    }
    mbar_init(s_full, 1);
    mbar_init(dp_full, 1);
    mbar_init(p_full, kWarps);
    mbar_init(ds_full, kWarps);
    mbar_init(final_bar, 1);
    fence_mbar_init_cluster();
  }
  if (warp == kMmaWarp) tmem_alloc<1>(smem_u32(tmem_slot), kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;

  if (warp == kTmaWarp) {
    if (lane == 0) {
      mbar_arrive_expect_tx(kv_full, 2 * kTile);
      for (int hf = 0; hf < Y::kBoxes; ++hf) {
        tma_load_3d(base + Y::kKvOffK + hf * kBox, &tmk, kv_full, hk * HD + 64 * hf, kt * kTk, b);
        tma_load_3d(base + Y::kKvOffV + hf * kBox, &tmv, kv_full, hk * HD + 64 * hf, kt * kTk, b);
      }
      int issued = 0;
      Step sp{hk * rep, kt};
      for (int t = 0; t < nsteps; ++t, next(sp)) {
        const int st = t & 1;
        if (t >= 2 && !mbar_wait(st_empty0 + 8u * st, ((t >> 1) & 1) ^ 1, a.wc)) { ok = false; break; }
        const uint32_t sb = base + Y::kKvOffStage + st * Y::kStageBytes;
        mbar_arrive_expect_tx(st_full0 + 8u * st, Y::kStageBytes);
        for (int hf = 0; hf < Y::kBoxes; ++hf) {
          tma_load_3d(sb + hf * kBox, &tmq, st_full0 + 8u * st, sp.h * HD + 64 * hf, sp.i * kTq, b);
          tma_load_3d(sb + kTile + hf * kBox, &tmdo, st_full0 + 8u * st, sp.h * HD + 64 * hf, sp.i * kTq, b);
        }
        issued = t + 1;
      }
      drain(kv_full, 0);
      for (int t = issued - 2 < 0 ? 0 : issued - 2; t < issued; ++t) drain(st_full0 + 8u * (t & 1), (t >> 1) & 1);
    }
  } else if (warp == kMmaWarp) {
    constexpr uint32_t idesc_s = idesc_bf16_f32(kTk, kTq, false, false);
    constexpr uint32_t idesc_g = idesc_bf16_f32(kTk, HD, false, true);
    const bool issuer = elect_one();
    auto stage = [&](int t) { return base + Y::kKvOffStage + (t & 1) * Y::kStageBytes; };
    auto issue_s = [&](int t) {  // S^T = K Q^T
      if (!issuer) return;
      mma_kmajor<HD>(tmem + kColS, base + Y::kKvOffK, stage(t), idesc_s);
      umma_commit<1>(s_full);
    };
    auto issue_dp = [&](int t) {  // dP^T = V dO^T
      if (!issuer) return;
      mma_kmajor<HD>(tmem + kColP, base + Y::kKvOffV, stage(t) + kTile, idesc_s);
      umma_commit<1>(dp_full);
    };
    if (!mbar_wait_warp(kv_full, 0, a.wc) || !mbar_wait_warp(st_full0, 0, a.wc)) ok = false;
    if (ok) {
      tc_fence_after();
      issue_s(0);
      issue_dp(0);
    }
    for (int t = 0; ok && t < nsteps; ++t) {
      // P^T is ready: dV, then the next scores over it, while dS^T is formed
      if (!mbar_wait_warp(p_full, t & 1, a.wc)) { ok = false; break; }
      tc_fence_after();
      if (issuer) mma_ts_tile(tmem + kColV, tmem + kColS, stage(t) + kTile, idesc_g, t > 0);  // dV += P^T dO
      if (t + 1 < nsteps) {
        if (!mbar_wait_warp(st_full0 + 8u * ((t + 1) & 1), ((t + 1) >> 1) & 1, a.wc)) { ok = false; break; }
        tc_fence_after();
        issue_s(t + 1);
      }
      // dS^T is ready: dK, then the next dP^T over it, while the next P^T is formed
      if (!mbar_wait_warp(ds_full, t & 1, a.wc)) { ok = false; break; }
      tc_fence_after();
      if (issuer) {
        mma_ts_tile(tmem + kColK, tmem + kColP, stage(t), idesc_g, t > 0);  // dK += dS^T Q
        umma_commit<1>(st_empty0 + 8u * (t & 1));
      }
      if (t + 1 < nsteps) issue_dp(t + 1);
    }
    if (issuer) umma_commit<1>(final_bar);
    __syncwarp();
    drain(final_bar, 0);
  } else {
    // key row rk of the tile (TMEM lane), queries 64 w .. 64 w + 63 of each query tile
    const int w = warp >> 2, rk = (warp & 3) * 32 + lane;
    const uint32_t lane_off = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const uint32_t scol = tmem + lane_off + kColS + 64u * w, pcol = tmem + lane_off + kColP + 64u * w;
    // Row rk of each step's query tile, its log-sum-exp (log2 units, warpgroup 0) or delta (1): loaded a
    // step ahead and handed to the other threads through shared memory; 0 past the sequence.
    float* const rows = reinterpret_cast<float*>(gbase + Y::kKvOffRow);
    Step sp{hk * rep, kt}, ahead = sp;
    auto fetch = [&]() {
      const int q = ahead.i * kTq + rk;
      const float* p = w == 0 ? a.lse : a.delta;
      return q < a.S ? __ldg(p + (static_cast<int64_t>(b) * a.nh + ahead.h) * a.S + q) * (w == 0 ? kLog2e : 1.0f) : 0.0f;
    };
    float row = fetch();
    for (int t = 0; t < nsteps; ++t, next(sp)) {
      // (every thread is past step t - 2, the buffer's last use, since the barrier of step t - 1)
      float* const lse = rows + (t & 1) * 2 * kTq;
      lse[w * kTq + rk] = row;
      next(ahead);
      if (t + 1 < nsteps) row = fetch();
      ok = bar_all(1, kElem, ok);
      if (!ok) break;
      const float4* const lse4 = reinterpret_cast<const float4*>(lse + 64 * w);
      const float4* const dlt4 = reinterpret_cast<const float4*>(lse + kTq + 64 * w);
      if (!mbar_wait_warp(s_full, t & 1, a.wc)) { ok = false; continue; }
      tc_fence_after();
      uint32_t sv[2][32], pv[2][32];
#pragma unroll
      for (int u = 0; u < 2; ++u) tmem_ld32(scol + 32u * u, sv[u]);
      tmem_ld_wait();
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const float4 l4 = lse4[(32 * u + i) / 4];
          const float lv[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
            sv[u][i + e] = __float_as_uint(fast_exp2(fmaf(__uint_as_float(sv[u][i + e]), a.scale_log2, -lv[e])));
        }
      // queries lo .. hi - 1 of the tile count for this key: from the diagonal on, and real
      const bool diag = sp.i == kt;
      const int lo = (diag ? rk : 0) - 64 * w, hi = min(kTq, a.S - sp.i * kTq) - 64 * w;
      const bool edge = diag || hi < 64;
      if (edge) {
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (32 * u + i < lo || 32 * u + i >= hi) sv[u][i] = 0u;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        uint32_t pp[16];
#pragma unroll
        for (int i = 0; i < 32; i += 2) pp[i / 2] = pack2(__uint_as_float(sv[u][i]), __uint_as_float(sv[u][i + 1]));
        tmem_st16(scol + 16u * u, pp);
      }
      tmem_st_wait();
      warp_arrive(p_full, lane);
      if (!mbar_wait_warp(dp_full, t & 1, a.wc)) { ok = false; continue; }
      tc_fence_after();
#pragma unroll
      for (int u = 0; u < 2; ++u) tmem_ld32(pcol + 32u * u, pv[u]);
      tmem_ld_wait();
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        uint32_t ds[16];
#pragma unroll
        for (int i = 0; i < 32; i += 4) {
          const float4 d4 = dlt4[(32 * u + i) / 4];
          const float dv[4] = {d4.x, d4.y, d4.z, d4.w};
          float e4[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            e4[e] = __uint_as_float(sv[u][i + e]) * (__uint_as_float(pv[u][i + e]) - dv[e]);
          ds[i / 2] = pack2(e4[0], e4[1]);
          ds[i / 2 + 1] = pack2(e4[2], e4[3]);
        }
        tmem_st16(pcol + 16u * u, ds);
      }
      tmem_st_wait();
      warp_arrive(ds_full, lane);
    }
    if (ok && mbar_wait_warp(final_bar, 0, a.wc)) {  // every MMA has completed (one phase)
      tc_fence_after();
      const int64_t ld = static_cast<int64_t>(a.nkv) * HD;
      const int first = kt * kTk + (warp & 3) * 32;  // the warp's first key
      uint16_t* dst = (w == 0 ? a.dk : a.dv) + (static_cast<int64_t>(b) * a.S + first) * ld + static_cast<int64_t>(hk) * HD;
      const uint32_t col = w == 0 ? kColK : kColV;  // warpgroup 0 writes dK, 1 dV
#pragma unroll
      for (int u = 0; u < HD / 32; ++u) {
        uint32_t o[32];
        tmem_ld32(tmem + lane_off + col + 32u * u, o);
        tmem_ld_wait();
        store_cols32(dst + 32 * u, ld, a.S - first, o, w == 0 ? a.scale : 1.0f, lane);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc<1>(tmem, kTmemCols);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 g_enc = nullptr;
std::once_flag g_enc_once;

// bf16 row-major [B, S, inner] tensor, 128-byte swizzled boxes of 64 columns x 128 tokens of one
// sequence; tokens past a sequence's end read as zeros.
bool tmap_rows(CUtensorMap* m, const void* ptr, uint64_t inner, uint64_t S, uint64_t B) {
  std::call_once(g_enc_once, [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_enc = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  });
  if (!g_enc) return false;
  const cuuint64_t dims[3] = {inner, S, B};
  const cuuint64_t strides[2] = {inner * 2, inner * 2 * S};
  const cuuint32_t box[3] = {64, 128, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return g_enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int sm_count() {
  int sm = 152, dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev);
  return sm;
}

template <int HD>
cudaError_t run_fwd(const void* q, const void* k, const void* v, void* out, float* lse, int32_t B, int32_t S, int32_t nh,
                    int32_t nkv, cudaStream_t st) {
  CUtensorMap tq, tk, tv;
  if (!tmap_rows(&tq, q, static_cast<uint64_t>(nh) * HD, S, B) ||
      !tmap_rows(&tk, k, static_cast<uint64_t>(nkv) * HD, S, B) ||
      !tmap_rows(&tv, v, static_cast<uint64_t>(nkv) * HD, S, B))
    return cudaErrorInvalidValue;
  TcAttnArgs a{};
  a.out = static_cast<uint16_t*>(out);
  a.lse = lse;
  a.B = B;
  a.S = S;
  a.nh = nh;
  a.nkv = nkv;
  a.scale_log2 = 1.4426950408889634f / sqrtf(static_cast<float>(HD));
  if (!launch_wait_ctl(&a.wc)) return cudaErrorInvalidDevice;
  cudaError_t e = cudaFuncSetAttribute(attn_tc_fwd_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       Lay<HD>::kSmem);
  if (e != cudaSuccess) return e;
  const int64_t items = static_cast<int64_t>((S + kTq - 1) / kTq) * nh * B;
  // persistent: one CTA per SM (the 512 TMEM columns allow no second), each taking every
  // gridDim-th work item
  attn_tc_fwd_kernel<HD><<<static_cast<unsigned>(std::min<int64_t>(items, sm_count())), kThreadsTc, Lay<HD>::kSmem,
                           st>>>(tq, tk, tv, a);
  return cudaGetLastError();
}

template <int HD>
cudaError_t run_bwd(const void* q, const void* k, const void* v, const void* dO, const float* lse, const float* delta,
                    void* dq, void* dk, void* dv, int32_t B, int32_t S, int32_t nh, int32_t nkv, cudaStream_t st) {
  CUtensorMap tq, tdo, tk, tv;
  if (!tmap_rows(&tq, q, static_cast<uint64_t>(nh) * HD, S, B) ||
      !tmap_rows(&tdo, dO, static_cast<uint64_t>(nh) * HD, S, B) ||
      !tmap_rows(&tk, k, static_cast<uint64_t>(nkv) * HD, S, B) ||
      !tmap_rows(&tv, v, static_cast<uint64_t>(nkv) * HD, S, B))
    return cudaErrorInvalidValue;
  TcBwdArgs a{};
  a.dq = static_cast<uint16_t*>(dq);
  a.dk = static_cast<uint16_t*>(dk);
  a.dv = static_cast<uint16_t*>(dv);
  a.lse = lse;
  a.delta = delta;
  a.B = B;
  a.S = S;
  a.nh = nh;
  a.nkv = nkv;
  a.scale = 1.0f / sqrtf(static_cast<float>(HD));
  a.scale_log2 = a.scale * kLog2e;
  if (!launch_wait_ctl(&a.wc)) return cudaErrorInvalidDevice;
  cudaError_t e = cudaFuncSetAttribute(attn_tc_dq_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       Lay<HD>::kDqSmem);
  if (e != cudaSuccess) return e;
  const int tiles = (S + kTq - 1) / kTq;
  const int64_t items = static_cast<int64_t>(tiles) * nh * B;
  attn_tc_dq_kernel<HD><<<static_cast<unsigned>(std::min<int64_t>(items, sm_count())), kThreadsDq, Lay<HD>::kDqSmem,
                          st>>>(tq, tdo, tk, tv, a);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = cudaFuncSetAttribute(attn_tc_dkdv_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay<HD>::kKvSmem);
  if (e != cudaSuccess) return e;
  attn_tc_dkdv_kernel<HD><<<dim3(tiles, nkv, B), kThreadsTc, Lay<HD>::kKvSmem, st>>>(tq, tdo, tk, tv, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_attention_fwd_tc(const void* q, const void* k, const void* v, void* out, float* lse, int32_t B,
                                    int32_t S, int32_t nh, int32_t nkv, int32_t d, cudaStream_t st) {
  return d == 128 ? run_fwd<128>(q, k, v, out, lse, B, S, nh, nkv, st)
                  : run_fwd<64>(q, k, v, out, lse, B, S, nh, nkv, st);
}

cudaError_t launch_attention_bwd_tc(const void* q, const void* k, const void* v, const void* dO, const float* lse,
                                    const float* delta, void* dq, void* dk, void* dv, int32_t B, int32_t S, int32_t nh,
                                    int32_t nkv, int32_t d, cudaStream_t st) {
  return d == 128 ? run_bwd<128>(q, k, v, dO, lse, delta, dq, dk, dv, B, S, nh, nkv, st)
                  : run_bwd<64>(q, k, v, dO, lse, delta, dq, dk, dv, B, S, nh, nkv, st);
}

}  // namespace catq
