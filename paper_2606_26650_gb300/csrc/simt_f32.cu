// simt_f32.cu — fp32 CUDA-core path of the three contractions, used when W and X are fp32
// (a tensor-core path cannot meet an fp32 tolerance).  Tiled FFMA GEMMs with fp32 accumulation
// and accurate tanhf.  The Eq. 6 weight is computed while its tile is staged into shared memory,
// and the dW contraction reduces straight into per-group partial sums (G = dY^T X is never
// stored).
//
// C[i][j] = sum_c A(i, c) B(j, c) with
//   FWD: i = m, j = n, c = k:  A = X[m][k],  B = Wq[n][k]
//   DX : i = m, j = k, c = n:  A = dY[m][n], B = Wq[n][k]
//   DW : i = n, j = k, c = m:  A = dY[m][n], B = X[m][k]
//
// A CTA of 256 threads owns TI x TJ outputs (8192 of them, 8 x 4 a thread: 3 16-byte shared loads
// for 32 multiply-adds) over a share of the contraction; the S CTAs of a cluster hold one tile's
// partial sums and add them through distributed shared memory in rank order, each finishing its
// part of the rows.  Slices of 16 are double-buffered, the next one's global loads in flight
// while one is multiplied.  Bound by the FMA pipe and, for FWD and DX, by the weight transform
// (two tanhf a weight and row tile, the cost of about 80 multiply-adds): tall tiles (TI = 256)
// transform each weight once per 256 rows, wide ones (TI = 32) serve few rows.  A whole step of the
// 512 x 512 layer on 1024 rows (the three contractions, loss and update), one GB300: 298 -> 104 us
// against 64 x 64 tiles with 4 x 4 outputs a thread, scalar loads, and the group's constants and
// the transform formed anew for every row tile of 64 (110, 128 and 116 us of it, 16 % of the FMA
// pipe, 64 to 128 CTAs).
#include <algorithm>

#include "launch.h"
#include "ptx_sm100.cuh"

namespace catq {
namespace {

constexpr int TK = 16;  // contraction slice
constexpr int kThr = 256;
constexpr int kMi = 8, kMj = 4;  // outputs of a thread
constexpr int kPad = 4;          // floats after a slice row (16-byte rows, two-way store conflicts)

enum : int { MODE_FWD = 0, MODE_DX = 1, MODE_DW = 2 };

struct SimtArgs {
  LayerDev L;
  StepScalars sc;
  const float* A;  // FWD: X [M,K]; DX: dY [M,N]; DW: dY [M,N]
  const float* B;  // DW: X [M,K]; otherwise unused (W comes from L)
  float* C;        // FWD: Y [M,N]; DX: dX [M,K]; DW: partials [3][N][K/P]
  int64_t M;
  int32_t P;       // DW partial chunk width
  int32_t splits;  // CTAs per tile (the cluster's size along z)
  const float* row_scale;  // FWD, nullable: Y row m times row_scale[m]
};

// N values at p, element q valid when q < limit (16- or 8-byte load when all are and `vec`).
template <int N>
__device__ __forceinline__ void load_run(const float* p, int64_t limit, bool vec, float (&v)[N]) {
  if (vec && limit >= N) {
    if constexpr (N == 2) {
      const float2 q = __ldg(reinterpret_cast<const float2*>(p));
      v[0] = q.x;
      v[1] = q.y;
    } else {
      static_assert(N % 4 == 0, "runs are 2 or a multiple of 4");
#pragma unroll
      for (int i = 0; i < N; i += 4) {
        const float4 q = __ldg(reinterpret_cast<const float4*>(p + i));
        v[i] = q.x;
        v[i + 1] = q.y;
        v[i + 2] = q.z;
        v[i + 3] = q.w;
      }
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = i < limit ? __ldg(p + i) : 0.0f;
}

// Staging of one operand, R rows (the tile's i or j) x TK contraction columns, by 256 threads with V
// consecutive values each.  C_MAJOR: memory runs along the rows (one run per contraction index),
// otherwise along the contraction.
template <int R, bool C_MAJOR>
struct Stage {
  static constexpr int V0 = R * TK / kThr;
  static constexpr int V = V0 > 4 ? 4 : V0;  // values per run
  static constexpr int kRuns = R * TK / (kThr * V);
  static constexpr int kPerLine = (C_MAJOR ? R : TK) / V;  // runs per memory line
  __device__ static __forceinline__ int row(int u) {
    const int e = threadIdx.x + u * kThr;
    return C_MAJOR ? (e % kPerLine) * V : e / kPerLine;
  }
  __device__ static __forceinline__ int col(int u) {
    const int e = threadIdx.x + u * kThr;
    return C_MAJOR ? e / kPerLine : (e % kPerLine) * V;
  }
  __device__ static __forceinline__ void store(float (*s)[R + kPad], int u, const float (&v)[V]) {
    const int r = row(u), c = col(u);
    if constexpr (C_MAJOR) {
      if constexpr (V == 4) *reinterpret_cast<float4*>(&s[c][r]) = make_float4(v[0], v[1], v[2], v[3]);
      else *reinterpret_cast<float2*>(&s[c][r]) = make_float2(v[0], v[1]);
    } else {
#pragma unroll
      for (int i = 0; i < V; ++i) s[c + i][r] = v[i];
    }
  }
};

template <int MODE, int TI, int TJ>
struct SimtSmem {
  static_assert(TI * TJ == kThr * kMi * kMj, "8 x 4 outputs a thread");
  union {
    struct {
      float As[2][TK][TI + kPad];
      float Bs[2][TK][TJ + kPad];
    };
    float out[TI][TJ];  // the CTA's partial sums
  };
};

template <int MODE, int TI, int TJ>
__global__ void __launch_bounds__(kThr, 2) simt_gemm_kernel(const __grid_constant__ SimtArgs a) {
  extern __shared__ __align__(16) uint8_t smem_raw[];
  using Smem = SimtSmem<MODE, TI, TJ>;
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  const LayerDev& L = a.L;
  const int64_t rowsI = MODE == MODE_DW ? L.N : a.M;
  const int64_t colsJ = MODE == MODE_FWD ? L.N : L.K;
  const int64_t depth = MODE == MODE_FWD ? L.K : (MODE == MODE_DX ? L.N : a.M);
  const int64_t i0 = static_cast<int64_t>(blockIdx.y) * TI;
  const int64_t j0 = static_cast<int64_t>(blockIdx.x) * TJ;
  const int rank = static_cast<int>(blockIdx.z), S = a.splits;
  const int64_t slices = (depth + TK - 1) / TK;
  const int64_t s0 = slices * rank / S, s1 = slices * (rank + 1) / S;
  constexpr int kTx = TJ / kMj;  // threads along j
  const int tx = threadIdx.x % kTx, ty = threadIdx.x / kTx;

  using SA = Stage<TI, MODE == MODE_DW>;
  using SB = Stage<TJ, MODE != MODE_FWD>;
  // 16-byte (8-byte) runs of A need rows of a whole number of them; K is a multiple of 4 always
  const bool vec_a = MODE == MODE_FWD || L.N % 4 == 0;
  const bool transform = MODE != MODE_DW && a.sc.phase != PHASE_TEACHER;
  float ra[SA::kRuns][SA::V], rb[SB::kRuns][SB::V];
  GroupRaw rg[MODE == MODE_DW ? 1 : SB::kRuns];
  int64_t have[SB::kRuns];
#pragma unroll
  for (int u = 0; u < SB::kRuns; ++u) have[u] = -1;

  auto fetch = [&](int64_t slice) {
    const int64_t c0 = slice * TK;
#pragma unroll
    for (int u = 0; u < SA::kRuns; ++u) {
      const int64_t i = i0 + SA::row(u), c = c0 + SA::col(u);
      if constexpr (MODE == MODE_DW)  // dY[m][n], runs along n
        load_run<SA::V>(a.A + c * L.N + i, c < depth ? rowsI - i : 0, vec_a, ra[u]);
      else  // X[m][k] or dY[m][n], runs along the contraction
        load_run<SA::V>(a.A + i * (MODE == MODE_FWD ? L.K : L.N) + c, i < rowsI ? depth - c : 0, vec_a, ra[u]);
    }
#pragma unroll
    for (int u = 0; u < SB::kRuns; ++u) {
      const int64_t j = j0 + SB::row(u), c = c0 + SB::col(u);
      const bool in = j < colsJ && c < depth;
      if constexpr (MODE == MODE_DW) {
        load_run<SB::V>(a.B + c * L.K + j, in ? colsJ - j : 0, true, rb[u]);
      } else {
        // W[n][k], runs along k: a run lies in one group (g and the run's start are multiples of 4)
        const int64_t n = MODE == MODE_FWD ? j : c, k = MODE == MODE_FWD ? c : j;
        load_run<SB::V>(static_cast<const float*>(L.W) + n * L.K + k, in ? L.K - k : 0, true, rb[u]);
        const int64_t g = in && transform ? n * L.groups_per_row + k / L.g : -1;
        if (g >= 0 && g != have[u]) rg[u] = group_raw(L, g);
        have[u] = g;
      }
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int u = 0; u < SA::kRuns; ++u) SA::store(sm.As[buf], u, ra[u]);
#pragma unroll
    for (int u = 0; u < SB::kRuns; ++u) {
      if constexpr (MODE != MODE_DW) {
        if (have[u] >= 0) {
          const GroupConst gc = group_const(rg[u]);
#pragma unroll
          for (int q = 0; q < SB::V; ++q)
            rb[u][q] = ternary_weight_f32(rb[u][q], gc, a.sc.s, a.sc.inv_2tanh_s, a.sc.phase, L.recon);
        }
      }
      SB::store(sm.Bs[buf], u, rb[u]);
    }
  };

  float acc[kMi][kMj] = {};
  if (s0 < s1) {
    fetch(s0);
    put(0);
    __syncthreads();
    for (int64_t s = s0; s < s1; ++s) {
      const int buf = static_cast<int>(s - s0) & 1;
      if (s + 1 < s1) fetch(s + 1);
#pragma unroll
      for (int c = 0; c < TK; ++c) {
        float av[kMi], bv[kMj];
#pragma unroll
        for (int u = 0; u < kMi; u += 4) {
          const float4 q = *reinterpret_cast<const float4*>(&sm.As[buf][c][ty * kMi + u]);
          av[u] = q.x;
          av[u + 1] = q.y;
          av[u + 2] = q.z;
          av[u + 3] = q.w;
        }
        const float4 q = *reinterpret_cast<const float4*>(&sm.Bs[buf][c][tx * kMj]);
        bv[0] = q.x;
        bv[1] = q.y;
        bv[2] = q.z;
        bv[3] = q.w;
#pragma unroll
        for (int u = 0; u < kMi; ++u)
#pragma unroll
          for (int v = 0; v < kMj; ++v) acc[u][v] = fmaf(av[u], bv[v], acc[u][v]);
      }
      if (s + 1 < s1) put(buf ^ 1);
      __syncthreads();
    }
  }

  // The partial tile goes to shared memory; each CTA adds its share of the rows over the cluster.
#pragma unroll
  for (int u = 0; u < kMi; ++u)
    *reinterpret_cast<float4*>(&sm.out[ty * kMi + u][tx * kMj]) =
        make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]);
  if (S > 1) cluster_sync_all(); else __syncthreads();
  const int r1 = TI * (rank + 1) / S;
  constexpr int kRowsAtOnce = kThr / kTx;
  // every thread of a warp takes part in the chunk sums of MODE_DW: the loop is uniform
  for (int rb0 = TI * rank / S; rb0 < r1; rb0 += kRowsAtOnce) {
    const int r = rb0 + ty;
    const int64_t i = i0 + r, j = j0 + tx * kMj;
    float y[kMj] = {};
    if (r < r1) {
      const uint32_t at = smem_u32(&sm.out[r][tx * kMj]);
      for (int p = 0; p < S; ++p) {
        const float4 q = S > 1 ? ld_cluster_f4(mapa_shared(at, p)) : *reinterpret_cast<const float4*>(&sm.out[r][tx * kMj]);
        y[0] += q.x;
        y[1] += q.y;
        y[2] += q.z;
        y[3] += q.w;
      }
    }
    const bool live = r < r1 && i < rowsI && j < colsJ;
    if constexpr (MODE != MODE_DW) {
      if (!live) continue;
      if (a.row_scale) {
        const float rs = __ldg(a.row_scale + i);
#pragma unroll
        for (int v = 0; v < kMj; ++v) y[v] *= rs;
      }
      float* dst = a.C + i * colsJ + j;
      if (colsJ % 4 == 0) {
        *reinterpret_cast<float4*>(dst) = make_float4(y[0], y[1], y[2], y[3]);
      } else {
#pragma unroll
        for (int v = 0; v < kMj; ++v)
          if (j + v < colsJ) dst[v] = y[v];
      }
    } else {
      // Chain rule on the thread's 4 columns (one group), then the sum over the P / 4 lanes of
      // the chunk of P columns (fixed xor order: deterministic).
      GradSums e{0.f, 0.f, 0.f};
      if (live) {
        const GroupConst gc = group_const(L, i * L.groups_per_row + j / L.g);
        if (gc.alpha != 0.0f) {
          const float4 w = __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(L.W) + i * L.K + j));
          const float wv[4] = {w.x, w.y, w.z, w.w};
          if (L.recon) {
            const float inv_k = 1.0f / (a.sc.s * a.sc.inv_2tanh_s);
#pragma unroll
            for (int v = 0; v < kMj; ++v)
              grad_element<false, true>(y[v], wv[v], gc, a.sc.s, a.sc.inv_2tanh_s, a.sc.phase, e, inv_k);
          } else {
#pragma unroll
            for (int v = 0; v < kMj; ++v) grad_element(y[v], wv[v], gc, a.sc.s, a.sc.inv_2tanh_s, a.sc.phase, e);
          }
        }
      }
      const int lanes = a.P / kMj;
      for (int o = 1; o < lanes; o <<= 1) {
        e.smu += __shfl_xor_sync(0xffffffffu, e.smu, o);
        e.salpha += __shfl_xor_sync(0xffffffffu, e.salpha, o);
        e.sdelta += __shfl_xor_sync(0xffffffffu, e.sdelta, o);
      }
      if (live && tx % lanes == 0) {
        const int64_t cpr = L.K / a.P, plane = L.N * cpr, idx = i * cpr + j / a.P;
        a.C[idx] = e.smu;
        a.C[plane + idx] = e.salpha;
        a.C[2 * plane + idx] = e.sdelta;
      }
    }
  }
  if (S > 1) cluster_sync_all();  // peers have read this CTA's partial sums
}

template <int MODE, int TI, int TJ>
cudaError_t launch(SimtArgs& a, int64_t rows, int64_t cols, int64_t depth, cudaStream_t st) {
  const int64_t ti = (rows + TI - 1) / TI, tj = (cols + TJ - 1) / TJ;
  if (ti > 65535) return cudaErrorInvalidValue;
  // shares of the contraction until every SM has about two CTAs, each with two slices or more
  int s = 1;
  while (s < 8 && ti * tj * s * 2 <= 4 * 152 && (depth + TK - 1) / TK >= 4 * s) s *= 2;
  a.splits = s;
  constexpr int smem = static_cast<int>(sizeof(SimtSmem<MODE, TI, TJ>));
  auto kern = simt_gemm_kernel<MODE, TI, TJ>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(tj), static_cast<unsigned>(ti), static_cast<unsigned>(s));
  cfg.blockDim = dim3(kThr);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = static_cast<unsigned>(s);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

// FWD and DX: the tile height by the least of padded rows (a multiply-add each per weight) and weight
// transforms (about 80, once per row tile; a copy's 8).
template <int MODE>
cudaError_t launch_rows(SimtArgs& a, int64_t cols, int64_t depth, cudaStream_t st) {
  const int xf = a.sc.phase == PHASE_TEACHER ? 8 : 80;
  auto cost = [&](int64_t ti) { return (a.M + ti - 1) / ti * (ti + xf); };
  const int64_t c32 = cost(32), c128 = cost(128), c256 = cost(256);
  if (c32 < c128 && c32 < c256) return launch<MODE, 32, 256>(a, a.M, cols, depth, st);
  if (c128 < c256) return launch<MODE, 128, 64>(a, a.M, cols, depth, st);
  return launch<MODE, 256, 32>(a, a.M, cols, depth, st);
}

}  // namespace

cudaError_t launch_simt_fwd(const LayerDev& L, StepScalars sc, const float* X, int64_t M, float* Y, cudaStream_t st,
                            const float* row_scale) {
  SimtArgs a{L, sc, X, nullptr, Y, M, 0, 1, row_scale};
  return launch_rows<MODE_FWD>(a, L.N, L.K, st);
}

cudaError_t launch_simt_dx(const LayerDev& L, StepScalars sc, const float* dY, int64_t M, float* dX, cudaStream_t st) {
  SimtArgs a{L, sc, dY, nullptr, dX, M, 0, 1, nullptr};
  return launch_rows<MODE_DX>(a, L.K, L.N, st);
}

cudaError_t launch_simt_dw(const LayerDev& L, StepScalars sc, const float* X, const float* dY, int64_t M,
                           float* partials, cudaStream_t st) {
  const int32_t P = L.g < kSimtTile ? L.g : kSimtTile;
  SimtArgs a{L, sc, dY, X, partials, M, P, 1, nullptr};
  return launch<MODE_DW, 128, 64>(a, L.N, L.K, M, st);
}

}  // namespace catq
