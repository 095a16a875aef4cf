// block.cu — the layers around the seven soft-ternary linears of one decoder block, for the
// block-output reconstruction step (§2.4, Eq. 7 over a window of one block): RMSNorm (with the
// residual add fused into the forward, and the residual and second upstream gradient fused
// into the backward; one CTA per long row, a team of lanes per short row such as an attention head),
// rotary position embedding, SwiGLU, the fp32 block output with the loss on it, and the row sums
// the attention backward needs.  The attention itself runs on tcgen05 (attn_tc.cu).
#include <cuda_bf16.h>

#include <algorithm>

#include "launch.h"
#include "ptx_sm100.cuh"

namespace catq {
namespace {

constexpr int kRowThreads = 256;

__device__ __forceinline__ float bf16_at(const uint16_t* p, int64_t i) { return __uint_as_float(uint32_t(p[i]) << 16); }
__device__ __forceinline__ uint16_t to_bf16(float v) { return static_cast<uint16_t>(pack_bf16x2(v, 0.0f) & 0xFFFFu); }

__device__ __forceinline__ float team_sum(float v, int team) {
  for (int o = team >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ float block_sum(float v, float* red) {
  v = team_sum(v, 32);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) red[w] = v;
  __syncthreads();
  float t = 0.0f;
#pragma unroll
  for (int i = 0; i < kRowThreads / 32; ++i) t += red[i];
  return t;
}

// ---------------------------------------------------------------- RMSNorm
// Both directions are bound by HBM: a row's 16-byte vectors (8 elements) are loaded once, kept
// as loaded (bf16 packed) in registers through the row's sum and unpacked again for the output,
// so that a thread holds many rows' or vectors' loads in flight.  A row of at most 1024 elements
// belongs to a team of lanes (16 lanes for a 128-wide attention head, so a warp holds two rows at
// a time, four times over), a longer one to a CTA; VPL vectors per thread.  On one GB300, against
// kernels that loaded 2-byte elements twice: backward of 8192 rows of 4096 (fp32 row, two
// gradients and the residual's, 403 MB) 124 -> 64 us = 6.3 TB/s, forward 76 -> 60 us; backward of
// 262144 head rows of 128 (201 MB) 64 -> 49 us, forward (134 MB) 47 -> 27 us.
__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = bf16lo_to_f32(w[i]);
    f[2 * i + 1] = bf16hi_to_f32(w[i]);
  }
}

__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
  return make_uint4(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3]), pack_bf16x2(f[4], f[5]),
                    pack_bf16x2(f[6], f[7]));
}

// Eight consecutive elements as loaded.
template <typename T>
struct Raw8;
template <>
struct Raw8<uint16_t> {
  uint4 q;
  __device__ __forceinline__ void load(const uint16_t* p) { q = *reinterpret_cast<const uint4*>(p); }
  __device__ __forceinline__ void zero() { q = make_uint4(0u, 0u, 0u, 0u); }
  __device__ __forceinline__ void get(float (&f)[8]) const { unpack8(q, f); }
};
template <>
struct Raw8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p) {
    a = reinterpret_cast<const float4*>(p)[0];
    b = reinterpret_cast<const float4*>(p)[1];
  }
  __device__ __forceinline__ void zero() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ void get(float (&f)[8]) const {
    f[0] = a.x; f[1] = a.y; f[2] = a.z; f[3] = a.w;
    f[4] = b.x; f[5] = b.y; f[6] = b.z; f[7] = b.w;
  }
};

__device__ __forceinline__ void load8(const uint16_t* p, float (&f)[8]) {
  unpack8(*reinterpret_cast<const uint4*>(p), f);
}
// The norm's weights carry no alignment beyond their type's: GVEC when they are 16-byte aligned.
template <bool GVEC>
__device__ __forceinline__ void load_gamma8(const float* p, float (&f)[8]) {
  if constexpr (GVEC) {
    Raw8<float> v;
    v.load(p);
    v.get(f);
  } else {
    // aligned vectors of the eight, the rest one by one: p is 4, 8 or 12 bytes past a 16-byte boundary, the
    // same in every thread (8192 rows of 4096 in bf16: forward 43 -> 32 us with 8 loads as 3 or 4)
    auto one = [&](int i) { f[i] = __ldg(p + i); };
    auto two = [&](int i) {
      const float2 v = __ldg(reinterpret_cast<const float2*>(p + i));
      f[i] = v.x; f[i + 1] = v.y;
    };
    auto four = [&](int i) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(p + i));
      f[i] = v.x; f[i + 1] = v.y; f[i + 2] = v.z; f[i + 3] = v.w;
    };
    const uint32_t off = (static_cast<uint32_t>(reinterpret_cast<uintptr_t>(p)) >> 2) & 3u;
    if (off == 2) {
      two(0); four(2); two(6);
    } else if (off == 1) {
      one(0); two(1); four(3); one(7);
    } else {
      one(0); four(1); two(5); one(7);
    }
  }
}

// One vector of the forward: h = x (+ residual in fp32, never rounded).
template <typename TX>
struct FwdVec {
  Raw8<TX> x;
  Raw8<uint16_t> res;
  __device__ __forceinline__ void load(const TX* xp, const uint16_t* rp, int64_t at) {
    x.load(xp + at);
    if (rp) res.load(rp + at);
  }
  __device__ __forceinline__ void h(bool with_res, float (&f)[8]) const {
    x.get(f);
    if (with_res) {
      float q[8];
      res.get(q);
#pragma unroll
      for (int i = 0; i < 8; ++i) f[i] += q[i];
    }
  }
  // its squares added to s; h stored when h_out is given
  __device__ __forceinline__ float sum(bool with_res, float* h_out, int64_t at, float s) const {
    float f[8];
    h(with_res, f);
    if (h_out) {
      reinterpret_cast<float4*>(h_out + at)[0] = make_float4(f[0], f[1], f[2], f[3]);
      reinterpret_cast<float4*>(h_out + at)[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) s = fmaf(f[i], f[i], s);
    return s;
  }
  // z = gamma * h * r
  template <bool GVEC>
  __device__ __forceinline__ void store_z(bool with_res, const float* gamma, int64_t col, float rr, uint16_t* z) const {
    float f[8], g[8];
    h(with_res, f);
    load_gamma8<GVEC>(gamma + col, g);
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = g[i] * f[i] * rr;
    *reinterpret_cast<uint4*>(z) = pack8(f);
  }
};

// One vector of the backward: dx = r u - h r^3 mean(u h) (+ dres), u = gamma (dy + dy2).
template <typename TH>
struct BwdVec {
  Raw8<TH> x;
  Raw8<uint16_t> dy, dy2, dres;
  __device__ __forceinline__ void load(const TH* xp, const uint16_t* d1, const uint16_t* d2, const uint16_t* dr,
                                       int64_t at) {
    dy.load(d1 + at);
    if (d2) dy2.load(d2 + at);
    x.load(xp + at);
    if (dr) dres.load(dr + at);
  }
  template <bool GVEC>
  __device__ __forceinline__ void u(bool two, const float* gamma, int64_t col, float (&f)[8]) const {
    float g[8];
    dy.get(f);
    if (two) {
      float q[8];
      dy2.get(q);
#pragma unroll
      for (int i = 0; i < 8; ++i) f[i] += q[i];
    }
    load_gamma8<GVEC>(gamma + col, g);
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] *= g[i];
  }
  template <bool GVEC>
  __device__ __forceinline__ float dot(bool two, const float* gamma, int64_t col, float s) const {
    float f[8], h[8];
    u<GVEC>(two, gamma, col, f);
    x.get(h);
#pragma unroll
    for (int i = 0; i < 8; ++i) s = fmaf(f[i], h[i], s);
    return s;
  }
  template <bool GVEC>
  __device__ __forceinline__ void store_dx(bool two, bool with_res, const float* gamma, int64_t col, float rr, float c,
                                           uint16_t* dx) const {
    float f[8], h[8];
    u<GVEC>(two, gamma, col, f);
    x.get(h);
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = rr * f[i] - h[i] * c;
    if (with_res) {
      dres.get(h);
#pragma unroll
      for (int i = 0; i < 8; ++i) f[i] += h[i];
    }
    *reinterpret_cast<uint4*>(dx) = pack8(f);
  }
};

// One CTA per row; rows of more than 8 VPL kRowThreads elements load their further vectors
// twice.
template <typename TX, bool GVEC, int VPL>
__global__ void __launch_bounds__(kRowThreads) rmsnorm_fwd_kernel(const TX* __restrict__ x,
                                                                   const uint16_t* __restrict__ res,
                                                                   const float* __restrict__ gamma, int64_t H,
                                                                   float eps, float* __restrict__ h_out,
                                                                   uint16_t* __restrict__ z, float* __restrict__ r) {
  __shared__ float red[kRowThreads / 32];
  const int64_t t = blockIdx.x, row = t * H;
  const int nvec = static_cast<int>(H / 8);
  FwdVec<TX> q[VPL];
  float ss = 0.0f;
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int v = threadIdx.x + k * kRowThreads;
    if (v < nvec) q[k].load(x, res, row + 8 * v);
  }
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int v = threadIdx.x + k * kRowThreads;
    if (v < nvec) ss = q[k].sum(res != nullptr, h_out, row + 8 * v, ss);
  }
  for (int v = threadIdx.x + VPL * kRowThreads; v < nvec; v += kRowThreads) {
    FwdVec<TX> w;
    w.load(x, res, row + 8 * v);
    ss = w.sum(res != nullptr, h_out, row + 8 * v, ss);
  }
  const float rr = rsqrtf(block_sum(ss, red) / static_cast<float>(H) + eps);
  if (threadIdx.x == 0) r[t] = rr;
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int v = threadIdx.x + k * kRowThreads;
    if (v < nvec) q[k].template store_z<GVEC>(res != nullptr, gamma, 8 * v, rr, z + row + 8 * v);
  }
  for (int v = threadIdx.x + VPL * kRowThreads; v < nvec; v += kRowThreads) {
    FwdVec<TX> w;
    w.load(x, res, row + 8 * v);
    w.template store_z<GVEC>(res != nullptr, gamma, 8 * v, rr, z + row + 8 * v);
  }
}

// dx may alias dy, dy2 or dres: a thread stores only vectors that it alone loads, after loading
// them for the last time.
template <typename TH, bool GVEC, int VPL>
__global__ void __launch_bounds__(kRowThreads) rmsnorm_bwd_kernel(const TH* __restrict__ x,
                                                                   const float* __restrict__ gamma,
                                                                   const float* __restrict__ r, const uint16_t* dy,
                                                                   const uint16_t* dy2, const uint16_t* dres,
                                                                   int64_t H, uint16_t* dx) {
  __shared__ float red[kRowThreads / 32];
  const int64_t t = blockIdx.x, row = t * H;
  const int nvec = static_cast<int>(H / 8);
  const bool two = dy2 != nullptr, with_res = dres != nullptr;
  BwdVec<TH> q[VPL];
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int v = threadIdx.x + k * kRowThreads;
    if (v < nvec) q[k].load(x, dy, dy2, dres, row + 8 * v);
  }
  const float rr = r[t];
  float sux = 0.0f;
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int v = threadIdx.x + k * kRowThreads;
    if (v < nvec) sux = q[k].template dot<GVEC>(two, gamma, 8 * v, sux);
  }
  for (int v = threadIdx.x + VPL * kRowThreads; v < nvec; v += kRowThreads) {
    BwdVec<TH> w;
    w.load(x, dy, dy2, nullptr, row + 8 * v);
    sux = w.template dot<GVEC>(two, gamma, 8 * v, sux);
  }
  const float c = block_sum(sux, red) / static_cast<float>(H) * rr * rr * rr;
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    const int v = threadIdx.x + k * kRowThreads;
    if (v < nvec) q[k].template store_dx<GVEC>(two, with_res, gamma, 8 * v, rr, c, dx + row + 8 * v);
  }
  for (int v = threadIdx.x + VPL * kRowThreads; v < nvec; v += kRowThreads) {
    BwdVec<TH> w;
    w.load(x, dy, dy2, dres, row + 8 * v);
    w.template store_dx<GVEC>(two, with_res, gamma, 8 * v, rr, c, dx + row + 8 * v);
  }
}

// Rows of at most 1024 elements: a team of `team` lanes (a power of two) per row, VPL vectors per
// lane, U rows of every team of a warp in flight at once.
constexpr int kRowWarps = kRowThreads / 32;

// Weights of less alignment pass through shared memory, loaded one by one but side by side (8 loads of a
// lane's 8 neighbours touch 32 sectors each; 8192 rows of 1024, backward in bf16: 21.7 -> 10.8 us).
template <bool GVEC, int CAP>
__device__ __forceinline__ const float* stage_gamma(const float* gamma, int H, float* shared) {
  if constexpr (GVEC) return gamma;
  for (int i = threadIdx.x; i < CAP && i < H; i += kRowThreads) shared[i] = __ldg(gamma + i);
  __syncthreads();
  return shared;
}

template <typename TX, bool GVEC, int VPL, int U>
__global__ void __launch_bounds__(kRowThreads) rmsnorm_fwd_team_kernel(const TX* __restrict__ x,
                                                                        const uint16_t* __restrict__ res,
                                                                        const float* __restrict__ gamma, int64_t T,
                                                                        int32_t H, int32_t team, float eps,
                                                                        float* __restrict__ h_out,
                                                                        uint16_t* __restrict__ z,
                                                                        float* __restrict__ r) {
  const int lane = threadIdx.x & 31, sub = lane & (team - 1), nvec = H / 8;
  const int per_warp = 32 / team;
  __shared__ __align__(16) float gs[GVEC ? 1 : 256 * VPL];
  const int64_t t0 =
      (blockIdx.x * static_cast<int64_t>(kRowWarps) + (threadIdx.x >> 5)) * per_warp * U + lane / team;
  FwdVec<TX> q[U][VPL];
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const int64_t t = t0 + k * per_warp;
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const int v = sub + u * team;
      if (t < T && v < nvec) q[k][u].load(x, res, t * H + 8 * v);
    }
  }
  const float* const g8 = stage_gamma<GVEC, 256 * VPL>(gamma, H, gs);
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const int64_t t = t0 + k * per_warp;
    float ss = 0.0f;
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const int v = sub + u * team;
      if (t < T && v < nvec) ss = q[k][u].sum(res != nullptr, h_out, t * H + 8 * v, ss);
    }
    const float rr = rsqrtf(team_sum(ss, team) / static_cast<float>(H) + eps);  // every lane of the warp
    if (t < T && sub == 0) r[t] = rr;
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const int v = sub + u * team;
      if (t < T && v < nvec) q[k][u].template store_z<true>(res != nullptr, g8, 8 * v, rr, z + t * H + 8 * v);
    }
  }
}

template <typename TH, bool GVEC, int VPL, int U>
__global__ void __launch_bounds__(kRowThreads) rmsnorm_bwd_team_kernel(const TH* __restrict__ x,
                                                                        const float* __restrict__ gamma,
                                                                        const float* __restrict__ r,
                                                                        const uint16_t* dy, const uint16_t* dy2,
                                                                        const uint16_t* dres, int64_t T, int32_t H,
                                                                        int32_t team, uint16_t* dx) {
  const int lane = threadIdx.x & 31, sub = lane & (team - 1), nvec = H / 8;
  const int per_warp = 32 / team;
  __shared__ __align__(16) float gs[GVEC ? 1 : 256 * VPL];
  const int64_t t0 =
      (blockIdx.x * static_cast<int64_t>(kRowWarps) + (threadIdx.x >> 5)) * per_warp * U + lane / team;
  const bool two = dy2 != nullptr, with_res = dres != nullptr;
  BwdVec<TH> q[U][VPL];
  float rr[U];
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const int64_t t = t0 + k * per_warp;
    rr[k] = t < T ? r[t] : 0.0f;
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const int v = sub + u * team;
      if (t < T && v < nvec) q[k][u].load(x, dy, dy2, dres, t * H + 8 * v);
    }
  }
  const float* const g8 = stage_gamma<GVEC, 256 * VPL>(gamma, H, gs);
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const int64_t t = t0 + k * per_warp;
    float sux = 0.0f;
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const int v = sub + u * team;
      if (t < T && v < nvec) sux = q[k][u].template dot<true>(two, g8, 8 * v, sux);
    }
    const float c = team_sum(sux, team) / static_cast<float>(H) * rr[k] * rr[k] * rr[k];
#pragma unroll
    for (int u = 0; u < VPL; ++u) {
      const int v = sub + u * team;
      if (t < T && v < nvec) q[k][u].template store_dx<true>(two, with_res, g8, 8 * v, rr[k], c, dx + t * H + 8 * v);
    }
  }
}

// ---------------------------------------------------------------- rotary embedding
// Element pair (i, i + d/2) of every head of token t (position s = t mod S) rotated by the
// angle s base^(-2i/d) (its negative for the inverse), in place.
__global__ void __launch_bounds__(kRowThreads) rope_kernel(uint16_t* __restrict__ x, int64_t T, int64_t S,
                                                            int32_t nheads, int32_t d, float log2_base,
                                                            int32_t inverse) {
  const int32_t half = d / 2;
  const int64_t pairs = T * nheads * half;
  for (int64_t e = blockIdx.x * (int64_t)kRowThreads + threadIdx.x; e < pairs; e += (int64_t)gridDim.x * kRowThreads) {
    const int32_t i = static_cast<int32_t>(e % half);
    const int64_t th = e / half;  // token * nheads + head
    const int64_t t = th / nheads;
    const float inv_freq = exp2f(-log2_base * (2.0f * i) / static_cast<float>(d));
    float sn, cs;
    sincosf(static_cast<float>(t % S) * inv_freq, &sn, &cs);
    if (inverse) sn = -sn;
    uint16_t* p = x + th * d;
    const float a = bf16_at(p, i), b = bf16_at(p, i + half);
    p[i] = to_bf16(a * cs - b * sn);
    p[i + half] = to_bf16(a * sn + b * cs);
  }
}

// Rows of 8 consecutive elements of d = 16 k (half = 8 k) heads: one thread per (token, 8
// consecutive i, run of `hpt` heads), its 8 angles computed once and applied to its heads with
// 16-byte loads and stores.  Bound by HBM (4 bytes an element); the head runs give the launch
// enough loads in flight (8192 tokens of 32 128-wide heads, 134 MB: 28 us with one thread per
// token and i over all heads, 23 with runs of 4).
__global__ void __launch_bounds__(kRowThreads) rope_vec_kernel(uint16_t* __restrict__ x, int64_t T, int64_t S,
                                                                int32_t nheads, int32_t d, float log2_base,
                                                                int32_t inverse, int32_t hpt) {
  const int32_t half = d / 2, groups = half / 8, runs = (nheads + hpt - 1) / hpt;
  const int64_t items = T * groups * runs;
  for (int64_t e = blockIdx.x * (int64_t)kRowThreads + threadIdx.x; e < items; e += (int64_t)gridDim.x * kRowThreads) {
    const int32_t i0 = static_cast<int32_t>(e % groups) * 8;
    const int64_t tr = e / groups;
    const int32_t h0 = static_cast<int32_t>(tr % runs) * hpt;
    const int64_t t = tr / runs;
    const int32_t h1 = min(h0 + hpt, nheads);
    // four heads' loads go out before any store, which the compiler could not move them over, and
    // the first four before the angles, which cover their latency
    constexpr int kAhead = 4;
    uint4 av[kAhead], bv[kAhead];
    auto load = [&](int32_t hb) {
#pragma unroll
      for (int u = 0; u < kAhead; ++u)
        if (hb + u < h1) {
          const uint16_t* p = x + (t * nheads + hb + u) * d + i0;
          av[u] = *reinterpret_cast<const uint4*>(p);
          bv[u] = *reinterpret_cast<const uint4*>(p + half);
        }
    };
    load(h0);
    const float pos = static_cast<float>(t % S);
    float cs[8], sn[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float inv_freq = exp2f(-log2_base * (2.0f * (i0 + j)) / static_cast<float>(d));
      sincosf(pos * inv_freq, &sn[j], &cs[j]);
      if (inverse) sn[j] = -sn[j];
    }
    for (int32_t hb = h0; hb < h1; hb += kAhead) {
      if (hb > h0) load(hb);
#pragma unroll
      for (int u = 0; u < kAhead; ++u)
        if (hb + u < h1) {
          uint16_t* p = x + (t * nheads + hb + u) * d + i0;
          float a[8], b[8], o[8], q[8];
          unpack8(av[u], a);
          unpack8(bv[u], b);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            o[j] = a[j] * cs[j] - b[j] * sn[j];
            q[j] = a[j] * sn[j] + b[j] * cs[j];
          }
          *reinterpret_cast<uint4*>(p) = pack8(o);
          *reinterpret_cast<uint4*>(p + half) = pack8(q);
        }
    }
  }
}

// ---------------------------------------------------------------- SwiGLU
// Eight elements per thread and iteration (16-byte loads and stores); block 0 takes the tail.
__device__ __forceinline__ float sigmoidf(float a) { return 1.0f / (1.0f + expf(-a)); }

__global__ void __launch_bounds__(kRowThreads) swiglu_fwd_kernel(const uint16_t* __restrict__ gt,
                                                                  const uint16_t* __restrict__ u, int64_t n,
                                                                  uint16_t* __restrict__ m) {
  const int64_t nvec = n / 8;
  for (int64_t e = blockIdx.x * (int64_t)kRowThreads + threadIdx.x; e < nvec; e += (int64_t)gridDim.x * kRowThreads) {
    float a[8], b[8], o[8];
    unpack8(reinterpret_cast<const uint4*>(gt)[e], a);
    unpack8(reinterpret_cast<const uint4*>(u)[e], b);
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] = a[i] * sigmoidf(a[i]) * b[i];
    reinterpret_cast<uint4*>(m)[e] = pack8(o);
  }
  if (blockIdx.x == 0)
    for (int64_t e = nvec * 8 + threadIdx.x; e < n; e += kRowThreads) {
      const float a = bf16_at(gt, e);
      m[e] = to_bf16(a * sigmoidf(a) * bf16_at(u, e));
    }
}

// d_gate = dm u sigma(a) (1 + a (1 - sigma(a))), d_up = dm a sigma(a).
__device__ __forceinline__ void swiglu_grad(float a, float b, float g, float& dg, float& du) {
  const float s = sigmoidf(a);
  dg = g * b * s * (1.0f + a * (1.0f - s));
  du = g * a * s;
}

__global__ void __launch_bounds__(kRowThreads) swiglu_bwd_kernel(const uint16_t* __restrict__ gt,
                                                                  const uint16_t* __restrict__ u,
                                                                  const uint16_t* __restrict__ dm, int64_t n,
                                                                  uint16_t* __restrict__ dgt,
                                                                  uint16_t* __restrict__ du) {
  const int64_t nvec = n / 8;
  for (int64_t e = blockIdx.x * (int64_t)kRowThreads + threadIdx.x; e < nvec; e += (int64_t)gridDim.x * kRowThreads) {
    float a[8], b[8], g[8], dg[8], dd[8];
    unpack8(reinterpret_cast<const uint4*>(gt)[e], a);
    unpack8(reinterpret_cast<const uint4*>(u)[e], b);
    unpack8(reinterpret_cast<const uint4*>(dm)[e], g);
#pragma unroll
    for (int i = 0; i < 8; ++i) swiglu_grad(a[i], b[i], g[i], dg[i], dd[i]);
    reinterpret_cast<uint4*>(dgt)[e] = pack8(dg);
    reinterpret_cast<uint4*>(du)[e] = pack8(dd);
  }
  if (blockIdx.x == 0)
    for (int64_t e = nvec * 8 + threadIdx.x; e < n; e += kRowThreads) {
      float dg, dd;
      swiglu_grad(bf16_at(gt, e), bf16_at(u, e), bf16_at(dm, e), dg, dd);
      dgt[e] = to_bf16(dg);
      du[e] = to_bf16(dd);
    }
}

// Block output in fp32, out = h + branch, and (with a teacher output) Eq. 7's loss: partial
// sums of (out - ref)^2 per CTA (compensated fp32, then fp64) and d_out = scale (out - ref)
// rounded once to bf16.  Eight elements per thread and iteration (count % 8 == 0).
__global__ void __launch_bounds__(kRowThreads) block_output_loss_kernel(const float* __restrict__ h,
                                                                         const uint16_t* __restrict__ branch,
                                                                         const float* __restrict__ ref, int64_t count,
                                                                         float scale, float* __restrict__ out,
                                                                         uint16_t* __restrict__ d_out,
                                                                         double* __restrict__ partials) {
  Sum2 acc{0.f, 0.f};
  const int64_t nvec = count / 8;
  for (int64_t i = blockIdx.x * (int64_t)kRowThreads + threadIdx.x; i < nvec; i += (int64_t)gridDim.x * kRowThreads) {
    const float4 h0 = reinterpret_cast<const float4*>(h)[2 * i], h1 = reinterpret_cast<const float4*>(h)[2 * i + 1];
    const uint4 bw = reinterpret_cast<const uint4*>(branch)[i];
    float o[8] = {h0.x + bf16lo_to_f32(bw.x), h0.y + bf16hi_to_f32(bw.x), h0.z + bf16lo_to_f32(bw.y),
                  h0.w + bf16hi_to_f32(bw.y), h1.x + bf16lo_to_f32(bw.z), h1.y + bf16hi_to_f32(bw.z),
                  h1.z + bf16lo_to_f32(bw.w), h1.w + bf16hi_to_f32(bw.w)};
    if (out) {
      reinterpret_cast<float4*>(out)[2 * i] = make_float4(o[0], o[1], o[2], o[3]);
      reinterpret_cast<float4*>(out)[2 * i + 1] = make_float4(o[4], o[5], o[6], o[7]);
    }
    if (ref) {
      const float4 r0 = reinterpret_cast<const float4*>(ref)[2 * i], r1 = reinterpret_cast<const float4*>(ref)[2 * i + 1];
      const float rv[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
      Sum2 local{0.f, 0.f};
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        o[q] -= rv[q];
        sum2_add(local, o[q] * o[q]);
      }
      acc = sum2_merge(acc, local);
      if (d_out) {
        uint4 w;
        w.x = pack_bf16x2(o[0] * scale, o[1] * scale);
        w.y = pack_bf16x2(o[2] * scale, o[3] * scale);
        w.z = pack_bf16x2(o[4] * scale, o[5] * scale);
        w.w = pack_bf16x2(o[6] * scale, o[7] * scale);
        reinterpret_cast<uint4*>(d_out)[i] = w;
      }
    }
  }
  if (!ref) return;
  __shared__ Sum2 red[kRowThreads / 32];
  acc = sum2_team(acc, 32);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x < 32) {
    Sum2 v = threadIdx.x < kRowThreads / 32 ? red[threadIdx.x] : Sum2{0.f, 0.f};
    v = sum2_team(v, 32);
    if (threadIdx.x == 0) partials[blockIdx.x] = sum2_value(v);
  }
}

// ---------------------------------------------------------------- attention
struct DeltaArgs {
  const uint16_t *o, *dO;
  float* delta;
  int32_t B, S, nh;
};

// delta[b, h, s] = sum over the head's columns of dO * O.  HD / 8 lanes per row, each one
// 16-byte vector of O and dO; a CTA takes as many consecutive tokens of one head as it has such
// teams (16 or 32, which divide S), so that their sums leave as whole sectors.  Bound by HBM:
// 134 MB of the 8B block's 4 x 2048 tokens in 25 us = 5.3 TB/s (a warp per row with 2-byte loads:
// 64).
template <int HD>
__global__ void __launch_bounds__(kRowThreads) attn_delta_kernel(const DeltaArgs a) {
  constexpr int kTeam = HD / 8, kTok = kRowThreads / kTeam;
  const int64_t blocks = static_cast<int64_t>(a.B) * (a.S / kTok) * a.nh;
  const int sub = threadIdx.x % kTeam, row = threadIdx.x / kTeam;
  for (int64_t w = blockIdx.x; w < blocks; w += gridDim.x) {
    const int h = static_cast<int>(w % a.nh);
    const int64_t tok = w / a.nh * kTok + row;
    const int64_t at = (tok * a.nh + h) * HD + 8 * sub;
    float o[8], d[8], s = 0.0f;
    load8(a.o + at, o);
    load8(a.dO + at, d);
#pragma unroll
    for (int i = 0; i < 8; ++i) s = fmaf(o[i], d[i], s);
    s = team_sum(s, kTeam);
    if (sub == 0) a.delta[(tok / a.S * a.nh + h) * a.S + tok % a.S] = s;
  }
}

int elem_grid(int64_t n) {
  int64_t b = (n + kRowThreads - 1) / kRowThreads;
  if (b < 1) b = 1;
  if (b > 152 * 16) b = 152 * 16;
  return static_cast<int>(b);
}

}  // namespace

namespace {

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Lanes per row of the team kernels: one vector per lane up to 256 elements (four rows of a team in
// flight, two of fp32 input; one where a launch is of no more than two CTAs an SM even so, since the
// shorter program starts sooner: 8 rows of 40, 2.9 -> 2.1 us), then 2 or 4 vectors per lane of a whole warp.
int row_team(int64_t H) {
  int team = 1;
  while (team < 32 && team * 8 < H) team *= 2;
  return team;
}

unsigned row_grid(int64_t T, int team, int in_flight) {
  const int64_t rows = static_cast<int64_t>(kRowWarps) * (32 / team) * in_flight;
  return static_cast<unsigned>((T + rows - 1) / rows);
}

template <typename TX, bool GVEC>
cudaError_t run_rmsnorm_fwd(const TX* x, const uint16_t* res, const float* gamma, int64_t T, int64_t H, float eps,
                            float* h_out, uint16_t* z, float* r, cudaStream_t st) {
  const int team = row_team(H), h32 = static_cast<int>(H);
  const unsigned rows = static_cast<unsigned>(T);
  constexpr int U = sizeof(TX) == 2 ? 4 : 2;
  if (H <= 256 && row_grid(T, team, 1) <= 2 * 152)
    rmsnorm_fwd_team_kernel<TX, GVEC, 1, 1><<<row_grid(T, team, 1), kRowThreads, 0, st>>>(x, res, gamma, T, h32, team,
                                                                                         eps, h_out, z, r);
  else if (H <= 256)
    rmsnorm_fwd_team_kernel<TX, GVEC, 1, U><<<row_grid(T, team, U), kRowThreads, 0, st>>>(x, res, gamma, T, h32, team,
                                                                                         eps, h_out, z, r);
  else if (H <= 512)
    rmsnorm_fwd_team_kernel<TX, GVEC, 2, 1><<<row_grid(T, team, 1), kRowThreads, 0, st>>>(x, res, gamma, T, h32, team,
                                                                                         eps, h_out, z, r);
  else if (H <= 1024)
    rmsnorm_fwd_team_kernel<TX, GVEC, 4, 1><<<row_grid(T, team, 1), kRowThreads, 0, st>>>(x, res, gamma, T, h32, team,
                                                                                         eps, h_out, z, r);
  else if (H <= 8 * kRowThreads)
    rmsnorm_fwd_kernel<TX, GVEC, 1><<<rows, kRowThreads, 0, st>>>(x, res, gamma, H, eps, h_out, z, r);
  else if (H <= 16 * kRowThreads)
    rmsnorm_fwd_kernel<TX, GVEC, 2><<<rows, kRowThreads, 0, st>>>(x, res, gamma, H, eps, h_out, z, r);
  else
    rmsnorm_fwd_kernel<TX, GVEC, 4><<<rows, kRowThreads, 0, st>>>(x, res, gamma, H, eps, h_out, z, r);
  return cudaGetLastError();
}

template <typename TH, bool GVEC>
cudaError_t run_rmsnorm_bwd(const TH* x, const float* gamma, const float* r, const uint16_t* dy, const uint16_t* dy2,
                            const uint16_t* dres, int64_t T, int64_t H, uint16_t* dx, cudaStream_t st) {
  const int team = row_team(H), h32 = static_cast<int>(H);
  const unsigned rows = static_cast<unsigned>(T);
  constexpr int U = sizeof(TH) == 2 ? 4 : 2;
  if (H <= 256 && row_grid(T, team, 1) <= 2 * 152)
    rmsnorm_bwd_team_kernel<TH, GVEC, 1, 1><<<row_grid(T, team, 1), kRowThreads, 0, st>>>(x, gamma, r, dy, dy2, dres, T,
                                                                                         h32, team, dx);
  else if (H <= 256)
    rmsnorm_bwd_team_kernel<TH, GVEC, 1, U><<<row_grid(T, team, U), kRowThreads, 0, st>>>(x, gamma, r, dy, dy2, dres, T,
                                                                                         h32, team, dx);
  else if (H <= 512)
    rmsnorm_bwd_team_kernel<TH, GVEC, 2, 1><<<row_grid(T, team, 1), kRowThreads, 0, st>>>(x, gamma, r, dy, dy2, dres, T,
                                                                                         h32, team, dx);
  else if (H <= 1024)
    rmsnorm_bwd_team_kernel<TH, GVEC, 4, 1><<<row_grid(T, team, 1), kRowThreads, 0, st>>>(x, gamma, r, dy, dy2, dres, T,
                                                                                         h32, team, dx);
  else if (H <= 8 * kRowThreads)
    rmsnorm_bwd_kernel<TH, GVEC, 1><<<rows, kRowThreads, 0, st>>>(x, gamma, r, dy, dy2, dres, H, dx);
  else if (H <= 16 * kRowThreads)
    rmsnorm_bwd_kernel<TH, GVEC, 2><<<rows, kRowThreads, 0, st>>>(x, gamma, r, dy, dy2, dres, H, dx);
  else
    rmsnorm_bwd_kernel<TH, GVEC, 4><<<rows, kRowThreads, 0, st>>>(x, gamma, r, dy, dy2, dres, H, dx);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_rmsnorm_fwd(const void* x, bool x_f32, const void* res, const float* gamma, int64_t T, int64_t H,
                               float eps, float* h_out, void* z, float* r, cudaStream_t st) {
  const auto* rp = static_cast<const uint16_t*>(res);
  auto* zp = static_cast<uint16_t*>(z);
  const auto* xf = static_cast<const float*>(x);
  const auto* xh = static_cast<const uint16_t*>(x);
  if (aligned16(gamma))
    return x_f32 ? run_rmsnorm_fwd<float, true>(xf, rp, gamma, T, H, eps, h_out, zp, r, st)
                 : run_rmsnorm_fwd<uint16_t, true>(xh, rp, gamma, T, H, eps, h_out, zp, r, st);
  return x_f32 ? run_rmsnorm_fwd<float, false>(xf, rp, gamma, T, H, eps, h_out, zp, r, st)
               : run_rmsnorm_fwd<uint16_t, false>(xh, rp, gamma, T, H, eps, h_out, zp, r, st);
}

cudaError_t launch_rmsnorm_bwd(const void* x, bool x_f32, const float* gamma, const float* r, const void* dy,
                               const void* dy2, const void* dres, int64_t T, int64_t H, void* dx, cudaStream_t st) {
  const auto* dyp = static_cast<const uint16_t*>(dy);
  const auto* dy2p = static_cast<const uint16_t*>(dy2);
  const auto* drp = static_cast<const uint16_t*>(dres);
  auto* dxp = static_cast<uint16_t*>(dx);
  const auto* xf = static_cast<const float*>(x);
  const auto* xh = static_cast<const uint16_t*>(x);
  if (aligned16(gamma))
    return x_f32 ? run_rmsnorm_bwd<float, true>(xf, gamma, r, dyp, dy2p, drp, T, H, dxp, st)
                 : run_rmsnorm_bwd<uint16_t, true>(xh, gamma, r, dyp, dy2p, drp, T, H, dxp, st);
  return x_f32 ? run_rmsnorm_bwd<float, false>(xf, gamma, r, dyp, dy2p, drp, T, H, dxp, st)
               : run_rmsnorm_bwd<uint16_t, false>(xh, gamma, r, dyp, dy2p, drp, T, H, dxp, st);
}

cudaError_t launch_rope(void* x, int64_t T, int64_t S, int32_t nheads, int32_t d, float base, int32_t inverse,
                        cudaStream_t st) {
  if (d % 16 == 0) {
    // heads per thread: the longest run (fewest repeated angles) that still gives every SM a full
    // set of threads
    int32_t hpt = 8;
    while (hpt > 1 && T * (d / 16) * ((nheads + hpt - 1) / hpt) < 152 * 2048) hpt /= 2;
    rope_vec_kernel<<<elem_grid(T * (d / 16) * ((nheads + hpt - 1) / hpt)), kRowThreads, 0, st>>>(
        static_cast<uint16_t*>(x), T, S, nheads, d, log2f(base), inverse, hpt);
  } else
    rope_kernel<<<elem_grid(T * nheads * (d / 2)), kRowThreads, 0, st>>>(static_cast<uint16_t*>(x), T, S, nheads, d,
                                                                          log2f(base), inverse);
  return cudaGetLastError();
}

cudaError_t launch_swiglu(const void* gt, const void* u, const void* dm, int64_t n, void* out, void* dgt, void* du,
                          cudaStream_t st) {
  if (!dm)
    swiglu_fwd_kernel<<<elem_grid((n + 7) / 8), kRowThreads, 0, st>>>(static_cast<const uint16_t*>(gt),
                                                             static_cast<const uint16_t*>(u), n,
                                                             static_cast<uint16_t*>(out));
  else
    swiglu_bwd_kernel<<<elem_grid((n + 7) / 8), kRowThreads, 0, st>>>(
        static_cast<const uint16_t*>(gt), static_cast<const uint16_t*>(u), static_cast<const uint16_t*>(dm), n,
        static_cast<uint16_t*>(dgt), static_cast<uint16_t*>(du));
  return cudaGetLastError();
}

cudaError_t launch_block_output_loss(const float* h, const void* branch, const float* ref, int64_t count,
                                     int32_t reduction, float* out, void* d_out, float* loss_out, double* partials,
                                     cudaStream_t st) {
  const int nb = ref ? recon_loss_blocks(count) : elem_grid(count / 8);
  const double inv = reduction == 0 ? 1.0 / static_cast<double>(count) : 1.0;
  block_output_loss_kernel<<<nb, kRowThreads, 0, st>>>(h, static_cast<const uint16_t*>(branch), ref, count,
                                                        static_cast<float>(2.0 * inv), out,
                                                        static_cast<uint16_t*>(d_out), partials);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !ref) return e;
  return launch_loss_final(partials, nb, inv, loss_out, st);
}

cudaError_t launch_attention(const AttnIo& io, int32_t B, int32_t S, int32_t nh, int32_t nkv, int32_t d, bool backward,
                             cudaStream_t st) {
  if (!backward) return launch_attention_fwd_tc(io.q, io.k, io.v, io.out, io.lse, B, S, nh, nkv, d, st);
  const DeltaArgs a{static_cast<const uint16_t*>(io.o), static_cast<const uint16_t*>(io.dO), io.delta, B, S, nh};
  const int64_t rows = static_cast<int64_t>(B) * S * nh;
  if (d == 128)
    attn_delta_kernel<128><<<elem_grid(rows * 16), kRowThreads, 0, st>>>(a);
  else
    attn_delta_kernel<64><<<elem_grid(rows * 8), kRowThreads, 0, st>>>(a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_attention_bwd_tc(io.q, io.k, io.v, io.dO, io.lse, io.delta, io.dq, io.dk, io.dv, B, S, nh, nkv, d, st);
}

}  // namespace catq
