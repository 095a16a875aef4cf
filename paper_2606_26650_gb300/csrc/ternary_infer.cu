// ternary_infer.cu — inference with the deployed form of a calibrated layer (App. B.2: only
// the ternary codes T and the group scale alpha are kept, W ~ alpha T, or W ~ alpha T + mu for
// the variant of the tab:mu ablation):
//   Y[b, n] = sum_k X[b, k] * (alpha[n, k / g] * T[n, k] + mu[n, k / g])
// reading T from the 2-bit codes catq_hard_ternarize_pack writes.  Decode-shaped (a few token
// rows), so the bound is HBM: every weight costs 0.25 byte of codes plus its share of a 4-byte
// group scale.
//
// Decoding 2-bit codes and multiplying them on the CUDA cores costs several instructions per
// weight, which binds long before HBM does.  Here the multiply-adds go to the tensor pipe
// (mma.sync m16n8k16, bf16 in, fp32 accumulate; a GEMV has too little work per weight for a
// tcgen05 tile to pay off), and decoding costs 10 integer instructions per 16 codes:
//
// * Code c (T = c - 1) sitting at bits 2i, 2i+1 of a 16-bit half, i < 3, is masked in place
//   and OR-ed into the bit pattern of bf16 128 (0x4300), whose mantissa unit is 1: the half
//   is the bf16 value 128 + c 4^i exactly.  One LOP3 makes two such values (the same position
//   in both halves of a 32-bit code word); positions 3..7 take the word shifted by 6 or 12.
// * The activation of that position enters the B operand pre-scaled by 4^-i (a power of two,
//   exact), so the product sums to  sum (128 4^-i + c) x  over the group's columns.
// * A second MMA per k step with constant A rows gives the same sum for c = 1 (T = 0),
//   sum (128 4^-i + 1) x, and the plain activation sum sum x; the first minus the second is
//   sum T x.  Per group: y += alpha (D - D_corr) + mu sum x.
//
// The k order inside an MMA is free as long as A and B agree: a thread's A columns
// {2q, 2q+1, 2q+8, 2q+9} are two positions of its own code word (lower and upper half), and
// its B rows are the activations of exactly those columns.
//
// A launch covers one or several layers (independent of each other).  Its work items are
// blocks of 16 R rows of a layer; a persistent CTA of 8 computing and 2 copying warps takes every
// gridDim-th item.  The copying warps stream the items' codes and group scales, in K slabs, through a
// ring of shared-memory buffers (asynchronous 16-byte copies: bulk copies of one row each are issued
// one after the other, 150 to 260 cycles a row), beside a few words on what the slab is, so that the
// computing warps touch neither the layer table nor any weight in global memory.  Those split each
// slab into contiguous K ranges, and their partial sums meet in shared memory in a fixed
// order (deterministic), summed while the next item's products run.  Token rows are taken 8 at a
// time (the MMA's N); all arithmetic after the MMAs is fp32, with one rounding of Y.
//
// A staged launch runs a chain of such layer sets in one cooperative launch (the layers of a
// decode step in dependency order: stage s + 1 may read what stage s wrote).  The work items
// of all stages form one stream; before its first item of a stage, a CTA arrives at the
// barriers of the stages it is done with and waits (bounded) until every CTA has arrived at
// the previous stage's.  The weights of the next items do not depend on earlier stages,
// so their copies are issued before the wait and the HBM stream does not drain at a stage
// boundary.
//
// What bounds it: the multiply-adds of a 128-column super-chunk (24 MMAs at 8 cycles and about 190
// other instructions for 32 rows) run at some 70 % of the MMA rate while they run; a third of
// the time goes to the ends of items, stages and launches.  Two 8B blocks (109 MB of codes, 18 us at the
// HBM rate), as eight launches in a graph / one staged call (with scales fetched where they are
// used and row-wise bulk copies, in parentheses): groups of 128, 1 token 86 us (84) / 95 (119), 8 tokens
// 92 (94) / 101 (139); groups of 64 with offsets, 1 token 97 (108) / 102 (144).  Four 1.7B blocks, 6
// tokens, groups of 64 with offsets, staged: 87 us (133).  (The figures in parentheses are of a kernel
// that copied a launch's first codes before the launch ahead of it had finished, which a pack or a
// copy just before does not allow: some 0.7 us a launch.)
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "launch.h"
#include "ptx_sm100.cuh"

namespace catq {
namespace {

constexpr int kMmaWarps = 8;                       // computing warps
constexpr int kCopyWarps = 2;                      // copying warps
constexpr int kThreads = (kMmaWarps + kCopyWarps) * 32;
constexpr int kMaxBufs = 4;                        // slab buffers
constexpr uint32_t kMagic = 0x43004300u;  // bf16 128.0 in both halves

// D += A B for one m16n8k16 tile (A row-major 16 x 16, B column-major 16 x 8, bf16).
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}

// Position p (0..7) of a code word's halves: which shifted copy of the word holds it at bits
// 2i..2i+1 (i < 3), the mask selecting it there, and its scale 4^i.
__host__ __device__ constexpr int pos_shift(int p) { return p < 3 ? 0 : (p < 6 ? 1 : 2); }
__host__ __device__ constexpr int pos_i(int p) { return p - 3 * pos_shift(p); }
__host__ __device__ constexpr uint32_t pos_mask(int p) { return 0x00030003u << (2 * pos_i(p)); }
// bf16 pairs: (128 + 4^i) for the correction row, 4^i for the activation-sum row, 4^-i for
// the activations.
__host__ __device__ constexpr uint32_t pos_corr(int p) { return kMagic | (0x00010001u << (2 * pos_i(p))); }
__host__ __device__ constexpr uint32_t pos_unit(int p) {
  return pos_i(p) == 0 ? 0x3F803F80u : (pos_i(p) == 1 ? 0x40804080u : 0x41804180u);
}
__host__ __device__ constexpr uint32_t pos_inv(int p) {
  return pos_i(p) == 0 ? 0x3F803F80u : (pos_i(p) == 1 ? 0x3E803E80u : 0x3D803D80u);
}

// The three shifted copies of a code word, and the magic constant held in a register, so
// that mask-and-insert is one three-input logic operation (a & mask | magic).
struct Shifted {
  uint32_t t[3];
  uint32_t magic;
};
__device__ __forceinline__ Shifted shifted(uint32_t w, uint32_t magic) {
  return Shifted{{w, w >> 6, w >> 12}, magic};
}

template <int P>
__device__ __forceinline__ uint32_t code_pair(const Shifted& s) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(s.t[pos_shift(P)]), "n"(pos_mask(P)), "r"(s.magic));
  return d;
}

// 16 or 4 bytes from global to shared memory, asynchronously (in this thread's open group of copies).
__device__ __forceinline__ void copy16_async(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void copy4_async(uint32_t dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
// The thread's arrival at an mbarrier, once all its copies so far have landed.
__device__ __forceinline__ void copies_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void copies_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// 32 bytes (aligned) of global memory.
__device__ __forceinline__ void ld_global_32(const void* p, uint4& lo, uint4& hi) {
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w), "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w)
               : "l"(p)
               : "memory");
}

__device__ __forceinline__ float ld_shared_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
  return v;
}

// An opaque copy of the magic constant (kept in a register instead of being folded into
// each logic operation as a second immediate).
__device__ __forceinline__ uint32_t magic_reg() {
  uint32_t m;
  asm volatile("mov.b32 %0, %1;" : "=r"(m) : "n"(kMagic));
  return m;
}

// Activation pair (x[p], x[p + 8]) of 16 consecutive bf16 (h0 = elements 0..7, h1 = 8..15),
// scaled by 4^-i of position p.
template <int P>
__device__ __forceinline__ uint32_t act_pair(const uint4& h0, const uint4& h1) {
  const uint32_t lo = (P / 2) == 0 ? h0.x : (P / 2) == 1 ? h0.y : (P / 2) == 2 ? h0.z : h0.w;
  const uint32_t hi = (P / 2) == 0 ? h1.x : (P / 2) == 1 ? h1.y : (P / 2) == 2 ? h1.z : h1.w;
  const uint32_t v = __byte_perm(lo, hi, (P & 1) ? 0x7632 : 0x5410);
  return pos_i(P) == 0 ? v : mul_bf16x2(v, pos_inv(P));
}

// VW consecutive code words of shared memory (one 4- or 8-byte load).
template <int VW>
__device__ __forceinline__ void ld_shared_words(uint32_t addr, uint32_t (&w)[VW]) {
  if constexpr (VW == 2)
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(addr));
  else
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(w[0]) : "r"(addr));
}

// MMA j of one code word of each of the thread's two rows: positions 2j and 2j + 1.
template <int J>
__device__ __forceinline__ void word_mma(float (&d)[4], const Shifted& r0, const Shifted& r1,
                                         const uint32_t (&xb)[8]) {
  mma_16816(d, code_pair<2 * J>(r0), code_pair<2 * J>(r1), code_pair<2 * J + 1>(r0), code_pair<2 * J + 1>(r1),
            xb[2 * J], xb[2 * J + 1]);
}

// One layer of a launch: its buffers, shape and code slabs (KS columns per slab, nslabs per
// token block), its group count per row, and its first work item.
struct InferLayer {
  const uint8_t* codes;
  const float* alpha;
  const float* mu;
  const uint16_t* X;
  uint16_t* Y;
  int64_t N, K, B;
  int32_t gpr;     // groups per row, K / g
  int32_t KS;      // code columns per slab (a multiple of 64 VW)
  int32_t nslabs;  // slabs per token block
  int32_t csh, ssh;  // log2 of the lanes that copy a row's codes, its scales
  int32_t wide;    // scales per copy, 4 or 1
  int32_t sld;     // row stride of a slab's scales in shared memory, words (4 times an odd number)
  int32_t item0;   // first work item of this layer
};

constexpr int kMaxInferLayers = 32;
constexpr int kMaxInferStages = 32;

struct InferArgs {
  int32_t n_layers;
  int32_t total_items;  // work items (16 R-row blocks) over all layers
  int32_t g;
  int32_t n_stages;     // staged launches: stages; 1 otherwise
  uint32_t* sync;       // staged launches: [kMaxInferStages] barrier counters, then the exit counter
  int32_t stage_end[kMaxInferStages];  // first item after each stage
  InferLayer L[kMaxInferLayers];
};

// Staged launches: arrive at stage barriers from, ..., to - 1 (one thread, after a CTA barrier that
// follows every thread's stores): one fence for all of them.
__device__ __forceinline__ void counters_arrive(uint32_t* ctr, int32_t from, int32_t to) {
  __threadfence();
  for (int32_t b = from; b < to; ++b) asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(ctr + b) : "memory");
}

__device__ __forceinline__ uint32_t counter_load(const uint32_t* ctr) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(ctr) : "memory");
  return v;
}

// Bounded wait until *ctr >= target: false on timeout (latched) or when another wait of the
// launch has given up.
__device__ __forceinline__ bool counter_wait(const uint32_t* ctr, uint32_t target, const WaitCtl& w) {
  if (counter_load(ctr) >= target) return true;
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    __nanosleep(20);
    if (counter_load(ctr) >= target) return true;
    if (aborted(w)) return false;
    if (globaltimer_ns() - t0 > w.timeout_ns) {
      signal_timeout(w);
      return false;
    }
  }
}

// A position in a CTA's stream of code slabs: work item t (a block of 16 R rows of layer l),
// token block b0 and slab.  Work items run t = blockIdx.x, blockIdx.x + gridDim.x, ...
struct Cursor {
  int32_t t, l, slab;
  int64_t b0;
};

// Move to item t, which lies in layer c.l or a later one.
__device__ __forceinline__ void cursor_at(Cursor& c, int32_t t, const InferArgs& a) {
  c.t = t;
  c.slab = 0;
  c.b0 = 0;
  if (t >= a.total_items) return;
  while (c.l + 1 < a.n_layers && t >= a.L[c.l + 1].item0) ++c.l;
}

__device__ __forceinline__ void cursor_next(Cursor& c, const InferArgs& a) {
  const InferLayer& L = a.L[c.l];
  if (++c.slab < L.nslabs) return;
  c.slab = 0;
  c.b0 += 8;
  if (c.b0 < L.B) return;
  cursor_at(c, c.t + static_cast<int32_t>(gridDim.x), a);
}

// What the computing warps need to know of a slab, written beside it by a copying warp: the layer's
// parameters and the arithmetic on them cost each computing warp some 1,000 cycles an item.
struct __align__(16) SlabInfo {
  const uint16_t* X;  // the first token's activations of the slab's first column
  uint16_t* Y;        // the first token's output of the item's first row
  int32_t ldx, ldy;   // their row strides (K, N)
  int32_t nb;         // token rows of the block, 1 .. 8
  int32_t rows;       // output rows of the item
  int32_t n_sc;       // super-chunks of the slab; 0: no slab, the stream has ended
  int32_t row_bytes;  // row stride of its codes in shared memory
  int32_t sld;        // row stride of its scales, bytes
  int32_t sc0;        // super-chunks between the start of its first group and its first column
  int32_t stage;
  int32_t place;      // 1: the token block's first slab, 2: its last
};
static_assert(sizeof(SlabInfo) == 64, "read as four 16-byte words");

// R: 16-row tiles per work item.  VW: code words per thread per super-chunk (a super-chunk is
// 64 VW columns and lies in one group).  MU: add mu times each group's activation sum.
// A persistent CTA of 8 computing and 2 copying warps walks its work items (over every layer of
// the launch) as one stream of code slabs through `nbuf` shared-memory buffers: the copying warps
// run ahead by that many slabs, whichever item, layer or stage they belong to, and the computing
// warps only wait for a slab to land and hand it back.  Each row's copy lands at a stride padded by
// 16 VW bytes, so the fragment reads (four lanes per row, eight rows per instruction) are free
// of bank conflicts; its groups' scales (and offsets) land beside it, since fetched where they are
// used each cost a trip to HBM.  One CTA barrier per work item: the partial sums' hand-over, in two
// alternating arrays.
template <int R, int VW, bool MU, bool STAGED>
__global__ void __launch_bounds__(kThreads, 2) ternary_mma_kernel(const __grid_constant__ InferArgs a,
                                                                 int32_t buf_bytes, int32_t nbuf, int32_t toks,
                                                                 const WaitCtl wc) {
  constexpr int ROWS = 16 * R;
  constexpr int NX = VW == 1 ? 4 : 2;
  constexpr int LDR = ROWS + 4;  // row stride of the partial sums: a warp's stores hit 32 banks
  extern __shared__ __align__(128) uint8_t ring[];  // nbuf slab buffers, then red[2][kMmaWarps][toks][LDR]
  __shared__ __align__(8) uint64_t bars[3 * kMaxBufs + 2];
  __shared__ SlabInfo infos[kMaxBufs];
  __shared__ SlabInfo handed[2];  // of the work items (token blocks) handed over
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t ring_base = smem_u32(ring);
  const uint32_t full = smem_u32(&bars[0]), empty = smem_u32(&bars[kMaxBufs]), info = smem_u32(&bars[2 * kMaxBufs]);
  const uint32_t summed = smem_u32(&bars[3 * kMaxBufs]);
  float* const red = reinterpret_cast<float*>(ring + nbuf * buf_bytes);
  if (threadIdx.x == 0) {
    for (int i = 0; i < nbuf; ++i) {
      mbar_init(info + 8 * i, 1);                // the slab's SlabInfo is written
      mbar_init(full + 8 * i, 32 * kCopyWarps);  // the copying warps' lanes
      mbar_init(empty + 8 * i, kMmaWarps);       // the computing warps
    }
    mbar_init(summed, kMmaWarps);
    mbar_init(summed + 8, kMmaWarps);
    fence_mbar_init_cluster();
  }
  // The next kernel of the stream may launch now (it waits for this one before it touches
  // anything this one writes).
  grid_launch_dependents();
  __syncthreads();

  if (warp >= kMmaWarps) {
    // codes of the slab at c: 16-byte pieces, 1 << csh lanes a row
    const int pw = warp - kMmaWarps;
    auto codes = [&](const Cursor& c, uint32_t base, auto hint) {
      constexpr bool kHint = decltype(hint)::value;
      const InferLayer& L = a.L[c.l];
      const int64_t n0 = static_cast<int64_t>(c.t - L.item0) * ROWS;
      const int32_t KS = L.KS, k0 = c.slab * KS, pieces = min(static_cast<int32_t>(L.K) - k0, KS) / 64;
      const int32_t nvalid = static_cast<int32_t>(min(L.N - n0, static_cast<int64_t>(ROWS)));
      const int32_t step = 1 << L.csh, rs = (kCopyWarps * 32) >> L.csh;
      const int32_t r0 = (lane >> L.csh) * kCopyWarps + pw;
      const int64_t ld = L.K / 4, row_step = rs * ld;
      const uint32_t row_bytes = static_cast<uint32_t>(KS / 4 + 16 * VW), dst_step = rs * row_bytes;
      const uint8_t* src = L.codes + (n0 + r0) * ld + k0 / 4;
      const uint32_t dst = base + r0 * row_bytes;
      for (int32_t j = lane & (step - 1); j < pieces; j += step) {
        if (kHint && (j & 1) != 0) continue;  // 32-byte sectors
        const uint8_t* p = src + 16 * j;
        uint32_t d = dst + 16 * j;
#pragma unroll 4
        for (int32_t r = r0; r < nvalid; r += rs) {
          if constexpr (kHint) prefetch_l2(p);
          else copy16_async(d, p);
          p += row_step;
          d += dst_step;
        }
      }
    };
    // the scales (and offsets) of the groups it touches, 1 << ssh lanes a row: 16-byte pieces where every
    // row's start on such a boundary, otherwise 4-byte pieces
    struct Scales {
      const float *alpha, *mu;  // of the lane's first row
      uint32_t dst;
      int32_t ng, nvalid, r0, rs, src_step, j0, j_step, wide, sld;
    };
    auto scales_of = [&](const Cursor& c, uint32_t base) {
      const InferLayer& L = a.L[c.l];
      const int64_t n0 = static_cast<int64_t>(c.t - L.item0) * ROWS;
      const int32_t KS = L.KS, k0 = c.slab * KS, cols = min(static_cast<int32_t>(L.K) - k0, KS);
      Scales f;
      const int32_t g0 = k0 / a.g;
      f.ng = (k0 + cols - 1) / a.g + 1 - g0;
      f.nvalid = static_cast<int32_t>(min(L.N - n0, static_cast<int64_t>(ROWS)));
      f.wide = L.wide;
      f.sld = L.sld;
      f.rs = (kCopyWarps * 32) >> L.ssh;
      f.r0 = (lane >> L.ssh) * kCopyWarps + pw;
      f.j0 = (lane & ((1 << L.ssh) - 1)) * f.wide;
      f.j_step = f.wide << L.ssh;
      f.src_step = f.rs * L.gpr;
      const int64_t src = (n0 + f.r0) * L.gpr + g0;
      f.alpha = L.alpha + src;
      f.mu = MU ? L.mu + src : nullptr;
      f.dst = base + ROWS * static_cast<uint32_t>(KS / 4 + 16 * VW) + f.r0 * f.sld * 4;
      return f;
    };
    auto scales = [&](const Scales& f, auto hint) {
      constexpr bool kHint = decltype(hint)::value;
      for (int32_t j = f.j0; j < f.ng; j += f.j_step) {
        if (kHint && (j & 7) != 0 && j + f.wide < f.ng) continue;  // 32-byte sectors, wherever they start
        const float* p = f.alpha + j;
        const float* m = f.mu + j;
        uint32_t d = f.dst + 4 * j;
#pragma unroll 4
        for (int32_t r = f.r0; r < f.nvalid; r += f.rs) {
          if constexpr (kHint) {
            prefetch_l2(p);
            if constexpr (MU) prefetch_l2(m);
          } else if (f.wide == 4) {
            copy16_async(d, p);
            if constexpr (MU) copy16_async(d + ROWS * f.sld * 4, m);
          } else {
            copy4_async(d, p);
            if constexpr (MU) copy4_async(d + ROWS * f.sld * 4, m);
          }
          p += f.src_step;
          m += f.src_step;
          d += f.rs * f.sld * 4;
        }
      }
    };
    int32_t stage = 0;
    auto describe = [&](const Cursor& c, int slot) {
      if (warp != kMmaWarps || lane != 0) return;
      SlabInfo f{};
      if (c.t < a.total_items) {
        const InferLayer& L = a.L[c.l];
        const int64_t n0 = static_cast<int64_t>(c.t - L.item0) * ROWS;
        const int32_t k0 = c.slab * L.KS;
        if constexpr (STAGED)
          while (c.t >= a.stage_end[stage]) ++stage;
        f.X = L.X + c.b0 * L.K + k0;
        f.Y = L.Y + c.b0 * L.N + n0;
        f.ldx = static_cast<int32_t>(L.K);
        f.ldy = static_cast<int32_t>(L.N);
        f.nb = static_cast<int32_t>(min(L.B - c.b0, static_cast<int64_t>(8)));
        f.rows = static_cast<int32_t>(min(L.N - n0, static_cast<int64_t>(ROWS)));
        f.n_sc = min(f.ldx - k0, L.KS) / (64 * VW);
        f.row_bytes = L.KS / 4 + 16 * VW;
        f.sld = L.sld * 4;
        f.sc0 = a.g == 64 * VW ? 0 : k0 % a.g / (64 * VW);
        f.stage = stage;
        f.place = (c.slab == 0 ? 1 : 0) | (c.slab + 1 == L.nslabs ? 2 : 0);
      }
      infos[slot] = f;
      mbar_arrive_local(info + 8 * slot);
    };
    constexpr std::false_type kCopy{};
    constexpr std::true_type kAsk{};
    // The kernel before may be the one that wrote the codes and scales (a pack, a copy), and its writes
    // are only sure to be seen past the wait: until then the first slabs are merely asked for in L2.
    Cursor c{};
    cursor_at(c, blockIdx.x, a);
    Cursor n = c;
    for (int i = 0; i < nbuf && n.t < a.total_items; ++i, cursor_next(n, a)) {
      if (STAGED && i == 0) continue;  // (no launch to wait for: copied right away)
      codes(n, 0, kAsk);
      scales(scales_of(n, 0), kAsk);
    }
    grid_dependency_wait();
    int slot = 0;
    uint32_t phase = 0;
    for (;;) {
      // a buffer's first use needs no wait: the phase before a barrier's first counts as passed
      if (!mbar_wait_warp(empty + 8 * slot, phase ^ 1u, wc)) break;
      if (c.t >= a.total_items) {
        describe(c, slot);
        break;
      }
      const uint32_t base = ring_base + slot * buf_bytes;
      codes(c, base, kCopy);
      describe(c, slot);
      scales(scales_of(c, base), kCopy);
      copies_arrive(full + 8 * slot);
      if (++slot == nbuf) {
        slot = 0;
        phase ^= 1u;
      }
      cursor_next(c, a);
    }
    copies_wait_all();
    return;
  }

  grid_dependency_wait();
  const int gid = lane >> 2, q = lane & 3;
  const uint32_t magic = magic_reg();
  const int32_t sc_per_group = a.g / (64 * VW);
  int slot = 0;
  uint32_t phase = 0;
  float acc[R][4];
  int32_t stage = 0, arrived = 0;  // staged: stage of the current item, barriers arrived at

  // Hand-overs: the warps' partial sums of a token block meet in shared memory, in a fixed order, and
  // are summed and stored only when the next block's products are done (or the stream or the
  // stage ends), so that no warp waits for the slowest one of the same block.  Two arrays suffice: a
  // warp writes the one of two blocks before once it has seen every warp hand over the block before,
  // which each did after its share of that sum.
  uint32_t given = 0, taken = 0;  // token blocks handed over, summed
  auto take = [&]() -> bool {
    if (taken == given) return true;
    const uint32_t p = taken & 1u;
    if (!mbar_wait_warp(summed + 8 * p, (taken >> 1) & 1u, wc)) return false;
    ++taken;
    const SlabInfo& h = handed[p];
    const float* const part = red + static_cast<int>(p) * kMmaWarps * toks * LDR;
    const int row = threadIdx.x % ROWS;
    for (int tok = threadIdx.x / ROWS; tok < h.nb; tok += kMmaWarps * 32 / ROWS) {
      float s = 0.0f;
#pragma unroll
      for (int w = 0; w < kMmaWarps; ++w) s += part[(w * toks + tok) * LDR + row];
      if (row < h.rows)
        h.Y[static_cast<int64_t>(tok) * h.ldy + row] = static_cast<uint16_t>(pack_bf16x2(s, 0.0f) & 0xFFFFu);
    }
    return true;
  };

  // Waits are bounded: a warp whose wait gives up tells the others at the CTA barrier that they reach
  // next, whichever it is, and all leave (a warp waiting for its hand-over gives up too).
  for (;;) {
    if (!mbar_wait_warp(info + 8 * slot, phase, wc)) {
      bar_all(1, kMmaWarps * 32, false);
      break;
    }
    const SlabInfo& f = infos[slot];
    const int32_t n_sc = f.n_sc;
    if (n_sc == 0) {
      bar_all(1, kMmaWarps * 32, take());
      break;
    }
    if constexpr (STAGED) {
      const int32_t st = f.stage;
      if (st > stage) {
        // This CTA has no items left in stages before st (items run in order).  Store its last
        // outputs there, arrive at those stages' barriers, then wait until every CTA has
        // arrived at stage st - 1's.
        if (!bar_all(1, kMmaWarps * 32, take())) break;
        bool good = true;
        if (threadIdx.x == 0) {
          counters_arrive(a.sync, arrived, st);
          good = counter_wait(a.sync + (st - 1), gridDim.x, wc);
        }
        arrived = st;
        stage = st;
        if (!bar_all(1, kMmaWarps * 32, good)) break;
      }
    }
    // this warp's contiguous range of the slab's super-chunks, and its first activations (token columns
    // past the block's rows read the first row's: their sums are computed and never stored, as are
    // those of rows past the layer's last, whose codes and scales are whatever lay there)
    const int32_t lo = n_sc * warp / kMmaWarps, hi = n_sc * (warp + 1) / kMmaWarps;
    const int32_t nb = f.nb, place = f.place;
    const uint4* const xbase =
        reinterpret_cast<const uint4*>(f.X + static_cast<int64_t>(gid < nb ? gid : 0) * f.ldx + 16 * VW * q);
    // (32 bytes at a time where X allows: half the passes through L1, which a load of eight token rows
    // at 16 bytes a lane keeps busy; two 8B blocks, 8 tokens: 10 us less, staged 129 -> 101.  A staged
    // launch's X may be an earlier stage's Y: plain loads, after the stage's acquire, or through L2 for
    // a single token, whose row is not read twice: 96 -> 92.)
    const bool x32 = (reinterpret_cast<uintptr_t>(xbase) & 31u) == 0 && (!STAGED || nb > 1);
    auto load_x = [&](int32_t sc, uint4 (&xv)[2 * VW]) {
      const uint4* xp = xbase + sc * (8 * VW);
      if (x32) {
#pragma unroll
        for (int i = 0; i < VW; ++i) ld_global_32(xp + 2 * i, xv[2 * i], xv[2 * i + 1]);
        return;
      }
#pragma unroll
      for (int i = 0; i < 2 * VW; ++i) xv[i] = STAGED ? __ldcg(xp + i) : __ldg(xp + i);
    };
    uint4 xs[NX][2 * VW];  // activations, up to NX super-chunks ahead
#pragma unroll
    for (int j = 0; j < NX; ++j)
      if (lo + j < hi) load_x(lo + j, xs[j]);
    if (place & 1) {
#pragma unroll
      for (int r = 0; r < R; ++r)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[r][e] = 0.0f;
    }
    const uint32_t row_bytes = static_cast<uint32_t>(f.row_bytes), sld = static_cast<uint32_t>(f.sld);
    const uint32_t tile = ring_base + slot * buf_bytes;
    // shared-memory address of the thread's words in row gid, and of that row's scale in the group
    // that the warp's range starts in; the super-chunks to the group's end
    const uint32_t rowa = tile + gid * row_bytes + VW * q * 4;
    uint32_t scale = tile + ROWS * row_bytes + gid * sld;
    int32_t left = 1;
    if (sc_per_group == 1) {
      scale += lo * 4;
    } else {
      const int32_t at = f.sc0 + lo, grp = at / sc_per_group;
      left = (grp + 1) * sc_per_group - at;
      scale += grp * 4;
    }
    if (!mbar_wait_warp(full + 8 * slot, phase, wc)) {
      bar_all(1, kMmaWarps * 32, false);
      break;
    }
    // one super-chunk: this thread's code words from shared memory, its activations xv
    auto step = [&](int32_t sc, const uint4 (&xv)[2 * VW]) {
      const uint32_t woff = static_cast<uint32_t>(sc * 16 * VW);
      float d[R][4], da[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        da[e] = 0.0f;
#pragma unroll
        for (int r = 0; r < R; ++r) d[r][e] = 0.0f;
      }
      uint32_t cw[R][2][VW];  // the thread's code words of rows gid and gid + 8 of each tile
#pragma unroll
      for (int r = 0; r < R; ++r) {
        ld_shared_words<VW>(rowa + (16 * r) * row_bytes + woff, cw[r][0]);
        ld_shared_words<VW>(rowa + (16 * r + 8) * row_bytes + woff, cw[r][1]);
      }
#pragma unroll
      for (int v = 0; v < VW; ++v) {
        uint32_t xb[8];
        const uint4 h0 = xv[2 * v], h1 = xv[2 * v + 1];
        xb[0] = act_pair<0>(h0, h1);
        xb[1] = act_pair<1>(h0, h1);
        xb[2] = act_pair<2>(h0, h1);
        xb[3] = act_pair<3>(h0, h1);
        xb[4] = act_pair<4>(h0, h1);
        xb[5] = act_pair<5>(h0, h1);
        xb[6] = act_pair<6>(h0, h1);
        xb[7] = act_pair<7>(h0, h1);
        // rows 0..7 of the constant tile: the correction sums; rows 8..15: activation sums
        mma_16816(da, pos_corr(0), pos_unit(0), pos_corr(1), pos_unit(1), xb[0], xb[1]);
        mma_16816(da, pos_corr(2), pos_unit(2), pos_corr(3), pos_unit(3), xb[2], xb[3]);
        mma_16816(da, pos_corr(4), pos_unit(4), pos_corr(5), pos_unit(5), xb[4], xb[5]);
        mma_16816(da, pos_corr(6), pos_unit(6), pos_corr(7), pos_unit(7), xb[6], xb[7]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const Shifted s0 = shifted(cw[r][0][v], magic), s1 = shifted(cw[r][1][v], magic);
          word_mma<0>(d[r], s0, s1, xb);
          word_mma<1>(d[r], s0, s1, xb);
          word_mma<2>(d[r], s0, s1, xb);
          word_mma<3>(d[r], s0, s1, xb);
        }
      }
      // a super-chunk lies in one group: scale (and offset) its sums
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float a0 = ld_shared_f32(scale + (16 * r) * sld);
        const float a1 = ld_shared_f32(scale + (16 * r + 8) * sld);
        acc[r][0] = fmaf(a0, d[r][0] - da[0], acc[r][0]);
        acc[r][1] = fmaf(a0, d[r][1] - da[1], acc[r][1]);
        acc[r][2] = fmaf(a1, d[r][2] - da[0], acc[r][2]);
        acc[r][3] = fmaf(a1, d[r][3] - da[1], acc[r][3]);
        if constexpr (MU) {
          const float m0 = ld_shared_f32(scale + (ROWS + 16 * r) * sld);
          const float m1 = ld_shared_f32(scale + (ROWS + 16 * r + 8) * sld);
          acc[r][0] = fmaf(m0, da[2], acc[r][0]);
          acc[r][1] = fmaf(m0, da[3], acc[r][1]);
          acc[r][2] = fmaf(m1, da[2], acc[r][2]);
          acc[r][3] = fmaf(m1, da[3], acc[r][3]);
        }
      }
      if (--left == 0) {
        scale += 4;
        left = sc_per_group;
      }
    };
    for (int32_t sc = lo; sc < hi; sc += NX) {
#pragma unroll
      for (int j = 0; j < NX; ++j) {
        if (sc + j >= hi) break;
        step(sc + j, xs[j]);
        if (sc + j + NX < hi) load_x(sc + j + NX, xs[j]);
      }
    }
    if (place & 2) {
      // the token block's last slab: sum the block before, hand this one over
      // D fragment: (row gid, tokens 2q, 2q + 1) and (row gid + 8, the same tokens)
      if (!take()) {
        bar_all(1, kMmaWarps * 32, false);
        break;
      }
      const uint32_t p = given & 1u;
      float* const part = red + (static_cast<int>(p) * kMmaWarps + warp) * toks * LDR;
#pragma unroll
      for (int e = 0; e < 2; ++e)
        if (2 * q + e < nb) {
          float* const to = part + (2 * q + e) * LDR + gid;
#pragma unroll
          for (int r = 0; r < R; ++r) {
            to[16 * r] = acc[r][e];
            to[16 * r + 8] = acc[r][2 + e];
          }
        }
      if (threadIdx.x == 0) handed[p] = f;
      __syncwarp();
      if (lane == 0) mbar_arrive_local(summed + 8 * p);
      ++given;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive_local(empty + 8 * slot);
    if (++slot == nbuf) {
      slot = 0;
      phase ^= 1u;
    }
  }
  if constexpr (STAGED) {
    // Arrive at the barriers still owed (every thread's stores came before the last CTA barrier), then
    // leave; the last CTA to leave (every other one has passed all its waits by then) zeroes the
    // counters for the next launch.
    if (threadIdx.x == 0) {
      counters_arrive(a.sync, arrived, a.n_stages - 1);
      const uint32_t prev = atomicAdd(a.sync + kMaxInferStages, 1u);
      if (prev == gridDim.x - 1) {
        for (int32_t b = 0; b < a.n_stages - 1; ++b) a.sync[b] = 0u;
        a.sync[kMaxInferStages] = 0u;
        __threadfence();
      }
    }
  }
}

// Dynamic shared memory of a CTA: half of an SM's, less its reserve and the static arrays.
constexpr int64_t kDynBytes = 112 * 1024;
// More than two slab buffers only up to this much of it: the rest caches activations (two 8B blocks, groups
// of 128, 8 tokens: 101 us staged and 92 in single launches so, 114 and 94 with a third buffer instead).
constexpr int64_t kRingBytes = 80 * 1024;

// log2 of the lanes that share n pieces of a row: the power of two up to a warp that covers them.
int32_t lanes_log2(int64_t n) {
  int32_t s = 0;
  while (s < 5 && (int64_t(1) << s) < n) ++s;
  return s;
}

// Row stride of a slab's scales, words: the groups that KS columns can touch, up to 4 times an odd
// number, so that 16-byte copies fit and the eight rows that a warp reads lie in different banks.
int64_t scale_stride(int64_t KS, int64_t g) { return (((KS % g == 0 ? KS / g : KS / g + 2) + 3) / 4 | 1) * 4; }

// Bytes of one slab buffer for KS columns: 16 R rows of codes, each padded by 16 VW bytes, and their
// groups' scales (and offsets).
int64_t slab_bytes(int64_t KS, int R, int VW, int64_t g, bool mu) {
  return 16 * R * (KS / 4 + 16 * VW + scale_stride(KS, g) * 4 * (mu ? 2 : 1));
}

// Code columns per slab for K: all of K when it fits one buffer, else the fewest equal slabs
// (multiples of 64 VW columns) that do.
int64_t slab_cols(int64_t K, int R, int VW, int64_t g, bool mu, int64_t cap) {
  const int64_t unit = 64 * VW;
  for (int64_t nslabs = 1;; ++nslabs) {
    const int64_t KS = ((K + nslabs - 1) / nslabs + unit - 1) / unit * unit;
    if (KS == unit || slab_bytes(KS, R, VW, g, mu) <= cap) return KS;
  }
}

// stage_of (nullable): the stage of each layer (non-decreasing from 0 in steps of 1); sync: the
// staged launch's counters (zero on entry and on exit).
template <int R, int VW>
cudaError_t launch_mma(const InferDesc* ls, int n, int32_t g, bool with_mu, const int32_t* stage_of, uint32_t* sync,
                       cudaStream_t st) {
  WaitCtl wc;
  if (!launch_wait_ctl(&wc)) return cudaErrorInvalidDevice;
  InferArgs a{};
  a.n_layers = n;
  a.g = g;
  a.n_stages = stage_of ? stage_of[n - 1] + 1 : 1;
  a.sync = sync;
  const int64_t toks = std::min<int64_t>(ls[0].B, 8);  // (the layers of a launch share B)
  const int64_t red_bytes = 2 * kMmaWarps * toks * (16 * R + 4) * 4;
  const int64_t cap = (kDynBytes - red_bytes) / 2 / 128 * 128;  // of a slab buffer
  int64_t items = 0, max_buf = 0;
  for (int i = 0; i < n; ++i) {
    InferLayer& L = a.L[i];
    L.codes = ls[i].codes;
    L.alpha = ls[i].alpha;
    L.mu = ls[i].mu;
    L.X = static_cast<const uint16_t*>(ls[i].X);
    L.Y = static_cast<uint16_t*>(ls[i].Y);
    L.N = ls[i].N;
    L.K = ls[i].K;
    L.B = ls[i].B;
    L.gpr = static_cast<int32_t>(ls[i].K / g);
    const int64_t KS = slab_cols(L.K, R, VW, g, with_mu, cap);
    L.KS = static_cast<int32_t>(KS);
    L.csh = lanes_log2(KS / 64);
    const bool al16 = (reinterpret_cast<uintptr_t>(L.alpha) & 15u) == 0 && (reinterpret_cast<uintptr_t>(L.mu) & 15u) == 0;
    L.wide = al16 && L.gpr % 4 == 0 && (KS >= L.K || KS % (4 * g) == 0) ? 4 : 1;
    L.ssh = lanes_log2(((KS % g == 0 ? KS / g : KS / g + 2) + L.wide - 1) / L.wide);
    L.sld = static_cast<int32_t>(scale_stride(KS, g));
    L.nslabs = static_cast<int32_t>((L.K + KS - 1) / KS);
    L.item0 = static_cast<int32_t>(items);
    items += (L.N + 16 * R - 1) / (16 * R);
    max_buf = std::max<int64_t>(max_buf, slab_bytes(KS, R, VW, g, with_mu));
    if (stage_of) a.stage_end[stage_of[i]] = static_cast<int32_t>(std::min<int64_t>(items, INT32_MAX));
  }
  if (items >= (int64_t(1) << 31)) return cudaErrorInvalidValue;
  if (items == 0) return cudaSuccess;
  a.total_items = static_cast<int32_t>(items);
  if (!stage_of) a.stage_end[0] = a.total_items;
  int64_t widest = 0;  // most items of one stage
  for (int32_t s = 0, prev = 0; s < a.n_stages; prev = a.stage_end[s], ++s)
    widest = std::max<int64_t>(widest, a.stage_end[s] - prev);
  const int buf_bytes = static_cast<int>((max_buf + 127) / 128 * 128);
  const int nbuf = static_cast<int>(
      std::max<int64_t>(2, std::min<int64_t>(kMaxBufs, (kRingBytes - red_bytes) / buf_bytes)));
  const int smem = nbuf * buf_bytes + static_cast<int>(red_bytes);
  int sm = 152;
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev);
  const bool staged = a.n_stages > 1;
  auto kern = staged ? (with_mu ? ternary_mma_kernel<R, VW, true, true> : ternary_mma_kernel<R, VW, false, true>)
                     : (with_mu ? ternary_mma_kernel<R, VW, true, false> : ternary_mma_kernel<R, VW, false, false>);
  // (the kernel's own state, which launches from other threads share: the most that any asks for)
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kDynBytes));
  if (e != cudaSuccess) return e;
  int64_t blocks = std::min<int64_t>(items, 2 * static_cast<int64_t>(sm));
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute attr[1];
  if (staged) {
    // every CTA must be resident at once (they wait on each other): a cooperative launch of
    // at most the co-resident CTAs, and no more than the widest stage has items
    int per_sm = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, static_cast<size_t>(smem));
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    blocks = std::min<int64_t>(widest, static_cast<int64_t>(per_sm) * sm);
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  } else {
    // programmatic dependent launch: this kernel may start while the previous one in the
    // stream finishes (see grid_dependency_wait in the kernel)
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
  }
  cfg.gridDim = dim3(static_cast<unsigned>(blocks));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = static_cast<size_t>(smem);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, a, buf_bytes, nbuf, static_cast<int32_t>(toks), wc);
}

template <int R>
cudaError_t launch_rows(const InferDesc* ls, int n, int32_t g, bool with_mu, const int32_t* stage_of, uint32_t* sync,
                        cudaStream_t st) {
  if (g % 128 == 0) return launch_mma<R, 2>(ls, n, g, with_mu, stage_of, sync, st);
  return launch_mma<R, 1>(ls, n, g, with_mu, stage_of, sync, st);
}

// 16-row tiles per work item (1 or 2: more hold more registers than two CTAs per SM allow
// without spills): the fewest rows on the busiest SM summed over the stages (two persistent
// CTAs per SM), then the most tiles per item (the correction MMAs and the activation
// preparation serve more rows).
int pick_rows(const InferDesc* ls, int n, const int32_t* stage_of) {
  int sm = 152;
  {
    int dev = 0;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sm, cudaDevAttrMultiProcessorCount, dev);
  }
  int best = 1;
  int64_t best_rows = -1;
  for (int r = 1; r <= 2; ++r) {
    int64_t busiest = 0, items = 0;
    for (int i = 0; i < n; ++i) {
      items += (ls[i].N + 16 * r - 1) / (16 * r);
      if (i + 1 == n || (stage_of && stage_of[i + 1] != stage_of[i])) {
        busiest += (items + 2 * sm - 1) / (2 * sm) * 16 * r;
        items = 0;
      }
    }
    if (best_rows < 0 || busiest <= best_rows) {
      best = r;
      best_rows = busiest;
    }
  }
  return best;
}

cudaError_t launch_infer(const InferDesc* ls, int n, int32_t g, const int32_t* stage_of, uint32_t* sync,
                         cudaStream_t st) {
  if (n < 1 || n > kMaxInferLayers) return cudaErrorInvalidValue;
  const bool with_mu = ls[0].mu != nullptr;
  for (int i = 1; i < n; ++i)
    if ((ls[i].mu != nullptr) != with_mu) return cudaErrorInvalidValue;
  if (stage_of) {
    if (stage_of[0] != 0 || !sync) return cudaErrorInvalidValue;
    for (int i = 1; i < n; ++i)
      if (stage_of[i] != stage_of[i - 1] && stage_of[i] != stage_of[i - 1] + 1) return cudaErrorInvalidValue;
    if (stage_of[n - 1] + 1 > kMaxInferStages) return cudaErrorInvalidValue;
  }
  if (pick_rows(ls, n, stage_of) == 2) return launch_rows<2>(ls, n, g, with_mu, stage_of, sync, st);
  return launch_rows<1>(ls, n, g, with_mu, stage_of, sync, st);
}

}  // namespace

int ternary_infer_max_layers() { return kMaxInferLayers; }

cudaError_t launch_ternary_infer_batched(const InferDesc* ls, int n, int32_t g, cudaStream_t st) {
  return launch_infer(ls, n, g, nullptr, nullptr, st);
}

int ternary_infer_max_stages() { return kMaxInferStages; }
size_t ternary_infer_sync_bytes() { return (kMaxInferStages + 1) * sizeof(uint32_t); }

cudaError_t launch_ternary_infer_staged(const InferDesc* ls, int n, const int32_t* stage_of, int32_t g, uint32_t* sync,
                                        cudaStream_t st) {
  if (!stage_of) return cudaErrorInvalidValue;
  return launch_infer(ls, n, g, stage_of, sync, st);
}

cudaError_t launch_ternary_infer(const uint8_t* codes, const float* alpha, const float* mu, int64_t N, int64_t K,
                                 int32_t g, const void* X, int64_t B, void* Y, cudaStream_t st) {
  const InferDesc d{codes, alpha, mu, N, K, X, B, Y};
  return launch_ternary_infer_batched(&d, 1, g, st);
}

}  // namespace catq
