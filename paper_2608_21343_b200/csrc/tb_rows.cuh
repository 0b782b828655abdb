// Device code of the two-step greedy decode (tb_rows.cu): rows of any vocabulary, fp32 or bf16, any strides with
// contiguous tokens, reduced to 32-byte summaries, and the decider that walks a stretch of one stream from summaries.
//
// Step 1 (frames_summary, one warp per row, independent of the graph state): the row's best root-boosted token, a bound on
// all others, its blank logit, and -- where asked for -- its log-softmax normaliser or its best duration.
// Step 2 (decide, one warp per stretch): the sequential part.  What bounds it is the chain state -> list -> logits ->
// token -> state: a trip to shared memory or L2 for each arrow and some 500 instructions, which a warp that is alone on
// its scheduler issues one every five to seven cycles; 3300 cycles in all, whatever number of rows are looked at.  So a
// round takes as many rows as can be foreseen: the summaries alone say which way most rows go, and the rows on that way
// (up to eight, of several frames) are decided at once, each under the state foreseen for it; three to four hold on
// average.  Rounds of the rows (t, k), (t+1, 0), .. under the current state only, which end with the first token, took
// twice as many.  A row the summaries cannot decide is read in full, but only for the tokens past a threshold (V = 8192:
// 190 000 cycles a row when every token was looked up, 20 000 so).  Nothing is asked into L2 ahead: a stretch's rows
// amount to more requests than its SM issues in the time (V = 8192: 203 us with it, 143 without).
// 32 fp32 streams of 500 frames, V = 1024: 197 us before these, 118 after.
//
// The code is kept small on purpose (no register-resident lists, loops not unrolled beyond what keeps loads in flight,
// options as uniform branches instead of instantiations): a chunk or a short utterance runs through it a few dozen times
// only, and a first version of 130-250 KB spent most of its time fetching instructions (a 100-frame utterance: 83 us,
// the same at 2 and at 16 stretches).
//
// Exactness: as in tb_greedy_fast.cu.  A summary's winner is accepted only when it clears every other token by a margin
// that dominates all roundings, or when no token that is not listed can reach the best of {blank, listed tokens}; else
// the row is evaluated exactly (exact_row).
#ifndef TB_ROWS_CUH_
#define TB_ROWS_CUH_

#include <cuda_bf16.h>

#include "tb_device.cuh"
#include "tb_launch.h"

namespace {

constexpr int kRowsPerFrame = 4;      // rows per frame (S) the summaries are laid out for
constexpr int kWalkBuf = 256;         // entries of a list put together by walking that are kept in shared memory

struct RowSum {      // 32 bytes, read as two 16-byte halves
  float y1;          // best root-boosted token value of the row (ties: lowest id)
  float y2b;         // upper bound on the root-boosted value of every other token
  float xb;          // blank logit
  float x1;          // raw logit of the best token
  float rootcw1;     // root arc weight of the best token's class (0 if none)
  int32_t rootdst1;  // root arc target of the best token's class (0 if none)
  uint32_t packed;   // id1 | kRsOvf | kRsGap | duration << 24
  float extra;       // the row's normaliser (log-softmax), or the logit of its best duration (TDT)
};
static_assert(sizeof(RowSum) == 32, "two 16-byte halves");
constexpr uint32_t kRsIdMask = 0x3FFFu, kRsOvf = 1u << 16, kRsGap = 1u << 17, kRsAbsent = 1u << 18;

__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t shared_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// ---- the graph's root in shared memory: weight and arc per class -------------------------------------------------
struct RootTab {
  float* w;          // [C] root arc weight (0 if none)
  uint16_t* arc;     // [C] root arc + 1 (0 if none)
  float* stats;      // beta_min, beta_max, largest |w|, number of root arcs
};
__host__ __device__ inline size_t root_tab_bytes(int C) {
  return ((static_cast<size_t>(C) * 4 + 15) & ~size_t(15)) + ((static_cast<size_t>(C) * 2 + 15) & ~size_t(15)) + 16;
}
__device__ __forceinline__ RootTab root_tab_at(unsigned char* mem, int C) {
  RootTab r;
  r.w = reinterpret_cast<float*>(mem);
  mem += (static_cast<size_t>(C) * 4 + 15) & ~size_t(15);
  r.arc = reinterpret_cast<uint16_t*>(mem);
  mem += (static_cast<size_t>(C) * 2 + 15) & ~size_t(15);
  r.stats = reinterpret_cast<float*>(mem);
  return r;
}
// Block-wide (three barriers); part: 3 floats per warp of scratch shared memory.
__device__ inline void root_tab_fill(const RootTab& r, const GraphPtrs& g, bool bound, float lam, int C, float* part) {
  const int tid = threadIdx.x, n = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = (n + 31) >> 5;
#pragma unroll 1
  for (int c = tid; c < C; c += n) { r.w[c] = 0.0f; r.arc[c] = 0; }
  __syncthreads();
  float bmin = 0.0f, bmax = 0.0f, R = 0.0f;
  if (bound) {
    const int a0 = g.arc_begin[0], e = g.arc_begin[1];
#pragma unroll 1
    for (int a = a0 + tid; a < e; a += n) {
      const int c = g.arc_cls[a];
      const float wv = __fadd_rn(0.0f, g.arc_w[a]);          // the walk's fl(acc + w) with acc = 0
      const float cb = __fmul_rn(lam, wv);
      if (c >= 0 && c < C) { r.w[c] = wv; r.arc[c] = static_cast<uint16_t>(a - a0 + 1); }
      bmin = fminf(bmin, cb); bmax = fmaxf(bmax, cb); R = fmaxf(R, fabsf(wv));
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    bmin = fminf(bmin, __shfl_xor_sync(0xffffffffu, bmin, off));
    bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, off));
    R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, off));
  }
  if (lane == 0) { part[3 * warp] = bmin; part[3 * warp + 1] = bmax; part[3 * warp + 2] = R; }
  __syncthreads();
  if (tid == 0) {
#pragma unroll 1
    for (int w2 = 1; w2 < nwarps; ++w2) {
      bmin = fminf(bmin, part[3 * w2]); bmax = fmaxf(bmax, part[3 * w2 + 1]); R = fmaxf(R, part[3 * w2 + 2]);
    }
    r.stats[0] = bmin; r.stats[1] = bmax; r.stats[2] = R;
    r.stats[3] = bound ? static_cast<float>(g.arc_begin[1] - g.arc_begin[0]) : 0.0f;
  }
  __syncthreads();
}

// ---- step 1: one row -> summary -----------------------------------------------------------------------------------
struct RowCtx {
  const float* rootw; const uint16_t* rootarc;   // RootTab
  const int32_t* cls;                            // device [V] token -> class
  const float* arc_w; const int32_t* arc_dst;    // the root's arcs
  float lam, beta_min, beta_max, bmag_max;       // bmag_max: bound on |lambda| * (|D(s)| + largest root weight) over all states s
  bool boosts, norm;                             // the root has arcs (which may weigh nothing); the row's normaliser is wanted
  uint32_t boost_a;                              // shared address of the table of root boosts per token (BoostTab; TAB only)
  int V, n_dur;
};

// G 16-byte blocks per lane: one group of a row is 32 * G blocks.
template <typename LT> struct RowBlock;
template <> struct RowBlock<uint16_t> {          // eight bf16 each
  static constexpr int E = 8;
  static constexpr uint32_t kNone = 0xFF80FF80u;   // -inf
  static __device__ __forceinline__ __nv_bfloat162 h2(uint32_t w) { __nv_bfloat162 r; *reinterpret_cast<uint32_t*>(&r) = w; return r; }
  template <int G> static __device__ __forceinline__ float max(const uint4 (&q)[G]) {
    __nv_bfloat162 m = h2(kNone);
#pragma unroll
    for (int u = 0; u < G; ++u) m = __hmax2(m, __hmax2(__hmax2(h2(q[u].x), h2(q[u].y)), __hmax2(h2(q[u].z), h2(q[u].w))));
    const uint32_t w = *reinterpret_cast<const uint32_t*>(&m);
    return fmaxf(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
  }
  static __device__ __forceinline__ float threshold(float t) { return __bfloat162float(__float2bfloat16_rd(t)); }
  // one bit per element of blocks u0 .. u0 + 3 at or above t (a value of `threshold`): bit 4 u + i + 16 h is half h of word i
  static constexpr int kUnits = 4;
  template <int G> static __device__ __forceinline__ uint32_t hits(const uint4 (&q)[G], int u0, float t) {
    const __nv_bfloat162 t2 = __float2bfloat162_rn(t);
    uint32_t r = 0;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      r |= __hge2_mask(h2(q[u0 + u].x), t2) & (0x00010001u << (4 * u));
      r |= __hge2_mask(h2(q[u0 + u].y), t2) & (0x00010001u << (4 * u + 1));
      r |= __hge2_mask(h2(q[u0 + u].z), t2) & (0x00010001u << (4 * u + 2));
      r |= __hge2_mask(h2(q[u0 + u].w), t2) & (0x00010001u << (4 * u + 3));
    }
    return r;
  }
  // the same for root-boosted values: cb holds a block's boosts, rounded up
  static __device__ __forceinline__ uint32_t boost(float cb) { return __bfloat16_as_ushort(__float2bfloat16_ru(cb)); }
  static constexpr float kBoostSlack = 0.0078125f;   // of |value| + largest boost: the roundings of the boost and of the sum
  static __device__ __forceinline__ uint32_t hits_boosted(const uint4& q, const uint4& cb, int u, float t) {
    const __nv_bfloat162 t2 = __float2bfloat162_rn(t);
    uint32_t r = __hge2_mask(__hadd2(h2(q.x), h2(cb.x)), t2) & (0x00010001u << (4 * u));
    r |= __hge2_mask(__hadd2(h2(q.y), h2(cb.y)), t2) & (0x00010001u << (4 * u + 1));
    r |= __hge2_mask(__hadd2(h2(q.z), h2(cb.z)), t2) & (0x00010001u << (4 * u + 2));
    r |= __hge2_mask(__hadd2(h2(q.w), h2(cb.w)), t2) & (0x00010001u << (4 * u + 3));
    return r;
  }
  static __device__ __forceinline__ int unit(int bit) { return (bit & 15) >> 2; }
  static __device__ __forceinline__ int elem(int bit) { return (bit & 3) * 2 + (bit >> 4); }
  template <typename F> static __device__ __forceinline__ void each2(const uint4& q, F f) {
#pragma unroll
    for (int i = 0; i < 4; ++i) { const uint32_t w = (&q.x)[i]; f(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u)); }
  }
};
template <> struct RowBlock<float> {             // four floats each
  static constexpr int E = 4;
  static constexpr uint32_t kNone = 0xFF800000u;
  template <int G> static __device__ __forceinline__ float max(const uint4 (&q)[G]) {
    float m = -INFINITY;
#pragma unroll
    for (int u = 0; u < G; ++u)
      m = fmaxf(m, fmaxf(fmaxf(__uint_as_float(q[u].x), __uint_as_float(q[u].y)), fmaxf(__uint_as_float(q[u].z), __uint_as_float(q[u].w))));
    return m;
  }
  static __device__ __forceinline__ float threshold(float t) { return t; }
  static constexpr int kUnits = 8;
  template <int G> static __device__ __forceinline__ uint32_t hits(const uint4 (&q)[G], int, float t) {
    uint32_t r = 0;
#pragma unroll
    for (int u = 0; u < G; ++u)
#pragma unroll
      for (int i = 0; i < 4; ++i) r |= __uint_as_float((&q[u].x)[i]) >= t ? 1u << (4 * u + i) : 0u;
    return r;
  }
  static __device__ __forceinline__ uint32_t boost(float cb) { return __float_as_uint(cb); }
  static constexpr float kBoostSlack = 0.0f;
  static __device__ __forceinline__ uint32_t hits_boosted(const uint4& q, const uint4& cb, int u, float t) {
    uint32_t r = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) r |= __fadd_rn(__uint_as_float((&q.x)[i]), __uint_as_float((&cb.x)[i])) >= t ? 1u << (4 * u + i) : 0u;
    return r;
  }
  static __device__ __forceinline__ int unit(int bit) { return bit >> 2; }
  static __device__ __forceinline__ int elem(int bit) { return bit & 3; }
  template <typename F> static __device__ __forceinline__ void each2(const uint4& q, F f) {
    f(__uint_as_float(q.x), __uint_as_float(q.y)); f(__uint_as_float(q.z), __uint_as_float(q.w));
  }
};
__device__ __forceinline__ float exp2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The root boost of every token, in the rows' element type, once for each way a row may be aligned: copy h begins with token
// h, so that the boosts of a row's aligned 16-byte blocks are aligned blocks themselves.  With it a row's candidates are the
// tokens whose root-boosted value reaches the row's raw maximum: three or four, where the tokens within the largest boost
// of the maximum are hundreds when boosts are several nats (lists of text, weighted by the length of a piece).
template <typename LT>
struct BoostTab {
  static __host__ __device__ constexpr size_t copy_bytes(int V) { return (static_cast<size_t>(V) * sizeof(LT) + 31) & ~size_t(15); }
  static __host__ __device__ constexpr size_t bytes(int V) { return 16 / sizeof(LT) * copy_bytes(V); }
};
// Block-wide, after root_tab_fill; the caller's next barrier completes it.
template <typename LT>
__device__ __forceinline__ void boost_tab_fill(unsigned char* tab, const RootTab& r, const int32_t* cls, float lam, int V) {
  using RB = RowBlock<LT>;
  const size_t stride = BoostTab<LT>::copy_bytes(V);
#pragma unroll 1
  for (int v = threadIdx.x; v < V; v += blockDim.x) {
    const uint32_t cb = RB::boost(__fmul_rn(lam, r.w[__ldg(cls + v)]));
#pragma unroll
    for (int h = 0; h < RB::E; ++h)
      if (v >= h) {
        if constexpr (sizeof(LT) == 2) reinterpret_cast<uint16_t*>(tab + h * stride)[v - h] = static_cast<uint16_t>(cb);
        else reinterpret_cast<uint32_t*>(tab + h * stride)[v - h] = cb;
      }
  }
}

// The rows of up to 32 frames by one warp: frames f0, f0 + step, ... (n of them), row k of a frame only when row k - 1 is
// likely to select a token (its best root-boosted token reaches the blank less a margin); a row left out is marked
// kRsAbsent, and a decider that gets there after all evaluates it exactly.  About half the rows of three per frame are
// never visited, and fewer still are read here.  sums: the summary of row 0 of frame 0.
//
// One row: a pass over its groups of 32 * G aligned 16-byte blocks for the maximum, then a pass for the few candidates --
// over the last group, still in registers, and from L1 over the groups before it.  The elements before the first and
// after the last aligned block are one per lane; nothing outside the row is read.  The next row's blocks are requested
// before a row's candidates are looked at, where a row is one group.  What is the same for all lanes is kept by lane i
// for frame i and finished for all frames of a pass at once (root arcs, normalisers, durations, the store).
//
// TAB: the candidates come from the table of root boosts (h.boost_a); else they are the tokens within the largest boost of
// the row's maximum.
template <typename LT, int G, bool TAB>
__device__ __forceinline__ void frames_summary(const RowCtx& h, const LT* base, int64_t st, int64_t ss, int S, int f0, int step, int n,
                                               RowSum* sums, int fmask, int lane) {
  using RB = RowBlock<LT>;
  constexpr int E = RB::E;
  const int V = h.V;
  const float kL2e = 1.4426950408889634f;
  unsigned todo = n >= 32 ? 0xFFFFFFFFu : (1u << n) - 1u;
  const float margin = 0.5f * h.beta_max;
#pragma unroll 1
  for (int k = 0; k < S; ++k) {
    // this lane's frame: what the warp finds out about its row
    float m_y1 = -INFINITY, m_y2 = -INFINITY, m_M = 0.0f, m_acc = 0.0f;
    int m_id = 0x7FFFFFFF;
    const LT* row0 = base + static_cast<int64_t>(f0) * st + static_cast<int64_t>(k) * ss;
    const int64_t fstep = static_cast<int64_t>(step) * st;
    uint4 q[G];
    float xs;
    const LT* row = nullptr;
    int hd = 0, nb = 0, sidx = 0;
    bool sok = false;
    auto begin = [&](int i) {                                  // geometry and first group of frame i's row
      row = row0 + static_cast<int64_t>(i) * fstep;
      hd = min(V, static_cast<int>((16u - static_cast<uint32_t>(reinterpret_cast<uintptr_t>(row) & 15)) & 15u) / static_cast<int>(sizeof(LT)));
      nb = (V - hd) / E;
      sidx = lane < hd ? lane : nb * E + lane;                 // this lane's element outside the blocks
      sok = sidx < V && lane < 2 * E;
      xs = -INFINITY;
      if (sok) xs = LogitLoad<LT>::at(row + sidx);
    };
    auto load = [&](int g) {
      const uint4* blk = reinterpret_cast<const uint4*>(row + hd) + lane;
#pragma unroll
      for (int u = 0; u < G; ++u) {
        q[u] = make_uint4(RB::kNone, RB::kNone, RB::kNone, RB::kNone);
        if (g + 32 * u + lane < nb) q[u] = __ldg(blk + g + 32 * u);
      }
    };
    unsigned left = todo;
    int i = __ffs(left) - 1;
    if (i >= 0) { begin(i); load(0); }
#pragma unroll 1
    while (left) {
      left &= left - 1u;
      const LT* rowi = row;
      const int hdi = hd, nbi = nb, si = sidx;
      const bool soki = sok;
      const float xsi = xs;
      const int inext = __ffs(left) - 1;
      float m = fmaxf(xsi, RB::template max<G>(q));
      int g_last = 0;
#pragma unroll 1
      for (int g = 32 * G; g < nb; g += 32 * G) { load(g); m = fmaxf(m, RB::template max<G>(q)); g_last = g; }
      const float mf = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(m)));
      // every token whose root-boosted value can reach that of the raw maximum has x >= m - (beta_max - beta_min); gamma
      // keeps a strict margin over all roundings
      const float gamma = (fabsf(mf) + fabsf(h.beta_max) + fabsf(h.beta_min)) * 0.0009765625f + 1e-30f;
      const float thr = RB::threshold(__fsub_rn(__fsub_rn(mf, __fsub_rn(h.beta_max, h.beta_min)), gamma));
      // tokens that are no candidates have root-boosted values of at most `others`: x < thr, hence <= fl(thr + beta_max); or,
      // TAB, by their boosted values themselves (some token's reaches mf + beta_min)
      const float others = TAB ? __fsub_rn(__fadd_rn(mf, h.beta_min), gamma) : __fadd_rn(thr, h.beta_max);
      // (no slack, no term: zero times an infinite maximum would be no number, and a row of -inf has its lowest token like any)
      float thr_b = others;
      if constexpr (TAB && RB::kBoostSlack > 0.0f) thr_b = __fsub_rn(others, RB::kBoostSlack * (fabsf(mf) + h.beta_max - h.beta_min));
      thr_b = TAB ? RB::threshold(thr_b) : 0.0f;
      // L = M + log(sum_v exp(x_v - M)): one fused multiply-add and one exponential per entry, see tb_fast_common.cuh
      float M = 0.0f, acc0 = 0.0f, acc1 = 0.0f;
      if (h.norm) M = fmaxf(mf, LogitLoad<LT>::at(rowi + V));
      const float nc = -__fmul_rn(M, kL2e);
      ValId b{-INFINITY, INT32_MAX};
      float sec = -INFINITY;
      auto offer = [&](int idx) {
        const float cb = h.boosts ? __fmul_rn(h.lam, h.rootw[__ldg(h.cls + idx)]) : 0.0f;
        const ValId c{__fadd_rn(LogitLoad<LT>::at(rowi + idx), cb), idx};
        if (better(c, b)) { sec = fmaxf(sec, b.v); b = c; } else { sec = fmaxf(sec, c.v); }
      };
#pragma unroll 1
      for (int g = g_last; g >= 0; g -= 32 * G) {
        if (g != g_last) load(g);
        if (h.norm) {
#pragma unroll
          for (int u = 0; u < G; ++u)
            RB::each2(q[u], [&](float x0, float x1) {
              acc0 = __fadd_rn(acc0, exp2_approx(__fmaf_rn(x0, kL2e, nc)));
              acc1 = __fadd_rn(acc1, exp2_approx(__fmaf_rn(x1, kL2e, nc)));
            });
        }
        uint32_t hits = 0u, hits2 = 0u;
        if constexpr (TAB) {
          const uint32_t at = h.boost_a + static_cast<uint32_t>(hdi) * static_cast<uint32_t>(BoostTab<LT>::copy_bytes(V)) + 16u * (g + lane);
#pragma unroll
          for (int u = 0; u < G; ++u)
            if (g + 32 * u + lane < nbi) {
              const uint4 cb = lds128(at + 512u * u);
              if (u < RB::kUnits) hits |= RB::hits_boosted(q[u], cb, u, thr_b); else hits2 |= RB::hits_boosted(q[u], cb, u - RB::kUnits, thr_b);
            }
        } else {
          hits = RB::template hits<G>(q, 0, thr);
          if constexpr (RB::kUnits < G) hits2 = RB::template hits<G>(q, RB::kUnits, thr);
        }
        if (g == 0 && inext >= 0) {                            // (q is free: the next row is on its way from here on)
          begin(inext);
          load(0);
        }
        int ub = g + lane;
#pragma unroll 1
        for (;;) {
          if (hits == 0u) {
            if (hits2 == 0u) break;
            hits = hits2; hits2 = 0u; ub += 32 * RB::kUnits;
          }
          const int bit = __ffs(hits) - 1;
          hits &= hits - 1u;
          const int bi = ub + 32 * RB::unit(bit);
          if (bi < nbi) offer(hdi + bi * E + RB::elem(bit));   // (places without a block pass only a threshold of -inf)
        }
      }
      if (soki && xsi >= thr) offer(si);
      if (h.norm) {
        float acc = __fadd_rn(acc0, acc1);
        if (soki) acc = __fadd_rn(acc, exp2_approx(__fmaf_rn(xsi, kL2e, nc)));
        if (lane == 0) acc = __fadd_rn(acc, exp2_approx(__fmaf_rn(LogitLoad<LT>::at(rowi + V), kL2e, nc)));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, off));
        if (lane == i) { m_M = M; m_acc = acc; }
      }
      // across the warp: best (value, lowest id) and the runner-up value
      const uint32_t key = order_key(b.v);
      const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
      const int idmin = static_cast<int>(__reduce_min_sync(0xffffffffu, key == kmax ? static_cast<uint32_t>(b.i) : 0x7FFFFFFFu));
      const uint32_t k2 = __reduce_max_sync(0xffffffffu, order_key((key == kmax && b.i == idmin) ? sec : b.v));
      if (lane == i) { m_y1 = order_key_inv(kmax); m_id = idmin; m_y2 = fmaxf(order_key_inv(k2), others); }
      i = inext;
    }
    // ---- lane i finishes frame i's row
    bool need = false;
    if (lane < n) {
      const int f = f0 + lane * step;
      uint4* o = reinterpret_cast<uint4*>(sums + (f & fmask) * S + k);
      uint4 w0 = make_uint4(0u, 0u, 0u, 0u), w1 = make_uint4(0u, 0u, kRsAbsent, 0u);
      if ((todo >> lane) & 1u) {
        const LT* r = row0 + static_cast<int64_t>(lane) * fstep;
        const bool ovf = m_id >= V;                            // no candidate at all (cannot happen with finite logits)
        const int id1 = ovf ? 0 : m_id;
        const int a1 = h.boosts ? h.rootarc[__ldg(h.cls + id1)] : 0;
        const float x1 = LogitLoad<LT>::at(r + id1), xb = LogitLoad<LT>::at(r + V);
        float cw = 0.0f, extra = 0.0f;
        int cd = 0, dur = 0;
        if (a1) { cw = __fadd_rn(0.0f, h.arc_w[a1 - 1]); cd = h.arc_dst[a1 - 1]; }
        if (h.norm && m_M != -INFINITY) {
          const float c_lo = __fmaf_rn(m_M, kL2e, -__fmul_rn(m_M, kL2e));      // what the rounding of M * log2(e) left out, exactly
          extra = __fadd_rn(m_M, __fsub_rn(logf(m_acc), __fmul_rn(c_lo, 0.6931471805599453f)));
        }
#pragma unroll 4
        for (int d = 0; d < h.n_dur; ++d) {                    // the row's best duration (lowest on ties)
          const float xd = LogitLoad<LT>::at(r + V + 1 + d);
          if (d == 0 || xd > extra) { extra = xd; dur = d; }
        }
        // the same margin as the decider's, with the largest scale any state can have
        const float tau = (fabsf(m_y1) + 4.0f * h.bmag_max) * 1.9073486328125e-6f + 1e-30f;
        w0 = make_uint4(__float_as_uint(m_y1), __float_as_uint(m_y2), __float_as_uint(xb), __float_as_uint(x1));
        w1 = make_uint4(__float_as_uint(cw), static_cast<uint32_t>(cd),
                        static_cast<uint32_t>(id1) | (ovf ? kRsOvf : 0u) | ((m_y1 - m_y2 > tau) ? kRsGap : 0u) | (static_cast<uint32_t>(dur) << 24),
                        __float_as_uint(extra));
        // (a row whose duration moves the cursor on has no row after it; normalisers are wanted for every row)
        need = h.norm || ((ovf || !(m_y1 + margin < xb)) && dur == 0);
      }
      o[0] = w0; o[1] = w1;
    }
    todo = __ballot_sync(0xffffffffu, need);
  }
  __syncwarp();
}

// ---- step 2: the decider -------------------------------------------------------------------------------------------

// What a decider needs to know about its stream's graph and rows; the same for all lanes.
template <typename LT>
struct DecideCtx {
  const LT* base;                  // row (frame 0 of the call, row 0) of the stream
  int64_t st, ss;                  // element strides: frame, row in frame
  int V, S, n_dur, tb;             // tb: bits of 2 * token in a list entry (tb_rs_tok_bits)
  bool bound, resolved, norm;
  int n_states, max_depth;
  float lam, R;                    // lambda; largest |root arc weight|
  const TbRsRec* rsrec;            // resolved lists, in the arena or in shared memory
  const TbRsEnt* rsent;
  const TbStateRec* strec;         // without resolved lists: what the suffix-chain walk reads
  const TbTokEnt* tokent;
  RootTab root;
  const int32_t* cls; const float* arc_w; const int32_t* arc_dst;
  uint32_t* bitmap;                // [(V + 32) / 32] shared memory of this warp, zero between uses
  TbRsEnt* walk_buf;               // [kWalkBuf] shared memory of this warp, and
  TbRsEnt* spill;                  // [V + 32] global memory: lists put together by walking (null: the lists are resolved)
  const TbDecodeParams* p;         // a graph whose lists are not there (not yet, in the chunk that binds it; or for want of room) is
  int slot;                        // walked from its flat arrays, with its slot's record (-1: it is not such a graph)
  int32_t* status;
};

// The tokens boosted by the non-root part of the current state's suffix chain: entries {target << tb | 2 * token, lb},
// lb = fl(lambda * fl(acc + w)).  Resolved lists are read where they lie.
struct TokList {
  const TbRsEnt* ent;
  int n;
  float D, bmag;
};
// {target << tb | 2 token} -> {2 token | target}: an integer minimum finds the lowest token and its target at once
__device__ __forceinline__ uint32_t td_pack(uint32_t dst_tok, int tb) { return __funnelshift_r(dst_tok, dst_tok, tb); }
__device__ __forceinline__ int td_tok(uint32_t td, int tb) { return static_cast<int>(td >> (33 - tb)); }
__device__ __forceinline__ int td_dst(uint32_t td, int tb) { return static_cast<int>(td & (0xFFFFFFFFu >> tb)); }

// One more entry of a list that is put together by walking, unless a chain state closer to the start listed the token.
template <typename LT>
__device__ __forceinline__ void walk_add(const DecideCtx<LT>& c, bool have, int tk, uint32_t dst, float w, float acc, int& n, int lane) {
  const bool fresh = have && !((c.bitmap[tk >> 5] >> (tk & 31)) & 1u);
  const unsigned mask = __ballot_sync(0xffffffffu, fresh);
  if (fresh) {
    atomicOr(&c.bitmap[tk >> 5], 1u << (tk & 31));
    TbRsEnt o;
    o.dst_tok = (dst << c.tb) | (2u * static_cast<uint32_t>(tk));
    o.lb = __fmul_rn(c.lam, __fadd_rn(acc, w));
    const int at = n + __popc(mask & ((1u << lane) - 1u));
    c.spill[at] = o;
    if (at < kWalkBuf) c.walk_buf[at] = o;
  }
  n += __popc(mask);
}
// The walk over a graph's flat arrays; sum: the suffix-link weights of the whole chain, in walk order.
template <typename LT>
__device__ __forceinline__ int walk_flat(const DecideCtx<LT>& c, int s, float& sum, int lane) {
  const GraphPtrs g = graph_of(c.p->arena, c.p->slots[c.slot]);
  const int32_t* ctb = c.p->class_tok;
  const int32_t* ctk = ctb + c.p->C + 1;
  int n = 0, u = s > 0 ? s : 0;
  float acc = 0.0f;
#pragma unroll 1
  for (int it = 0; u != 0; ++it) {
    if (it > c.max_depth + 1) { if (lane == 0) atomicOr(c.status, TB_STATUS_WALK_TOO_DEEP); break; }
    const int a1 = g.arc_begin[u + 1], nu = g.fail[u];
    const float bw = g.bw[u];
#pragma unroll 1
    for (int a = g.arc_begin[u] + lane; __any_sync(0xffffffffu, a < a1); a += 32) {
      int q = 0, q1 = 0;
      uint32_t dst = 0;
      float w = 0.0f;
      if (a < a1) { const int cl = g.arc_cls[a]; q = ctb[cl]; q1 = ctb[cl + 1]; dst = static_cast<uint32_t>(g.arc_dst[a]); w = g.arc_w[a]; }
#pragma unroll 1
      for (; __any_sync(0xffffffffu, q < q1); ++q) walk_add(c, q < q1, q < q1 ? ctk[q] : 0, dst, w, acc, n, lane);
    }
    __syncwarp();
    acc = __fadd_rn(acc, bw);
    u = nu > 0 && nu < c.n_states ? nu : 0;
  }
  sum = acc;
  return n;
}

// The list of state s (warp-wide); W: groups of 32 entries of a chain state that are asked for at once.
template <typename LT, int W>
__device__ __forceinline__ TokList list_of(const DecideCtx<LT>& c, int s, int lane) {
  TokList L;
  if (c.resolved) {
    L.ent = c.rsent; L.n = 0; L.D = 0.0f; L.bmag = fabsf(c.lam) * c.R;
    if (s > 0) {                                              // (the root's list is empty)
      const uint4 r = *reinterpret_cast<const uint4*>(c.rsrec + s);
      L.ent += r.x; L.n = static_cast<int>(r.y); L.D = __uint_as_float(r.z); L.bmag = __uint_as_float(r.w);
    }
    return L;
  }
  // Chain walk: the chain state closest to s first; a token whose class a closer state lists is in the bitmap already.
  // acc = suffix-link weights crossed so far, in walk order.
  int n = 0;
  float acc = 0.0f;
  int u = s > 0 ? s : 0;
  if (c.slot >= 0) { n = walk_flat(c, s, acc, lane); u = 0; }
  uint4 rec = make_uint4(0u, 0u, 0u, 0u);                     // TbStateRec
  if (u != 0) rec = *reinterpret_cast<const uint4*>(c.strec + u);
#pragma unroll 1
  for (int it = 0; u != 0; ++it) {
    if (it > c.max_depth + 1) { if (lane == 0) atomicOr(c.status, TB_STATUS_WALK_TOO_DEEP); break; }
    // the next chain state's record is requested before this state's arcs are: the two trips to L2 overlap
    const int nu = (static_cast<int>(rec.z) > 0 && static_cast<int>(rec.z) < c.n_states) ? static_cast<int>(rec.z) : 0;
    uint4 nrec = rec;
    if (nu > 0) nrec = *reinterpret_cast<const uint4*>(c.strec + nu);
    const int e1 = static_cast<int>(rec.y);
    // (where an entry leads: the state's record and its first arcs are asked into L2, in case the entry is taken)
    auto take = [&](bool have, const uint4& ent) {            // TbTokEnt
      if (have) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(c.strec + ent.z));
        asm volatile("prefetch.global.L2 [%0];" ::"l"(c.tokent + ent.w));
      }
      walk_add(c, have, static_cast<int>(ent.x & 0xFFFFu), ent.z, __uint_as_float(ent.y), acc, n, lane);
    };
    if constexpr (W > 1) {
#pragma unroll 1
      for (int e0 = static_cast<int>(rec.x); e0 < e1; e0 += 32 * W) {
        uint4 ent[W];
#pragma unroll
        for (int u = 0; u < W; ++u) {
          const int e = e0 + 32 * u + lane;
          ent[u] = make_uint4(0u, 0u, 0u, 0u);
          if (e < e1) ent[u] = *reinterpret_cast<const uint4*>(c.tokent + e);
        }
#pragma unroll
        for (int u = 0; u < W; ++u) {
          if (u > 0 && e0 + 32 * u >= e1) break;
          take(e0 + 32 * u + lane < e1, ent[u]);
        }
      }
    } else {
#pragma unroll 2
      for (int e = static_cast<int>(rec.x) + lane; __any_sync(0xffffffffu, e < e1); e += 32) {
        uint4 ent = make_uint4(0u, 0u, 0u, 0u);
        if (e < e1) ent = *reinterpret_cast<const uint4*>(c.tokent + e);
        take(e < e1, ent);
      }
    }
    __syncwarp();
    acc = __fadd_rn(acc, __uint_as_float(rec.w));
    u = nu;
    rec = nrec;
  }
  L.n = n; L.D = acc; L.bmag = fabsf(c.lam) * (fabsf(acc) + c.R);
  L.ent = n <= kWalkBuf ? c.walk_buf : c.spill;
#pragma unroll 1
  for (int i = lane; i < n; i += 32) c.bitmap[(L.ent[i].dst_tok & ((1u << c.tb) - 1u)) >> 6] = 0u;
  __syncwarp();
  return L;
}

struct RowPick { float val; int tok, next, dur; float xdur; };   // tok == V: blank

// Exact evaluation of one row under the current state by the whole warp.
template <typename LT>
__device__ __forceinline__ RowPick exact_row(const DecideCtx<LT>& c, const TokList& L, const LT* row, int s, int lane) {
  using RB = RowBlock<LT>;
  ValId best{LogitLoad<LT>::at(row + c.V), c.V};
  int bn = s;
#pragma unroll 1
  for (int i = lane; i < L.n; i += 32) {
    const TbRsEnt e = L.ent[i];
    const int tk = static_cast<int>((e.dst_tok & ((1u << c.tb) - 1u)) >> 1);
    if (tk >= c.V) continue;                                   // (padding)
    atomicOr(&c.bitmap[tk >> 5], 1u << (tk & 31));
    const ValId o{__fadd_rn(LogitLoad<LT>::at(row + tk), e.lb), tk};
    if (better(o, best)) { best = o; bn = static_cast<int>(e.dst_tok >> c.tb); }
  }
  __syncwarp();
  // A token outside the list is worth looking up only where its logit alone could bring it past the best so far (`slack`
  // covers all roundings): the row is compared with that threshold, 16 bytes at a time.
  const float B = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(best.v)));
  const float U = c.bound ? c.lam * L.D + c.root.stats[1] : 0.0f;
  const float slack = (fabsf(B) + fabsf(U) + L.bmag) * 3.814697265625e-6f + 1e-30f;
  // (a best that is infinite bounds nothing: its difference from the slack is no number, and every token is looked up)
  const float bound_x = B - U - slack;
  const float thr = RB::threshold(fabsf(bound_x) < INFINITY ? bound_x : -INFINITY);
  auto offer = [&](int tk) {
    float v = LogitLoad<LT>::at(row + tk);
    int nx = -1;
    if (c.bound) {
      const int cl = __ldg(c.cls + tk);
      v = __fadd_rn(v, __fmul_rn(c.lam, __fadd_rn(L.D, c.root.w[cl])));
      nx = c.root.arc[cl];
      nx = nx ? -1 - nx : 0;                                   // (the arc's target is looked up for the winner only)
    }
    const ValId o{v, tk};
    if (!((c.bitmap[tk >> 5] >> (tk & 31)) & 1u) && better(o, best)) { best = o; bn = nx; }
  };
  const int hd = min(c.V, static_cast<int>((16u - static_cast<uint32_t>(reinterpret_cast<uintptr_t>(row) & 15)) & 15u) / static_cast<int>(sizeof(LT)));
  const int nb = (c.V - hd) / RB::E;
#pragma unroll 1
  for (int g = lane; __any_sync(0xffffffffu, g < nb); g += 32 * 4) {
    uint4 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      q[u] = make_uint4(RB::kNone, RB::kNone, RB::kNone, RB::kNone);
      if (g + 32 * u < nb) q[u] = __ldg(reinterpret_cast<const uint4*>(row + hd) + g + 32 * u);
    }
    uint32_t hits = RB::template hits<4>(q, 0, thr);
#pragma unroll 1
    while (hits) {
      const int bit = __ffs(hits) - 1, bi = g + 32 * RB::unit(bit);
      hits &= hits - 1u;
      if (bi < nb) offer(hd + bi * RB::E + RB::elem(bit));
    }
  }
  const int edge = lane < hd ? lane : nb * RB::E + lane;         // this lane's token outside the aligned blocks
  if (lane < 2 * RB::E && edge < c.V) offer(edge);
  __syncwarp();
#pragma unroll 1
  for (int i = lane; i < L.n; i += 32) c.bitmap[(L.ent[i].dst_tok & ((1u << c.tb) - 1u)) >> 6] = 0u;
  __syncwarp();
  const uint32_t key = order_key(best.v);
  const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
  const uint32_t idmin = __reduce_min_sync(0xffffffffu, key == kmax ? static_cast<uint32_t>(best.i) : 0xFFFFFFFFu);
  const unsigned who = __ballot_sync(0xffffffffu, key == kmax && static_cast<uint32_t>(best.i) == idmin);
  const int src = __ffs(who) - 1;
  RowPick pk;
  pk.dur = 0; pk.xdur = 0.0f;
#pragma unroll 1
  for (int d = 0; d < c.n_dur; ++d) {                          // the row's best duration (lowest on ties)
    const float xd = LogitLoad<LT>::at(row + c.V + 1 + d);
    if (d == 0 || xd > pk.xdur) { pk.xdur = xd; pk.dur = d; }
  }
  pk.val = __shfl_sync(0xffffffffu, best.v, src);
  pk.tok = static_cast<int>(idmin);
  pk.next = __shfl_sync(0xffffffffu, bn, src);
  if (pk.tok == c.V) pk.next = s;
  else if (!c.bound) pk.next = -1;
  else if (pk.next < 0) pk.next = c.arc_dst[-pk.next - 2];     // -1 - (arc + 1) -> arc
  return pk;
}

// Where a decider stands.
struct Cursor {
  int t, k, s;          // frame, row in frame, graph state
  int n_out, nv;        // tokens emitted, row values logged
  bool failed;
  int met;              // frame start at which it met a later stretch of the stream (-1: none)
  bool listed;          // list is that of state s
  TokList list;
};
// Where its results go.
struct DecideOut {
  int32_t* tok; int32_t* frm; int32_t* dur;   // emitted tokens, their frames, durations (dur may be null)
  float* vals;                                // value of every visited row, in order
  int cap;                                    // places in tok / frm
  // a stretch of an offline decode (SEG): the graph state at every frame start it answers for, [first, next), and how
  // much it had logged there; past `next` it stops where its state is the one recorded there
  volatile int32_t* trace; int2* trace_aux;
  int first, next;
  bool is_last;
};

// Decides the rows from the cursor on, up to frame `end` (exclusive).  Summaries of row k of frame f are at shared
// address sum_a + (((f - f0) & mask) * S + k) * 32; SEG: that is a ring of mask + 1 frames which the decider fills itself
// from gsum (the summary of row 0 of frame 0), else they are all in place.  f0: the frame the rows (c.base) start at.
// WALK: for lists that are put together by walking.  A lane's entries of a list whose logits are on their way at once, and groups of a chain state's entries,
// are more then: a state of 64 streams with lists of 1000 own phrases and 4000 shared ones has about 140 entries, of which the logits, all over their row, took
// 4400 of a round's 9500 cycles and the walk 3600.  A call took 1283 us with 4 entries and 2 groups, 1169 with 8 and 2, 1119 with 8 and 4, 1096 with 12 and 4,
// 1117 with 16 and 4, 1203 with 8 and 8.  (Resolved lists are shorter: 32 fp32 streams of 500 frames 152 us with 4 entries, 162 with 12.  Rows
// brought into shared memory ahead of their rounds leave L1 too little: 1369.)
template <typename LT, bool SEG, bool WALK>
__device__ __forceinline__ void decide(const DecideCtx<LT>& c, Cursor& cu, const DecideOut& o, const RowSum* gsum,
                                       uint32_t sum_a, int mask, int f0, int end, int lane) {
  const int S = c.S, V = c.V, tb = c.tb;
  constexpr int kIn = WALK ? 12 : 4, kWalk = WALK ? 4 : 1;
  const bool tdt = !SEG && c.n_dur > 0;
  int t = cu.t, k = cu.k, s = cu.s, n_out = cu.n_out, nv = cu.nv;
  bool listed = cu.listed;
  int still = 0;                               // tokens in a row that left the (non-root) state what it was
  TokList L = cu.list;
  const uint32_t none = (2u * static_cast<uint32_t>(V)) << (32 - tb), tmask = (1u << tb) - 1u;
  // what a row adds to the score: its value less its normaliser, or plus its duration's logit
  auto adjust = [&](float v, float extra) { return c.norm ? __fsub_rn(v, extra) : tdt ? __fadd_rn(v, extra) : v; };
  auto trace = [&](int fs, int st_, int n_tok, int n_val) {
    if (SEG && fs >= o.first && fs < o.next) { o.trace_aux[fs] = make_int2(n_tok, n_val); o.trace[fs] = st_; }
  };
  if (SEG && lane == 0 && k == 0) trace(t, s, n_out, nv);
  int loaded = t & ~7, refill = t;            // SEG: frames up to `loaded` have been asked for; the next group is due at frame `refill`
  const int max_rounds = (end - t) * (S + 1) + 8;
#pragma unroll 1
  for (int it = 0; t < end; ++it) {
    if (it >= max_rounds) { if (lane == 0) atomicOr(c.status, TB_STATUS_STEP_LIMIT); cu.failed = true; break; }
    if (SEG) {
      if (k == 0 && t >= o.next && !o.is_last) {
        if (!c.bound || o.trace[t] == s) { cu.met = t; break; }     // (unbound: no graph state, the owner's decode from here is this one's)
      }
      // the ring, in groups of eight frames: the round's window is in place, the next group is on its way
      if (t >= refill) {
        do {
          const int nq = min(8, end - loaded) * S * 2;
          const uint4* src = reinterpret_cast<const uint4*>(gsum + static_cast<int64_t>(loaded) * S);
          const uint32_t dst = sum_a + static_cast<uint32_t>((loaded & mask) * S) * 32u;
#pragma unroll
          for (int i = 0; i < 8 * kRowsPerFrame * 2; i += 32)
            if (i + lane < nq) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * (i + lane)), "l"(src + i + lane) : "memory");
          asm volatile("cp.async.commit_group;" ::: "memory");
          loaded += 8;
        } while (loaded < t + 24);
        refill = (t & ~7) + 8;
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncwarp();
      }
    }
    if (!listed) { L = list_of<LT, kWalk>(c, s, lane); listed = true; }
    // One round: up to eight rows in the order they are visited in, a group of lanes each.  Which rows those are, and the
    // graph state each is visited in, is predicted from the summaries alone -- a row selects its best plain token, which
    // leads to a root arc's target, or blank -- and every group then decides its row exactly under the state predicted for
    // it.  The round ends with the first row that goes another way (a token of the list, most often) or has to be
    // evaluated in full.  Longer lists get more lanes per row, and fewer rows.
    const int left = end - 1 - t;              // frames after the current one
    const int sh = L.n <= 32 ? 2 : L.n <= 128 ? 3 : 4, G = 1 << sh;
    auto summary_at = [&](int q, int j) { return sum_a + static_cast<uint32_t>(((t + q - f0) & mask) * S + j) * 32u; };
    // (after a token the state is the root most often; one that has repeated itself, as lists with repeated tokens make a
    // state do for hundreds of frames, is taken to go on doing so)
    const bool stay = still >= 4;
    auto pred_tok = [&](float y1, float xb, bool seen) { return stay || (seen ? y1 : __fadd_rn(y1, __fmul_rn(c.lam, L.D))) >= xb; };
    // where a row leads, as 4 * frame + row
    auto next_at = [&](int q, int j, bool tk, int dur) {
      if (tdt && (!tk || dur > 0)) return 4 * (q + max(dur, 1));
      return tk && j + 1 < S ? 4 * q + j + 1 : 4 * q + 4;
    };
    // ---- the path: lane 4 q + j stands for row (t + q, j); lane 31 is where it leaves the window
    int sel = 31, tok_before = -1;             // this lane's row on the path, and the lane of the last token before it
    int plain_a;                               // where the best plain token of row (lane >> 2, lane & 3) leads
    {
      const int q = lane >> 2, j = lane & 3;
      const uint32_t a = summary_at(q, min(j, S - 1));
      const uint4 h1 = lds128(a + 16u), h0 = lds128(a);
      plain_a = c.bound ? static_cast<int>(h1.y) : -1;
      const float y1 = __uint_as_float(h0.x), xb = __uint_as_float(h0.z);
      const int dur = tdt ? static_cast<int>(h1.z >> 24) : 0;
      const bool tk_s = pred_tok(y1, xb, false), tk_0 = pred_tok(y1, xb, true);
      uint32_t step = static_cast<uint32_t>(min(next_at(q, j, tk_s, dur), 31)) << 1 | (tk_s ? 1u : 0u) |
                      static_cast<uint32_t>(min(next_at(q, j, tk_0, dur), 31)) << 17 | (tk_0 ? 1u << 16 : 0u);
      if (lane == 31) step = 31u << 1 | 31u << 17;
      int cur = k, last = -1, half = 0;
      const int group = lane >> sh;
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        if (group == g) { sel = cur; tok_before = last; }
        if (g == 7) break;
        const uint32_t w = __shfl_sync(0xffffffffu, step, cur) >> half;
        if (w & 1u) { last = cur; half = 16; }
        cur = static_cast<int>((w >> 1) & 31u);
      }
    }
    // ---- this lane's row, state and list
    const int rq = sel >> 2, rj = min(sel & 3, S - 1);
    const bool exists = sel != 31 && rq <= left;
    const uint32_t a = summary_at(rq, rj);
    const uint4 q1 = lds128(a + 16u), q0 = lds128(a);
    const int before = __shfl_sync(0xffffffffu, plain_a, tok_before & 31);
    const int ls = tok_before >= 0 && !stay ? before : s;
    TokList ll = L;
    bool lane_ok = true;
    if (ls != s) {
      ll.n = 0; ll.D = 0.0f; ll.bmag = fabsf(c.lam) * c.R;
      if (ls > 0) {
        lane_ok = c.resolved && ls < c.n_states;
        if (lane_ok) {
          const uint4 rec = *reinterpret_cast<const uint4*>(c.rsrec + ls);
          ll.ent = c.rsent + rec.x; ll.n = static_cast<int>(rec.y); ll.D = __uint_as_float(rec.z); ll.bmag = __uint_as_float(rec.w);
          lane_ok = ll.n <= 8 * G;
        }
      }
    }
    if (!lane_ok || !exists) ll.n = 0;
    const LT* row = c.base + static_cast<int64_t>(t - f0 + min(rq, left)) * c.st + static_cast<int64_t>(rj) * c.ss;
    const float y1 = __uint_as_float(q0.x), y2b = __uint_as_float(q0.y), xb = __uint_as_float(q0.z), x1 = __uint_as_float(q0.w);
    const uint32_t id1x2 = 2u * (q1.z & kRsIdMask);
    const int plain_next = c.bound ? static_cast<int>(q1.y) : -1, pred_next = stay ? s : plain_next;
    float lv = -INFINITY;
    uint32_t lt = none;
    bool in_deep = false;
#pragma unroll 1
    for (int i0 = lane & (G - 1); i0 < ll.n; i0 += kIn * G) {
      uint2 e[kIn];
      float x[kIn];
#pragma unroll
      for (int u = 0; u < kIn; ++u) {
        e[u] = make_uint2(2u * static_cast<uint32_t>(V), 0xFF800000u);
        if (i0 + u * G < ll.n) e[u] = *reinterpret_cast<const uint2*>(ll.ent + i0 + u * G);
      }
#pragma unroll
      for (int u = 0; u < kIn; ++u) x[u] = LogitLoad<LT>::at(row + ((e[u].x & tmask) >> 1));
#pragma unroll
      for (int u = 0; u < kIn; ++u) {
        const uint32_t td = td_pack(e[u].x, tb);
        const float v = __fadd_rn(x[u], __uint_as_float(e[u].y));
        if (v > lv || (v == lv && td < lt)) { lv = v; lt = td; }
        in_deep |= (e[u].x & tmask) == id1x2;
      }
    }
    // the group's best (largest value, then lowest token), in all its lanes
    auto join = [&](int off) {
      const float ov = __shfl_xor_sync(0xffffffffu, lv, off);
      const uint32_t ot = __shfl_xor_sync(0xffffffffu, lt, off);
      if (ov > lv || (ov == lv && ot < lt)) { lv = ov; lt = ot; }
    };
    join(1); join(2);
#pragma unroll 1
    for (int off = 4; off < G; off <<= 1) join(off);
    in_deep = ((__ballot_sync(0xffffffffu, in_deep) >> (lane & -G)) & ((1u << G) - 1u)) != 0u;
    // the row's pick: the best plain token is exact when the summary's winner is not listed and clears the others by the
    // rounding margin (at the root it is exact by construction); else it is bounded from above
    const float extra = __uint_as_float(q1.w);
    const int id1 = static_cast<int>(id1x2 >> 1), dur = tdt ? static_cast<int>(q1.z >> 24) : 0;
    float wv = lv;
    int wtok = td_tok(lt, tb), wnext = td_dst(lt, tb);
    bool rescan = (q1.z & (kRsOvf | kRsAbsent)) != 0;
    {
      const bool plain_ok = !in_deep && ((q1.z & kRsGap) != 0 || ls <= 0);
      const float nd = __fadd_rn(x1, __fmul_rn(c.lam, __fadd_rn(ll.D, __uint_as_float(q1.x))));
      const float ub = (in_deep ? y2b : y1) + c.lam * ll.D;
      const float tau = (fabsf(y1) + 4.0f * ll.bmag) * 3.814697265625e-6f + 1e-30f;
      rescan = rescan || (!plain_ok && !(fmaxf(wv, xb) > ub + tau));
      if (plain_ok && (nd > wv || (nd == wv && id1 < wtok))) { wv = nd; wtok = id1; wnext = plain_next; }
    }
    const bool blank = !(wv >= xb);                            // (a tie with blank goes to the token)
    // ---- as far as the rows went as predicted, and the first that did not
    const bool lead = (lane & (G - 1)) == 0, ready = lead && exists && lane_ok && !rescan;
    const bool as_pred = blank ? !pred_tok(y1, xb, tok_before >= 0) : pred_tok(y1, xb, tok_before >= 0) && wnext == pred_next;
    const unsigned ready_m = __ballot_sync(0xffffffffu, ready), blank_m = __ballot_sync(0xffffffffu, blank);
    const unsigned bad = __ballot_sync(0xffffffffu, lead && !(ready && as_pred));
    const unsigned cut = bad & (0u - bad);
    const unsigned cm = ready_m & ((cut - 1u) | cut);          // (cut == 0: all)
    int tok = V, tnext = s;                                    // where the round leads (tok == V: the state stays)
    if (cm != 0u) {
      const unsigned tm = cm & ~blank_m, upto = 0xFFFFFFFFu >> (31 - lane);
      const bool mine = (cm >> lane) & 1u;
      const int ntok = n_out + __popc(tm & upto), nval = nv + __popc(cm & upto);
      const int after = blank ? ls : wnext, at = next_at(rq, rj, !blank, dur);
      if (mine) {
        o.vals[nval - 1] = adjust(blank ? xb : wv, extra);
        if (!blank && ntok <= o.cap) {
          o.tok[ntok - 1] = wtok; o.frm[ntok - 1] = t + rq;
          if (!SEG && o.dur) o.dur[ntok - 1] = dur;
        }
        if ((at & 3) == 0) trace(t + rq + 1, after, ntok, nval);
      }
      nv += __popc(cm);
      n_out += __popc(tm);
      const int hi = 31 - __clz(cm);
      const int pos = __shfl_sync(0xffffffffu, at, hi);
      tnext = __shfl_sync(0xffffffffu, after, hi);
      still = s > 0 && tnext == s && ((tm >> hi) & 1u) ? still + __popc(tm) : 0;
      if (tnext != s) tok = 0;
      t += pos >> 2;
      k = pos & 3;
    } else {                                                   // the current row, in full
      const RowPick pk = exact_row(c, L, c.base + static_cast<int64_t>(t - f0) * c.st + static_cast<int64_t>(k) * c.ss, s, lane);
      tok = pk.tok; tnext = pk.next;
      still = s > 0 && tok != V && tnext == s ? still + 1 : 0;
      if (lane == 0) o.vals[nv] = adjust(pk.val, tdt ? pk.xdur : extra);
      ++nv;
      if (tok != V) {
        if (lane == 0 && n_out < o.cap) {
          o.tok[n_out] = tok; o.frm[n_out] = t;
          if (!SEG && o.dur) o.dur[n_out] = pk.dur;
        }
        ++n_out;
      }
      const int at = next_at(0, k, tok != V, pk.dur);
      if (lane == 0 && (at & 3) == 0) trace(t + 1, tnext, n_out, nv);
      t += at >> 2;
      k = at & 3;
    }
    if (tok != V && tnext != s && c.bound) {
      if (tnext < 0 || tnext >= c.n_states) { if (lane == 0) atomicOr(c.status, TB_STATUS_BAD_STATE); tnext = 0; }
      s = tnext;
      listed = false;
    }
  }
  if (SEG) asm volatile("cp.async.wait_all;" ::: "memory");
  cu.t = t; cu.k = k; cu.s = s; cu.n_out = n_out; cu.nv = nv; cu.listed = listed; cu.list = L;
}

}  // namespace

#endif  // TB_ROWS_CUH_
