// Beam pre-pass: every logit row to its few best root-boosted tokens, ahead of the steps and independent of every hypothesis.
#include "tb_rows.cuh"

namespace {

// One warp per row.  With the rows of a stream shared by its hypotheses, the order of a row's tokens that no hypothesis' state
// boosts is, up to rounding, the order of their root-boosted values y -- so a step only needs the first few of them.
// Bound by instruction issue.  A block takes a stretch of rows of one stream and lays out its root boosts per token once (four
// copies, the h-th beginning with token h, so that the boosts of a row's aligned 16-byte pieces are aligned as well); a row's
// values then take one addition each.  The top_m + 1 best come without rounds of picking: a threshold that as many of the lanes' best values
// (two per lane where one is too few) reach bounds the last of them from below; the row's tokens at or above that -- 1.3 times as many as are wanted, on average -- are collected and put in order by counting, for
// each, those before it.  Values that are no numbers come first, as their keys do, wherever in the row they are.  32 x 1000 rows of 1024 bf16, K = 4 (16 entries): 84 us token by token with a class and a root weight looked up for
// each, 53 so (10 by their bytes); 32 x 200 rows, K = 32 (44 entries): 26 us; 128 x 16 rows, K = 4: 11 to 21 us, 10 so.
constexpr int kTopWarps = 8;
constexpr int kTopGroup = 4;           // 16-byte pieces of a row a lane has at hand
constexpr int kTopCap = 128;           // tokens collected at a time
static_assert(kTopCap > TB_MAX_BEAM + 13, "more than any row keeps");
__host__ __device__ inline size_t boost_copy_bytes(int V) { return (static_cast<size_t>(V) * 4 + 31) & ~size_t(15); }

template <typename LT>
__global__ void __launch_bounds__(kTopWarps * 32, 3) k_beam_topm(const LT* logits, int32_t T, int32_t E, int32_t V, int32_t C,
                                                              int64_t stream_stride, int64_t frame_stride, int64_t row_stride,
                                                              const int32_t* n_frames, const TbSlotRec* slots, const unsigned char* arena,
                                                              const int32_t* cls, int32_t top_m, int32_t rows_per_warp, int32_t blocks_per_stream,
                                                              TbTopEnt* out) {
  using RB = RowBlock<LT>;
  constexpr int EB = RB::E, G = kTopGroup;
  pdl_chain();
  extern __shared__ __align__(16) unsigned char dyn[];
  const size_t copy = boost_copy_bytes(V);
  unsigned char* tab = dyn;                                                       // [4] copies of the tokens' boosts
  uint64_t* cand = reinterpret_cast<uint64_t*>(dyn + 4 * copy) + (threadIdx.x >> 5) * kTopCap;
  float* rootcw = reinterpret_cast<float*>(dyn + 4 * copy + kTopWarps * kTopCap * sizeof(uint64_t));   // [C] root arc weight per class
  const int b = blockIdx.x / blocks_per_stream, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int want = top_m + 1;
  const bool both = want > 28;
  int end = T;
  if (n_frames) end = max(0, min(T, n_frames[b]));
  const int rows = end * E, r0 = (blockIdx.x - b * blocks_per_stream) * rows_per_warp * kTopWarps;
  if (r0 >= rows) return;
  const int r1 = min(rows, r0 + rows_per_warp * kTopWarps);
  const LT* base = logits + static_cast<int64_t>(b) * stream_stride;
  auto row_at = [&](int r) { const int t = r / E; return base + static_cast<int64_t>(t) * frame_stride + static_cast<int64_t>(r - t * E) * row_stride; };
  uint4 q[G];
  const LT* row = nullptr;
  int hd = 0, nb = 0;
  auto begin = [&](int r) {                                     // geometry of row r: elements before its first aligned piece, pieces
    row = row_at(r);
    hd = min(V, static_cast<int>((16u - static_cast<uint32_t>(reinterpret_cast<uintptr_t>(row) & 15)) & 15u) / static_cast<int>(sizeof(LT)));
    nb = (V - hd) / EB;
  };
  auto load = [&](int g) {
    const uint4* p = reinterpret_cast<const uint4*>(row + hd) + lane;
#pragma unroll
    for (int u = 0; u < G; ++u) {
      q[u] = make_uint4(RB::kNone, RB::kNone, RB::kNone, RB::kNone);
      if (g + 32 * u + lane < nb) q[u] = __ldg(p + g + 32 * u);
    }
  };
  int r = r0 + warp;
  if (r < r1) { begin(r); load(0); }                            // (the first row is on its way while the table is laid out)
  const TbSlotRec rec = slots[b];
  const bool bound = rec.n_states > 0;
  const GraphPtrs g = graph_of(arena, rec);
  for (int c = threadIdx.x; c < C; c += blockDim.x) rootcw[c] = 0.0f;
  __syncthreads();
  if (bound) {
    const int e = g.arc_begin[1];
    for (int a = g.arc_begin[0] + threadIdx.x; a < e; a += blockDim.x) {
      const int c = g.arc_cls[a];
      if (c >= 0 && c < C) rootcw[c] = __fadd_rn(0.0f, g.arc_w[a]);
    }
  }
  __syncthreads();
  for (int v = threadIdx.x; v < V; v += blockDim.x) {
    const float cb = bound ? __fmul_rn(g.lambda, rootcw[__ldg(cls + v)]) : 0.0f;
#pragma unroll
    for (int h = 0; h < 4; ++h)
      if (v >= h) reinterpret_cast<float*>(tab + h * copy)[v - h] = cb;
  }
  __syncthreads();
#pragma unroll 1
  for (; r < r1; r += kTopWarps) {
    const LT* rowi = row;
    const int hdi = hd, nbi = nb;
    // the boosts of piece bi of this row
    const unsigned char* boosts = tab + (hdi & 3) * copy + 4 * (hdi - (hdi & 3));
    float y[G * EB];
    auto values = [&](int g0) {
#pragma unroll
      for (int u = 0; u < G; ++u) {
        const int bi = min(g0 + 32 * u + lane, max(nbi - 1, 0));
        float x[EB];
        int n = 0;
        RB::each2(q[u], [&](float a, float c) { x[n++] = a; x[n++] = c; });
#pragma unroll
        for (int e = 0; e < EB; e += 4) {
          const float4 cb = *reinterpret_cast<const float4*>(boosts + 4 * (EB * bi + e));
          y[u * EB + e] = __fadd_rn(x[e], cb.x); y[u * EB + e + 1] = __fadd_rn(x[e + 1], cb.y);
          y[u * EB + e + 2] = __fadd_rn(x[e + 2], cb.z); y[u * EB + e + 3] = __fadd_rn(x[e + 3], cb.w);
        }
      }
    };
    // the lane's best and second best value (of those that are numbers)
    float m1 = -INFINITY, m2 = -INFINITY;
    auto best_of = [&]() {
      if (both) {
#pragma unroll
        for (int i = 0; i < G * EB; ++i) { m2 = fmaxf(m2, min_nan(m1, y[i])); m1 = fmaxf(m1, y[i]); }
      } else {
#pragma unroll
        for (int i = 0; i < G * EB; ++i) m1 = fmaxf(m1, y[i]);
      }
    };
    const int sidx = lane < hdi ? lane : nbi * EB + lane;       // this lane's token outside the pieces
    const bool sok = lane < 2 * EB && sidx < V;
    const float* boost0 = reinterpret_cast<const float*>(tab);
    float ys = -INFINITY;
    if (sok) ys = __fadd_rn(LogitLoad<LT>::at(rowi + sidx), boost0[sidx]);
    m1 = fmaxf(m1, ys);
    int g_last = 0;
    values(0);
    best_of();
#pragma unroll 1
    for (int g0 = 32 * G; g0 < nbi; g0 += 32 * G) { load(g0); values(g0); best_of(); g_last = g0; }
    // a threshold that as many as are wanted of the lanes' values reach, and hardly more: halving between the least and the largest
    float thr = -INFINITY;                                      // (fewer values than that: all tokens are looked at)
    {
      auto reach = [&](float t) {
        int n = __popc(__ballot_sync(0xffffffffu, m1 >= t));
        if (both) n += __popc(__ballot_sync(0xffffffffu, m2 >= t));
        return n >= want;
      };
      const float least = both && m2 > -INFINITY ? m2 : m1;
      float hi = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(m1)));
      float lo = order_key_inv(__reduce_min_sync(0xffffffffu, least > -INFINITY ? order_key(least) : 0xFFFFFFFFu));
      if (reach(lo)) {
        thr = lo;
#pragma unroll 1
        for (int i = 0; i < 7; ++i) {
          const float t = 0.5f * lo + 0.5f * hi;
          if (reach(t)) { lo = t; thr = t; } else { hi = t; }
        }
      }
    }
    // candidates as value key << 32 | inverted token, all different
    uint64_t lim = static_cast<uint64_t>(order_key(thr)) << 32;
    bool ahead = false, taken = false;                          // the next row has been asked for; its pieces were overwritten
    int n;
#pragma unroll 1
    for (;;) {
      n = 0;
      const uint32_t lim_key = static_cast<uint32_t>(lim >> 32);
      const float lim_v = lim_key < 0x007FFFFFu ? -INFINITY : order_key_inv(lim_key);
      auto note = [&](bool have, float v, int tok) {
        const uint64_t k = static_cast<uint64_t>(order_key(v)) << 32 | (0xFFFFFFFFu - static_cast<uint32_t>(tok));
        const bool hit = have && k >= lim;
        const unsigned mask = __ballot_sync(0xffffffffu, hit);
        const int at = n + __popc(mask & ((1u << lane) - 1u));
        if (hit && at < kTopCap) cand[at] = k;
        n += __popc(mask);
      };
#pragma unroll 1
      for (int g0 = g_last; g0 >= 0; g0 -= 32 * G) {
        if (g0 != g_last || ahead) {                            // (not at hand any more)
          const LT* keep_row = row; const int keep_hd = hd, keep_nb = nb;
          row = rowi; hd = hdi; nb = nbi;
          load(g0);
          values(g0);
          taken = ahead;
          row = keep_row; hd = keep_hd; nb = keep_nb;
        }
        uint32_t hits = 0u;
#pragma unroll
        for (int u = 0; u < G; ++u)
#pragma unroll
          for (int e = 0; e < EB; ++e) hits |= !(y[u * EB + e] < lim_v) ? 1u << (u * EB + e) : 0u;     // (what is no number, too: its key decides)
#pragma unroll 1
        while (__any_sync(0xffffffffu, hits != 0u) && n < kTopCap) {
          const int bit = max(__ffs(hits) - 1, 0), bi = g0 + 32 * (bit / EB) + lane, tok = hdi + bi * EB + bit % EB;
          const bool have = hits != 0u && bi < nbi;             // (places without a piece pass only a threshold of -inf)
          hits &= hits - 1u;
          note(have, have ? __fadd_rn(LogitLoad<LT>::at(rowi + tok), boost0[tok]) : 0.0f, tok);
        }
      }
      if (n < kTopCap) note(sok, ys, sidx);
      n = min(n, kTopCap);
      __syncwarp();
      if (!ahead) {
        ahead = true;
        if (r + kTopWarps < r1) { begin(r + kTopWarps); load(0); }
      }
      if (n < kTopCap) break;
      // more than can be held: the want-th of those that were bounds the row's from below more tightly (and lim rises, as they
      // are all different and more than are wanted)
      uint64_t next = 0ull;
#pragma unroll 1
      for (int i = lane; i < n; i += 32) {
        const uint64_t k = cand[i];
        int before = 0;
#pragma unroll 4
        for (int j = 0; j < n; ++j) before += cand[j] > k ? 1 : 0;
        if (before == want - 1) next = k;
      }
      const unsigned who = __ballot_sync(0xffffffffu, next != 0ull);
      next = __shfl_sync(0xffffffffu, next, __ffs(who) - 1);
      __syncwarp();
      lim = next;
    }
    if (taken && r + kTopWarps < r1) load(0);
    TbTopEnt* o = out + (static_cast<int64_t>(b) * T * E + r) * want;
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += 64) {
      const int i = i0 + lane, i2 = i + 32;
      const uint64_t ka = i < n ? cand[i] : 0ull, kb = i2 < n ? cand[i2] : 0ull;
      int ma = 0, mb = 0;
      if (n - i0 <= 32) {
#pragma unroll 4
        for (int j = 0; j < n; ++j) ma += cand[j] > ka ? 1 : 0;
      } else {
#pragma unroll 4
        for (int j = 0; j < n; ++j) { const uint64_t c = cand[j]; ma += c > ka ? 1 : 0; mb += c > kb ? 1 : 0; }
      }
      auto put = [&](uint64_t k, int m) {
        const int tok = static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(k));
        TbTopEnt e;
        e.y = order_key_inv(static_cast<uint32_t>(k >> 32));
        if (m == top_m) { e.x = LogitLoad<LT>::at(rowi + V); e.tok_cls = 0u; }
        else { e.x = LogitLoad<LT>::at(rowi + tok); e.tok_cls = static_cast<uint32_t>(tok) | (static_cast<uint32_t>(__ldg(cls + tok)) << 16); }
        o[m] = e;
      };
      if (i < n && ma <= top_m) put(ka, ma);
      if (i2 < n && mb <= top_m) put(kb, mb);
    }
    for (int m = n + lane; m <= top_m; m += 32) {               // fewer tokens in the row
      TbTopEnt e;
      e.y = -INFINITY; e.x = m == top_m ? LogitLoad<LT>::at(rowi + V) : -INFINITY; e.tok_cls = m == top_m ? 0u : 0xFFFFu;
      o[m] = e;
    }
    __syncwarp();                                               // (cand is written again)
  }
}

}  // namespace

int tb_launch_beam_topm(const void* logits, int dtype, int32_t B, int32_t T, int32_t E, int32_t V, int32_t C,
                        int64_t stream_stride, int64_t frame_stride, int64_t row_stride, const int32_t* n_frames,
                        const TbSlotRec* slots, const unsigned char* arena, const int32_t* cls, int32_t top_m,
                        TbTopEnt* out, int32_t n_sm, cudaStream_t stream) {
  const size_t smem = 4 * boost_copy_bytes(V) + kTopWarps * kTopCap * sizeof(uint64_t) + static_cast<size_t>(C) * 4;
  // rows per warp: enough blocks for every SM's three places twice over, before a block's table serves more rows
  const int64_t rows = static_cast<int64_t>(T) * E, all = rows * B;
  int64_t per = all / (static_cast<int64_t>(n_sm > 0 ? n_sm : 1) * 6 * kTopWarps);     // (0: the device did not tell)
  per = per < 1 ? 1 : per > 16 ? 16 : per;
  const int blocks = static_cast<int>((rows + per * kTopWarps - 1) / (per * kTopWarps));
  auto launch = [&](auto* fn, auto* x) -> int {
    if (smem > 16 * 1024 && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess) { cudaGetLastError(); return TB_ERR_INVALID_ARG; }
    return tb_launch_chained(fn, dim3(static_cast<unsigned>(blocks) * B), dim3(kTopWarps * 32), smem, stream, x, T, E, V, C, stream_stride, frame_stride, row_stride, n_frames, slots, arena, cls,
                             top_m, static_cast<int32_t>(per), blocks, out) == TB_OK ? TB_OK : TB_ERR_CUDA;
  };
  const int rc = dtype == TB_BF16 ? launch(k_beam_topm<uint16_t>, static_cast<const uint16_t*>(logits)) : launch(k_beam_topm<float>, static_cast<const float*>(logits));
  if (rc != TB_OK) return rc;
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}
