// Greedy decode in two steps, for what the pipelined kernels (tb_greedy_fast.cu, tb_greedy_seg.cu) do not cover: fp32
// logits, vocabularies beyond 2047 tokens, rows that are not packed; for calls where those are the slower ones (lists of more than
// 48 KB, lists walked along the suffix chain: two_step in tb_batch.cu); and for streaming chunks, where both steps run in the block of a slot.
//
// Offline: k_row_sums reduces every row of the call to a 32-byte summary (one warp per row, all SMs, one pass over HBM),
// then k_decide_rows walks the streams, one block per stream, one warp per stretch of it.  Every stretch but the first
// starts a few frames early in the root state, records the graph state at the frame starts it answers for, and decodes
// past its end until its state is the one recorded there, so that the chain of stretches is the sequential decode (the
// scheme of tb_greedy_seg.cu, inside one block); the block then copies the chain's tokens out and adds its row values one
// by one in visiting order.  The second launch is a programmatic dependent of the first: its blocks set up (root tables,
// the stream's lists in shared memory) while the last rows are reduced.
//
// Streaming (k_chunk_rows): one block per slot; its warps reduce the chunk's rows, sixteen frames at a time, to
// summaries in shared memory, and warp 0 decides them.
#include "tb_rows.cuh"

#include "tb_launch.h"

namespace {

constexpr int kSumThreads = 256;
constexpr int kDecMaxSegs = 16;     // stretches (warps) per stream
constexpr int kDecWarm = 8;         // frames a stretch decodes before the first frame it answers for
constexpr int kDecRing = 32;        // frames of summaries a decider keeps in shared memory
constexpr int kTraceSmem = 8192;    // streams of up to this many frames keep their trace in shared memory
constexpr int kChunkThreads = 256;
constexpr int kPiece = 16;          // frames a slot's block reduces at a time

inline size_t up256(size_t x) { return (x + 255) & ~static_cast<size_t>(255); }

struct RowsParams {
  TbDecodeParams d;
  RowSum* sums;               // [n_streams][frames * S]
  int32_t frames_per_warp;    // step 1: frames whose rows one warp reduces (at most 32)
  int32_t nseg;
  int32_t cache_bytes;        // shared memory for a copy of the stream's lists (0: none fits)
  int32_t* log_tok; int32_t* log_frm; float* log_val; int64_t log_stride;   // [n_streams][log_stride]
  int32_t* trace; int2* aux;  // [n_streams][frames + 1]
  // Room for lists put together by walking, [n_streams][spills][V + 32]: one per stretch, or -- when the lists of all graphs were
  // resolved at the launch -- a single one.  A captured launch is replayed with whatever graphs are bound by then; a stream
  // whose lists are to be walked after all is decoded as one stretch.
  TbRsEnt* spill;
  int32_t spills;
  // where each stretch's part of a stream's logs begins (tabulated: a division in 64 bits takes as long as a frame)
  int64_t seg_at[kDecMaxSegs + 1];
};

// what a stretch's part of the logs has to hold, in frames: from its warmed-up start to the end of the stream
inline int64_t seg_frames(int64_t frames, int nseg, int i) {
  const int64_t f = (frames * (nseg - i) + nseg - 1) / nseg + kDecWarm + 1;
  return f < frames ? f : frames;
}

__device__ __forceinline__ RowCtx row_ctx(const TbDecodeParams& p, const TbSlotRec& rec, const GraphPtrs& g, const RootTab& root) {
  RowCtx h;
  const bool bound = rec.n_states > 0;
  h.rootw = root.w; h.rootarc = root.arc; h.cls = p.cls;
  h.arc_w = g.arc_w; h.arc_dst = g.arc_dst;
  h.lam = bound ? rec.lambda : 0.0f;
  h.beta_min = root.stats[0]; h.beta_max = root.stats[1];
  h.bmag_max = fabsf(h.lam) * ((bound ? rec.d_max : 0.0f) + root.stats[2]);
  h.boosts = root.stats[3] > 0.0f;
  h.norm = p.normalize != 0;
  h.V = p.V; h.n_dur = p.n_dur;
  h.boost_a = 0u;
  return h;
}
template <typename LT>
__device__ __forceinline__ DecideCtx<LT> decide_ctx(const TbDecodeParams& p, const TbSlotRec& rec, const GraphPtrs& g, const RootTab& root,
                                                    const unsigned char* blob, int slot, const LT* base, uint32_t* bitmap, TbRsEnt* walk_buf,
                                                    TbRsEnt* spill) {
  DecideCtx<LT> c;
  c.base = base; c.st = p.st; c.ss = p.ss; c.V = p.V; c.S = p.S; c.n_dur = p.n_dur;
  c.tb = tb_rs_tok_bits(p.V); c.norm = p.normalize != 0;
  c.bound = rec.n_states > 0;
  c.resolved = !c.bound || (rec.n_rsent >= 0 && rec.lists_ready);
  c.n_states = rec.n_states; c.max_depth = rec.max_depth;
  c.lam = c.bound ? rec.lambda : 0.0f; c.R = root.stats[2];
  c.rsrec = reinterpret_cast<const TbRsRec*>(blob + rec.off_rsrec);
  c.rsent = reinterpret_cast<const TbRsEnt*>(p.arena + rec.rsent_at);
  c.strec = reinterpret_cast<const TbStateRec*>(blob + rec.off_strec);
  c.tokent = reinterpret_cast<const TbTokEnt*>(blob + rec.off_tokent);
  c.root = root; c.cls = p.cls; c.arc_w = g.arc_w; c.arc_dst = g.arc_dst;
  c.bitmap = bitmap; c.walk_buf = walk_buf; c.spill = spill; c.status = p.status;
  c.p = &p; c.slot = !c.resolved && rec.n_rsent >= 0 ? slot : -1;
  return c;
}

// ---- step 1 -------------------------------------------------------------------------------------------------------
// Bound by HBM for wide rows (16 KB a row at V = 8192), by instruction issue for narrow ones.  A block reduces a stretch
// of frames of one stream, so that its root tables are built once for them; warp w takes frames w, w + 8, ... of it.
template <typename LT, int G, bool TAB>
__global__ void __launch_bounds__(kSumThreads, G == 4 ? 3 : 2) k_row_sums(const __grid_constant__ RowsParams P) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ float part[3 * kSumThreads / 32];
  // (the second step's blocks read the graphs before their own wait: they may start only once this launch's wait is over)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const TbDecodeParams& p = P.d;
  constexpr int kWarps = kSumThreads / 32;
  const int b = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int end = p.lengths ? p.lengths[b] : p.frames;
  end = max(0, min(end, p.frames));
  const int f0 = blockIdx.x * P.frames_per_warp * kWarps, nf = min(P.frames_per_warp * kWarps, end - f0);
  if (nf <= 0) return;
  const TbSlotRec rec = p.slots[b];
  const GraphPtrs g = graph_of(p.arena, rec);
  const RootTab root = root_tab_at(dyn, p.C);
  root_tab_fill(root, g, rec.n_states > 0, rec.lambda, p.C, part);
  RowCtx h = row_ctx(p, rec, g, root);
  if (TAB) {
    unsigned char* tab = dyn + root_tab_bytes(p.C);
    boost_tab_fill<LT>(tab, root, p.cls, h.lam, p.V);
    h.boost_a = shared_u32(tab);
    __syncthreads();
  }
  if (warp < nf)
    frames_summary<LT, G, TAB>(h, reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.sb, p.st, p.ss, p.S, f0 + warp, kWarps,
                          (nf - warp + kWarps - 1) / kWarps, P.sums + static_cast<int64_t>(b) * p.frames * p.S, -1, lane);
}

// ---- step 2 -------------------------------------------------------------------------------------------------------
struct DecSmem { int root, bitmap, walk, ring, trace, misc, cache, total; };
__host__ __device__ inline DecSmem dec_smem(int V, int C, int S, int frames, int nseg, int cache_bytes, int spills) {
  DecSmem s;
  int o = 0;
  s.root = o; o += static_cast<int>(root_tab_bytes(C));
  s.bitmap = o; o += nseg * (((V + 32) / 32 * 4 + 15) & ~15);
  s.walk = o; o += spills * kWalkBuf * 8;
  s.ring = o; o += nseg * kDecRing * S * 32;
  s.trace = o; o += frames <= kTraceSmem ? ((frames + 1) * 4 + 15) & ~15 : 0;
  s.misc = o; o += kDecMaxSegs * 3 * 32 + 64;
  s.cache = o; o += (cache_bytes + 15) & ~15;
  s.total = o;
  return s;
}

template <typename LT, bool WALK>
__global__ void __launch_bounds__(32 * kDecMaxSegs, 1) k_decide_rows(const __grid_constant__ RowsParams P) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ float part[3 * kDecMaxSegs];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const TbDecodeParams& p = P.d;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthreads = blockDim.x, S = p.S;
  const DecSmem so = dec_smem(p.V, p.C, S, p.frames, P.nseg, P.cache_bytes, P.spills);
  const TbSlotRec rec = p.slots[b];
  const bool bound = rec.n_states > 0;
  const unsigned char* blob = p.arena + rec.blob_off;
  const GraphPtrs g = graph_of(p.arena, rec);
  int end = p.lengths ? p.lengths[b] : p.frames;
  end = max(0, min(end, p.frames));
  // stretches of this stream: nseg pieces of Lf frames (the last one shorter)
  const bool walks = bound && !(rec.n_rsent >= 0 && rec.lists_ready);
  int nseg = walks && P.spills < P.nseg ? 1 : max(1, min(P.nseg, end / kDecWarm));
  const int Lf = max(1, (end + nseg - 1) / nseg);
  nseg = max(1, (end + Lf - 1) / Lf);
  const RootTab root = root_tab_at(dyn + so.root, p.C);
  root_tab_fill(root, g, bound, rec.lambda, p.C, part);
  const int bm_words = (p.V + 32) / 32, bm_stride = (bm_words * 4 + 15) & ~15;
#pragma unroll 1
  for (int i = tid; i < P.nseg * bm_stride / 4; i += nthreads) reinterpret_cast<uint32_t*>(dyn + so.bitmap)[i] = 0u;
  int32_t* trace = p.frames <= kTraceSmem ? reinterpret_cast<int32_t*>(dyn + so.trace) : P.trace + static_cast<int64_t>(b) * (p.frames + 1);
#pragma unroll 1
  for (int i = tid; i <= end; i += nthreads) trace[i] = INT32_MIN;          // (no state: nothing recorded yet)
  const int tail = rec.blob_bytes - rec.off_rsrec;
  const bool cached = bound && !walks && tail <= P.cache_bytes;
  if (cached) {                                                             // (the records, then the entries)
    const uint4* src = reinterpret_cast<const uint4*>(blob + rec.off_rsrec);
    const uint4* ent = reinterpret_cast<const uint4*>(p.arena + rec.rsent_at) - rec.n_states;
    uint4* dst = reinterpret_cast<uint4*>(dyn + so.cache);
    for (int i = tid; i < (tail >> 4); i += nthreads) dst[i] = (i < rec.n_states ? src : ent)[i];
  }
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");                        // the rows' summaries are in place
  // stretch results: {tokens, values, state, frame it stopped at}, {met, failed}
  int4* res = reinterpret_cast<int4*>(dyn + so.misc);
  const int64_t seg_off = P.seg_at[min(warp, kDecMaxSegs - 1)];
  const int64_t log0 = static_cast<int64_t>(b) * P.log_stride;
  if (warp < nseg) {
    DecideCtx<LT> c = decide_ctx<LT>(p, rec, g, root, blob, b, reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.sb,
                                     reinterpret_cast<uint32_t*>(dyn + so.bitmap + warp * bm_stride), reinterpret_cast<TbRsEnt*>(dyn + so.walk) + min(warp, P.spills - 1) * kWalkBuf,
                                     P.spill + (static_cast<int64_t>(b) * P.spills + min(warp, P.spills - 1)) * (p.V + 32));
    if (cached) {
      c.rsrec = reinterpret_cast<const TbRsRec*>(dyn + so.cache);
      c.rsent = reinterpret_cast<const TbRsEnt*>(dyn + so.cache + 16 * rec.n_states);
    }
    DecideOut o;
    o.first = warp * Lf; o.is_last = warp == nseg - 1; o.next = o.is_last ? end : min(end, (warp + 1) * Lf);
    o.tok = P.log_tok + log0 + seg_off; o.frm = P.log_frm + log0 + seg_off; o.dur = nullptr;
    o.vals = P.log_val + log0 + seg_off;
    o.cap = static_cast<int>(P.seg_at[warp + 1] - seg_off);
    o.trace = trace; o.trace_aux = P.aux + static_cast<int64_t>(b) * (p.frames + 1);
    Cursor cu;
    cu.t = max(0, o.first - ((bound && warp > 0) ? kDecWarm : 0)); cu.k = 0; cu.s = bound ? 0 : -1;
    cu.n_out = cu.nv = 0; cu.failed = false; cu.met = -1; cu.listed = false;
    if (warp == 0) o.first = INT32_MAX;                                     // (nobody needs the first stretch's records)
    decide<LT, true, WALK>(c, cu, o, P.sums + static_cast<int64_t>(b) * p.frames * S,
                               shared_u32(dyn + so.ring) + warp * kDecRing * S * 32, kDecRing - 1, 0, end, lane);
    if (lane == 0) {
      res[2 * warp] = make_int4(cu.n_out, cu.nv, cu.s, cu.met >= 0 ? cu.met : cu.t);
      res[2 * warp + 1] = make_int4(cu.met >= 0 ? 1 : 0, cu.failed ? 1 : 0, 0, 0);
    }
  }
  __threadfence_block();
  __syncthreads();
  // ---- the chain of stretches: {stretch, first token, end token, output offset}, {first value, end value, values before it}
  int4* hops = res + 2 * kDecMaxSegs;
  int* vars = reinterpret_cast<int*>(hops + 2 * kDecMaxSegs);
  const int2* aux = P.aux + static_cast<int64_t>(b) * (p.frames + 1);
  if (tid == 0) {
    int seg = 0, ptok = 0, pval = 0, n = 0, n_val = 0, cnt = 0, fin_state = bound ? 0 : -1, fin_t = 0, bad = 0;
#pragma unroll 1
    for (int hop = 0; hop < nseg && !bad && end > 0; ++hop) {
      const int4 ra = res[2 * seg], rb = res[2 * seg + 1];
      if (rb.y || ra.x < ptok || ra.y < pval) { bad = 1; break; }
      hops[2 * cnt] = make_int4(seg, ptok, ra.x, n);
      hops[2 * cnt + 1] = make_int4(pval, ra.y, n_val, 0);
      ++cnt;
      n += ra.x - ptok; n_val += ra.y - pval;
      fin_state = ra.z; fin_t = ra.w;
      if (!rb.x) break;                                   // decoded to the end of the stream
      const int j = min(ra.w / Lf, nseg - 1);             // the owner of frame start ra.w
      if (j <= seg) { bad = 1; break; }
      const int2 a = aux[ra.w];
      seg = j; ptok = a.x; pval = a.y;
      if (hop == nseg - 1) bad = 1;                       // a chain longer than the number of stretches
    }
    if (bad) atomicOr(p.status, TB_STATUS_STEP_LIMIT);
    vars[0] = cnt; vars[1] = n; vars[2] = fin_state; vars[3] = fin_t; vars[4] = n_val;
  }
  __syncthreads();
  const int cnt = vars[0];
  int32_t* o_tok = p.out_tokens + static_cast<int64_t>(b) * p.out_cap;
  int32_t* o_frm = p.out_frames + static_cast<int64_t>(b) * p.out_cap;
  // A warp per link of the chain copies its tokens out.  The score is the sum of the visited rows' values in visiting order:
  // they are brought into shared memory (the rings are free now), all links at once, a window of them at a time, and added
  // one by one by a single thread.
  float* vbuf = reinterpret_cast<float*>(dyn + so.ring);
  const int vcap = P.nseg * kDecRing * S * 8, n_val = vars[4];
  float score = 0.0f;
#pragma unroll 1
  for (int w0 = 0; w0 == 0 || w0 < n_val; w0 += vcap) {
    if (warp < cnt) {
      const int4 ha = hops[2 * warp], hb = hops[2 * warp + 1];
      const int64_t off = log0 + P.seg_at[ha.x];
      const int v0 = max(hb.x, hb.x + w0 - hb.z), v1 = min(hb.y, hb.x + w0 + vcap - hb.z);
#pragma unroll 4
      for (int v = v0 + lane; v < v1; v += 32) vbuf[hb.z + v - hb.x - w0] = P.log_val[off + v];
      if (w0 == 0) {
#pragma unroll 4
        for (int j = ha.y + lane; j < ha.z; j += 32) {
          const int at = ha.w + j - ha.y;
          if (at < p.out_cap) { o_tok[at] = P.log_tok[off + j]; o_frm[at] = P.log_frm[off + j]; }
        }
      }
    }
    __syncthreads();
    if (tid == 0) {
      const int filled = min(n_val - w0, vcap);
      int i = 0;
#pragma unroll 1
      for (; i + 32 <= filled; i += 32) {
        float4 v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = *reinterpret_cast<const float4*>(vbuf + i + 4 * u);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          score = __fadd_rn(score, v[u].x); score = __fadd_rn(score, v[u].y); score = __fadd_rn(score, v[u].z); score = __fadd_rn(score, v[u].w);
        }
      }
#pragma unroll 1
      for (; i < filled; ++i) score = __fadd_rn(score, vbuf[i]);
    }
    if (w0 + vcap < n_val) __syncthreads();
  }
  if (tid == 0) {
    // (a graph of more states than a list entry has room for, bound since the launch was captured; asked here, at the end: up
    // front the question cost k_chunk_rows 50 bytes of spilled registers a thread and 7 %)
    if (rec.n_states > (1 << (32 - tb_rs_tok_bits(p.V)))) atomicOr(p.status, TB_STATUS_BAD_STATE);
    p.out_counts[b] = vars[1]; p.out_scores[b] = score; p.out_states[b] = vars[2];
    if (p.out_cursors) p.out_cursors[b] = vars[3];
  }
}

// ---- streaming chunks -----------------------------------------------------------------------------------------------
struct ChunkSmem { int root, bitmap, walk, sums, vals, total; };
__host__ __device__ inline ChunkSmem chunk_smem(int V, int C, int S, bool walk) {
  ChunkSmem s;
  int o = 0;
  s.root = o; o += static_cast<int>(root_tab_bytes(C));
  s.bitmap = o; o += ((V + 32) / 32 * 4 + 15) & ~15;
  s.walk = o; o += walk ? kWalkBuf * 8 : 0;
  s.sums = o; o += kPiece * S * 32;
  s.vals = o; o += kPiece * S * 4;
  s.total = (o + 15) & ~15;
  return s;
}

// One block per slot.  A slot that is re-bound with this launch first brings its new graph's image from page-locked host
// memory into its arena block (see TbInlineBinds); every other block is on its way already.
template <typename LT>
__global__ void __launch_bounds__(kChunkThreads, 3) k_chunk_rows(const __grid_constant__ TbDecodeParams p,
                                                                 const __grid_constant__ TbInlineBinds ib, TbRsEnt* spill) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ float part[3 * kChunkThreads / 32];
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nthreads = blockDim.x, nwarps = nthreads >> 5, S = p.S;
  // the first rows of the chunk's frames are asked into L2 now: their trip from HBM overlaps the set-up
  {
    const int lines = (p.V * static_cast<int>(sizeof(LT)) + 127) >> 7, nfr = min(p.frames, kPiece);
#pragma unroll 1
    for (int i = tid; i < nfr * lines; i += nthreads) {
      const int f = i / lines;
      const LT* row = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.sb + static_cast<int64_t>(f) * p.st;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const unsigned char*>(row) + min((i - f * lines) * 128, p.V * static_cast<int>(sizeof(LT)))));
    }
  }
  const ChunkSmem so = chunk_smem(p.V, p.C, S, spill != nullptr);
  TbSlotRec rec = p.slots[b];
  bool rebound = false;
  if (ib.n > 0) {
    int hit = -1;
#pragma unroll 1
    for (int i = 0; i < ib.n; ++i) if (ib.slot[i] == b) hit = i;
    if (hit >= 0) {
      const unsigned char* src = ib.src[hit];
      const int32_t bytes = ib.bytes[hit];
      rec = ib.rec[hit];
      rebound = true;
      pull_image<12>(src, ib.arena + rec.blob_off, bytes);
      if (tid == 0) ib.slots[b] = rec;
    }
  }
  const bool bound = rec.n_states > 0;
  const unsigned char* blob = p.arena + rec.blob_off;
  const GraphPtrs g = graph_of(p.arena, rec);
  TbSlotState st = p.sstate[b];
  if (rebound) { st.state = bound ? 0 : -1; st.t = 0; st.k = 0; st.score = 0.0f; st.n_emitted = 0; st.chunk_base = 0; }
  const int t0 = st.chunk_base, valid = p.lengths ? p.lengths[b] : INT32_MAX;
  const int end = min(t0 + p.frames, valid);
  const RootTab root = root_tab_at(dyn + so.root, p.C);
  uint32_t* bitmap = reinterpret_cast<uint32_t*>(dyn + so.bitmap);
#pragma unroll 1
  for (int i = tid; i < (p.V + 32) / 32; i += nthreads) bitmap[i] = 0u;
  root_tab_fill(root, g, bound, rec.lambda, p.C, part);
  const RowCtx h = row_ctx(p, rec, g, root);
  const LT* base = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.sb;
  RowSum* sums = reinterpret_cast<RowSum*>(dyn + so.sums);
  float* vals = reinterpret_cast<float*>(dyn + so.vals);
  int* cursor_t = reinterpret_cast<int*>(part);              // (free again: the frame cursor, from warp 0 to the others)

  DecideCtx<LT> c = decide_ctx<LT>(p, rec, g, root, blob, b, base, bitmap, reinterpret_cast<TbRsEnt*>(dyn + so.walk), spill ? spill + static_cast<int64_t>(b) * (p.V + 32) : nullptr);
  Cursor cu;
  DecideOut o;
  float score = st.score;
  cu.t = st.t; cu.k = st.k; cu.s = bound ? st.state : -1; cu.n_out = cu.nv = 0; cu.failed = false; cu.met = -1; cu.listed = false;
  if (warp == 0) {
    if (bound && (cu.s < 0 || cu.s >= rec.n_states)) { if (lane == 0) atomicOr(p.status, TB_STATUS_BAD_STATE); cu.s = 0; }
    const int64_t at = static_cast<int64_t>(b) * p.out_cap;
    o.tok = p.out_tokens + at; o.frm = p.out_frames + at; o.dur = p.out_durs ? p.out_durs + at : nullptr;
    o.vals = vals; o.cap = p.out_cap; o.trace = nullptr; o.trace_aux = nullptr; o.first = o.next = 0; o.is_last = true;
  }
  int t = cu.t;
#pragma unroll 1
  for (int f0 = t0; f0 < end; f0 += kPiece) {
    const int f1 = min(f0 + kPiece, end), ff = max(t, f0);   // (frames behind the cursor are not looked at)
    if (ff + warp < f1)
      frames_summary<LT, 4, false>(h, base, p.st, p.ss, S, ff - t0 + warp, nwarps, (f1 - ff - warp + nwarps - 1) / nwarps, sums, kPiece - 1, lane);
    __syncthreads();
    if (warp == 0) {
      if (cu.t < f1) {
        cu.nv = 0;
        decide<LT, false, false>(c, cu, o, nullptr, shared_u32(sums), kPiece - 1, t0, f1, lane);
        __syncwarp();
        if (lane == 0) {
#pragma unroll 4
          for (int i = 0; i < cu.nv; ++i) score = __fadd_rn(score, vals[i]);
        }
      }
      if (lane == 0) *cursor_t = cu.t;
    }
    if (f1 < end) {
      __syncthreads();
      t = *cursor_t;
      __syncthreads();                                       // (read by everyone before it is written again)
    }
  }
  if (tid == 0) {
    p.out_counts[b] = cu.n_out;
    p.out_scores[b] = score;
    p.out_states[b] = cu.s;
    if (p.out_cursors) p.out_cursors[b] = cu.t;
    if (c.n_states > (1 << (32 - c.tb))) atomicOr(p.status, TB_STATUS_BAD_STATE);   // (as in k_decide_rows)
    st.state = cu.s; st.t = cu.t; st.k = cu.k; st.score = score; st.n_emitted += cu.n_out;
    st.chunk_base = t0 + p.frames; st.pad0 = 0; st.pad1 = 0;
    p.sstate[b] = st;
  }
}

bool rows_apply(const TbDecodeParams& d, int32_t max_states) {
  if (d.sv != 1 || d.S > kRowsPerFrame || d.V > TB_MAX_VOCAB || d.C > 0xFFFF) return false;
  if (reinterpret_cast<uintptr_t>(d.logits) & (d.dtype == TB_BF16 ? 1 : 3)) return false;
  return max_states <= (1 << (32 - tb_rs_tok_bits(d.V)));
}

struct RowsLayout { size_t sums, log_tok, log_frm, log_val, trace, aux, spill, total; int64_t log_stride; };
int spills_of(int nseg, bool all_resolved) { return all_resolved ? 1 : nseg; }
RowsLayout rows_layout(const TbDecodeParams& d, int nseg, bool all_resolved) {
  RowsLayout l;
  const size_t n = static_cast<size_t>(d.n_streams);
  int64_t fr = 0;
  for (int i = 0; i < nseg; ++i) fr += seg_frames(d.frames, nseg, i);
  l.log_stride = fr * d.S;
  size_t o = 0;
  l.sums = o; o += up256(n * d.frames * d.S * sizeof(RowSum));
  l.log_tok = o; o += up256(n * l.log_stride * 4);
  l.log_frm = o; o += up256(n * l.log_stride * 4);
  l.log_val = o; o += up256(n * l.log_stride * 4);
  l.trace = o; o += d.frames <= kTraceSmem ? 0 : up256(n * (static_cast<size_t>(d.frames) + 1) * 4);
  l.aux = o; o += up256(n * (static_cast<size_t>(d.frames) + 1) * 8);
  l.spill = o; o += up256(n * spills_of(nseg, all_resolved) * (static_cast<size_t>(d.V) + 32) * 8);
  l.total = o;
  return l;
}

}  // namespace

bool tb_rows_plan(const TbDecodeParams& d, int32_t max_cache_bytes, int32_t max_states, int32_t all_resolved, float root_span, int32_t n_sm,
                  int32_t max_smem, TbRowsPlan* plan) {
  if (d.persistent || d.n_dur != 0 || n_sm < 1 || !rows_apply(d, max_states)) return false;
  if (d.n_streams > 65535) return false;                     // (step 1 has the streams in the grid's second dimension)
  int nseg = static_cast<int>(d.frames / 12);
  nseg = nseg < 1 ? 1 : nseg > kDecMaxSegs ? kDecMaxSegs : nseg;
  // lists in shared memory where they fit beside the rest, with every stream's block resident at once if that is possible
  const int per_sm = d.n_streams <= n_sm ? 1 : 2;
  int cache = all_resolved ? max_cache_bytes : 0;
  const int spills = spills_of(nseg, all_resolved != 0);
  int smem = dec_smem(d.V, d.C, d.S, d.frames, nseg, cache, spills).total;
  if (smem > max_smem / per_sm - 2048) { cache = 0; smem = dec_smem(d.V, d.C, d.S, d.frames, nseg, 0, spills).total; }
  if (smem > max_smem - 2048) return false;
  plan->nseg = nseg; plan->cache_bytes = cache; plan->smem = smem; plan->all_resolved = all_resolved; plan->root_span = root_span;
  plan->scratch_bytes = rows_layout(d, nseg, all_resolved != 0).total;
  return true;
}

int tb_launch_rows(const TbDecodeParams& d, const TbRowsPlan& plan, int32_t n_sm, void* scratch, cudaStream_t stream) {
  RowsParams P;
  P.d = d;
  const RowsLayout l = rows_layout(d, plan.nseg, plan.all_resolved != 0);
  unsigned char* sb = static_cast<unsigned char*>(scratch);
  P.sums = reinterpret_cast<RowSum*>(sb + l.sums);
  P.log_tok = reinterpret_cast<int32_t*>(sb + l.log_tok);
  P.log_frm = reinterpret_cast<int32_t*>(sb + l.log_frm);
  P.log_val = reinterpret_cast<float*>(sb + l.log_val);
  P.log_stride = l.log_stride;
  P.seg_at[0] = 0;
  for (int i = 0; i < kDecMaxSegs; ++i) P.seg_at[i + 1] = P.seg_at[i] + (i < plan.nseg ? seg_frames(d.frames, plan.nseg, i) * d.S : 0);
  P.trace = reinterpret_cast<int32_t*>(sb + l.trace);
  P.aux = reinterpret_cast<int2*>(sb + l.aux);
  P.spill = reinterpret_cast<TbRsEnt*>(sb + l.spill);
  P.spills = spills_of(plan.nseg, plan.all_resolved != 0);
  P.nseg = plan.nseg; P.cache_bytes = plan.cache_bytes;
  // frames per block: enough blocks to fill the GPU several times over, at least a frame per warp
  const int64_t all = static_cast<int64_t>(d.frames) * d.n_streams;
  int64_t per = all / (static_cast<int64_t>(n_sm) * 8 * kSumThreads / 32);
  per = per < 1 ? 1 : per > 16 ? 16 : per;
  P.frames_per_warp = static_cast<int32_t>(per);
  // a row of up to 128 blocks of 16 bytes is one group of four per lane, a wider one takes groups of eight
  const bool narrow = d.V * (d.dtype == TB_BF16 ? 2 : 4) <= 128 * 16 + 15;
  // The table of root boosts, where boosts beyond a nat or so make candidates of hundreds of tokens, a block has rows to use it on,
  // and two blocks' tables leave L1 its half of an SM.  64 x 750 rows of three with text lists, boosts of 2 to 3 nats, 125 to 440
  // candidates: 326 us without, 149 with it.  Token lists, V = 1024, whole decodes without and with it, by the boost of a first
  // token: 0.5 144 and 159 us, 1.0 267 and 268, 1.2 346 and 342, 1.6 520 and 497, 3.0 1865 and 1741; V = 256, fp32: 1.0 304 and 304,
  // 1.6 1463 and 1456.  (Between 1.1 and 1.6 nats the line hardly matters.)
  const size_t tab = d.dtype == TB_BF16 ? BoostTab<uint16_t>::bytes(d.V) : BoostTab<float>::bytes(d.V);
  const bool with_tab = plan.root_span > 1.5f && per >= 2 && tab <= 40 * 1024;
  void (*f1)(RowsParams);
  if (d.dtype == TB_BF16)
    f1 = narrow ? (with_tab ? k_row_sums<uint16_t, 4, true> : k_row_sums<uint16_t, 4, false>) : with_tab ? k_row_sums<uint16_t, 8, true> : k_row_sums<uint16_t, 8, false>;
  else
    f1 = narrow ? (with_tab ? k_row_sums<float, 4, true> : k_row_sums<float, 4, false>) : with_tab ? k_row_sums<float, 8, true> : k_row_sums<float, 8, false>;
  void (*f2)(RowsParams) = plan.all_resolved ? (d.dtype == TB_BF16 ? k_decide_rows<uint16_t, false> : k_decide_rows<float, false>)
                                             : d.dtype == TB_BF16 ? k_decide_rows<uint16_t, true> : k_decide_rows<float, true>;
  const size_t smem1 = root_tab_bytes(d.C) + (with_tab ? tab : 0);
  if (smem1 > 24 * 1024 && cudaFuncSetAttribute(f1, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem1)) != cudaSuccess) {
    cudaGetLastError();
    return TB_ERR_CUDA;
  }
  if (cudaFuncSetAttribute(f2, cudaFuncAttributeMaxDynamicSharedMemorySize, plan.smem) != cudaSuccess) { cudaGetLastError(); return TB_ERR_CUDA; }
  if (tb_launch_chained(f1, dim3(static_cast<unsigned>((d.frames + per * kSumThreads / 32 - 1) / (per * kSumThreads / 32)), d.n_streams), dim3(kSumThreads), smem1, stream, P) != TB_OK)
    return TB_ERR_CUDA;
  if (cudaGetLastError() != cudaSuccess) return TB_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(d.n_streams); cfg.blockDim = dim3(32 * plan.nseg); cfg.dynamicSmemBytes = plan.smem; cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, f2, P) == cudaSuccess ? TB_OK : (cudaGetLastError(), TB_ERR_CUDA);
}

int tb_launch_chunk_rows(const TbDecodeParams& d, int32_t max_states, int32_t n_sm, int32_t max_smem, TbRsEnt* spill, cudaStream_t stream,
                         const TbInlineBinds* binds) {
  if (!d.persistent || !rows_apply(d, max_states)) return 1;
  const int smem = chunk_smem(d.V, d.C, d.S, spill != nullptr).total;
  if (smem > max_smem - 2048) return 1;
  TbInlineBinds ib;
  if (binds) ib = *binds; else ib.n = 0;
  if (ib.n < 0 || ib.n > TB_INLINE_BINDS || (ib.n > 0 && (!ib.arena || !ib.slots))) return TB_ERR_INVALID_ARG;
  void (*fn)(TbDecodeParams, TbInlineBinds, TbRsEnt*) = d.dtype == TB_BF16 ? k_chunk_rows<uint16_t> : k_chunk_rows<float>;
  if (smem > 24 * 1024 && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) { cudaGetLastError(); return TB_ERR_CUDA; }
  // eight warps a slot; six when only four such blocks (80 registers a thread) bring all slots onto the GPU at once
  const int threads = d.n_streams <= 3 * n_sm ? kChunkThreads : kChunkThreads * 3 / 4;
  fn<<<d.n_streams, threads, smem, stream>>>(d, ib, spill);
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}
