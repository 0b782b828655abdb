// General decode kernels: one thread block per stream (or per stream's beam), any strides,
// any vocabulary up to TB_MAX_VOCAB, RNNT and TDT, offline and streaming.  Every row is
// evaluated exactly as the arithmetic contract in tb.h states.  These kernels are the
// reference device path; the pipelined greedy kernels cover packed bf16 rows, the two-step and
// chunk kernels (tb_rows.cu) the rest of what has contiguous tokens, and this one what is left:
// other token strides, more than four rows a frame, chunks of a few frames.
#include <cfloat>
#include <type_traits>

#include "tb_device.cuh"
#include "tb_launch.h"

namespace {

constexpr int kThreads = 256;
constexpr int kBeamList = 64;   // boosted tokens per hypothesis kept for the next-state lookup of the beam step

struct ChainSmem {
  int32_t state[TB_CHAIN_MAX];
  float acc[TB_CHAIN_MAX];
  int32_t len;
};

// Shared state of one block's sequential decode.
struct StepSmem {
  ValId red[kThreads / 32 + 1];
  ChainSmem chain;
  int32_t t, k, s, tok, go;
};

// Token view of the current graph state, for graphs that carry resolved lists (see TbRsRec):
// instead of walking the suffix chain into a class-indexed bonus vector, the state's finished list
// is scattered into two token-indexed arrays; a token that is not in the list ("plain") gets
// fl(lambda * fl(D + root arc weight of its class)) and the root arc's target.
struct TokView {
  float* rootcw;      // [C] root arc weight per class (0 if none)
  int32_t* rootdst;   // [C] root arc target per class (0 if none)
  float* tok_lb;      // [V] finished additive term of a listed token
  int32_t* tok_dst;   // [V] target state of a listed token, -1: not listed
  uint16_t* cur_tok;  // tokens of the list now scattered (to undo it)
  int32_t n;
  float D;
};
__host__ __device__ inline size_t tokview_bytes(int V, int C) {
  return static_cast<size_t>(C) * 8 + static_cast<size_t>(V) * 8 + ((static_cast<size_t>(V) * 2 + 8 + 15) & ~size_t(15));
}
// The beam kernels' auxiliary shared memory behind the candidate arrays: class vectors or the token view.
__host__ __device__ inline size_t beam_aux_bytes(int V, int C, int tokview) {
  size_t a = static_cast<size_t>(C) * 8;
  if (tokview && tokview_bytes(V, C) > a) a = tokview_bytes(V, C);
  return (a + 15) & ~size_t(15);
}
__device__ inline void tokview_init(TokView& tv, unsigned char* mem, int V, int C, const GraphPtrs& g) {
  tv.rootcw = reinterpret_cast<float*>(mem);
  tv.rootdst = reinterpret_cast<int32_t*>(mem + 4 * static_cast<size_t>(C));
  tv.tok_lb = reinterpret_cast<float*>(mem + 8 * static_cast<size_t>(C));
  tv.tok_dst = reinterpret_cast<int32_t*>(mem + 8 * static_cast<size_t>(C) + 4 * static_cast<size_t>(V));
  tv.cur_tok = reinterpret_cast<uint16_t*>(mem + 8 * static_cast<size_t>(C) + 8 * static_cast<size_t>(V));
  tv.n = 0; tv.D = 0.0f;
  for (int c = threadIdx.x; c < C; c += blockDim.x) { tv.rootcw[c] = 0.0f; tv.rootdst[c] = 0; }
  for (int v = threadIdx.x; v < V; v += blockDim.x) tv.tok_dst[v] = -1;
  __syncthreads();
  const int e = g.arc_begin[1];
  for (int a = g.arc_begin[0] + threadIdx.x; a < e; a += blockDim.x) {
    const int c = g.arc_cls[a];
    if (c >= 0 && c < C) { tv.rootcw[c] = __fadd_rn(0.0f, g.arc_w[a]); tv.rootdst[c] = g.arc_dst[a]; }
  }
  __syncthreads();
}
// The same tables, already filled by an earlier tokview_init of this block with the same arguments.
__device__ inline void tokview_attach(TokView& tv, unsigned char* mem, int V, int C) {
  tv.rootcw = reinterpret_cast<float*>(mem);
  tv.rootdst = reinterpret_cast<int32_t*>(mem + 4 * static_cast<size_t>(C));
  tv.tok_lb = reinterpret_cast<float*>(mem + 8 * static_cast<size_t>(C));
  tv.tok_dst = reinterpret_cast<int32_t*>(mem + 8 * static_cast<size_t>(C) + 4 * static_cast<size_t>(V));
  tv.cur_tok = reinterpret_cast<uint16_t*>(mem + 8 * static_cast<size_t>(C) + 8 * static_cast<size_t>(V));
  tv.n = 0; tv.D = 0.0f;
}
// Block-wide: replace the scattered list by that of state s (the root's list is empty, D = 0).
__device__ inline void tokview_enter(TokView& tv, const unsigned char* blob, const TbSlotRec& rec, int32_t s, int V,
                                     int32_t* status) {
  for (int i = threadIdx.x; i < tv.n; i += blockDim.x) {
    const int tk = tv.cur_tok[i];
    if (tk < V) tv.tok_dst[tk] = -1;
  }
  __syncthreads();
  if (s < 0 || s >= rec.n_states) { if (threadIdx.x == 0) atomicOr(status, TB_STATUS_BAD_STATE); s = 0; }
  const TbRsRec r = reinterpret_cast<const TbRsRec*>(blob + rec.off_rsrec)[s];
  const TbRsEnt* ent = reinterpret_cast<const TbRsEnt*>(blob + rec.off_rsent) + r.begin;
  const int n = min(r.count, V + 4);
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const TbRsEnt e = ent[i];
    const int tk = static_cast<int>((e.dst_tok & ((1u << TB_RS_TOK_BITS) - 1u)) >> 1);   // padding entries carry token V
    if (tk < V) { tv.tok_lb[tk] = e.lb; tv.tok_dst[tk] = static_cast<int32_t>(e.dst_tok >> TB_RS_TOK_BITS); }
    tv.cur_tok[i] = static_cast<uint16_t>(tk);
  }
  __syncthreads();
  tv.n = n; tv.D = r.D;
}

template <typename LT>
__global__ void __launch_bounds__(kThreads) k_decode_general(TbDecodeParams p, TbInlineBinds ib) {
  extern __shared__ __align__(16) unsigned char dyn[];
  float* bvec = reinterpret_cast<float*>(dyn);
  int32_t* nvec = reinterpret_cast<int32_t*>(dyn + sizeof(float) * p.C);
  __shared__ StepSmem sm;
  __shared__ float fred[kThreads / 32];

  const int b = blockIdx.x;
  TbSlotRec rec = p.slots[b];
  // A bind that travels with this launch (streaming chunks): the block of a re-bound slot brings the new graph's
  // image from page-locked host memory into its arena block itself, then stores the slot's new record; every other
  // block is on its way already.
  bool rebound = false;
  if (ib.n > 0) {
    int hit = -1;
#pragma unroll
    for (int i = 0; i < TB_INLINE_BINDS; ++i)
      if (i < ib.n && ib.slot[i] == b) hit = i;
    if (hit >= 0) {
      const unsigned char* src = nullptr;
      int32_t bytes = 0;
#pragma unroll
      for (int i = 0; i < TB_INLINE_BINDS; ++i)
        if (hit == i) { src = ib.src[i]; bytes = ib.bytes[i]; rec = ib.rec[i]; }
      rebound = true;
      pull_image<8>(src, ib.arena + rec.blob_off, bytes);
      if (threadIdx.x == 0) ib.slots[b] = rec;
    }
  }
  const bool bound = rec.n_states > 0;
  const GraphPtrs g = graph_of(p.arena, rec);
  const unsigned char* blob = p.arena + rec.blob_off;
  // resolved lists: token view instead of a chain walk (a graph bound with this launch has its lists derived behind it)
  const bool use_tv = bound && rec.n_rsent >= 0 && rec.lists_ready && p.tokview;
  TokView tv;
  if (use_tv) tokview_init(tv, dyn, p.V, p.C, g);
  const LT* base = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.sb;
  const int V = p.V;

  // where this call starts and ends for the stream
  int32_t t0 = 0, end, s, t, k, n_total = 0;
  float score;
  if (p.persistent) {
    TbSlotState st = p.sstate[b];
    if (rebound) { st.state = rec.n_states > 0 ? 0 : -1; st.t = 0; st.k = 0; st.score = 0.0f; st.n_emitted = 0; st.chunk_base = 0; }
    t0 = st.chunk_base; s = st.state; t = st.t; k = st.k; score = st.score; n_total = st.n_emitted;
    int32_t valid = p.lengths ? p.lengths[b] : INT32_MAX;
    end = min(t0 + p.frames, valid);
  } else {
    s = bound ? 0 : -1; t = 0; k = 0; score = 0.0f;
    int32_t len = p.lengths ? p.lengths[b] : p.frames;
    end = max(0, min(len, p.frames));
  }
  if (!bound) s = -1;
  int32_t n_out = 0;
  int32_t built_for = -2;  // state the bonus vector currently describes

  const int64_t max_steps = static_cast<int64_t>(p.frames) * p.S;
  for (int64_t it = 0; t < end; ++it) {
    if (it >= max_steps) {  // every step emits or closes a frame, so this cannot happen
      if (threadIdx.x == 0) atomicOr(p.status, TB_STATUS_STEP_LIMIT);
      break;
    }
    if (bound && built_for != s) {
      if (use_tv) tokview_enter(tv, blob, rec, s, V, p.status);
      else build_bonus(g, s, p.C, bvec, nvec, sm.chain.state, sm.chain.acc, &sm.chain.len, p.status);
      built_for = s;
    }
    const LT* row = base + static_cast<int64_t>(t - t0) * p.st + static_cast<int64_t>(k) * p.ss;
    float lse = 0.0f;
    if (p.normalize) {
      // log-softmax fused into the selection: L = m + log(sum_v exp(x_v - m)) over the row's V+1 entries, in
      // float with a fixed order of additions (per thread by index, then lanes, then warps), so that a launch
      // repeats bit for bit; every entry becomes x_v - L before its bonus is added
      float m = -INFINITY;
      for (int v = threadIdx.x; v <= V; v += kThreads) m = fmaxf(m, LogitLoad<LT>::at(row + static_cast<int64_t>(v) * p.sv));
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
      if ((threadIdx.x & 31) == 0) fred[threadIdx.x >> 5] = m;
      __syncthreads();
      m = fred[0];
      for (int w2 = 1; w2 < kThreads / 32; ++w2) m = fmaxf(m, fred[w2]);
      __syncthreads();
      float sum = 0.0f;
      for (int v = threadIdx.x; v <= V; v += kThreads) sum = __fadd_rn(sum, expf(__fsub_rn(LogitLoad<LT>::at(row + static_cast<int64_t>(v) * p.sv), m)));
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) sum = __fadd_rn(sum, __shfl_xor_sync(0xffffffffu, sum, off));
      if ((threadIdx.x & 31) == 0) fred[threadIdx.x >> 5] = sum;
      __syncthreads();
      sum = fred[0];
      for (int w2 = 1; w2 < kThreads / 32; ++w2) sum = __fadd_rn(sum, fred[w2]);
      __syncthreads();
      lse = m == -INFINITY ? 0.0f : __fadd_rn(m, logf(sum));
    }
    ValId best{-INFINITY, INT32_MAX};
    for (int v = threadIdx.x; v <= V; v += kThreads) {
      float x = LogitLoad<LT>::at(row + static_cast<int64_t>(v) * p.sv);
      if (p.normalize) x = __fsub_rn(x, lse);
      float val = x;
      if (bound && v < V) {
        if (use_tv) {
          const float lb = tv.tok_dst[v] >= 0 ? tv.tok_lb[v]
                                              : __fmul_rn(g.lambda, __fadd_rn(tv.D, tv.rootcw[__ldg(p.cls + v)]));
          val = __fadd_rn(x, lb);
        } else {
          val = __fadd_rn(x, __fmul_rn(g.lambda, bvec[__ldg(p.cls + v)]));
        }
      }
      ValId c{val, v};
      if (better(c, best)) best = c;
    }
    best = block_best(best, sm.red);
    // every thread now holds the same (value, token); all of them advance the same cursor
    const int tok = best.i;
    float add = best.v;
    int dur = 0;
    if (p.n_dur > 0) {
      float bd = 0.0f;
      for (int d = 0; d < p.n_dur; ++d) {
        float xd = LogitLoad<LT>::at(row + static_cast<int64_t>(V + 1 + d) * p.sv);
        if (d == 0 || xd > bd) { bd = xd; dur = d; }
      }
      add = __fadd_rn(add, bd);
    }
    score = __fadd_rn(score, add);
    if (tok == V) {
      t += (p.n_dur > 0) ? max(dur, 1) : 1;
      k = 0;
    } else {
      if (threadIdx.x == 0 && n_out < p.out_cap) {
        const int64_t o = static_cast<int64_t>(b) * p.out_cap + n_out;
        p.out_tokens[o] = tok;
        p.out_frames[o] = t;
        if (p.out_durs) p.out_durs[o] = dur;
      }
      ++n_out;
      if (bound) s = use_tv ? (tv.tok_dst[tok] >= 0 ? tv.tok_dst[tok] : tv.rootdst[__ldg(p.cls + tok)]) : nvec[__ldg(p.cls + tok)];
      if (p.n_dur > 0 && dur > 0) { t += dur; k = 0; }
      else { ++k; if (k == p.S) { ++t; k = 0; } }
    }
    __syncthreads();  // nvec / bvec are read above and may be rebuilt next
  }

  if (threadIdx.x == 0) {
    p.out_counts[b] = n_out;
    p.out_scores[b] = score;
    p.out_states[b] = s;
    if (p.out_cursors) p.out_cursors[b] = t;
    if (p.persistent) {
      TbSlotState st;
      st.state = s; st.t = t; st.k = k; st.score = score; st.n_emitted = n_total + n_out;
      st.chunk_base = t0 + p.frames; st.pad0 = 0; st.pad1 = 0;
      p.sstate[b] = st;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// beam step
// ---------------------------------------------------------------------------------------------

struct BeamKey {  // order: value descending, token key ascending, parent ascending
  float v;
  int32_t tkey, par;
};
// One beam expansion of the block's stream (the body of k_beam_step; k_beam_frames calls it once per row).
// threads of a beam block: more warps than the general kernel's hide the latencies of its short dependent phases; 17
// warps take a row of 1025 logits (vocabularies of about a thousand pieces) in two strides instead of three
constexpr int kBeamThreads = 544;
constexpr int kBeamPref = 5;   // elements of a shared row each thread may hold ahead of time (rows up to 5 * kBeamThreads wide)
// xpre / xpre_valid: this thread's elements of the stream's shared row, fetched ahead by the previous step of the same
// launch; next_row: where the next step's shared row starts (null: none), fetched while this step selects.
// What a beam block keeps in shared memory besides its candidate arrays: the stream's hypotheses from step to step,
// and the working set of a step.
constexpr int kHistBins = 128, kSurvivors = 512;   // of a team step: histogram bins, candidates that may be picks
struct BeamShared {
  ChainSmem chain;
  // token-view path: per hypothesis a copy of its state's short list, to find the next state of a pick
  uint16_t hl_tok[TB_MAX_BEAM][kBeamList];
  int32_t hl_dst[TB_MAX_BEAM][kBeamList];
  int32_t hl_n[TB_MAX_BEAM];                                 // -1: list too long, walk the chain instead
  int32_t h_beg[TB_MAX_BEAM], h_cnt[TB_MAX_BEAM];
  float h_D[TB_MAX_BEAM];
  unsigned long long red64[2][kBeamThreads / 32];   // the warps' best keys, two copies used in turn by the selection rounds
  float h_score[TB_MAX_BEAM];
  int32_t h_state[TB_MAX_BEAM];
  uint8_t h_live[TB_MAX_BEAM];
  unsigned long long h_hash[TB_MAX_BEAM];   // identity of the hypothesis' token sequence
  int32_t h_len[TB_MAX_BEAM];
  BeamKey sel[TB_MAX_BEAM];
  float root_wmax;                   // largest |root arc weight| of the stream's graph (filled with the root tables)
  int32_t team_done;                 // steps the team has just taken
  int32_t taken[3];                  // steps of this launch so far, by kind (TbBeamParams::taken)
  // the team's steps (beam_team_run); two copies of what one step still reads while the next one writes
  float w_ub[2][TB_MAX_BEAM];                            // what the K-th pick has to clear on behalf of each hypothesis
  __align__(16) int32_t hist[2][kHistBins];              // candidates by value
  __align__(16) unsigned long long sk[kSurvivors + 64];  // the candidates that may be picks: keys, target states
  int32_t sd[kSurvivors + 1];
  int32_t ord[TB_MAX_BEAM];                              // the K best of them, best first
  int32_t n_surv[2], cmd, done;
  __align__(16) uint32_t hlow[TB_MAX_BEAM];              // low words of the sequences' hashes
  uint4 no_rec;                                          // the empty list (unbound streams)
};

// A token sequence's identity with one more token: a 64-bit mix of the sequence so far and the token.
__device__ __forceinline__ unsigned long long beam_extend(unsigned long long h, int token) {
  h = (h ^ static_cast<unsigned long long>(token + 1)) * 0xff51afd7ed558ccdull;
  h ^= h >> 33;
  return h + 0x9e3779b97f4a7c15ull;
}

template <typename LT>
__device__ __forceinline__ void beam_step_body(const TbBeamParams& p, BeamShared& sh, LT (&xpre)[kBeamPref], bool& xpre_valid,
                                               const LT* next_row) {
  extern __shared__ __align__(16) unsigned char dyn[];
  const int V = p.V, K = p.K, W = V + 1;
  float* cand = reinterpret_cast<float*>(dyn);                         // [K, V+1]
  const int WW = (W + 31) >> 5;
  uint32_t* ovr = reinterpret_cast<uint32_t*>(dyn + ((static_cast<size_t>(K) * W * sizeof(float) + 15) & ~size_t(15)));   // [K, WW] bits: the value in cand is a boosted one
  unsigned char* aux = reinterpret_cast<unsigned char*>(ovr) + ((static_cast<size_t>(K) * WW * sizeof(uint32_t) + 15) & ~size_t(15));
  float* bvec = reinterpret_cast<float*>(aux);                         // [C]   (chain-walk path)
  int32_t* nvec = reinterpret_cast<int32_t*>(bvec + p.C);              // [C]
  ChainSmem& chain = sh.chain;
  auto& hl_tok = sh.hl_tok; auto& hl_dst = sh.hl_dst; auto& hl_n = sh.hl_n;
  auto& h_beg = sh.h_beg; auto& h_cnt = sh.h_cnt; auto& h_D = sh.h_D;
  auto& red64 = sh.red64;
  auto& h_score = sh.h_score; auto& h_state = sh.h_state; auto& h_live = sh.h_live; auto& h_hash = sh.h_hash; auto& h_len = sh.h_len;
  auto& sel = sh.sel;
  float& root_wmax = sh.root_wmax;

  const int b = blockIdx.x;
  const TbSlotRec rec = p.slots[b];
  const bool bound = rec.n_states > 0;
  const GraphPtrs g = graph_of(p.arena, rec);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned char* blob = p.arena + rec.blob_off;
  const bool use_tv = bound && rec.n_rsent >= 0 && p.tokview;
  // rows shared by the hypotheses of a stream (hyp_stride 0) depend on nothing that is loaded below: fetch this
  // thread's elements now, so that their latency overlaps the loads of the slot record, states and lists
  constexpr int kPref = kBeamPref;
  const bool pref = use_tv && p.hyp_stride == 0 && W <= kPref * kBeamThreads;
  if (pref && !xpre_valid) {
    const LT* row0 = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.stream_stride;
#pragma unroll
    for (int j = 0; j < kPref; ++j) {
      const int v = threadIdx.x + j * kBeamThreads;
      if (v < W) xpre[j] = LogitLoad<LT>::raw(row0 + v);
    }
  }
  TokView tv;
  if (use_tv) {
    if (p.tv_ready) tokview_attach(tv, aux, V, p.C);      // a later step of the same launch: the root tables are there
    else {
      tokview_init(tv, aux, V, p.C, g);
      if (warp == 0) {
        float r = 0.0f;
        for (int c = lane; c < p.C; c += 32) r = fmaxf(r, fabsf(tv.rootcw[c]));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) r = fmaxf(r, __shfl_xor_sync(0xffffffffu, r, off));
        if (lane == 0) root_wmax = r;
      }
    }
  } else if (!p.tv_ready && threadIdx.x == 0) {
    root_wmax = 0.0f;
  }

  if (threadIdx.x < K) {
    if (p.tv_ready) {
      // a later step of the same launch: the previous step left its hypotheses in shared memory
      if (p.new_frame) h_live[threadIdx.x] = static_cast<uint8_t>(h_score[threadIdx.x] != -INFINITY);
    } else {
      const int64_t o = static_cast<int64_t>(b) * K + threadIdx.x;
      float sc = p.scores[o];
      h_score[threadIdx.x] = sc;
      h_state[threadIdx.x] = p.states[o];
      h_live[threadIdx.x] = p.new_frame ? static_cast<uint8_t>(sc != -INFINITY) : p.live[o];
      h_hash[threadIdx.x] = p.fresh ? 0ull : p.hash_in[o];
      h_len[threadIdx.x] = p.fresh ? 0 : p.len_in[o];
    }
  }
  __syncthreads();
  if (p.merge) {
    // hypotheses that have emitted the same token sequence are one transcript: the first in selection order (the
    // best) stays, the others become empty places before anything is expanded
    bool dup = false;
    if (threadIdx.x < K && h_score[threadIdx.x] != -INFINITY) {
      const int k = threadIdx.x;
      for (int j = 0; j < k; ++j)
        if (h_score[j] != -INFINITY && h_len[j] == h_len[k] && h_hash[j] == h_hash[k] && h_state[j] == h_state[k]) { dup = true; break; }
    }
    __syncthreads();
    if (dup) { h_score[threadIdx.x] = -INFINITY; h_state[threadIdx.x] = -1; h_live[threadIdx.x] = 0; }
    __syncthreads();
  }
  if (p.prune_delta >= 0.0f) {
    // still at the frame start: whatever scores below the best by more than the threshold becomes an empty place
    bool drop = false;
    if (threadIdx.x < K) {
      float best = -INFINITY;
      for (int j = 0; j < K; ++j) best = fmaxf(best, h_score[j]);
      const float sc = h_score[threadIdx.x];
      drop = sc != -INFINITY && sc < __fsub_rn(best, p.prune_delta);
    }
    __syncthreads();
    if (drop) { h_score[threadIdx.x] = -INFINITY; h_state[threadIdx.x] = -1; h_live[threadIdx.x] = 0; }
    __syncthreads();
  }

  auto make_key = [](float v, int tkey, int k) -> unsigned long long {
    const uint32_t lo = 0xFFFFFFFFu - (static_cast<uint32_t>(tkey) * 32u + static_cast<uint32_t>(k));
    return (static_cast<unsigned long long>(order_key(v)) << 32) | lo;
  };
  // this thread's two best candidates, collected by the sweep below
  unsigned long long m1 = 0ull, m2 = 0ull;
  auto offer = [&](unsigned long long kk) { if (kk > m1) { m2 = m1; m1 = kk; } else if (kk > m2) m2 = kk; };
  // all candidate values of the live hypotheses
  if (use_tv) {
    // every hypothesis at once: its state's record, then all plain values, then the listed tokens on top
    if (threadIdx.x < K) {
      const int k = threadIdx.x;
      int32_t st = h_state[k];
      if (st < 0 || st >= rec.n_states) { if (h_score[k] != -INFINITY && h_live[k]) atomicOr(p.status, TB_STATUS_BAD_STATE); st = 0; }
      const TbRsRec r = reinterpret_cast<const TbRsRec*>(blob + rec.off_rsrec)[st];
      h_beg[k] = r.begin; h_cnt[k] = r.count; h_D[k] = r.D;
      hl_n[k] = r.count <= kBeamList ? r.count : -1;
    }
    for (int i = threadIdx.x; i < K * WW; i += kBeamThreads) ovr[i] = 0u;
    __syncthreads();
    const LT* base = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.stream_stride;
    // the boosted tokens of every hypothesis first: their values go to cand and are marked, so that the sweep over
    // all candidates below leaves them alone -- and sees every candidate's final value, which lets each thread
    // collect its best keys on the way instead of scanning cand again afterwards
    {
      const TbRsEnt* ent = reinterpret_cast<const TbRsEnt*>(blob + rec.off_rsent);
      for (int k = 0; k < K; ++k) {
        if (h_score[k] == -INFINITY || !h_live[k]) continue;
        for (int i = threadIdx.x; i < h_cnt[k]; i += kBeamThreads) {
          const TbRsEnt e = ent[h_beg[k] + i];
          const int tk = static_cast<int>((e.dst_tok & ((1u << TB_RS_TOK_BITS) - 1u)) >> 1);   // padding entries carry token V
          if (i < kBeamList) { hl_tok[k][i] = static_cast<uint16_t>(tk); hl_dst[k][i] = static_cast<int32_t>(e.dst_tok >> TB_RS_TOK_BITS); }
          if (tk < V) {
            const float x = LogitLoad<LT>::at(base + static_cast<int64_t>(k) * p.hyp_stride + tk);
            cand[static_cast<size_t>(k) * W + tk] = __fadd_rn(h_score[k], __fadd_rn(x, e.lb));
            atomicOr(&ovr[k * WW + (tk >> 5)], 1u << (tk & 31));
          }
        }
      }
    }
    __syncthreads();
    if (pref) {
      // the row sits in registers: every index below is a compile-time constant
#pragma unroll
      for (int j = 0; j < kPref; ++j) {
        const int v = threadIdx.x + j * kBeamThreads;
        if (v < W) {
          const float plain_w = v < V ? tv.rootcw[__ldg(p.cls + v)] : 0.0f;
          const float x = LogitLoad<LT>::widen(xpre[j]);
          for (int k = 0; k < K; ++k) {
            if (h_score[k] == -INFINITY || !h_live[k]) continue;
            float c;
            if ((ovr[k * WW + (v >> 5)] >> (v & 31)) & 1u) {
              c = cand[static_cast<size_t>(k) * W + v];
            } else {
              const float val = v < V ? __fadd_rn(x, __fmul_rn(g.lambda, __fadd_rn(h_D[k], plain_w))) : x;
              c = __fadd_rn(h_score[k], val);
              cand[static_cast<size_t>(k) * W + v] = c;
            }
            offer(make_key(c, v, k));
          }
        }
      }
    } else {
      for (int v = threadIdx.x; v < W; v += kBeamThreads) {
        const float plain_w = v < V ? tv.rootcw[__ldg(p.cls + v)] : 0.0f;
        for (int k = 0; k < K; ++k) {
          if (h_score[k] == -INFINITY || !h_live[k]) continue;
          float c;
          if ((ovr[k * WW + (v >> 5)] >> (v & 31)) & 1u) {
            c = cand[static_cast<size_t>(k) * W + v];
          } else {
            const float x = LogitLoad<LT>::at(base + static_cast<int64_t>(k) * p.hyp_stride + v);
            const float val = v < V ? __fadd_rn(x, __fmul_rn(g.lambda, __fadd_rn(h_D[k], plain_w))) : x;
            c = __fadd_rn(h_score[k], val);
            cand[static_cast<size_t>(k) * W + v] = c;
          }
          offer(make_key(c, v, k));
        }
      }
    }
    __syncthreads();
  } else {
    for (int k = 0; k < K; ++k) {
      if (h_score[k] == -INFINITY || !h_live[k]) continue;  // uniform across the block
      if (bound) build_bonus(g, h_state[k], p.C, bvec, nvec, chain.state, chain.acc, &chain.len, p.status);
      const LT* row = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.stream_stride +
                      static_cast<int64_t>(k) * p.hyp_stride;
      const float sc = h_score[k];
      for (int v = threadIdx.x; v < W; v += kBeamThreads) {
        float x = LogitLoad<LT>::at(row + v);
        float val = (bound && v < V) ? __fadd_rn(x, __fmul_rn(g.lambda, bvec[__ldg(p.cls + v)])) : x;
        const float c = __fadd_rn(sc, val);
        cand[static_cast<size_t>(k) * W + v] = c;
        offer(make_key(c, v, k));
      }
      __syncthreads();
    }
  }
  // a frozen hypothesis is carried as one candidate (thread k offers it)
  if (threadIdx.x < K && h_score[threadIdx.x] != -INFINITY && !h_live[threadIdx.x]) offer(make_key(h_score[threadIdx.x], V + 1, threadIdx.x));

  // K rounds of selection.  A candidate's place in the order (value descending, token key ascending,
  // parent ascending) is one 64-bit key: the order-preserving image of the value above the inverted
  // (token key, parent) pair; keys are distinct, 0 means "none".  Every thread keeps the two best keys among its own
  // candidates -- tokens v = tid, tid + kBeamThreads, ... of every live hypothesis, plus (thread k) the carried candidate of a
  // frozen hypothesis k -- that have not been picked yet.
  // the row of the next step is requested now: its trip from HBM overlaps the selection rounds
  xpre_valid = false;
  if (pref && next_row) {
#pragma unroll
    for (int j = 0; j < kPref; ++j) {
      const int v = threadIdx.x + j * kBeamThreads;
      if (v < W) xpre[j] = LogitLoad<LT>::raw(next_row + v);
    }
    xpre_valid = true;
  }
  unsigned long long mine = m1, spare = m2;
  bool have_spare = true;
  // The largest of the lanes' keys.
  auto warp_best = [](unsigned long long k) -> unsigned long long {
    const uint32_t hi = static_cast<uint32_t>(k >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? static_cast<uint32_t>(k) : 0u);
    return (static_cast<unsigned long long>(mh) << 32) | ml;
  };
  // When a thread's two are used up, its warp looks for the next two, a hypothesis a lane: all others wait for it.  (By the thread alone, hypothesis after
  // hypothesis, this was most of a step: 8 streams of 120 steps, V = 1024, K = 4 932 us, K = 12 3100, K = 32
  // 14 020; so 877, 2064 and 5010.)
  static_assert(TB_MAX_BEAM <= 32, "a lane each");
  auto look_again = [&](unsigned long long limit, int thread, unsigned long long& first, unsigned long long& second) {
    unsigned long long m = 0ull, n = 0ull;
    if (lane < K && h_score[lane] != -INFINITY) {
      if (!h_live[lane]) {
        if (thread == lane) { const unsigned long long kk = make_key(h_score[lane], V + 1, lane); m = kk < limit ? kk : 0ull; }
      } else {
        const float* ck = cand + static_cast<size_t>(lane) * W;
        for (int v = thread; v < W; v += kBeamThreads) {
          const unsigned long long kk = make_key(ck[v], v, lane);
          if (kk < limit) { if (kk > m) { n = m; m = kk; } else if (kk > n) n = kk; }
        }
      }
    }
    first = warp_best(m);
    second = warp_best(m == first ? n : m);
  };
  for (int r = 0; r < K; ++r) {
    const unsigned long long wb = warp_best(mine);
    if (lane == 0) red64[r & 1][warp] = wb;
    __syncthreads();                     // (one barrier per round: the next round writes the other copy)
    unsigned long long best = red64[r & 1][0];
#pragma unroll
    for (int w2 = 1; w2 < kBeamThreads / 32; ++w2) { const unsigned long long o = red64[r & 1][w2]; if (o > best) best = o; }
    if (threadIdx.x == 0) {
      BeamKey c{-INFINITY, INT32_MAX, INT32_MAX};
      if (best != 0ull) {
        const uint32_t lo = 0xFFFFFFFFu - static_cast<uint32_t>(best & 0xFFFFFFFFull);
        c.tkey = static_cast<int32_t>(lo >> 5); c.par = static_cast<int32_t>(lo & 31u);
        c.v = c.tkey == V + 1 ? h_score[c.par] : cand[static_cast<size_t>(c.par) * W + c.tkey];
      }
      sel[r] = c;
    }
    const unsigned own = __ballot_sync(0xffffffffu, best != 0ull && mine == best);
    if (own != 0u) {                                             // one of this warp's threads owned the pick: its next best
      const int src = __ffs(own) - 1;
      if (__shfl_sync(0xffffffffu, have_spare ? 1 : 0, src)) {
        if (lane == src) { mine = spare; have_spare = false; }
      } else {
        unsigned long long m, n;
        look_again(best, 32 * warp + src, m, n);
        if (lane == src) { mine = m; spare = n; have_spare = true; }
      }
    }
  }
  __syncthreads();

  // new hypotheses, the hypothesis tree
  int32_t parent = -1, token = -1, state = -1;
  uint8_t lv = 0;
  float sc = -INFINITY;
  unsigned long long nh = 0ull;
  int32_t nl = 0;
  if (threadIdx.x < K) {
    const int r = threadIdx.x;
    const BeamKey c = sel[r];
    const int64_t o = static_cast<int64_t>(b) * K + r;
    if (c.par != INT32_MAX) {
      parent = c.par; sc = c.v;
      token = (c.tkey == V + 1) ? -1 : c.tkey;
      state = h_state[parent];
      if (token >= 0 && token != V) {
        if (use_tv && hl_n[parent] >= 0) {
          int nx = tv.rootdst[__ldg(p.cls + token)];          // a pick that the parent's list does not hold is a plain token
          for (int i = 0; i < hl_n[parent]; ++i)
            if (hl_tok[parent][i] == token) { nx = hl_dst[parent][i]; break; }
          state = nx;
        } else if (bound) {
          state = walk_next(g, state, __ldg(p.cls + token), p.status);
        }
        lv = h_live[parent];
      }
    }
    p.scores[o] = sc; p.states[o] = state; p.live[o] = lv;
    p.out_parent[o] = parent; p.out_token[o] = token;
    {
      if (parent >= 0) {
        nh = h_hash[parent]; nl = h_len[parent];
        if (token >= 0 && token != V) { nh = beam_extend(nh, token); ++nl; }
      }
      p.hash_out[o] = nh; p.len_out[o] = nl;
    }
    if (p.tree) {
      const int64_t at = p.tree_cap > 0 ? static_cast<int64_t>(b) * p.tree_cap + (p.step % p.tree_cap)
                                        : static_cast<int64_t>(p.step) * p.B + b;
      p.tree[at * K + r] = make_int2(parent, token);
    }
  }
  // ... and in shared memory, for the next step of a launch that runs several (read by every thread above: wait)
  __syncthreads();
  if (threadIdx.x < K) {
    h_score[threadIdx.x] = sc; h_state[threadIdx.x] = state; h_live[threadIdx.x] = lv;
    h_hash[threadIdx.x] = nh; h_len[threadIdx.x] = nl;
  }
}

template <typename LT>
__global__ void __launch_bounds__(kBeamThreads) k_beam_step(TbBeamParams p) {
  LT xpre[kBeamPref] = {};
  bool xpre_valid = false;
  __shared__ BeamShared sh;
  beam_step_body<LT>(p, sh, xpre, xpre_valid, static_cast<const LT*>(nullptr));
}


// ---- steps taken by a team of warps ---------------------------------------------------------------------------------
// With the rows reduced ahead of the steps (k_beam_topm) a hypothesis' candidates are the tokens its graph state lists
// (exact values from their entries), its blank, and the first tokens of the reduced row that the state does not list: a
// few dozen instead of vocab + 1.  Every token outside the reduced row has y <= y_next, hence a value of at most
// score + y_next + lambda * D plus roundings; a step is valid when its K-th pick clears that bound for every hypothesis
// by a margin that dominates the roundings (2^-18 of the operands' scale).
//
// beam_team_run lets min(K, 16) worker warps (at least four) and a keeper take such steps one after the other; worker w
// works for hypotheses w and w + 16.  Per step
//   1. every listed token, the first eight of the reduced row per hypothesis and the blanks go into a histogram of values
//      (128 bins of 1/8 below a reference above the best hypothesis);
//   2. every worker finds the bin in which the K-th best of these lies -- a lower bound on the K-th pick -- and notes its
//      candidates in that bin or above it (over the whole beam K and a few more) with their target states;
//   3. these are ranked by counting the keys above each (few: by every warp for itself; many: shared out);
//   4. every warp now knows the K picks and which of them are its hypotheses, asks for their lists and goes on with the
//      next step, while the keeper checks the bound, writes the tree and fetches rows; its verdict is read at the next
//      barrier.
// A step is a chain of short phases, so what counts is the number of dependent instructions on it and its trips to memory:
// two barriers (three with many candidates), rows and reduced rows by asynchronous copies ahead of time, values kept in
// registers from 1 to 2, few branches, nothing on the way that divides.  (Guessing the bound from the steps before instead
// of the histogram needed 1.6 to 2.3 passes per step and was slower.)
// A step the team cannot take (the bound not cleared, too many candidates in the bin) is left untouched: the run ends
// before it and the whole block does that step with beam_step_body.  Same arithmetic and order of candidates, hence the
// same results bit for bit.
constexpr int kTeamRecCache = 48 << 10;   // shared memory for a copy of the stream's list records (graphs of up to 3072 states)
constexpr float kHistAbove = 6.0f, kHistPerUnit = 8.0f;   // the reference's distance above score + best plain value; bins per unit
constexpr int kTeamRows = 3;              // rows (and reduced rows) in shared memory
// Narrow beams take their steps with one warp (tb_beam_solo.cuh); what that cannot take goes to the team.
constexpr int kSoloBeam = 8;              // hypotheses at most
constexpr int kSoloRows = 4;              // rows brought at a time (two such groups in shared memory)
constexpr int kSoloPlain = 8;             // tokens of a reduced row that are looked at (merging and pruning, with twelve K = 5 1360 us a call, 1307 with eight, K = 8 1335 and 1296)
// Wider ones by a crew of warps, four hypotheses each (tb_beam_crew.cuh); what that cannot take goes to the team as well.
constexpr int kCrewBeam = 32, kCrewWarps = kCrewBeam / 4;
constexpr int kCrewRows = 2;              // rows brought at a time (two such groups in shared memory)
constexpr int kCrewPlain = 16;            // tokens of a reduced row that are looked at
constexpr int kCrewVocab = 16;            // rows of fewer tokens are left to the team (see beam_team_setup)
constexpr int kWholeRows = 4;             // (in the place of a width class) neither: steps by the whole block only

__host__ __device__ inline int team_warps(int K) { return K > 16 ? 16 : K < 4 ? 4 : K; }
__device__ __forceinline__ unsigned long long beam_key(float v, int tkey, int k) {
  const uint32_t lo = 0xFFFFFFFFu - (static_cast<uint32_t>(tkey) * 32u + static_cast<uint32_t>(k));
  return (static_cast<unsigned long long>(order_key(v)) << 32) | lo;
}
__device__ __forceinline__ float beam_key_value(unsigned long long key) {
  return order_key_inv(static_cast<uint32_t>(key >> 32));
}
template <typename LT> __device__ __forceinline__ float beam_smem_logit(const unsigned char* row, int idx);
template <> __device__ __forceinline__ float beam_smem_logit<uint16_t>(const unsigned char* row, int idx) {
  return __uint_as_float(static_cast<uint32_t>(*reinterpret_cast<const uint16_t*>(row + 2 * idx)) << 16);
}
template <> __device__ __forceinline__ float beam_smem_logit<float>(const unsigned char* row, int idx) {
  return *reinterpret_cast<const float*>(row + 4 * idx);
}
__device__ __forceinline__ void beam_cp_async16(unsigned char* dst_smem, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(dst_smem))), "l"(src) : "memory");
}
// Starts the copy of one row (its 16-byte aligned superset) into buf, n threads sharing the pieces; a 16-byte piece that
// is not wholly inside the tensor [lo, hi) is assembled from the elements that are.
template <typename LT>
__device__ __forceinline__ void beam_fetch_row(unsigned char* buf, const LT* row, int W, const unsigned char* lo,
                                               const unsigned char* hi, int tid, int n) {
  const unsigned char* rp = reinterpret_cast<const unsigned char*>(row);
  const int off = static_cast<int>(reinterpret_cast<uintptr_t>(rp) & 15);
  const unsigned char* a0 = rp - off;
  const int nchunks = (off + W * static_cast<int>(sizeof(LT)) + 15) >> 4;
#pragma unroll 1
  for (int c = tid; c < nchunks; c += n) {
    const unsigned char* ac = a0 + 16 * c;
    if (ac >= lo && ac + 16 <= hi) {
      beam_cp_async16(buf + 16 * c, ac);
    } else {
#pragma unroll 1
      for (int e = 0; e < 16; e += static_cast<int>(sizeof(LT)))
        if (ac + e >= lo && ac + e + sizeof(LT) <= hi) *reinterpret_cast<LT*>(buf + 16 * c + e) = *reinterpret_cast<const LT*>(ac + e);
    }
  }
}
// Shared memory of the team behind the block's other arrays: row buffers, reduced rows, the copy of the list records.
struct TeamSmem { int row, row_stride, top, top_stride, recs, total; };
__host__ __device__ inline TeamSmem team_smem(int rows, int V, int elem, int top_m, int rec_bytes) {
  TeamSmem t;
  t.row_stride = (((V + 1) * elem + 16 + 15) & ~15) + 16;
  t.row = 0;
  t.top_stride = ((top_m + 1) * 12 + 15) & ~15;
  t.top = rows * t.row_stride;
  t.recs = t.top + rows * t.top_stride;
  t.total = t.recs + rec_bytes;
  return t;
}
__device__ __forceinline__ unsigned char* team_base(const TbBeamParams& p, unsigned char* dyn) {
  const int W = p.V + 1, WW = (W + 31) >> 5;
  unsigned char* ovr = dyn + ((static_cast<size_t>(p.K) * W * sizeof(float) + 15) & ~size_t(15));
  return ovr + ((static_cast<size_t>(p.K) * WW * sizeof(uint32_t) + 15) & ~size_t(15)) + beam_aux_bytes(p.V, p.C, p.tokview);
}
// Shared-memory atomics under a predicate, without a branch.
__device__ __forceinline__ uint32_t beam_smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void shared_or(uint32_t* p, uint32_t v, bool yes) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q red.shared.or.b32 [%0], %1; }" ::"r"(beam_smem_addr(p)), "r"(v), "r"(yes ? 1u : 0u) : "memory");
}
__device__ __forceinline__ void shared_add(int32_t* p, int v, bool yes) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %2, 0; @q red.shared.add.u32 [%0], %1; }" ::"r"(beam_smem_addr(p)), "r"(v), "r"(yes ? 1u : 0u) : "memory");
}
__device__ __forceinline__ void shared_put(unsigned long long* pk, unsigned long long key, int32_t* pd, int32_t d, bool yes) {
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %4, 0; @q st.shared.u64 [%0], %1; @q st.shared.u32 [%2], %3; }" ::"r"(beam_smem_addr(pk)), "l"(key),
               "r"(beam_smem_addr(pd)), "r"(d), "r"(yes ? 1u : 0u) : "memory");
}
__device__ __forceinline__ int shared_fetch_add(int32_t* p, int v, bool yes) {
  int r = 0;
  asm volatile("{ .reg .pred q; setp.ne.u32 q, %3, 0; @q atom.shared.add.u32 %0, [%1], %2; }" : "+r"(r) : "r"(beam_smem_addr(p)), "r"(v), "r"(yes ? 1u : 0u) : "memory");
  return r;
}
__device__ __forceinline__ void beam_team_barrier(int n_threads) { asm volatile("bar.sync 1, %0;" ::"r"(n_threads) : "memory"); }

// Whether the team's steps apply to this launch and this block's stream.
__device__ __forceinline__ bool beam_team_applies(const TbBeamParams& p) {
  if (p.top_base == nullptr || p.tensor_lo == nullptr) return false;
  const TbSlotRec& rec = p.slots[blockIdx.x];
  return rec.n_states <= 0 || (rec.n_rsent >= 0 && p.tokview);
}
// Block-wide, once per launch: the stream's hypotheses and root tables into shared memory, and its list records if they
// fit (returns whether they do).
__device__ inline bool beam_begin(const TbBeamParams& p, BeamShared& sh, unsigned char* dyn, const unsigned long long* hash_in,
                                  const int32_t* len_in, bool team, const TeamSmem& tm) {
  const int tid = threadIdx.x, lane = tid & 31, K = p.K, b = blockIdx.x;
  const TbSlotRec& rec = p.slots[b];
  const bool bound = rec.n_states > 0, use_tv = bound && rec.n_rsent >= 0 && p.tokview;
  const int W = p.V + 1, WW = (W + 31) >> 5;
  unsigned char* aux = dyn + ((static_cast<size_t>(K) * W * sizeof(float) + 15) & ~size_t(15)) + ((static_cast<size_t>(K) * WW * sizeof(uint32_t) + 15) & ~size_t(15));
  float* rootcw = reinterpret_cast<float*>(aux);               // (see tokview_attach)
  int32_t* rootdst = reinterpret_cast<int32_t*>(aux + 4 * static_cast<size_t>(p.C));
  const bool cached = use_tv && team && static_cast<int64_t>(rec.n_states) * 16 <= p.rec_cache_bytes;
  if (cached) {
    const unsigned char* src = p.arena + rec.blob_off + rec.off_rsrec;
    unsigned char* dst = team_base(p, dyn) + tm.recs;
    for (int i = tid; i < rec.n_states; i += blockDim.x) beam_cp_async16(dst + 16 * i, src + 16 * i);
  }
  if (tid < K) {
    const int64_t o = static_cast<int64_t>(b) * K + tid;
    sh.h_score[tid] = p.scores[o]; sh.h_state[tid] = p.states[o]; sh.h_live[tid] = p.live[o];
    sh.h_hash[tid] = p.fresh ? 0ull : hash_in[o];
    sh.h_len[tid] = p.fresh ? 0 : len_in[o];
  }
  if (tid == 0) { sh.root_wmax = 0.0f; sh.no_rec = make_uint4(0u, 0u, 0u, 0u); sh.taken[0] = sh.taken[1] = sh.taken[2] = 0; }
  if (use_tv) {
    const GraphPtrs g = graph_of(p.arena, rec);
    const int a0 = g.arc_begin[0], a1 = g.arc_begin[1];
    for (int c = tid; c < p.C; c += blockDim.x) { rootcw[c] = 0.0f; rootdst[c] = 0; }
    __syncthreads();
    uint32_t r = 0u;                                           // (|w| >= 0: ordered like its bits)
    for (int a = a0 + tid; a < a1; a += blockDim.x) {
      const int c = g.arc_cls[a];
      const float w = __fadd_rn(0.0f, g.arc_w[a]);
      if (c >= 0 && c < p.C) { rootcw[c] = w; rootdst[c] = g.arc_dst[a]; r = max(r, __float_as_uint(fabsf(w))); }
    }
    r = __reduce_max_sync(0xffffffffu, r);
    if (lane == 0 && r != 0u) atomicMax(reinterpret_cast<unsigned int*>(&sh.root_wmax), r);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  return cached;
}

// Takes the steps sidx, sidx + 1, ... of the block's stream as long as it can; returns how many it took.  Called by the
// team's warps; the hypotheses are read from and left in sh.h_*.  H: hypotheses per worker.  hashA / hashB, lenA / lenB: the two halves of the
// sequence records; step s writes half ((par0 + s) & 1 ? A : B), which only matters for the last one.
template <typename LT, int H>
__device__ __forceinline__ int beam_team_run(const TbBeamParams& p, BeamShared& sh, unsigned char* dyn, int32_t sidx, const int32_t n_steps,
                                             const int32_t E, const int64_t frame_stride, const int64_t row_stride,
                                             const int32_t rows_per_stream, const int32_t step_base, unsigned long long* hashA,
                                             unsigned long long* hashB, int32_t* lenA, int32_t* lenB, const int32_t par0,
                                             const bool recs_cached, const TeamSmem& tm) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x, K = p.K, V = p.V, W = V + 1, M = p.top_m, WW = (W + 31) >> 5;
  const int nw = team_warps(K), team = 32 * nw + 32;
  const bool keeper = warp == nw;                              // the warp that keeps the books
  const TbSlotRec& rec = p.slots[b];
  const int n_states = rec.n_states;
  const bool bound = n_states > 0;
  const float lam = bound ? rec.lambda : 0.0f;
  const unsigned char* blob = p.arena + rec.blob_off;
  uint32_t* ovr = reinterpret_cast<uint32_t*>(dyn + ((static_cast<size_t>(K) * W * sizeof(float) + 15) & ~size_t(15)));
  unsigned char* aux = reinterpret_cast<unsigned char*>(ovr) + ((static_cast<size_t>(K) * WW * sizeof(uint32_t) + 15) & ~size_t(15));
  const float* rootcw = reinterpret_cast<const float*>(aux);             // (see tokview_attach)
  const int32_t* rootdst = reinterpret_cast<const int32_t*>(aux + 4 * static_cast<size_t>(p.C));
  unsigned char* tb_ = team_base(p, dyn);
  const uint4* rsrec = !bound ? reinterpret_cast<const uint4*>(&sh.no_rec) : recs_cached ? reinterpret_cast<const uint4*>(tb_ + tm.recs) : reinterpret_cast<const uint4*>(blob + rec.off_rsrec);
  const uint2* ent = reinterpret_cast<const uint2*>(blob + rec.off_rsent);
  constexpr uint32_t kTok = (1u << TB_RS_TOK_BITS) - 1u;
  const float root_wmax = sh.root_wmax;
  // The rows: fr_* is the row that is fetched next (its frame and row in the frame, its buffer), off0 and off1
  // are the byte offsets of the current and the next row within their first 16-byte pieces, buf the current row's buffer.
  int e_cur = sidx % E, e_f = e_cur, buf = 0, buf_f = 0, s_f = sidx;
  const LT* row_f = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.stream_stride +
                    static_cast<int64_t>(sidx / E) * frame_stride + static_cast<int64_t>(e_cur) * row_stride;
  const unsigned char* top_f = reinterpret_cast<const unsigned char*>(p.top_base + (static_cast<int64_t>(b) * rows_per_stream + sidx) * (M + 1));
  const int64_t to_frame = frame_stride - static_cast<int64_t>(E - 1) * row_stride;
  int off0 = 0, off1 = 0;
  auto fetch = [&]() {                                         // one row and its reduced row, by the keeper: one group of copies
    off0 = off1;
    off1 = static_cast<int>(reinterpret_cast<uintptr_t>(row_f) & 15);
    if (keeper && s_f < n_steps) {
      beam_fetch_row<LT>(tb_ + tm.row + buf_f * tm.row_stride, row_f, W, p.tensor_lo, p.tensor_hi, lane, 32);
      unsigned char* dst = tb_ + tm.top + buf_f * tm.top_stride;
#pragma unroll 1
      for (int c = lane; c < ((M + 1) * 12) >> 4; c += 32) beam_cp_async16(dst + 16 * c, top_f + 16 * c);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    ++s_f;
    buf_f = buf_f == kTeamRows - 1 ? 0 : buf_f + 1;
    if (++e_f == E) { e_f = 0; row_f += to_frame; } else row_f += row_stride;
    top_f += (M + 1) * 12;
  };
  // This warp's hypotheses, warp and (beams wider than sixteen) warp + 16: score, graph state, list, first 32 * kEnt entries
  // (kEnt per lane).  live / have: bit k, hypothesis k can be expanded / has a score; best: the best score.
  constexpr int kEnt = 1;
  float ws[H], D[H];
  int st[H], beg[H], cnt[H];
  uint2 en[H][kEnt];
  unsigned live, have;
  bool long_lists = false;                                     // some list of this warp's has more entries than that
  float best;
  // lane k: the token sequence of hypothesis k (in the keeper, and in every warp where equal sequences are merged)
  const bool hashes = keeper || p.merge;
  unsigned long long hh = 0ull;
  int32_t hl = 0;
  // The hypotheses as the next step sees them, from lane r's (all warps alike): at a frame start all with a score are
  // live, equal sequences are merged (the first stays) and what scores far below the best is dropped.  Then every worker
  // takes its own and asks for their lists.
  auto prepare = [&](bool frame_start, float sc, int32_t dst, bool lv) {
    if (frame_start) {
      lv = sc != -INFINITY;
      if (p.merge) {
        // earlier hypotheses with the same low word of the hash (there is hardly ever one: a compare each, no matching
        // instruction, which goes value by value)
        sh.hlow[lane] = lv ? static_cast<uint32_t>(hh) : static_cast<uint32_t>(-1 - lane);      // (all warps write the same)
        __syncwarp();
        unsigned same = 0u;
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const uint4 q = *reinterpret_cast<const uint4*>(&sh.hlow[j]);
          const uint32_t me = static_cast<uint32_t>(hh);
          same |= (q.x == me ? 1u << j : 0u) | (q.y == me ? 2u << j : 0u) | (q.z == me ? 4u << j : 0u) | (q.w == me ? 8u << j : 0u);
        }
        same = lv ? same & ((1u << lane) - 1u) : 0u;
        bool dup = false;
#pragma unroll 1
        while (__any_sync(0xffffffffu, same != 0u)) {          // equal hashes: lengths and states as well?
          const int j = same ? __ffs(same) - 1 : lane;
          const int32_t lj = __shfl_sync(0xffffffffu, hl, j), sj = __shfl_sync(0xffffffffu, dst, j);
          const bool vj = __shfl_sync(0xffffffffu, sc != -INFINITY ? 1 : 0, j) != 0;
          const unsigned long long hj = (static_cast<unsigned long long>(__shfl_sync(0xffffffffu, static_cast<uint32_t>(hh >> 32), j)) << 32) |
                                        __shfl_sync(0xffffffffu, static_cast<uint32_t>(hh), j);
          if (same && vj && hj == hh && lj == hl && sj == dst) { dup = true; same = 0u; }
          same &= same - 1u;
        }
        if (dup) { sc = -INFINITY; lv = false; }
      }
      if (p.prune_delta >= 0.0f) {
        const float top1 = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(sc)));
        if (sc != -INFINITY && sc < __fsub_rn(top1, p.prune_delta)) { sc = -INFINITY; lv = false; }
      }
    }
    live = __ballot_sync(0xffffffffu, lv && sc != -INFINITY);
    have = __ballot_sync(0xffffffffu, sc != -INFINITY);
    best = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(sc)));
    if (!keeper) {
      long_lists = false;
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int k = min(warp + 16 * h, 31);                  // (a warp without a hypothesis: one without a score)
        ws[h] = __shfl_sync(0xffffffffu, sc, k);
        st[h] = __shfl_sync(0xffffffffu, dst, k);
        const uint4 r = rsrec[static_cast<unsigned>(st[h]) < static_cast<unsigned>(n_states) ? st[h] : 0];
        beg[h] = static_cast<int>(r.x); cnt[h] = static_cast<int>(r.y); D[h] = __uint_as_float(r.z);
#pragma unroll
        for (int u = 0; u < kEnt; ++u) {
          en[h][u] = make_uint2(2u * static_cast<uint32_t>(V), 0u);
          if (32 * u + lane < cnt[h]) en[h][u] = ent[beg[h] + 32 * u + lane];
        }
        long_lists |= cnt[h] > 32 * kEnt && ((live >> k) & 1u);
      }
    }
  };

#pragma unroll 1
  for (int i = tid; i < K * WW; i += team) ovr[i] = 0u;
#pragma unroll 1
  for (int i = tid; i < 2 * kHistBins; i += team) (&sh.hist[0][0])[i] = 0;
  if (tid < 2) sh.n_surv[tid] = 0;
  if (tid == 0) sh.cmd = 0;
  fetch();
  fetch();
  {
    float sc = -INFINITY; int32_t dst = -1; bool lv = false;
    if (lane < K) { sc = sh.h_score[lane]; dst = sh.h_state[lane]; lv = sh.h_live[lane] != 0; hh = sh.h_hash[lane]; hl = sh.h_len[lane]; }
    if (keeper && bound && lane < K && sc != -INFINITY && (dst < 0 || dst >= n_states)) atomicOr(p.status, TB_STATUS_BAD_STATE);   // (read as the root)
    prepare(e_cur == 0, sc, dst, lv);
  }
  int32_t tree_at = 0;                                         // where the step's nodes go in a ring
  if (p.tree_cap > 0) tree_at = (step_base + sidx) % p.tree_cap;
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  beam_team_barrier(team);
  int done = 0;
#pragma unroll 1
  for (;; ++sidx) {
    const int par = sidx & 1;
    const unsigned char* row = tb_ + tm.row + buf * tm.row_stride + off0;
    const TbTopEnt* top = reinterpret_cast<const TbTopEnt*>(tb_ + tm.top + buf * tm.top_stride);
    int32_t* hist = sh.hist[par];
    const bool over = sidx >= n_steps;                         // (only the last step's verdict is still to come)
    const int hp = H > 1 ? (lane >> 3) & 1 : 0, kp = warp + 16 * hp, j0 = lane & 7;
    const bool kp_ok = lane < 8 * H && kp < K && !keeper, alive = kp_ok && ((have >> (kp & 31)) & 1u), lvp = kp_ok && ((live >> (kp & 31)) & 1u);
    const float scp = H > 1 && hp ? ws[H - 1] : ws[0], Dp = H > 1 && hp ? D[H - 1] : D[0];
    uint32_t* ovr_p = ovr + min(kp, K - 1) * WW;
    float ref = 0.0f, vp = -INFINITY, vb = -INFINITY, vl[H][kEnt];
    bool listed[H][kEnt], pun = false, pin = false;
    int bl[H][kEnt], bp = 0, bb = 0, ptok = V;
    uint32_t pcls = 0u;
    auto bin_of = [&](float v) { return max(0, min(kHistBins - 1, __float2int_rz((ref - v) * kHistPerUnit))); };
    auto plain_value = [&](float x, uint32_t cl) {
      return __fadd_rn(scp, bound ? __fadd_rn(x, __fmul_rn(lam, __fadd_rn(Dp, rootcw[cl]))) : x);
    };
    auto listed_value = [&](int h, const uint2& e, int tk) {
      return __fadd_rn(ws[h], __fadd_rn(beam_smem_logit<LT>(row, tk), __uint_as_float(e.y)));
    };
    // ---- 1. values into the histogram.  A lane keeps the values of its entries per hypothesis, of its token of the reduced
    // row (eight lanes per hypothesis: hypothesis kp) and of the blank.  (Written without branches: a lone warp pays about
    // 45 cycles for each.)
    if (!keeper && !over) {
      const float xb = top[M].x, y_next = top[M].y;
      const TbTopEnt tt = top[j0];                             // (M >= 15)
      ref = best + fmaxf(xb, top[0].y) + kHistAbove;
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int k = warp + 16 * h;
        const bool lk = k < K && ((live >> (k & 31)) & 1u);
        uint32_t* ov = ovr + min(k, K - 1) * WW;
#pragma unroll
        for (int u = 0; u < kEnt; ++u) {
          const int tk = static_cast<int>((en[h][u].x & kTok) >> 1);       // (padding entries and unused lanes carry token V)
          listed[h][u] = tk < V && lk;
          shared_or(&ov[tk >> 5], 1u << (tk & 31), listed[h][u]);
          vl[h][u] = listed_value(h, en[h][u], tk);
          bl[h][u] = bin_of(vl[h][u]);
          shared_add(&hist[bl[h][u]], 1, listed[h][u]);
        }
      }
      if (long_lists) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const int k = warp + 16 * h;
          if (k < K && ((live >> (k & 31)) & 1u))
#pragma unroll 1
            for (int i0 = 32 * kEnt; i0 < cnt[h]; i0 += 32) {
              uint2 e = make_uint2(2u * static_cast<uint32_t>(V), 0u);
              if (i0 + lane < cnt[h]) e = ent[beg[h] + i0 + lane];
              const int t2 = static_cast<int>((e.x & kTok) >> 1);
              shared_or(&ovr[k * WW + (t2 >> 5)], 1u << (t2 & 31), t2 < V);
              shared_add(&hist[bin_of(listed_value(h, e, t2))], 1, t2 < V);
            }
        }
      }
      ptok = static_cast<int>(tt.tok_cls & 0xFFFFu); pcls = tt.tok_cls >> 16;
      pin = lvp && ptok < V;                                   // (token >= V: the row has fewer tokens)
      vp = plain_value(tt.x, pcls);
      bp = bin_of(vp);
      vb = lvp ? __fadd_rn(scp, xb) : scp;                     // the blank, or a frozen hypothesis carried
      bb = bin_of(vb);
      shared_add(&hist[bb], 1, alive && j0 == 0);
      // what the K-th pick has to clear on behalf of this hypothesis (-inf: nothing)
      const float scale = fabsf(scp) + fabsf(y_next) + 2.0f * fabsf(lam) * (fabsf(Dp) + root_wmax);
      const float ub = (scp + y_next) + lam * Dp + scale * 3.814697265625e-6f + 1e-30f;     // 2^-18 of the scale
      if (j0 == 0 && kp_ok) sh.w_ub[par][kp] = lvp && y_next != -INFINITY ? ub : -INFINITY;
      __syncwarp();
      const uint32_t bits = ovr_p[min(ptok, V) >> 5];
      pun = pin & !((bits >> (ptok & 31)) & 1u);
      shared_add(&hist[bp], 1, pun);
    }
    beam_team_barrier(team);                                   // the histogram is complete; the keeper has judged the step before
    if (sh.cmd != 0) break;
    fetch();
    // ---- 2. the bin up to which candidates may be picks
    if (keeper) {
      *reinterpret_cast<int4*>(&sh.hist[par ^ 1][4 * lane]) = make_int4(0, 0, 0, 0);
      if (lane == 0) sh.n_surv[par ^ 1] = 0;
      asm volatile("cp.async.wait_group 1;" ::: "memory");     // the next step's row and reduced row are there
    } else {
      int bstar;
      {
        const int4 h4 = *reinterpret_cast<const int4*>(hist + 4 * lane);
        const int c1 = h4.x, c2 = c1 + h4.y, c3 = c2 + h4.z, mine = c3 + h4.w;
        int incl;
        if (K <= 8) {                                          // counts up to K in unary: a ballot per unit instead of a scan
          incl = 0;
#pragma unroll
          for (int u = 0; u < 8; ++u) incl += __popc(__ballot_sync(0xffffffffu, mine > u) & (0xFFFFFFFFu >> (31 - lane)));
        } else {
          incl = mine;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) { const int v = __shfl_up_sync(0xffffffffu, incl, o); incl += lane >= o ? v : 0; }
        }
        const unsigned reach = __ballot_sync(0xffffffffu, incl >= K);
        const int above = incl - (K <= 8 ? min(mine, 8) : mine);
        const int d = (above + c1 < K ? 1 : 0) + (above + c2 < K ? 1 : 0) + (above + c3 < K ? 1 : 0);
        const int at = __shfl_sync(0xffffffffu, 4 * lane + d, reach ? __ffs(reach) - 1 : 0);
        bstar = reach ? at : kHistBins - 1;                    // (fewer than K: all of them)
      }
      // a lane's candidates take places one after the other
      int mine = 0;
#pragma unroll
      for (int h = 0; h < H; ++h)
#pragma unroll
        for (int u = 0; u < kEnt; ++u) { listed[h][u] = listed[h][u] && bl[h][u] <= bstar; mine += listed[h][u] ? 1 : 0; }
      const bool inp = pun && bp <= bstar, inb = alive && j0 == 0 && bb <= bstar;
      mine += (inp ? 1 : 0) + (inb ? 1 : 0);
      int at = shared_fetch_add(&sh.n_surv[par], mine, mine > 0);
      auto put = [&](bool yes, float v, int tkey, int k, int32_t dst) {
        shared_put(&sh.sk[min(at, kSurvivors)], beam_key(v, tkey, k), &sh.sd[min(at, kSurvivors)], dst, yes);     // (one place for what does not fit)
        at += yes ? 1 : 0;
      };
#pragma unroll
      for (int h = 0; h < H; ++h)
#pragma unroll
        for (int u = 0; u < kEnt; ++u)
          put(listed[h][u], vl[h][u], static_cast<int>((en[h][u].x & kTok) >> 1), warp + 16 * h, static_cast<int32_t>(en[h][u].x >> TB_RS_TOK_BITS));
      put(inp, vp, ptok, kp, bound ? rootdst[pcls] : -1);
      put(inb, vb, lvp ? V : V + 1, kp, H > 1 && hp ? st[H - 1] : st[0]);
      auto note = [&](bool yes, float v, int tkey, int k, int32_t dst) {
        yes = yes && bin_of(v) <= bstar;
        at = shared_fetch_add(&sh.n_surv[par], 1, yes);
        put(yes, v, tkey, k, dst);
      };
      if (long_lists) {
#pragma unroll
        for (int h = 0; h < H; ++h) {
          const int k = warp + 16 * h;
          if (k < K && ((live >> (k & 31)) & 1u))
#pragma unroll 1
            for (int i0 = 32 * kEnt; i0 < cnt[h]; i0 += 32) {
              uint2 e = make_uint2(2u * static_cast<uint32_t>(V), 0u);
              if (i0 + lane < cnt[h]) e = ent[beg[h] + i0 + lane];
              const int t2 = static_cast<int>((e.x & kTok) >> 1);
              note(t2 < V, listed_value(h, e, t2), t2, k, static_cast<int32_t>(e.x >> TB_RS_TOK_BITS));
            }
        }
      }
      // further tokens of the reduced row, eight at a time, while the group's last one is still within the bins wanted
      // (the order of the reduced row holds up to roundings: a margin of 2^-18 of the scale).  The last bin has no lower end -- values
      // 10 below the best and less, where a first step of K = 32 finds most of its picks --, down to the -inf that fill the
      // places nothing else is left for; where the reference is infinite only infinite values are in the other bins.
      const float slack = (fabsf(scp) + fabsf(ref) + fabsf(top[0].y) + 2.0f * fabsf(lam) * (fabsf(Dp) + root_wmax) + 32.0f) * 3.814697265625e-6f;
      const float lowest = bstar == kHistBins - 1 ? -INFINITY : fminf(ref - slack - static_cast<float>(bstar + 1) * (1.0f / kHistPerUnit), FLT_MAX);
      auto within = [&](float v) { return v >= lowest; };
      unsigned more = __ballot_sync(0xffffffffu, pin && within(vp)) & 0x8080u;
#pragma unroll 1
      for (int j = j0 + 8; more != 0u; j += 8) {
        const bool on = ((more >> (lane | 7)) & 1u) && j < M;
        const TbTopEnt t = top[min(j, M)];
        const int tk = static_cast<int>(t.tok_cls & 0xFFFFu);
        const bool good = on && tk < V;
        const float v = plain_value(t.x, t.tok_cls >> 16);
        const uint32_t bits = ovr_p[min(tk, V) >> 5];
        note(good & !((bits >> (tk & 31)) & 1u), v, tk, kp, bound ? rootdst[t.tok_cls >> 16] : -1);
        more = __ballot_sync(0xffffffffu, good && within(v)) & 0x8080u;
      }
      __syncwarp();
#pragma unroll
      for (int h = 0; h < H; ++h)                              // the bitmaps are left clean
#pragma unroll
        for (int u = 0; u < kEnt; ++u)
          if (warp + 16 * h < K) ovr[(warp + 16 * h) * WW + static_cast<int>((en[h][u].x & kTok) >> 6)] = 0u;
      if (long_lists) {
#pragma unroll
        for (int h = 0; h < H; ++h)
          if (warp + 16 * h < K)
#pragma unroll 1
            for (int i = lane; i < WW; i += 32) ovr[(warp + 16 * h) * WW + i] = 0u;
      }
    }
    beam_team_barrier(team);                                   // the candidates are noted
    // ---- 3. ranks
    const int n = min(sh.n_surv[par], kSurvivors + 1);
    if (n <= 32) {
      // few: every warp ranks all of them by itself (lane i: candidate i)
      const unsigned long long key = sh.sk[lane];
      int c = 0;
#pragma unroll 1
      for (int i0 = 0; i0 < n; i0 += 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) { const unsigned long long o = sh.sk[i0 + i]; c += (i0 + i < n) & (o > key) ? 1 : 0; }
      }
      if (lane < n && c < K) sh.ord[c] = lane;                 // (all warps write the same)
      __syncwarp();
    } else {
      // eight lanes per candidate count the keys above it
#pragma unroll 1
      for (int t0 = 4 * warp; t0 < n && n <= kSurvivors; t0 += 4 * nw + 4) {
        const int t = min(t0 + (lane >> 3), n - 1);
        const unsigned long long key = sh.sk[t];
        int c = 0;
#pragma unroll 1
        for (int i0 = j0; i0 - j0 < n; i0 += 64) {
#pragma unroll
          for (int i = 0; i < 64; i += 8) { const unsigned long long o = sh.sk[i0 + i]; c += (i0 + i < n) & (o > key) ? 1 : 0; }
        }
        c += __shfl_xor_sync(0xffffffffu, c, 1);
        c += __shfl_xor_sync(0xffffffffu, c, 2);
        c += __shfl_xor_sync(0xffffffffu, c, 4);
        if (c < K && j0 == 0) sh.ord[c] = t;                   // (the last candidate may be ranked more than once: the same)
      }
      beam_team_barrier(team);
    }
    // ---- 4. the picks: lane r, pick r (in every warp)
    const bool picked = n <= kSurvivors && lane < min(n, K);
    const int pick = picked ? sh.ord[lane] : 0;
    const unsigned long long pick_key = sh.sk[pick];
    const int32_t pick_dst = sh.sd[pick];
    const unsigned long long key = picked ? pick_key : 0ull;
    const int32_t dst = picked ? pick_dst : -1;
    const uint32_t l2 = 0xFFFFFFFFu - static_cast<uint32_t>(key & 0xFFFFFFFFull);
    const int parent = key != 0ull ? static_cast<int>(l2 & 31u) : -1, tkey = static_cast<int>(l2 >> 5);
    const float sc = key != 0ull ? beam_key_value(key) : -INFINITY;
    const bool emits = parent >= 0 && tkey < V;
    const bool lv = emits && ((live >> (parent & 31)) & 1u);
    const bool last = sidx + 1 >= n_steps, frame_next = e_cur + 1 == E;
    if (hashes) {
      const int from = parent >= 0 ? parent : lane;
      unsigned long long nh = (static_cast<unsigned long long>(__shfl_sync(0xffffffffu, static_cast<uint32_t>(hh >> 32), from)) << 32) |
                              __shfl_sync(0xffffffffu, static_cast<uint32_t>(hh), from);
      hl = __shfl_sync(0xffffffffu, hl, from) + (emits ? 1 : 0);
      hh = parent < 0 ? 0ull : emits ? beam_extend(nh, tkey) : nh;
      if (parent < 0) hl = 0;
    }
    if (keeper) {
      // does the K-th pick clear everything that was not looked at?
      const float c_k = __shfl_sync(0xffffffffu, sc, K - 1);
      const float ub = sh.w_ub[par][lane];
      const bool okk = (lane >= K) | (ub == -INFINITY) | (c_k > ub);
      if (__all_sync(0xffffffffu, okk) && n <= kSurvivors) {
        const int32_t token = parent < 0 || tkey == V + 1 ? -1 : tkey;
        if (lane < K) {
          sh.h_score[lane] = sc; sh.h_state[lane] = dst; sh.h_live[lane] = lv ? 1 : 0; sh.h_hash[lane] = hh; sh.h_len[lane] = hl;
          if (p.tree) {
            const int64_t at = p.tree_cap > 0 ? static_cast<int64_t>(b) * p.tree_cap + tree_at : static_cast<int64_t>(step_base + sidx) * p.B + b;
            p.tree[at * K + lane] = make_int2(parent, token);
          }
          if (last) {
            const int64_t o = static_cast<int64_t>(b) * K + lane;
            p.scores[o] = sc; p.states[o] = dst; p.live[o] = lv ? 1 : 0;
            p.out_parent[o] = parent; p.out_token[o] = token;
            const bool odd = ((par0 + sidx) & 1) != 0;
            (odd ? hashA : hashB)[o] = hh; (odd ? lenA : lenB)[o] = hl;
          }
        }
        if (lane == 0) { sh.done = done + 1; if (last) sh.cmd = 1; }
      } else if (lane == 0) {
        sh.done = done; sh.cmd = 2;
      }
    }
    ++done;
    if (!last) prepare(frame_next, sc, dst, lv);
    e_cur = frame_next ? 0 : e_cur + 1;
    buf = buf == kTeamRows - 1 ? 0 : buf + 1;
    if (++tree_at == p.tree_cap) tree_at = 0;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  return sh.done;
}

// The steps of this launch go to the batch's counts (thread 0 has written them).
__device__ __forceinline__ void beam_count(const TbBeamParams& p, const BeamShared& sh) {
  if (threadIdx.x == 0 && p.taken) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (sh.taken[i] > 0) atomicAdd(p.taken + i, static_cast<unsigned long long>(sh.taken[i]));
  }
}

// Steps sidx to end - 1 of a launch's n_steps by the whole block.
template <typename LT>
__device__ __forceinline__ void beam_block_steps(const TbBeamParams& p, BeamShared& sh, int32_t sidx, const int32_t end, const int32_t n_steps, const int32_t E,
                                                 const int64_t frame_stride, const int64_t row_stride, const int32_t step_base, unsigned long long* hashA,
                                                 unsigned long long* hashB, int32_t* lenA, int32_t* lenB, const int32_t par0) {
  LT xpre[kBeamPref] = {};
  bool xpre_valid = false;
  const LT* stream_base = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(blockIdx.x) * p.stream_stride;
#pragma unroll 1
  for (; sidx < end; ++sidx) {
    const int32_t t = sidx / E, e = sidx - t * E;
    TbBeamParams q = p;
    q.logits = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(t) * frame_stride + static_cast<int64_t>(e) * row_stride;
    q.hyp_stride = 0;
    q.new_frame = e == 0 ? 1 : 0;
    q.merge = e == 0 ? p.merge : 0;
    q.prune_delta = e == 0 ? p.prune_delta : -1.0f;
    q.fresh = 0;
    q.tv_ready = 1;
    q.step = step_base + sidx;
    const bool odd = ((par0 + sidx) & 1) != 0;
    q.hash_in = odd ? hashB : hashA; q.hash_out = odd ? hashA : hashB; q.len_in = odd ? lenB : lenA; q.len_out = odd ? lenA : lenB;
    const int32_t nt = e + 1 < E ? t : t + 1, ne = e + 1 < E ? e + 1 : 0;
    const LT* next_row = sidx + 1 < n_steps ? stream_base + static_cast<int64_t>(nt) * frame_stride + static_cast<int64_t>(ne) * row_stride : nullptr;
    beam_step_body<LT>(q, sh, xpre, xpre_valid, next_row);
    __syncthreads();
  }
}

// The same in a function of its own: its registers do not weigh on the other steps', nor theirs on its (see beam_all_steps).
template <typename LT>
__device__ __noinline__ void beam_block_steps_apart(const TbBeamParams& p, BeamShared& sh, const int32_t sidx, const int32_t end, const int32_t n_steps, const int32_t E,
                                                    const int64_t frame_stride, const int64_t row_stride, const int32_t step_base, unsigned long long* hashA,
                                                    unsigned long long* hashB, int32_t* lenA, int32_t* lenB, const int32_t par0) {
  __builtin_assume(__isShared(&sh));
  beam_block_steps<LT>(p, sh, sidx, end, n_steps, E, frame_stride, row_stride, step_base, hashA, hashB, lenA, lenB, par0);
}

// All steps of one stream of a launch without reduced rows, or without room for the team's (large vocabularies, odd strides).  A kernel of its own:
// what the other steps keep in shared memory and in registers is not there.
template <typename LT>
__device__ __forceinline__ void beam_whole_steps(const TbBeamParams& p, BeamShared& sh, unsigned char* dyn, const int32_t n_steps, const int32_t E,
                                                 const int64_t frame_stride, const int64_t row_stride, const int32_t step_base, unsigned long long* hashA,
                                                 unsigned long long* hashB, int32_t* lenA, int32_t* lenB, const int32_t par0) {
  const bool odd0 = (par0 & 1) != 0;
  beam_begin(p, sh, dyn, odd0 ? hashB : hashA, odd0 ? lenB : lenA, false, TeamSmem());
  beam_block_steps<LT>(p, sh, 0, n_steps, n_steps, E, frame_stride, row_stride, step_base, hashA, hashB, lenA, lenB, par0);
  if (threadIdx.x == 0) sh.taken[2] = n_steps;
  beam_count(p, sh);
}

#include "tb_beam_solo.cuh"
using BeamCrewAhead = BeamAhead<kCrewRows, kCrewPlain, kCrewBeam>;
#include "tb_beam_crew.cuh"

// All steps of one stream of a multi-step launch: a warp or the team takes what it can, the block the rest.
// WIDTH: 0 up to kSoloBeam / 2 hypotheses, 1 up to kSoloBeam, 2 up to 16, 3 more.  (A kernel each: in one kernel the registers and the code of one weighed on the others --
// 32 streams of 1000 steps, K = 32, 4384 us with the single warp's steps beside the team's, 3740 with the team's alone; K = 12 2633 and 2406.)
// The block's steps are a function apart but for WIDTH 1, whose own leave the compiler with no spilled registers: K = 5 1185 us apart and 1172 in place, K = 8 1256
// and 1243; K = 4 875 apart and 982 in place.
template <typename LT, int WIDTH>
__device__ __forceinline__ void beam_all_steps(const TbBeamParams& p, BeamShared& sh, unsigned char* dyn, const int32_t n_steps, const int32_t E,
                                               const int64_t frame_stride, const int64_t row_stride, const int32_t rows_per_stream,
                                               const int32_t step_base, unsigned long long* hashA, unsigned long long* hashB, int32_t* lenA,
                                               int32_t* lenB, const int32_t par0) {
  const bool fast = beam_team_applies(p);
  const TeamSmem tm = team_smem(p.rows_kept, p.V, sizeof(LT), p.top_m, p.rec_cache_bytes);
  const bool odd0 = (par0 & 1) != 0;
  const bool solo = fast && p.rows_kept > kTeamRows;            // steps by a warp or a crew (the launcher made room for their rows)
  using Ahead = typename std::conditional<WIDTH <= 1, BeamSolo, BeamCrewAhead>::type;
  __shared__ Ahead so;
  {                                           // the first rows are on their way while the tables are laid out
    const int row = static_cast<int>(threadIdx.x >> 5) - (kBeamThreads / 32 - Ahead::kRows);     // (a row each by the block's last warps)
    if (solo && row >= 0 && row < n_steps) BeamSoloRows<LT>(p, row, E, frame_stride, row_stride, rows_per_stream).fetch(p, team_base(p, dyn), tm, row);
  }
  const bool recs_cached = beam_begin(p, sh, dyn, odd0 ? hashB : hashA, odd0 ? lenB : lenA, fast, tm);
  // what the warp's steps keep behind dyn begins empty, and again after a step by the block
  auto clear = [&]() {
    for (int i = threadIdx.x; i < p.K * (p.V + 1); i += kBeamThreads) reinterpret_cast<uint32_t*>(dyn)[i] = 0u;
    if (threadIdx.x == 0) so.stamp = 0u;
    __syncthreads();
  };
  bool clean = false;
  int32_t backoff = 0;                        // steps the block takes beside one that the team could not take
  int32_t team_steps = 1;                     // steps the team takes when the warp could not
  int32_t sidx = 0;
#pragma unroll 1
  while (sidx < n_steps) {
    if (solo && backoff == 0) {               // (after the block's steps the team tries first)
      if (!clean) { clear(); clean = true; }
      const BeamSoloRows<LT> at(p, sidx, E, frame_stride, row_stride, rows_per_stream);
      const bool fetched = sidx == 0;
      const int warp = threadIdx.x >> 5;
      int d = 0;
      if constexpr (WIDTH <= 1) {
        if (warp == 0)
          d = beam_solo_run<LT, WIDTH == 0 ? 4 : 8>(p, sh, so, dyn, sidx, n_steps, E, recs_cached, tm);
        else if (warp == 1)
          beam_serve<LT, kSoloPlain>(p, sh, so, dyn, tm, sidx, n_steps, at, fetched, step_base, hashA, hashB, lenA, lenB, par0, 64);
      } else {
        __shared__ BeamCrew cr;
        static_assert(sizeof(BeamShared) + sizeof(BeamCrewAhead) + sizeof(BeamCrew) + 200 * 1024 <= 227 * 1024, "beside the launcher's 200 KB");
        const int n_warps = (p.K + 3) >> 2;
        if (warp < n_warps)
          d = beam_crew_run<LT>(p, sh, so, cr, dyn, sidx, n_steps, E, recs_cached, tm);
        else if (warp == n_warps)
          beam_serve<LT, kCrewPlain>(p, sh, so, dyn, tm, sidx, n_steps, at, fetched, step_base, hashA, hashB, lenA, lenB, par0, 32 * n_warps + 32);
      }
      if (threadIdx.x == 0) { sh.team_done = d; sh.taken[0] += d; }
      __syncthreads();
      d = sh.team_done;
      __syncthreads();                          // (read by everyone before a later run writes it again)
      sidx += d;
      if (sidx >= n_steps) break;
      team_steps = d == 0 ? min(2 * team_steps, 32) : 1;
    }
    if (fast) {
      const int32_t stop = solo ? min(n_steps, sidx + team_steps) : n_steps;
      if (threadIdx.x < 32 * (team_warps(p.K) + 1)) {
        const int d = beam_team_run<LT, WIDTH == 3 ? 2 : 1>(p, sh, dyn, sidx, stop, E, frame_stride, row_stride, rows_per_stream, step_base, hashA, hashB, lenA,
                                                            lenB, par0, recs_cached, tm);
        if (threadIdx.x == 0) { sh.team_done = d; sh.taken[1] += d; }
      }
      __syncthreads();
      const int d = sh.team_done;
      __syncthreads();                          // (read by everyone before a later run writes it again)
      sidx += d;
      if (sidx >= n_steps) break;
      backoff = d == 0 ? min(2 * backoff + 1, 32) : 0;
      if (sidx >= stop) continue;               // (the warp goes on)
    }
    clean = false;
    const int32_t end = fast ? min(n_steps, sidx + backoff + 1) : n_steps;
    if constexpr (WIDTH == 1)
      beam_block_steps<LT>(p, sh, sidx, end, n_steps, E, frame_stride, row_stride, step_base, hashA, hashB, lenA, lenB, par0);
    else
      beam_block_steps_apart<LT>(p, sh, sidx, end, n_steps, E, frame_stride, row_stride, step_base, hashA, hashB, lenA, lenB, par0);
    if (threadIdx.x == 0) sh.taken[2] += end - sidx;
    sidx = end;
  }
  beam_count(p, sh);
}

// T frames of E rows in one launch: the block loops over the expansions of its stream; every hypothesis of the
// stream reads row (t, e).
template <typename LT, int WIDTH>
__global__ void __launch_bounds__(kBeamThreads, 1) k_beam_frames(const __grid_constant__ TbBeamParams p, int32_t T, int32_t E, int64_t frame_stride,
                                                          int64_t row_stride) {
  __shared__ BeamShared sh;
  extern __shared__ __align__(16) unsigned char dyn_all[];
  if constexpr (WIDTH == kWholeRows)
    beam_whole_steps<LT>(p, sh, dyn_all, T * E, E, frame_stride, row_stride, p.step, const_cast<unsigned long long*>(p.hash_in), p.hash_out, const_cast<int32_t*>(p.len_in), p.len_out, 0);
  else
    beam_all_steps<LT, WIDTH>(p, sh, dyn_all, T * E, E, frame_stride, row_stride, T * E, p.step, const_cast<unsigned long long*>(p.hash_in), p.hash_out,
                       const_cast<int32_t*>(p.len_in), p.len_out, 0);
}

// A chunk of streaming beam decoding: slot by slot, n_frames[slot] frames (at most T) of E rows; each slot has its own
// position in its own tree ring and its own parity of the sequence-record halves, so that slots start, pause and end
// independently of each other (Sec. 2.3: hypotheses kept across chunks; Sec. 2.2 para. 4: slots re-bound in between).
template <typename LT, int WIDTH>
__global__ void __launch_bounds__(kBeamThreads, 1) k_beam_chunk(const __grid_constant__ TbBeamParams p, int32_t T, int32_t E, int64_t frame_stride,
                                                         int64_t row_stride, const int32_t* n_frames, int32_t* slot_pos,
                                                         unsigned long long* hash, int32_t* len, size_t n_hyp) {
  // (chained, but its long steps are not shared with the next launch's blocks: 117 us a chunk of 128 slots with an early start
  // of what follows, 114 without; k_beam_frames is not chained at all, the wait alone cost its step loop 2 %)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ BeamShared sh;
  extern __shared__ __align__(16) unsigned char dyn_all[];
  const int b = blockIdx.x;
  const int32_t nf = n_frames ? max(0, min(T, n_frames[b])) : T;
  const int32_t pos0 = slot_pos[b];
  if (nf > 0) {
    if constexpr (WIDTH == kWholeRows)
      beam_whole_steps<LT>(p, sh, dyn_all, nf * E, E, frame_stride, row_stride, pos0, hash, hash + n_hyp, len, len + n_hyp, pos0);
    else
      beam_all_steps<LT, WIDTH>(p, sh, dyn_all, nf * E, E, frame_stride, row_stride, T * E, pos0, hash, hash + n_hyp, len, len + n_hyp, pos0);
  }
  if (threadIdx.x == 0) slot_pos[b] = pos0 + nf * E;
}

struct SlotList { int32_t slot[TB_BIND_PAIRS]; };
// A new utterance on some slots (or on all): position 0 in the slot's tree, every hypothesis' sequence empty.
// With `scores` given, the slots' rows of the caller's [n_slots, K] arrays are set up as well: hypothesis 0 with score 0
// in the root state (state -1 on an unbound slot), the others empty.
__global__ void k_beam_reset_slots(int32_t* slot_pos, unsigned long long* hash, int32_t* len, size_t n_hyp, int32_t max_beam,   // (max_beam: records per slot)
                                   int32_t n, SlotList sl, int32_t all_slots, const TbSlotRec* slots, int32_t K,
                                   float* scores, int32_t* states, uint8_t* live) {
  pdl_chain();
  const int i = blockIdx.x;
  if (i >= n) return;
  const int slot = all_slots ? i : sl.slot[i];
  if (threadIdx.x == 0) slot_pos[slot] = 0;
  for (int k = threadIdx.x; k < max_beam; k += blockDim.x) {
    const size_t o = static_cast<size_t>(slot) * max_beam + k;
    hash[o] = 0ull; hash[n_hyp + o] = 0ull; len[o] = 0; len[n_hyp + o] = 0;
  }
  if (scores) {
    const bool bound = slots[slot].n_states > 0;
    for (int k = threadIdx.x; k < K; k += blockDim.x) {
      const size_t o = static_cast<size_t>(slot) * K + k;
      scores[o] = k == 0 ? 0.0f : -INFINITY;
      states[o] = (k == 0 && bound) ? 0 : -1;
      live[o] = 0;
    }
  }
}

// The tokens of every hypothesis a stream holds, walked back to the start of its utterance.  The walk is a chain of
// dependent look-ups, a step at a time, so the steps are cut into pieces walked at the same time, one warp each: (a) from
// every hypothesis at a piece's end to its start, counting tokens; (b) the pieces' maps composed from the last to the first
// give, per hypothesis, where it enters each piece and where its tokens there end in the transcript; (c) the pieces again,
// now writing.  A warp reads the nodes of 32 / K steps per register, eight registers at a time, and follows the parents with
// shuffles.  1000 steps of 32 streams: 17 us at K = 4, 28 at K = 32 (one warp for the whole chain, nodes staged in shared memory
// ahead of it: 75 and 100 us in a session of 3000 steps).
// RING: the stream's own ring of tree_cap steps at position slot_pos[slot] (streaming); else the batch-wide tree
// [n_steps, B, K].  sl / use_list: the slots to walk (output row i belongs to sl.slot[i]); else slot = block index.
constexpr int kBtWarps = 16;
constexpr int kBtMin = 16;         // steps of a piece at least
constexpr int kBtRegs = 8;
template <bool RING>
__global__ void __launch_bounds__(32 * kBtWarps) k_beam_backtrace(const int2* tree, int32_t tree_cap, const int32_t* slot_pos, int32_t n_steps,
                                                                  int32_t B, int32_t K, int32_t V, int32_t max_len, int32_t* out_tokens,
                                                                  int32_t* out_lens, int32_t* status, const __grid_constant__ SlotList sl,
                                                                  int32_t use_list) {
  pdl_chain();
  __shared__ int2 piece[kBtWarps][TB_MAX_BEAM];              // (a) where a hypothesis at the piece's end stood at its start, its tokens
  __shared__ int2 enter[kBtWarps][TB_MAX_BEAM];              // (b) which one a hypothesis of the last step was at the piece's end, tokens up to there
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = use_list ? sl.slot[blockIdx.x] : blockIdx.x;
  const int32_t pos = RING ? slot_pos[b] : n_steps;
  const int32_t first = RING ? max(0, pos - tree_cap) : 0;
  if (RING && pos > tree_cap && threadIdx.x == 0) atomicOr(status, TB_STATUS_STEP_LIMIT);   // the utterance is longer than the ring: its start is gone
  const int32_t n = pos - first;
  const int pieces = max(1, min(kBtWarps, n / kBtMin)), per = (n + pieces - 1) / pieces;
  const int32_t lo = first + warp * per, hi = min(pos, lo + per);
  const int2* base = RING ? tree + static_cast<int64_t>(b) * tree_cap * K : tree + static_cast<int64_t>(b) * K;
  const int64_t stride = RING ? K : static_cast<int64_t>(B) * K;
  const int spr = 32 / K, my_step = lane / K, my_k = lane - my_step * K;      // steps per register; this lane's node in it
  const int64_t row = (static_cast<int64_t>(blockIdx.x) * K + lane) * max_len;
  // from hypothesis `cur` after step hi - 1 back to before step lo; at: one past the last token's place
  auto walk = [&](int& cur, int& at, bool write) {
#pragma unroll 1
    for (int32_t top = hi; top > lo; top -= kBtRegs * spr) {
      int2 e[kBtRegs];
#pragma unroll
      for (int r = 0; r < kBtRegs; ++r) {                      // register r: steps top - (r + 1) * spr ... top - r * spr - 1
        const int32_t sidx = top - (r + 1) * spr + my_step;
        e[r] = make_int2(-1, -1);
        if (my_step < spr && sidx >= lo) e[r] = __ldg(base + static_cast<int64_t>(RING ? sidx % tree_cap : sidx) * stride + my_k);
      }
#pragma unroll
      for (int r = 0; r < kBtRegs; ++r) {
#pragma unroll 1
        for (int j = spr - 1; j >= 0 && top - (r + 1) * spr + j >= lo; --j) {
          const int from = j * K + max(cur, 0);
          const int px = __shfl_sync(0xffffffffu, e[r].x, from), tk = __shfl_sync(0xffffffffu, e[r].y, from);
          const bool tok = cur >= 0 && tk >= 0 && tk != V;
          at -= tok ? 1 : 0;
          if (write && tok && at < max_len) out_tokens[row + at] = tk;
          cur = cur >= 0 ? px : -1;
        }
      }
    }
  };
  int cur = lane < K ? lane : -1, at = 0;
  if (warp < pieces) {
    walk(cur, at, false);
    piece[warp][lane] = make_int2(cur, -at);
  }
  __syncthreads();
  if (warp == 0) {
    int total = 0, c = lane < K ? lane : -1;
    for (int w = pieces - 1; w >= 0; --w) {
      const int2 q = piece[w][max(c, 0)];
      enter[w][lane] = make_int2(c, total);                    // (tokens after the piece, for now)
      total += c >= 0 ? q.y : 0;
      c = c >= 0 ? q.x : -1;
    }
    for (int w = 0; w < pieces; ++w) enter[w][lane].y = total - enter[w][lane].y;
    if (lane < K) out_lens[static_cast<int64_t>(blockIdx.x) * K + lane] = total;
  }
  __syncthreads();
  if (warp < pieces) {
    const int2 q = enter[warp][lane];
    cur = q.x; at = q.y;
    walk(cur, at, true);
  }
}

__global__ void k_publish_slot(TbSlotRec* slots, TbSlotState* sstate, int32_t slot, TbSlotRec rec) {
  if (threadIdx.x == 0) {
    slots[slot] = rec;
    TbSlotState st;
    st.state = rec.n_states > 0 ? 0 : -1; st.t = 0; st.k = 0; st.score = 0.0f; st.n_emitted = 0;
    st.chunk_base = 0; st.pad0 = 0; st.pad1 = 0;
    sstate[slot] = st;
  }
}

template <typename F>
int set_smem(F* fn, size_t bytes) {
  // (the default limit of 48 KB counts the kernel's static shared memory too -- up to 28 KB here -- so the opt-in
  //  starts well below it)
  if (bytes > 16 * 1024) {
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes)) != cudaSuccess) {
      cudaGetLastError();
      return TB_ERR_INVALID_ARG;
    }
  }
  return TB_OK;
}

}  // namespace

int tb_launch_decode_general(const TbDecodeParams& p_in, cudaStream_t stream, const TbInlineBinds* binds) {
  TbDecodeParams p = p_in;
  TbInlineBinds ib;
  if (binds) ib = *binds; else ib.n = 0;
  if (ib.n < 0 || ib.n > TB_INLINE_BINDS || (ib.n > 0 && (!p.persistent || !ib.arena || !ib.slots))) return TB_ERR_INVALID_ARG;
  size_t smem = static_cast<size_t>(p.C) * (sizeof(float) + sizeof(int32_t));
  // graphs with resolved lists exist only for vocabularies whose token view fits comfortably
  p.tokview = 2 * (p.V + 1) <= (1 << TB_RS_TOK_BITS) ? 1 : 0;
  if (p.tokview && tokview_bytes(p.V, p.C) > smem) smem = tokview_bytes(p.V, p.C);
  int rc;
  if (p.dtype == TB_BF16) {
    if ((rc = set_smem(k_decode_general<uint16_t>, smem)) != TB_OK) return rc;
    k_decode_general<uint16_t><<<p.n_streams, kThreads, smem, stream>>>(p, ib);
  } else {
    if ((rc = set_smem(k_decode_general<float>, smem)) != TB_OK) return rc;
    k_decode_general<float><<<p.n_streams, kThreads, smem, stream>>>(p, ib);
  }
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_beam_step(const TbBeamParams& p_in, cudaStream_t stream) {
  TbBeamParams p = p_in;
  p.tokview = 2 * (p.V + 1) <= (1 << TB_RS_TOK_BITS) ? 1 : 0;
  const size_t aux = beam_aux_bytes(p.V, p.C, p.tokview);
  const size_t smem = ((static_cast<size_t>(p.K) * (p.V + 1) * sizeof(float) + 15) & ~size_t(15)) +
                      ((static_cast<size_t>(p.K) * ((p.V + 1 + 31) >> 5) * sizeof(uint32_t) + 15) & ~size_t(15)) + aux;
  if (smem > 200 * 1024) return TB_ERR_INVALID_ARG;
  int rc;
  if (p.dtype == TB_BF16) {
    if ((rc = set_smem(k_beam_step<uint16_t>, smem)) != TB_OK) return rc;
    k_beam_step<uint16_t><<<p.B, kBeamThreads, smem, stream>>>(p);
  } else {
    if ((rc = set_smem(k_beam_step<float>, smem)) != TB_OK) return rc;
    k_beam_step<float><<<p.B, kBeamThreads, smem, stream>>>(p);
  }
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

// Calls f with the width class of beam_all_steps, or kWholeRows, as a compile-time constant.
template <typename F>
static int beam_width_class(const TbBeamParams& p, F f) {
  if (!p.tensor_lo) return f(std::integral_constant<int, kWholeRows>{});     // (see beam_team_setup)
  const int K = p.K;
  if (K <= kSoloBeam / 2) return f(std::integral_constant<int, 0>{});
  if (K <= kSoloBeam) return f(std::integral_constant<int, 1>{});
  if (K <= 16) return f(std::integral_constant<int, 2>{});
  return f(std::integral_constant<int, 3>{});
}

// The team's steps (beam_team_run) read rows through buffers behind the block's other shared memory and need the extent
// of the logits tensor; without either (odd strides, no room) they stay off.
static void beam_team_setup(TbBeamParams* p, int32_t T, int32_t E, int64_t frame_stride, int64_t row_stride, size_t* smem) {
  constexpr size_t kMost = 200 * 1024;
  p->tensor_lo = nullptr; p->tensor_hi = nullptr; p->rec_cache_bytes = 0; p->rows_kept = 0;
  if (!p->top_base || p->stream_stride < 0 || frame_stride < 0 || row_stride < 0) return;
  const int elem = p->dtype == TB_BF16 ? 2 : 4;
  p->rows_kept = p->K <= kSoloBeam ? 2 * kSoloRows : 2 * kCrewRows;
  size_t more = team_smem(p->rows_kept, p->V, elem, p->top_m, 0).total;
  // (Steps of nearly as many places as there are tokens and hypotheses to fill them need a second look each: 32 streams of 200 steps, V = 8: K = 9 427 us by the
  // team, 440 by a crew, K = 24 648 and 632, K = 32 607 and 723; V = 17: 425 and 355, 649 and 458, 606 and 468.  A single warp: V = 8, K = 8 399 and 207.)
  if ((p->K > kSoloBeam && p->V < kCrewVocab) || *smem + more > kMost) {
    p->rows_kept = kTeamRows;
    more = team_smem(kTeamRows, p->V, elem, p->top_m, 0).total;
  }
  if (*smem + more > kMost) return;
  *smem += more;
  p->rec_cache_bytes = static_cast<int32_t>((kMost - *smem < static_cast<size_t>(kTeamRecCache) ? kMost - *smem : static_cast<size_t>(kTeamRecCache)) & ~size_t(15));
  *smem += p->rec_cache_bytes;
  const int64_t last = static_cast<int64_t>(p->B - 1) * p->stream_stride + static_cast<int64_t>(T - 1) * frame_stride +
                       static_cast<int64_t>(E - 1) * row_stride + p->V;
  p->tensor_lo = static_cast<const unsigned char*>(p->logits);
  p->tensor_hi = p->tensor_lo + static_cast<size_t>(last + 1) * elem;
}

int tb_launch_beam_frames(const TbBeamParams& p_in, int32_t T, int32_t E, int64_t frame_stride, int64_t row_stride,
                          cudaStream_t stream) {
  TbBeamParams p = p_in;
  p.tokview = 2 * (p.V + 1) <= (1 << TB_RS_TOK_BITS) ? 1 : 0;
  const size_t aux = beam_aux_bytes(p.V, p.C, p.tokview);
  size_t smem = ((static_cast<size_t>(p.K) * (p.V + 1) * sizeof(float) + 15) & ~size_t(15)) +
                ((static_cast<size_t>(p.K) * ((p.V + 1 + 31) >> 5) * sizeof(uint32_t) + 15) & ~size_t(15)) + aux;
  beam_team_setup(&p, T, E, frame_stride, row_stride, &smem);
  if (smem > 200 * 1024) return TB_ERR_INVALID_ARG;
  auto launch = [&](auto* fn) -> int {
    const int rc = set_smem(fn, smem);
    if (rc == TB_OK) fn<<<p.B, kBeamThreads, smem, stream>>>(p, T, E, frame_stride, row_stride);
    return rc;
  };
  const int rc = beam_width_class(p, [&](auto w) {
    return p.dtype == TB_BF16 ? launch(k_beam_frames<uint16_t, decltype(w)::value>) : launch(k_beam_frames<float, decltype(w)::value>);
  });
  if (rc != TB_OK) return rc;
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_beam_backtrace(const int2* tree, int32_t n_steps, int32_t B, int32_t K, int32_t V, int32_t max_len,
                             int32_t* out_tokens, int32_t* out_lens, cudaStream_t stream) {
  SlotList none;
  none.slot[0] = 0;
  if (tb_launch_chained(k_beam_backtrace<false>, dim3(B), dim3(32 * kBtWarps), 0, stream, tree, 0, nullptr, n_steps, B, K, V, max_len, out_tokens, out_lens, nullptr, none, 0) != TB_OK) return TB_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

// End of stream: every hypothesis that stops in a graph state is charged that state's final weight,
// score' = fl(score + fl(lambda * final(state))).  Unbound slots, state -1 and empty places (-inf) stay as they are.
__global__ void k_final_weights(const TbSlotRec* slots, const unsigned char* arena, int32_t B, int32_t K, float* scores,
                                const int32_t* states, int32_t* status) {
  pdl_chain();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * K) return;
  const TbSlotRec rec = slots[i / K];
  const int32_t s = states[i];
  if (rec.n_states <= 0 || s < 0) return;
  if (s >= rec.n_states) { atomicOr(status, TB_STATUS_BAD_STATE); return; }
  const float fin = reinterpret_cast<const float*>(arena + rec.blob_off + rec.off_final)[s];
  const float sc = scores[i];
  if (sc == -INFINITY) return;
  scores[i] = __fadd_rn(sc, __fmul_rn(rec.lambda, fin));
}

int tb_launch_final_weights(const TbSlotRec* slots, const unsigned char* arena, int32_t B, int32_t K, float* scores,
                            const int32_t* states, int32_t* status, cudaStream_t stream) {
  const int n = B * K;
  if (tb_launch_chained(k_final_weights, dim3((n + 127) / 128), dim3(128), 0, stream, slots, arena, B, K, scores, states, status) != TB_OK) return TB_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

__global__ void k_publish_model(TbSlotRec* model_recs, int32_t model_id, TbSlotRec rec) {
  if (threadIdx.x == 0) model_recs[model_id] = rec;
}

struct BindPairs { int32_t slot[TB_BIND_PAIRS]; int32_t model[TB_BIND_PAIRS]; };
__global__ void k_bind_models(TbSlotRec* slots, TbSlotState* sstate, const TbSlotRec* model_recs, int32_t n, BindPairs pr) {
  const int i = threadIdx.x;
  if (i >= n) return;
  TbSlotRec rec;
  if (pr.model[i] >= 0) rec = model_recs[pr.model[i]];
  else memset(&rec, 0, sizeof rec);
  slots[pr.slot[i]] = rec;
  TbSlotState st;
  st.state = rec.n_states > 0 ? 0 : -1; st.t = 0; st.k = 0; st.score = 0.0f; st.n_emitted = 0;
  st.chunk_base = 0; st.pad0 = 0; st.pad1 = 0;
  sstate[pr.slot[i]] = st;
}

int tb_launch_publish_model(TbSlotRec* model_recs, int32_t model_id, const TbSlotRec& rec, cudaStream_t stream) {
  k_publish_model<<<1, 32, 0, stream>>>(model_recs, model_id, rec);
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_bind_models(TbSlotRec* slots, TbSlotState* sstate, const TbSlotRec* model_recs, int32_t n,
                          const int32_t* slot_of, const int32_t* model_of, cudaStream_t stream) {
  if (n < 1 || n > TB_BIND_PAIRS) return TB_ERR_INVALID_ARG;
  BindPairs pr;
  for (int i = 0; i < TB_BIND_PAIRS; ++i) { pr.slot[i] = i < n ? slot_of[i] : 0; pr.model[i] = i < n ? model_of[i] : -1; }
  k_bind_models<<<1, TB_BIND_PAIRS, 0, stream>>>(slots, sstate, model_recs, n, pr);
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_publish_slot(TbSlotRec* slots, TbSlotState* sstate, int32_t slot, const TbSlotRec& rec,
                           cudaStream_t stream) {
  k_publish_slot<<<1, 32, 0, stream>>>(slots, sstate, slot, rec);
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

namespace {
// Many slots published at once: the records and their slot indices were copied to the device with the graphs.
__global__ void k_publish_slots(TbSlotRec* slots, TbSlotState* sstate, int32_t n, const TbSlotRec* recs, const int32_t* slot_of) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const TbSlotRec rec = recs[i];
  slots[slot_of[i]] = rec;
  TbSlotState st;
  st.state = rec.n_states > 0 ? 0 : -1; st.t = 0; st.k = 0; st.score = 0.0f; st.n_emitted = 0;
  st.chunk_base = 0; st.pad0 = 0; st.pad1 = 0;
  sstate[slot_of[i]] = st;
}

// Binds carried out by one launch (see TbInlineBinds): block i brings the image of bind i from page-locked host
// memory, read in place, into its arena block, then stores the slot's record and starts the slot's stream afresh.
constexpr int kPullThreads = 512;
__global__ void __launch_bounds__(kPullThreads) k_pull_binds(TbInlineBinds ib, TbSlotState* sstate) {
  pdl_chain();
  const int i = blockIdx.x;
  const unsigned char* src = nullptr;
  int32_t bytes = 0, slot = -1;
  TbSlotRec rec;
#pragma unroll
  for (int j = 0; j < TB_INLINE_BINDS; ++j)
    if (i == j) { src = ib.src[j]; bytes = ib.bytes[j]; slot = ib.slot[j]; rec = ib.rec[j]; }
  if (i >= ib.n || slot < 0) return;
  pull_image<8>(src, ib.arena + rec.blob_off, bytes);
  if (threadIdx.x == 0) {
    ib.slots[slot] = rec;
    TbSlotState st;
    st.state = rec.n_states > 0 ? 0 : -1; st.t = 0; st.k = 0; st.score = 0.0f; st.n_emitted = 0;
    st.chunk_base = 0; st.pad0 = 0; st.pad1 = 0;
    sstate[slot] = st;
  }
}

__global__ void k_final_weights_slots(const TbSlotRec* slots, const unsigned char* arena, int32_t n, SlotList sl, int32_t K,
                                      float* scores, const int32_t* states, int32_t* status) {
  pdl_chain();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n * K) return;
  const int slot = sl.slot[i / K];
  const int64_t o = static_cast<int64_t>(slot) * K + i % K;
  const TbSlotRec rec = slots[slot];
  const float sc = scores[o];
  const int32_t st = states[o];
  if (rec.n_states <= 0 || st < 0 || sc == -INFINITY) return;
  if (st >= rec.n_states) { atomicOr(status, TB_STATUS_BAD_STATE); return; }
  const float fw = reinterpret_cast<const float*>(arena + rec.blob_off + rec.off_final)[st];
  scores[o] = __fadd_rn(sc, __fmul_rn(rec.lambda, fw));
}
}  // namespace

int tb_launch_beam_chunk(const TbBeamParams& p_in, int32_t T, int32_t E, int64_t frame_stride, int64_t row_stride,
                         const int32_t* n_frames, int32_t* slot_pos, unsigned long long* hash, int32_t* len, size_t n_hyp,
                         cudaStream_t stream) {
  TbBeamParams p = p_in;
  p.tokview = 2 * (p.V + 1) <= (1 << TB_RS_TOK_BITS) ? 1 : 0;
  const size_t aux = beam_aux_bytes(p.V, p.C, p.tokview);
  size_t smem = ((static_cast<size_t>(p.K) * (p.V + 1) * sizeof(float) + 15) & ~size_t(15)) +
                ((static_cast<size_t>(p.K) * ((p.V + 1 + 31) >> 5) * sizeof(uint32_t) + 15) & ~size_t(15)) + aux;
  beam_team_setup(&p, T, E, frame_stride, row_stride, &smem);
  if (smem > 200 * 1024) return TB_ERR_INVALID_ARG;
  auto launch = [&](auto* fn) -> int {
    const int rc = set_smem(fn, smem);
    if (rc != TB_OK) return rc;
    return tb_launch_chained(fn, dim3(p.B), dim3(kBeamThreads), smem, stream, p, T, E, frame_stride, row_stride, n_frames, slot_pos, hash, len, n_hyp) == TB_OK ? TB_OK : TB_ERR_CUDA;
  };
  const int rc = beam_width_class(p, [&](auto w) {
    return p.dtype == TB_BF16 ? launch(k_beam_chunk<uint16_t, decltype(w)::value>) : launch(k_beam_chunk<float, decltype(w)::value>);
  });
  if (rc != TB_OK) return rc;
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_beam_reset_slots(int32_t* slot_pos, unsigned long long* hash, int32_t* len, size_t n_hyp, int32_t max_beam,
                               int32_t n, const int32_t* slots, int32_t all_slots, const TbSlotRec* slot_recs, int32_t K,
                               float* scores, int32_t* states, uint8_t* live, cudaStream_t stream) {
  if (n < 1 || (!all_slots && n > TB_BIND_PAIRS)) return TB_ERR_INVALID_ARG;
  SlotList sl;
  for (int i = 0; i < TB_BIND_PAIRS; ++i) sl.slot[i] = (!all_slots && i < n) ? slots[i] : 0;
  if (tb_launch_chained(k_beam_reset_slots, dim3(n), dim3(32), 0, stream, slot_pos, hash, len, n_hyp, max_beam, n, sl, all_slots, slot_recs, K, scores, states, live) != TB_OK) return TB_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_beam_backtrace_slots(const int2* tree, int32_t tree_cap, const int32_t* slot_pos, int32_t n_slots, int32_t K,
                                   int32_t V, int32_t max_len, int32_t* out_tokens, int32_t* out_lens, int32_t* status,
                                   const int32_t* slot_list, cudaStream_t stream) {
  // slot_list (host, n_slots entries, at most TB_BIND_PAIRS): the slots to walk; null: slots 0 .. n_slots-1
  if (slot_list && n_slots > TB_BIND_PAIRS) return TB_ERR_INVALID_ARG;
  SlotList sl;
  for (int i = 0; i < TB_BIND_PAIRS; ++i) sl.slot[i] = (slot_list && i < n_slots) ? slot_list[i] : 0;
  if (tb_launch_chained(k_beam_backtrace<true>, dim3(n_slots), dim3(32 * kBtWarps), 0, stream, tree, tree_cap, slot_pos, 0, n_slots, K, V, max_len, out_tokens, out_lens, status, sl,
                                                                slot_list ? 1 : 0) != TB_OK) return TB_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_final_weights_slots(const TbSlotRec* slots, const unsigned char* arena, int32_t n, const int32_t* slot_list,
                                  int32_t K, float* scores, const int32_t* states, int32_t* status, cudaStream_t stream) {
  if (n < 1 || n > TB_BIND_PAIRS) return TB_ERR_INVALID_ARG;
  SlotList sl;
  for (int i = 0; i < TB_BIND_PAIRS; ++i) sl.slot[i] = i < n ? slot_list[i] : 0;
  const int total = n * K;
  if (tb_launch_chained(k_final_weights_slots, dim3((total + 127) / 128), dim3(128), 0, stream, slots, arena, n, sl, K, scores, states, status) != TB_OK) return TB_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_publish_slots(TbSlotRec* slots, TbSlotState* sstate, int32_t n, const TbSlotRec* recs, const int32_t* slot_of,
                            cudaStream_t stream) {
  if (n < 1) return TB_ERR_INVALID_ARG;
  k_publish_slots<<<(n + 63) / 64, 64, 0, stream>>>(slots, sstate, n, recs, slot_of);
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}

int tb_launch_pull_binds(const TbInlineBinds& ib, TbSlotState* sstate, cudaStream_t stream) {
  if (ib.n < 1 || ib.n > TB_INLINE_BINDS || !ib.arena || !ib.slots || !sstate) return TB_ERR_INVALID_ARG;
  k_pull_binds<<<ib.n, kPullThreads, 0, stream>>>(ib, sstate);
  return cudaGetLastError() == cudaSuccess ? TB_OK : TB_ERR_CUDA;
}
