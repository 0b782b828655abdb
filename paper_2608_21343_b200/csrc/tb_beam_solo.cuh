// Beam steps of narrow beams by a single warp (part of tb_decode.cu, behind the team's steps, whose parts it uses).
#ifndef TB_BEAM_SOLO_CUH_
#define TB_BEAM_SOLO_CUH_

// The candidates of a team's step -- listed tokens, blank, the first tokens of the reduced row -- of a beam of up to KG hypotheses fit
// one warp: 32 / KG lanes per hypothesis.  A lane keeps the values of its two or three best candidates and the lower words of their keys (the order of the
// general step), the picks are the largest of the lanes' best, one after the other by two warp reductions each, and the next step starts from
// registers: no barriers, no shared counters, no candidates written out and read back.  A second warp brings rows and
// reduced rows into shared memory and keeps the books, kSoloRows steps at a time, one barrier of two warps for as many steps.
// Bound by the latency of a step's dependent instructions (one issued every four to five cycles): about 1650 cycles at K = 4 by a call's time; when counted, of 1500 of
// an average step the values of the plain tokens took 110, of up to two listed tokens a lane 120 and of longer lists 230 on average, what is kept of the plain
// ones and the blank 220, picks 245 (60 each), where they lead 125, their records and lists 330.  The team's step took 3500.  32 streams of 1000 steps,
// V = 1024, lists of 300 phrases, whole call with transcripts, by the team and so: K = 1 1869 and 802 us, K = 2 1901 and 809, K = 4 1950 and 881, K = 5 2083
// and 1172, K = 8 2191 and 1243; merging and pruning K = 4 2091 and 912, K = 5 2241 and 1273, K = 8 2388 and 1330.  (Wider
// beams would have two lanes a hypothesis, which a first step's picks do not fit.)
// A step is untouched and left to the team when a lane might have held one pick more than it keeps, when the K-th pick does not
// clear the bound on the tokens that were not looked at (as in the team's step, with the first token behind those looked at), and when a value that it weighs is
// no number (a row's tokens with such values are the first of its reduced form, so that one of them is weighed).
__device__ __forceinline__ void beam_group_barrier(int n_threads) { asm volatile("bar.sync 2, %0;" ::"r"(n_threads) : "memory"); }

// The logit at 2 * token of a row in shared memory.
template <typename LT> __device__ __forceinline__ float beam_smem_logit2(const unsigned char* row, uint32_t token2);
template <> __device__ __forceinline__ float beam_smem_logit2<uint16_t>(const unsigned char* row, uint32_t token2) {
  return __uint_as_float(static_cast<uint32_t>(*reinterpret_cast<const uint16_t*>(row + token2)) << 16);
}
template <> __device__ __forceinline__ float beam_smem_logit2<float>(const unsigned char* row, uint32_t token2) {
  return *reinterpret_cast<const float*>(row + 2 * token2);
}

// What the serving warp prepares per row, and what the steps leave it: rows brought R at a time, PLAIN tokens of a reduced row, PLACES hypotheses at most.
template <int R, int PLAIN, int PLACES>
struct BeamAhead {
  static constexpr int kRows = R;
  struct Row { float xb, y_next; uint32_t at, unused; };       // blank, value of the first token not looked at, where the row begins (behind dyn)
  uint4 plain[2 * R][PLAIN];                                   // per token looked at: logit, its class' root weight, token, the root arc's target
  Row row[2 * R];
  uint32_t pick[2 * R][PLACES];                                // 32 * token key + parent of every place's pick, all ones: none
  uint32_t stamp;                                              // the last step's number, in the upper bits (see beam_solo_run)
};
using BeamSolo = BeamAhead<kSoloRows, kSoloPlain, kSoloBeam>;

// Row sidx of the block's stream, the way from a frame's last row to the next frame, and the row's reduced form.
template <typename LT>
struct BeamSoloRows {
  const LT* row;
  const unsigned char* top;
  int64_t row_stride, to_frame;
  int e, E, top_bytes;
  __device__ __forceinline__ BeamSoloRows(const TbBeamParams& p, int32_t sidx, int32_t E_, int64_t frame_stride, int64_t row_stride_, int32_t rows_per_stream) {
    const int b = blockIdx.x;
    E = E_; e = sidx % E; row_stride = row_stride_; to_frame = frame_stride - static_cast<int64_t>(E - 1) * row_stride;
    row = reinterpret_cast<const LT*>(p.logits) + static_cast<int64_t>(b) * p.stream_stride + static_cast<int64_t>(sidx / E) * frame_stride + static_cast<int64_t>(e) * row_stride;
    top_bytes = (p.top_m + 1) * 12;
    top = reinterpret_cast<const unsigned char*>(p.top_base + (static_cast<int64_t>(b) * rows_per_stream + sidx) * (p.top_m + 1));
  }
  __device__ __forceinline__ void fetch(const TbBeamParams& p, unsigned char* mem, const TeamSmem& tm, int place) const {      // (by a warp)
    const int lane = threadIdx.x & 31;
    beam_fetch_row<LT>(mem + tm.row + place * tm.row_stride, row, p.V + 1, p.tensor_lo, p.tensor_hi, lane, 32);
    unsigned char* dst = mem + tm.top + place * tm.top_stride;
#pragma unroll 1
    for (int c = lane; c < top_bytes >> 4; c += 32) beam_cp_async16(dst + 16 * c, top + 16 * c);
  }
  __device__ __forceinline__ void next() {
    top += top_bytes;
    if (++e == E) { e = 0; row += to_frame; } else row += row_stride;
  }
};

// The second warp: brings rows sidx, sidx + 1, ... into the buffers and keeps the books of the steps before: the tree, and what
// identifies the hypotheses' token sequences.  (fetched: the first rows are on their way already.)  sh.cmd holds the number of the barrier that ends the run, sh.done the steps
// taken by then.  P: tokens of a reduced row that the steps look at; n_threads: of the group barrier, the steps' warps and this one.
template <typename LT, int P, typename Ahead>
__device__ __forceinline__ void beam_serve(const TbBeamParams& p, BeamShared& sh, Ahead& so, unsigned char* dyn, const TeamSmem& tm, int32_t sidx,
                                                const int32_t n_steps, BeamSoloRows<LT> at, bool fetched, const int32_t step_base, unsigned long long* hashA, unsigned long long* hashB,
                                                int32_t* lenA, int32_t* lenB, const int32_t par0, const int n_threads) {
  constexpr int R = Ahead::kRows;
  const int lane = threadIdx.x & 31, b = blockIdx.x, K = p.K, V = p.V, W = V + 1, M = p.top_m;
  const bool bound = p.slots[b].n_states > 0;
  const int WW = (W + 31) >> 5;
  const unsigned char* aux = dyn + ((static_cast<size_t>(K) * W * sizeof(float) + 15) & ~size_t(15)) + ((static_cast<size_t>(K) * WW * sizeof(uint32_t) + 15) & ~size_t(15));
  const float* rootcw = reinterpret_cast<const float*>(aux);    // (see tokview_attach)
  const int32_t* rootdst = reinterpret_cast<const int32_t*>(aux + 4 * static_cast<size_t>(p.C));
  unsigned char* mem = team_base(p, dyn);
  int step = sidx;                                              // the next one to be entered in the books
  const int32_t first = sidx;
  int tree_at = p.tree_cap > 0 ? (step_base + sidx) % p.tree_cap : 0;
  unsigned long long hh = 0ull;                                 // lane k: the sequence of hypothesis k
  int32_t hl = 0;
  if (lane < K) { hh = sh.h_hash[lane]; hl = sh.h_len[lane]; }
  const volatile int32_t* cmd = &sh.cmd;
  int buf = 0, book = 0;
#pragma unroll 1
  for (int n = 1;; ++n) {
    int rows = 0;
#pragma unroll 1
    for (; rows < R && sidx < n_steps; ++rows, ++sidx) {
      if (!fetched) at.fetch(p, mem, tm, buf + rows);
      if (lane == 0) so.row[buf + rows].at = static_cast<uint32_t>(mem - dyn) + tm.row + (buf + rows) * tm.row_stride + static_cast<uint32_t>(reinterpret_cast<uintptr_t>(at.row) & 15u);
      at.next();
    }
    fetched = false;
    // the steps before the last barrier (the rows are on their way)
    const bool end = n > 1 && *cmd == n - 1;
    const int32_t upto = end ? first + *const_cast<volatile int32_t*>(&sh.done) : first + max(n - 2, 0) * R;
#pragma unroll 1
    for (; step < upto; ++step) {
      const uint32_t l2 = lane < K ? so.pick[book][lane] : 0xFFFFFFFFu;
      const bool some = l2 != 0xFFFFFFFFu;
      const int parent = some ? static_cast<int>(l2 & 31u) : -1, tkey = static_cast<int>(l2 >> 5), from = some ? parent : lane;
      const bool emits = some && tkey < V;
      const unsigned long long nh = (static_cast<unsigned long long>(__shfl_sync(0xffffffffu, static_cast<uint32_t>(hh >> 32), from)) << 32) |
                                    __shfl_sync(0xffffffffu, static_cast<uint32_t>(hh), from);
      const int nl = __shfl_sync(0xffffffffu, hl, from) + (emits ? 1 : 0);
      hh = !some ? 0ull : emits ? beam_extend(nh, tkey) : nh;
      hl = some ? nl : 0;
      if (lane < K) {
        const int32_t token = !some || tkey == V + 1 ? -1 : tkey;
        if (p.tree) {
          const int64_t at = p.tree_cap > 0 ? static_cast<int64_t>(b) * p.tree_cap + tree_at : static_cast<int64_t>(step_base + step) * p.B + b;
          p.tree[at * K + lane] = make_int2(parent, token);
        }
        if (step + 1 == n_steps) {
          const int64_t o = static_cast<int64_t>(b) * K + lane;
          p.out_parent[o] = parent; p.out_token[o] = token;
          const bool odd = ((par0 + step) & 1) != 0;
          (odd ? hashA : hashB)[o] = hh; (odd ? lenA : lenB)[o] = hl;
        }
      }
      if (++tree_at == p.tree_cap) tree_at = 0;
      book = (book + 1) & (2 * R - 1);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    if (end) break;
#pragma unroll 1
    for (int i = lane; i < rows * P; i += 32) {
      const int r = buf + i / P, q = i % P;
      const TbTopEnt* t = reinterpret_cast<const TbTopEnt*>(mem + tm.top + r * tm.top_stride);
      const uint32_t tc = t[q].tok_cls, cl = tc >> 16;
      so.plain[r][q] = make_uint4(__float_as_uint(t[q].x), bound ? __float_as_uint(rootcw[cl]) : 0u, tc & 0xFFFFu, bound ? static_cast<uint32_t>(rootdst[cl]) : 0u);
      // (no finite value left: nothing was left out.  The steps' bound is then below any finite pick, where -inf would make it no number)
      if (q == 0) { so.row[r].xb = t[M].x; so.row[r].y_next = t[P].y == -INFINITY ? -FLT_MAX : t[P].y; }
    }
    beam_group_barrier(n_threads);                                       // group n is there, group n - 1 has been read
    buf ^= R;
  }
  if (lane < K) { sh.h_hash[lane] = hh; sh.h_len[lane] = hl; }
}

// Takes the steps sidx, sidx + 1, ... like beam_team_run; returns how many.  Called by warp 0 (warp 1 serves it).
template <typename LT, int KG>
__device__ __forceinline__ int beam_solo_run(const TbBeamParams& p, BeamShared& sh, BeamSolo& so, unsigned char* dyn, int32_t sidx, const int32_t n_steps,
                                             const int32_t E, const bool recs_cached, const TeamSmem& tm) {
  constexpr int L = 32 / KG, NP = kSoloPlain / L;              // lanes per hypothesis; tokens of the reduced row per lane
  constexpr int NE = 4;                                         // 16-byte pieces (two entries) of a list that a lane has at hand
  constexpr bool kThree = KG > 4;                               // a lane keeps three candidates (else two)
  const int lane = threadIdx.x & 31, b = blockIdx.x, K = p.K, V = p.V, W = V + 1;
  const int hyp = lane / L, j = lane % L;
  const bool mine = hyp < K;                                    // this lane's hypothesis exists
  const TbSlotRec& rec = p.slots[b];
  const int n_states = rec.n_states;
  const bool bound = n_states > 0;
  const float lam = bound ? rec.lambda : 0.0f;
  const unsigned char* blob = p.arena + rec.blob_off;
  unsigned char* mem = team_base(p, dyn);
  const uint4* rsrec = !bound ? reinterpret_cast<const uint4*>(&sh.no_rec) : reinterpret_cast<const uint4*>(blob + rec.off_rsrec);
  const uint4* recs_smem = reinterpret_cast<const uint4*>(mem + tm.recs);
  const uint2* ent = reinterpret_cast<const uint2*>(blob + rec.off_rsent);
  constexpr uint32_t kTok = (1u << TB_RS_TOK_BITS) - 1u;
  constexpr int kDstBits = 32 - TB_RS_TOK_BITS;
  constexpr uint32_t kMinusInf = 0x007FFFFFu, kPlusInf = 0xFF800000u;     // order_key of the infinities
  const float lam2 = 2.0f * fabsf(lam), root_wmax = sh.root_wmax;
  // Where each candidate leads: a word per hypothesis and token, target state below the number of the step it was written in
  // (which also says whether the hypothesis lists the token).  The block's steps have their candidates there.
  unsigned char* my_lead = dyn + 4 * (mine ? hyp : 0) * W;
  const uint32_t c_own = 0xFFFFFFFFu - static_cast<uint32_t>(hyp);                           // (the lower word of a key: see beam_key)
  uint32_t stamp = so.stamp;                                    // this step's number, in the upper bits
  int e_cur = sidx % E;
  // this lane's hypothesis: score, state, whether it can be expanded, and (merging) what identifies its token sequence
  float sc = -INFINITY;
  int st = -1, hl = 0;
  bool lv = false;
  unsigned long long hh = 0ull;
  if (mine) { sc = sh.h_score[hyp]; st = sh.h_state[hyp]; lv = sh.h_live[hyp] != 0; hh = sh.h_hash[hyp]; hl = sh.h_len[hyp]; }
  if (bound && mine && j == 0 && sc != -INFINITY && (st < 0 || st >= n_states)) atomicOr(p.status, TB_STATUS_BAD_STATE);   // (read as the root)
  // its list: sum of suffix-link weights, entries, this lane's first ones
  const uint4 pad = make_uint4(2u * static_cast<uint32_t>(V), 0xFF800000u, 2u * static_cast<uint32_t>(V), 0xFF800000u);
  float D = 0.0f;
  int cnt = 0;
  const uint4* list = nullptr;
  uint4 en[NE];
  auto ask = [&](int s) {                                       // for the list of state s
    const int at = static_cast<unsigned>(s) < static_cast<unsigned>(n_states) ? s : 0;
    const uint4 r = recs_cached ? recs_smem[at] : rsrec[at];
    D = __uint_as_float(r.z);
    cnt = static_cast<int>(r.y);                                // (a multiple of four)
    list = reinterpret_cast<const uint4*>(ent + r.x) + j;
#pragma unroll
    for (int u = 0; u < NE; ++u) { en[u] = pad; if (2 * (j + u * L) < cnt) en[u] = list[u * L]; }
  };
  // the hypothesis as the next step sees it (see beam_team_run)
  auto enter = [&](bool frame_start) {
    if (frame_start) {
      if (p.merge) {
        bool dup = false;
        const uint32_t me = static_cast<uint32_t>(hh);
        bool same = false;
#pragma unroll
        for (int d = 1; d < KG; ++d) same |= (__shfl_up_sync(0xffffffffu, me, d * L) == me) & (hyp >= d);
        if (__any_sync(0xffffffffu, same && sc != -INFINITY)) {
#pragma unroll 1
          for (int d = 1; d < K; ++d) {
            const uint32_t lo = __shfl_up_sync(0xffffffffu, me, d * L), hi = __shfl_up_sync(0xffffffffu, static_cast<uint32_t>(hh >> 32), d * L);
            const int32_t lj = __shfl_up_sync(0xffffffffu, hl, d * L), sj = __shfl_up_sync(0xffffffffu, st, d * L);
            const float cj = __shfl_up_sync(0xffffffffu, sc, d * L);
            dup |= hyp >= d && cj != -INFINITY && lo == me && hi == static_cast<uint32_t>(hh >> 32) && lj == hl && sj == st;
          }
          if (dup) sc = -INFINITY;
        }
      }
      if (p.prune_delta >= 0.0f) {
        const float top1 = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(sc)));
        if (sc < __fsub_rn(top1, p.prune_delta)) sc = -INFINITY;
      }
      lv = true;
    }
    lv = lv && sc != -INFINITY;
  };
  if (lane == 0) *const_cast<volatile int32_t*>(&sh.cmd) = 0;
  __syncwarp();
  ask(st);
  enter(e_cur == 0);
  int done = 0, slot = 0, n_bar = 0;
#pragma unroll 1
  for (; sidx < n_steps; ++sidx) {
    if ((slot & (kSoloRows - 1)) == 0) { beam_group_barrier(64); ++n_bar; }
    const BeamSolo::Row ro = so.row[slot];
    const unsigned char* row = dyn + ro.at;
    stamp += 1u << kDstBits;
    if (stamp == 0u) {                                          // (the numbers begin again)
      __syncwarp();
#pragma unroll 4
      for (int i = lane; i < K * W; i += 32) reinterpret_cast<uint32_t*>(dyn)[i] = 0u;
      __syncwarp();
      stamp = 1u << kDstBits;
    }
    // ---- the lane's best candidates: largest value, then lowest token.  A lane's listed tokens come in ascending order, so among
    // them, and for the blank, which comes last of all, a tie stays with what is there.
    float v1 = -INFINITY, v2 = -INFINITY, v3 = -INFINITY, rest = -INFINITY;     // (rest: the best value that is not kept; no number if any value is none)
    uint32_t c1 = 0u, c2 = 0u, c3 = 0u;                        // the lower words of the keys
    auto keep = [&](float v, uint32_t c, bool g1, bool g2, bool g3) {           // (g: comes before the first, second, third)
      if (kThree) {
        rest = max_nan(rest, min_nan(v3, v));
        v3 = fmaxf(v3, fminf(v2, v));
        c3 = g2 ? c2 : g3 ? c : c3;
      } else {
        rest = max_nan(rest, min_nan(v2, v));
      }
      v2 = fmaxf(v2, fminf(v1, v));
      v1 = fmaxf(v1, v);
      c2 = g1 ? c1 : g2 ? c : c2;
      c1 = g1 ? c : c1;
    };
    const float msc = lv ? sc : -INFINITY;                     // (what cannot be expanded has only itself to offer)
    float pv[NP];
    uint32_t ptk[NP], pdst[NP];
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      const uint4 t = so.plain[slot][j + u * L];
      const float x = __uint_as_float(t.x);
      ptk[u] = t.z;                                            // (V or more: the row has fewer tokens)
      pdst[u] = t.w;
      pv[u] = __fadd_rn(msc, bound ? __fadd_rn(x, __fmul_rn(lam, __fadd_rn(D, __uint_as_float(t.y)))) : x);
    }
    const float scale = fabsf(sc) + fabsf(ro.y_next) + lam2 * (fabsf(D) + root_wmax);
    const float ub = (sc + ro.y_next) + lam * D + scale * 3.814697265625e-6f + 1e-30f;       // 2^-18 of the scale
    // two listed tokens
    auto listed = [&](const uint4& e) {
      const uint32_t t0 = e.x & kTok, t1 = e.z & kTok;         // 2 * token (padding carries token V and -inf)
      const float x0 = beam_smem_logit2<LT>(row, t0), x1 = beam_smem_logit2<LT>(row, t1);
      *reinterpret_cast<uint32_t*>(my_lead + 2 * t0) = stamp | (e.x >> TB_RS_TOK_BITS);
      *reinterpret_cast<uint32_t*>(my_lead + 2 * t1) = stamp | (e.z >> TB_RS_TOK_BITS);
      const float a0 = __fadd_rn(msc, __fadd_rn(x0, __uint_as_float(e.y))), a1 = __fadd_rn(msc, __fadd_rn(x1, __uint_as_float(e.w)));
      keep(a0, c_own - 16u * t0, a0 > v1, a0 > v2, a0 > v3);
      keep(a1, c_own - 16u * t1, a1 > v1, a1 > v2, a1 > v3);
    };
    listed(en[0]);
    const int n_list = lv ? cnt : 0;
    if (__any_sync(0xffffffffu, n_list > 2 * L)) {
      listed(en[1]);
      if (__any_sync(0xffffffffu, n_list > 4 * L)) {
        uint4 a = pad, c = pad;
        if (2 * (j + NE * L) < cnt) a = list[NE * L];
        if (2 * (j + NE * L + L) < cnt) c = list[NE * L + L];
        listed(en[2]); listed(en[3]);
#pragma unroll 1
        for (int i = NE * L; __any_sync(0xffffffffu, 2 * i < n_list); i += 2 * L) {
          listed(a); listed(c);
          a = c = pad;                                         // (the next ones are on their way)
          if (2 * (i + j + 2 * L) < cnt) a = list[i + 2 * L];
          if (2 * (i + j + 3 * L) < cnt) c = list[i + 3 * L];
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int u = 0; u < NP; ++u) {
      uint32_t* at = reinterpret_cast<uint32_t*>(my_lead + 4 * min(ptk[u], static_cast<uint32_t>(V)));
      const bool ok = (ptk[u] < static_cast<uint32_t>(V)) & ((*at >> kDstBits) != (stamp >> kDstBits)) & lv;
      *(ok ? at : reinterpret_cast<uint32_t*>(my_lead + 4 * V)) = stamp | pdst[u];           // (nobody reads the blank's)
      const float v = ok ? pv[u] : -INFINITY;
      const uint32_t c = c_own - 32u * ptk[u];
      keep(v, c, v > v1 || (v == v1 && c > c1), v > v2 || (v == v2 && c > c2), kThree && (v > v3 || (v == v3 && c > c3)));
    }
    {
      const float v = j == L - 1 ? (lv ? __fadd_rn(sc, ro.xb) : sc) : -INFINITY;              // the blank, or a frozen hypothesis carried
      keep(v, c_own - 32u * static_cast<uint32_t>(lv ? V : V + 1), v > v1, v > v2, v > v3);
    }
    // ---- the picks, best first: pick r is noted by the lanes of place r
    uint32_t ph = 0u, pl = 0u, kth = 0u, top1 = 0u, h1 = order_key(v1), h2 = order_key(v2), h3 = kThree ? order_key(v3) : kMinusInf;
#pragma unroll
    for (int r = 0; r < KG; ++r) {
      const uint32_t mh = __reduce_max_sync(0xffffffffu, h1);
      const uint32_t ml = __reduce_max_sync(0xffffffffu, h1 == mh ? c1 : 0u);
      const bool win = h1 == mh && c1 == ml;
      if (hyp == r) { ph = mh; pl = ml; }
      if (r == 0) top1 = mh;
      if (r == K - 1) kth = mh;
      h1 = win ? h2 : h1; c1 = win ? c2 : c1;
      h2 = win ? h3 : h2; c2 = win ? c3 : c2;
      h3 = win ? kMinusInf : h3;
    }
    // ---- the next step's hypotheses and their lists
    __syncwarp();
    const bool some = mine && ph > kMinusInf;                  // (-inf: an empty place)
    const uint32_t l2 = some ? ~pl : 0xFFFFFFFFu;
    const int tkey = static_cast<int>(l2 >> 5), parent = some ? static_cast<int>(l2 & 31u) : 0, from = some ? parent * L : lane;
    const bool emits = some && tkey < V;
    const int32_t goes = static_cast<int32_t>(reinterpret_cast<const uint32_t*>(dyn)[min(parent, K - 1) * W + min(tkey, V)] & ((1u << kDstBits) - 1u)), stays = __shfl_sync(0xffffffffu, st, from);
    const bool plv = __shfl_sync(0xffffffffu, lv ? 1 : 0, from) != 0;
    const float c_k = order_key_inv(kth);
    const bool out = h1 == kMinusInf && rest >= c_k && rest > -INFINITY;   // (this lane's are used up, and it had one more)
    // (infinite values: differences with them are no numbers.  A value that is none leaves a kept value without its token.)
    if (__any_sync(0xffffffffu, out || (lv && !(c_k > ub)) || top1 >= kPlusInf || rest != rest)) break;
    st = !some || !bound ? -1 : emits ? goes : stays;
    ask(st);
    if (mine && j == 0) so.pick[slot][hyp] = l2;
    sc = some ? order_key_inv(ph) : -INFINITY;
    lv = emits && plv;
    if (p.merge) {
      const unsigned long long nh = (static_cast<unsigned long long>(__shfl_sync(0xffffffffu, static_cast<uint32_t>(hh >> 32), from)) << 32) |
                                    __shfl_sync(0xffffffffu, static_cast<uint32_t>(hh), from);
      const int nl = __shfl_sync(0xffffffffu, hl, from) + (emits ? 1 : 0);
      hh = !some ? 0ull : emits ? beam_extend(nh, tkey) : nh;
      hl = some ? nl : 0;
    }
    ++done;
    slot = (slot + 1) & (2 * kSoloRows - 1);
    e_cur = e_cur + 1 == E ? 0 : e_cur + 1;
    if (sidx + 1 < n_steps) enter(e_cur == 0);
  }
  if (lane == 0) { so.stamp = stamp; *const_cast<volatile int32_t*>(&sh.done) = done; *const_cast<volatile int32_t*>(&sh.cmd) = n_bar + 1; }
  if (mine && j == 0) {
    if (sidx >= n_steps) {
      const int64_t o = static_cast<int64_t>(b) * K + hyp;
      p.scores[o] = sc; p.states[o] = st; p.live[o] = lv ? 1 : 0;
    }
    // (for the team or the block, should they take the next step; what a frame's start has dropped they drop as well)
    sh.h_score[hyp] = sc; sh.h_state[hyp] = st; sh.h_live[hyp] = lv ? 1 : 0;
  }
  __syncwarp();
  beam_group_barrier(64);
  return done;
}

#endif  // TB_BEAM_SOLO_CUH_
