// Beam steps of wide beams by a crew of warps, four hypotheses each (part of tb_decode.cu, behind the single warp's steps, whose parts it uses).
#ifndef TB_BEAM_CREW_CUH_
#define TB_BEAM_CREW_CUH_

// Eight lanes weigh a hypothesis' candidates as the single warp's steps do (tb_beam_solo.cuh) and keep their best three (with two the first look is shorter, but
// settles 30 of 1000 steps less in the slowest of 32 streams).  What is left is to find the K
// best of up to 3 * 256 candidates that eight warps hold in registers:
//   A. every lane's best value goes to shared memory.  The least of 32 groups' best values is a lower bound on the K-th pick; every warp counts the values that
//      reach one of as many places between it and the best, and the highest place that K reach is the bound (a search by all warps for themselves, each over
//      all values, took 1450 cycles, this one 950);
//   B. the candidates that reach it (K and about a quarter as many again) are noted with where they lead;
//   C. each is ranked by counting the keys above it, four lanes a candidate, and goes to its place.
// Four barriers of the crew a step; a ninth warp brings rows and keeps the books (beam_serve).  The team's step (beam_team_run), which takes what this one cannot,
// puts every candidate into a histogram in shared memory, goes through long lists twice, and has all of its seventeen warps keep the books: the instructions
// that four schedulers issue for it bound it (6900 cycles at K = 32); this one is bound by the latency of a step's chain, 3400 cycles at K = 12 and 4600 at K = 32.
// 32 streams of 1000 steps, V = 1024, lists of 300 phrases, merging and pruning, whole call with transcripts, by the team and so: K = 9 2617 and 1801 us,
// K = 12 2922 and 1817, K = 16 3360 and 1948, K = 24 4042 and 2163, K = 32 4442 and 2447; a chunk of 8 frames of 64 slots, two rows each, one of them
// new and one ending, with all its calls: K = 12 115 and 92 us, K = 16 126 and 97, K = 24 151 and 117, K = 32 154 and 125.
// Where a lane might have held one pick more than it keeps, or the K-th pick does not clear the bound on the tokens that were not looked at, the crew takes a second look
// (beam_crew_look).  A step that this does not settle, or with a value that is infinite or no number in it, is untouched and left to the team.
__device__ __forceinline__ void beam_crew_barrier(int n_threads) { asm volatile("bar.sync 1, %0;" ::"r"(n_threads) : "memory"); }

struct BeamCrew {
  float best[32 * kCrewWarps];                                 // every lane's best value
  __align__(16) unsigned long long place[kCrewBeam];           // the picks' keys, best first
  int32_t goes[kCrewBeam];                                     // and where they lead
  uint32_t limit[2][kCrewWarps];                                // order_key of what the K-th pick has to clear on behalf of the warp's hypotheses (0: nothing)
  int32_t reach[kCrewWarps];                                   // how many of the lanes' best values reach the warp's place
  uint32_t limit_more[kCrewWarps];                              // the same of a second look
  int32_t n_found, n_more;
};

// The places of the n candidates in sh.sk, for those that have one: each is ranked by counting the keys above it, four lanes a candidate.
__device__ __forceinline__ void beam_crew_rank(BeamShared& sh, BeamCrew& cr, const int n, const int K, const int n_warps) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (n > kSurvivors) return;
#pragma unroll 1
  for (int t0 = 8 * warp; t0 < n; t0 += 8 * n_warps) {
    const int t = min(t0 + (lane >> 2), n - 1);
    const unsigned long long key = sh.sk[t];
    int c = 0;
#pragma unroll 2
    for (int i0 = 0; i0 < n; i0 += 16) {
      const int i = i0 + 4 * (lane & 3);
      const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(&sh.sk[i]), u = *reinterpret_cast<const ulonglong2*>(&sh.sk[i + 2]);
      c += (i < n) & (o.x > key) ? 1 : 0;
      c += (i + 1 < n) & (o.y > key) ? 1 : 0;
      c += (i + 2 < n) & (u.x > key) ? 1 : 0;
      c += (i + 3 < n) & (u.y > key) ? 1 : 0;
    }
    c += __shfl_xor_sync(0xffffffffu, c, 1);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    if (c < K && (lane & 3) == 0) { cr.place[c] = key; cr.goes[c] = sh.sd[t]; }      // (the last candidate may be ranked more than once: the same)
  }
}

// A second look at a step that the first one could not settle, when a lane might have held one pick more than it keeps or the K-th pick (kth, its order_key, of those
// that were looked at; K or more have it, or it is that of -inf) does not clear the bound: all candidates of every hypothesis that reach kth -- listed tokens,
// blank, all tokens of the reduced row -- are noted and ranked, a warp a hypothesis.  The places are in cr.place then; returns how many candidates there
// were, or -1 if the step is not settled (the K-th does not clear the bound on the tokens behind the reduced row, fewer than K finite ones, too many, a value that is no
// number).
// Steps of which one hypothesis has most of the picks need it: nearly all of a beam that is pruned to one at every frame, a new stream's first, one of a hundred
// elsewhere.  They went to the team, whose run starts cold: 32 streams of 400 frames, one row each, peaked, pruned to within 1 of the best: K = 17 2170 us a call, K = 32
// 2320 (1745 and 2050 by the team alone), so 1074 and 1490; a chunk of 4 frames of 128 slots, two rows each, K = 32: 58.6 and 39.8 us.
// A function of its own: its registers do not weigh on the first look's.
template <typename LT>
__device__ __noinline__ int beam_crew_look(const TbBeamParams& p, BeamShared& sh, BeamCrew& cr, unsigned char* dyn, const unsigned char* row, const unsigned char* reduced,
                                           const uint4* recs, const uint2* ent, const float psc, const int pst, const bool plv, const uint32_t kth, const uint32_t stamp, const float lam,
                                           const float lam2, const int n_states) {
  __builtin_assume(__isShared(&sh)); __builtin_assume(__isShared(&cr)); __builtin_assume(__isShared(dyn)); __builtin_assume(__isShared(row)); __builtin_assume(__isShared(reduced));
  constexpr uint32_t kTok = (1u << TB_RS_TOK_BITS) - 1u, kMinusInf = 0x007FFFFFu;
  constexpr int kDstBits = 32 - TB_RS_TOK_BITS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, K = p.K, V = p.V, W = V + 1, M = p.top_m;
  const int n_warps = (K + 3) >> 2, crew = 32 * n_warps;
  const bool bound = n_states > 0;
  const TbTopEnt* top = reinterpret_cast<const TbTopEnt*>(reduced);
  const unsigned char* aux = dyn + ((static_cast<size_t>(K) * W * sizeof(float) + 15) & ~size_t(15)) + ((static_cast<size_t>(K) * ((W + 31) >> 5) * sizeof(uint32_t) + 15) & ~size_t(15));
  const float* rootcw = reinterpret_cast<const float*>(aux);    // (see tokview_attach)
  const int32_t* rootdst = reinterpret_cast<const int32_t*>(aux + 4 * static_cast<size_t>(p.C));
  const float least = order_key_inv(kth), xb = top[M].x, y_next = top[M].y;
  uint32_t limit = 0u;
  bool none = false;                                           // a value that is no number
#pragma unroll 1
  for (int k = warp; k < K; k += n_warps) {
    const float sc = __shfl_sync(0xffffffffu, psc, k);
    const int st = __shfl_sync(0xffffffffu, pst, k);
    const bool lv = __shfl_sync(0xffffffffu, plv ? 1 : 0, k) != 0;
    if (sc == -INFINITY) continue;
    const uint32_t c_own = 0xFFFFFFFFu - static_cast<uint32_t>(k);
    const uint32_t* lead = reinterpret_cast<const uint32_t*>(dyn) + static_cast<size_t>(k) * W;
    auto offer = [&](bool have, float v, uint32_t c, int32_t d) {
      none |= have && v != v;
      const bool yes = have && v >= least && v > -INFINITY;
      const unsigned who = __ballot_sync(0xffffffffu, yes);
      if (who == 0u) return;
      int at = shared_fetch_add(&cr.n_more, __popc(who), lane == 0);
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(who & ((1u << lane) - 1u));
      at = min(at, kSurvivors);
      const unsigned long long key = (static_cast<unsigned long long>(order_key(v)) << 32) | c;
      shared_put(&sh.sk[at], key, &sh.sd[at], d, yes);
    };
    offer(lane == 0, lv ? __fadd_rn(sc, xb) : sc, c_own - 32u * static_cast<uint32_t>(lv ? V : V + 1), st);
    if (!lv) continue;
    const uint4 r = recs[static_cast<unsigned>(st) < static_cast<unsigned>(n_states) ? st : 0];
    const float D = __uint_as_float(r.z);
#pragma unroll 1
    for (int q0 = 0; q0 < M; q0 += 32) {
      const int q = min(q0 + lane, M - 1);
      const uint32_t tc = top[q].tok_cls, tok = tc & 0xFFFFu, cl = tc >> 16;
      const float x = top[q].x, w = bound ? rootcw[cl] : 0.0f;
      const bool have = q0 + lane < M && tok < static_cast<uint32_t>(V) && (lead[min(tok, static_cast<uint32_t>(V))] >> kDstBits) != (stamp >> kDstBits);
      offer(have, __fadd_rn(sc, bound ? __fadd_rn(x, __fmul_rn(lam, __fadd_rn(D, w))) : x), c_own - 32u * tok, bound ? rootdst[cl] : 0);
    }
    const uint4* list = reinterpret_cast<const uint4*>(ent + r.x);
    const int pieces = static_cast<int>(r.y) >> 1;
#pragma unroll 1
    for (int i0 = 0; i0 < pieces; i0 += 32) {
      const bool have = i0 + lane < pieces;
      uint4 e = make_uint4(2u * static_cast<uint32_t>(V), 0xFF800000u, 2u * static_cast<uint32_t>(V), 0xFF800000u);
      if (have) e = list[i0 + lane];
      const uint32_t t0 = e.x & kTok, t1 = e.z & kTok;
      offer(have, __fadd_rn(sc, __fadd_rn(beam_smem_logit2<LT>(row, t0), __uint_as_float(e.y))), c_own - 16u * t0, static_cast<int32_t>(e.x >> TB_RS_TOK_BITS));
      offer(have, __fadd_rn(sc, __fadd_rn(beam_smem_logit2<LT>(row, t1), __uint_as_float(e.w))), c_own - 16u * t1, static_cast<int32_t>(e.z >> TB_RS_TOK_BITS));
    }
    limit = max(limit, kMinusInf);                             // (places that no finite value is left for are the general step's)
    if (y_next != -INFINITY) {
      const float scale = fabsf(sc) + fabsf(y_next) + lam2 * (fabsf(D) + sh.root_wmax);
      limit = max(limit, order_key((sc + y_next) + lam * D + scale * 3.814697265625e-6f + 1e-30f));     // (see beam_crew_run)
    }
  }
  if (__any_sync(0xffffffffu, none)) limit = 0xFFFFFFFFu;
  if (lane == 0) cr.limit_more[warp] = limit;
  beam_crew_barrier(crew);
  const int n = *const_cast<volatile int32_t*>(&cr.n_more);
  beam_crew_rank(sh, cr, n, K, n_warps);
  beam_crew_barrier(crew);
  const uint32_t last = n >= K ? static_cast<uint32_t>(cr.place[K - 1] >> 32) : kMinusInf;
  return n > kSurvivors || __any_sync(0xffffffffu, lane < n_warps && cr.limit_more[lane & (kCrewWarps - 1)] >= last) ? -1 : n;
}

// Takes the steps sidx, sidx + 1, ... like beam_team_run; returns how many.  Called by the first (K + 3) / 4 warps (the next one serves them).
template <typename LT>
__device__ __forceinline__ int beam_crew_run(const TbBeamParams& p, BeamShared& sh, BeamCrewAhead& so, BeamCrew& cr, unsigned char* dyn, int32_t sidx,
                                             const int32_t n_steps, const int32_t E, const bool recs_cached, const TeamSmem& tm) {
  constexpr int L = 8, NP = kCrewPlain / L;                     // lanes per hypothesis; tokens of the reduced row per lane
  constexpr int NE = 4;                                         // 16-byte pieces (two entries) of a list that a lane has at hand
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, b = blockIdx.x, K = p.K, V = p.V, W = V + 1;
  const int n_warps = (K + 3) >> 2, crew = 32 * n_warps;
  const int hyp = 4 * warp + lane / L, j = lane % L;
  const bool mine = hyp < K;                                    // this lane's hypothesis exists
  const TbSlotRec& rec = p.slots[b];
  const int n_states = rec.n_states;
  const bool bound = n_states > 0;
  const float lam = bound ? rec.lambda : 0.0f;
  const unsigned char* blob = p.arena + rec.blob_off;
  unsigned char* mem = team_base(p, dyn);
  const uint4* recs = !bound ? reinterpret_cast<const uint4*>(&sh.no_rec) : recs_cached ? reinterpret_cast<const uint4*>(mem + tm.recs) : reinterpret_cast<const uint4*>(blob + rec.off_rsrec);
  const uint2* ent = reinterpret_cast<const uint2*>(blob + rec.off_rsent);
  constexpr uint32_t kTok = (1u << TB_RS_TOK_BITS) - 1u;
  constexpr int kDstBits = 32 - TB_RS_TOK_BITS;
  constexpr uint32_t kMinusInf = 0x007FFFFFu, kPlusInf = 0xFF800000u;     // order_key of the infinities
  const float lam2 = 2.0f * fabsf(lam), root_wmax = sh.root_wmax, parts = 1.0f / static_cast<float>(n_warps + 1);
  unsigned char* my_lead = dyn + 4 * (mine ? hyp : 0) * W;      // where each candidate leads (see beam_solo_run); only this warp's lanes use it
  const uint32_t c_own = 0xFFFFFFFFu - static_cast<uint32_t>(hyp);                           // (the lower word of a key: see beam_key)
  uint32_t stamp = so.stamp;
  int e_cur = sidx % E;
  // lane k: hypothesis k, in every warp alike -- score, state, whether it can be expanded, and (merging) what identifies its token sequence
  float psc = -INFINITY;
  int pst = -1, phl = 0;
  bool plv = false;
  unsigned long long phh = 0ull;
  if (lane < K) { psc = sh.h_score[lane]; pst = sh.h_state[lane]; plv = sh.h_live[lane] != 0; phh = sh.h_hash[lane]; phl = sh.h_len[lane]; }
  if (bound && warp == 0 && psc != -INFINITY && (pst < 0 || pst >= n_states)) atomicOr(p.status, TB_STATUS_BAD_STATE);   // (read as the root)
  // this lane's hypothesis: score, state, whether it can be expanded; its list: sum of suffix-link weights, entries, this lane's first ones
  float sc = -INFINITY, D = 0.0f;
  int st = -1, cnt = 0;
  bool lv = false;
  const uint4 pad = make_uint4(2u * static_cast<uint32_t>(V), 0xFF800000u, 2u * static_cast<uint32_t>(V), 0xFF800000u);
  const uint4* list = nullptr;
  uint4 en[NE];
  auto ask = [&]() {                                            // for the list of the lane's hypothesis
    st = __shfl_sync(0xffffffffu, pst, hyp);
    const int at = mine && static_cast<unsigned>(st) < static_cast<unsigned>(n_states) ? st : 0;
    const uint4 r = recs[at];
    D = __uint_as_float(r.z);
    cnt = mine ? static_cast<int>(r.y) : 0;                     // (a multiple of four)
    list = reinterpret_cast<const uint4*>(ent + r.x) + j;
#pragma unroll
    for (int u = 0; u < NE; ++u) { en[u] = pad; if (2 * (j + u * L) < cnt) en[u] = list[u * L]; }
  };
  auto merge = [&]() {                                          // of equal sequences in the same state the first stays
    bool dup = false;
#pragma unroll 1
    for (int d = 1; d < K; ++d) {
      const uint32_t lo = __shfl_up_sync(0xffffffffu, static_cast<uint32_t>(phh), d), hi = __shfl_up_sync(0xffffffffu, static_cast<uint32_t>(phh >> 32), d);
      const int32_t lj = __shfl_up_sync(0xffffffffu, phl, d), sj = __shfl_up_sync(0xffffffffu, pst, d);
      const float cj = __shfl_up_sync(0xffffffffu, psc, d);
      dup |= lane >= d && cj != -INFINITY && lo == static_cast<uint32_t>(phh) && hi == static_cast<uint32_t>(phh >> 32) && lj == phl && sj == pst;
    }
    if (dup) psc = -INFINITY;
  };
  // the hypotheses as the next step sees them (see beam_team_run).  A warp looks for earlier sequences equal to its own four hypotheses' only (by
  // the low words of the hashes first): of others it needs the best score, which is the first's, and no more.
  auto enter = [&](bool frame_start, bool first) {
    if (frame_start) {
      if (p.merge) {
        if (first) {
          merge();
        } else {
          sh.hlow[lane] = psc != -INFINITY ? static_cast<uint32_t>(phh) : static_cast<uint32_t>(-1 - lane);    // (all warps write the same)
          __syncwarp();
          const uint32_t me = sh.hlow[min(hyp, 31)];
          const uint4 q = *reinterpret_cast<const uint4*>(&sh.hlow[4 * j]);
          const int i = 4 * j;
          const bool same = ((q.x == me) & (i < hyp)) | ((q.y == me) & (i + 1 < hyp)) | ((q.z == me) & (i + 2 < hyp)) | ((q.w == me) & (i + 3 < hyp));
          if (__any_sync(0xffffffffu, same)) merge();
        }
      }
      if (p.prune_delta >= 0.0f) {
        const float top1 = order_key_inv(__reduce_max_sync(0xffffffffu, order_key(psc)));
        if (psc < __fsub_rn(top1, p.prune_delta)) psc = -INFINITY;
      }
      plv = true;
    }
    plv = plv && psc != -INFINITY;
    sc = __shfl_sync(0xffffffffu, psc, hyp);
    lv = __shfl_sync(0xffffffffu, plv ? 1 : 0, hyp) != 0 && mine;
    if (!mine) sc = -INFINITY;
  };
  if (warp == 0 && lane == 0) { *const_cast<volatile int32_t*>(&sh.cmd) = 0; cr.n_found = cr.n_more = 0; }     // (seen by all after the first group barrier)
  __syncwarp();
  ask();
  enter(e_cur == 0, true);
  int done = 0, slot = 0, n_bar = 0;
#pragma unroll 1
  for (; sidx < n_steps; ++sidx) {
    if ((slot & (kCrewRows - 1)) == 0) { beam_group_barrier(crew + 32); ++n_bar; }
    const BeamCrewAhead::Row ro = so.row[slot];
    const unsigned char* row = dyn + ro.at;
    stamp += 2u << kDstBits;                                    // (the next number marks the plain tokens)
    if (stamp == 0u) {                                          // (the numbers begin again)
      __syncwarp();
#pragma unroll 4
      for (int i = lane; i < min(4, K - 4 * warp) * W; i += 32) reinterpret_cast<uint32_t*>(dyn)[4 * warp * W + i] = 0u;
      __syncwarp();
      stamp = 2u << kDstBits;
    }
    // ---- the lane's best candidates (see beam_solo_run)
    float v1 = -INFINITY, v2 = -INFINITY, v3 = -INFINITY, rest = -INFINITY;
    uint32_t c1 = 0u, c2 = 0u, c3 = 0u;
    auto keep = [&](float v, uint32_t c, bool g1, bool g2, bool g3) {
      rest = max_nan(rest, min_nan(v3, v));
      v3 = fmaxf(v3, fminf(v2, v));
      c3 = g2 ? c2 : g3 ? c : c3;
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
      *(ok ? at : reinterpret_cast<uint32_t*>(my_lead + 4 * V)) = (stamp + (1u << kDstBits)) | pdst[u];           // (nobody reads the blank's)
      const float v = ok ? pv[u] : -INFINITY;
      const uint32_t c = c_own - 32u * ptk[u];
      keep(v, c, v > v1 || (v == v1 && c > c1), v > v2 || (v == v2 && c > c2), v > v3 || (v == v3 && c > c3));
    }
    {
      const float v = j == L - 1 ? (lv ? __fadd_rn(sc, ro.xb) : sc) : -INFINITY;              // the blank, or a frozen hypothesis carried
      keep(v, c_own - 32u * static_cast<uint32_t>(lv ? V : V + 1), v > v1, v > v2, v > v3);
    }
    // ---- A. a lower bound on the K-th pick
    cr.best[32 * warp + lane] = v1;
    {
      const uint32_t l = max(lv ? order_key(ub) : 0u, rest > -INFINITY ? order_key(rest) : 0u);
      const uint32_t lim = __reduce_max_sync(0xffffffffu, rest != rest ? 0xFFFFFFFFu : l);
      if (lane == 0) cr.limit[sidx & 1][warp] = lim;
    }
    // (where the lane's candidates lead: tokens through the table, others stay)
    auto leads = [&](uint32_t c) {
      const uint32_t tkey = (c_own - c) >> 5;
      const int32_t to = static_cast<int32_t>(*reinterpret_cast<const uint32_t*>(my_lead + 4 * min(tkey, static_cast<uint32_t>(V))) & ((1u << kDstBits) - 1u));
      return tkey < static_cast<uint32_t>(V) ? to : st;
    };
    __syncwarp();
    const int32_t d1 = leads(c1), d2 = leads(c2), d3 = leads(c3);
    beam_crew_barrier(crew);
    float floor_v;
    uint32_t top1;
    {
      float q[kCrewWarps], m = -INFINITY;
#pragma unroll
      for (int i = 0; i < kCrewWarps; ++i) { q[i] = i < n_warps ? cr.best[32 * i + lane] : -INFINITY; m = fmaxf(m, q[i]); }
      top1 = __reduce_max_sync(0xffffffffu, order_key(m));
      const float lo = order_key_inv(__reduce_min_sync(0xffffffffu, order_key(m))), range = order_key_inv(top1) - lo;     // (32 values reach lo)
      // every warp counts the values that reach one place between it and the best
      const float part = range * parts, mid = lo + static_cast<float>(warp + 1) * part;
      int c = 0;
#pragma unroll
      for (int i = 0; i < kCrewWarps; ++i) c += q[i] >= mid ? 1 : 0;
      c = __reduce_add_sync(0xffffffffu, c);
      if (lane == 0) cr.reach[warp] = c;
      beam_crew_barrier(crew);
      const int ok = __popc(__ballot_sync(0xffffffffu, lane < n_warps && cr.reach[lane & (kCrewWarps - 1)] >= K));
      floor_v = ok > 0 ? lo + static_cast<float>(ok) * part : lo;
    }
    // ---- B. the candidates that reach it
    const unsigned b1 = __ballot_sync(0xffffffffu, v1 >= floor_v && v1 > -INFINITY), b2 = __ballot_sync(0xffffffffu, v2 >= floor_v && v2 > -INFINITY),
                   b3 = __ballot_sync(0xffffffffu, v3 >= floor_v && v3 > -INFINITY);
    const int n1 = __popc(b1), n2 = __popc(b2), n_mine = n1 + n2 + __popc(b3);
    int at = shared_fetch_add(&cr.n_found, n_mine, lane == 0);
    at = __shfl_sync(0xffffffffu, at, 0);
    const unsigned below = (1u << lane) - 1u;
    auto note = [&](unsigned who, int o, float v, uint32_t c, int32_t d) {
      o = min(o + __popc(who & below), kSurvivors);
      const unsigned long long key = (static_cast<unsigned long long>(order_key(v)) << 32) | c;
      shared_put(&sh.sk[o], key, &sh.sd[o], d, (who >> lane) & 1u);
    };
    note(b1, at, v1, c1, d1);
    note(b2, at + n1, v2, c2, d2);
    note(b3, at + n1 + n2, v3, c3, d3);
    beam_crew_barrier(crew);
    // ---- C. their ranks
    int n = *const_cast<volatile int32_t*>(&cr.n_found);
    beam_crew_rank(sh, cr, n, K, n_warps);
    beam_crew_barrier(crew);
    // ---- the next step's hypotheses and their lists
    unsigned long long key = lane < min(n, K) ? cr.place[lane] : 0ull;
    // (infinite values: differences with them are no numbers; limit 0: nothing was left out)
    const uint32_t kth = n >= K ? __shfl_sync(0xffffffffu, static_cast<uint32_t>(key >> 32), K - 1) : kMinusInf;
    const uint32_t limit = __reduce_max_sync(0xffffffffu, lane < n_warps ? cr.limit[sidx & 1][lane & (kCrewWarps - 1)] : 0u);
    if (n > kSurvivors || max(top1, limit) >= kPlusInf) break;
    if (limit >= kth) {
      n = beam_crew_look<LT>(p, sh, cr, dyn, row, mem + tm.top + slot * tm.top_stride, recs, ent, psc, pst, plv, kth, stamp, lam, lam2, bound ? n_states : 0);
      if (n < 0) break;
      key = lane < min(n, K) ? cr.place[lane] : 0ull;
    }
    const bool some = lane < min(n, K);
    const uint32_t l2 = some ? ~static_cast<uint32_t>(key) : 0xFFFFFFFFu;
    const int tkey = static_cast<int>(l2 >> 5), from = some ? static_cast<int>(l2 & 31u) : lane;
    const bool emits = some && tkey < V;
    if (warp == 0) {
      if (lane == 0) cr.n_found = cr.n_more = 0;
      if (lane < K) so.pick[slot][lane] = l2;
    }
    pst = some && bound ? cr.goes[lane] : -1;
    ask();
    psc = some ? beam_key_value(key) : -INFINITY;
    plv = emits;
    if (p.merge) {
      const unsigned long long nh = (static_cast<unsigned long long>(__shfl_sync(0xffffffffu, static_cast<uint32_t>(phh >> 32), from)) << 32) |
                                    __shfl_sync(0xffffffffu, static_cast<uint32_t>(phh), from);
      const int nl = __shfl_sync(0xffffffffu, phl, from) + (emits ? 1 : 0);
      phh = !some ? 0ull : emits ? beam_extend(nh, tkey) : nh;
      phl = some ? nl : 0;
    }
    ++done;
    slot = (slot + 1) & (2 * kCrewRows - 1);
    e_cur = e_cur + 1 == E ? 0 : e_cur + 1;
    if (sidx + 1 < n_steps) enter(e_cur == 0, false);
  }
  if (warp == 0) {
    if (lane == 0) { so.stamp = stamp; *const_cast<volatile int32_t*>(&sh.done) = done; *const_cast<volatile int32_t*>(&sh.cmd) = n_bar + 1; }
    if (lane < K) {
      if (sidx >= n_steps) {
        const int64_t o = static_cast<int64_t>(b) * K + lane;
        p.scores[o] = psc; p.states[o] = pst; p.live[o] = plv ? 1 : 0;
      }
      // (for the team or the block, should they take the next step; at a frame's start they merge and drop for themselves)
      sh.h_score[lane] = psc; sh.h_state[lane] = pst; sh.h_live[lane] = plv ? 1 : 0;
    }
  }
  __syncwarp();
  beam_group_barrier(crew + 32);
  return done;
}

#endif  // TB_BEAM_CREW_CUH_
