"""Performance cases: the work that a user of this library has it do, through the public calls of ``binding``.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes what a recogniser has in
hand before the call (logits on the device, compiled and bound lists), ``run`` is one pass: an utterance batch, or one
chunk of a streaming session.  Inputs follow the library's synthetic workloads (``workloads``): N(0,1) token logits,
blank +3, phrases with Zipf-distributed classes, some of them planted in the logits in random casing; they are drawn
on the GPU because they are large.

Kinds of case:
  greedy      a batch of utterances, lists bound before the pass            (tb_greedy_decode)
  fresh       the same where every stream brings a new list: compile, bind, decode in the pass
  beam        a batch of utterances by beam search with transcripts         (tb_beam_frames, tb_beam_backtrace)
  chunk       one chunk of a streaming session, RNNT or TDT, with the streams that start with it  (tb_stream_chunk_binds)
  beam_chunk  one chunk of a streaming beam search, with the streams that start and end with it   (tb_beam_chunk, ...)
"""
import math

import numpy as np
import torch

from paper_2608_21343_b200 import binding as tb
from paper_2608_21343_b200 import workloads as W

GREEDY = dict(kind="greedy", S=3, dtype="bf16", lists="tokens", shared=0, len_lo=1, len_hi=6, plants=20, ragged=False,
              log_softmax=False)
ENDLESS = 1 << 30      # valid_frames of a live stream: its end is not known yet
ROTATION = 8           # chunks of logits a streaming session cycles through (a joint network's ring of buffers)


def listed():
    return [
        # The smallest offline call: a few short utterances, full-precision logits, small vocabulary (configuration 1).
        dict(GREEDY, name="greedy_tiny_f32", B=4, T=100, V=256, dtype="f32", phrases=10, len_hi=4, plants=10),
        # The production batch: 128 streams of a minute, a list of 100 phrases each (configuration 2, the headline).
        dict(GREEDY, name="greedy_batch", B=128, T=750, V=1024, phrases=100),
        # Large personal lists: 1000 own phrases and 4000 shared distractors per stream (configuration 3).
        dict(GREEDY, name="greedy_large_lists", B=64, T=750, V=1024, phrases=1000, shared=4000, len_lo=3, len_hi=10, plants=50),
        # Logits as a joint network without reduced precision leaves them (fp32), utterances of different lengths.
        dict(GREEDY, name="greedy_f32", B=32, T=500, V=1024, dtype="f32", phrases=100, ragged=True),
        # A multilingual vocabulary (the largest the library takes), a small batch of half a minute.
        dict(GREEDY, name="greedy_wide_vocab", B=16, T=375, V=8192, phrases=200, ragged=True),
        # Lists given as text over a piece vocabulary (every casing and segmentation), scores normalised per row.
        dict(GREEDY, name="greedy_text_log_softmax", B=64, T=750, V=1019, lists="text", phrases=100, log_softmax=True),
        # A new session's streams bring their own lists: compile and bind are paid in the pass.
        dict(GREEDY, name="fresh_lists", kind="fresh", B=16, T=250, V=1024, phrases=500, plants=10),
        # Beam search over an utterance batch with transcripts (configuration 4), and as wide as the library goes with
        # equal transcripts merged and the beam pruned.
        dict(kind="beam", name="beam_4", B=32, T=500, E=2, V=1024, K=4, dtype="bf16", phrases=300, plants=20, merge=False, prune=-1.0),
        dict(kind="beam", name="beam_32", B=32, T=500, E=2, V=1024, K=32, dtype="bf16", phrases=300, plants=20, merge=True, prune=10.0),
        # Streaming: the busy server (512 slots, TDT, five new streams with a chunk: configuration 5), and a small one
        # (RNNT, a new stream now and then), where the latency of one call is what counts.
        dict(kind="chunk", name="stream_tdt_512", slots=512, chunk=8, S=3, V=1024, n_dur=5, dtype="bf16", phrases=500, new=5, every=1),
        dict(kind="chunk", name="stream_rnnt_16", slots=16, chunk=8, S=3, V=1024, n_dur=0, dtype="bf16", phrases=200, new=1, every=7),
        # Streaming beam search: 128 slots, one stream ends and one starts with each chunk.
        dict(kind="beam_chunk", name="stream_beam_128", slots=128, chunk=8, E=2, V=1024, K=4, dtype="bf16", phrases=500, new=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["greedy", "greedy", "greedy", "greedy", "fresh", "beam", "beam", "chunk", "chunk", "beam_chunk"])
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    if kind in ("greedy", "fresh"):
        c = dict(GREEDY, kind=kind, B=_log(rng, 1, 160), T=_log(rng, 40, 900), S=rng.choice([1, 2, 3, 3, 4]), V=_log(rng, 200, 8192),
                 dtype=dtype, phrases=_log(rng, 10, 400), len_hi=rng.randint(4, 8), plants=rng.randint(5, 30), ragged=rng.random() < 0.5)
        most = 590e6               # the bytes of greedy_batch's logits
        if kind == "fresh":
            c.update(B=_log(rng, 1, 24), T=_log(rng, 40, 300), phrases=_log(rng, 20, 500), plants=5)
        elif rng.random() < 0.15:
            c.update(shared=_log(rng, 500, 3500), phrases=_log(rng, 100, 1000), B=_log(rng, 1, 64), V=_log(rng, 500, 2000), len_lo=3, len_hi=10)
        elif rng.random() < 0.2:   # (text lists: V is what the piece vocabulary of about that size comes to)
            c.update(lists="text", V=_log(rng, 200, 1800), B=_log(rng, 1, 64), log_softmax=rng.random() < 0.5, dtype="bf16", phrases=_log(rng, 20, 150))
        elif rng.random() < 0.25:
            c.update(V=_log(rng, 200, 2040), dtype="bf16", log_softmax=True)
        row = c["S"] * (c["V"] + 1) * (2 if c["dtype"] == "bf16" else 4)
        c["T"] = min(c["T"], int(2.5e6 / c["V"]))     # (greedy_wide_vocab is the longest sequence of wide rows)
        c["B"] = max(1, min(c["B"], int(most / (row * c["T"]))))
        return c
    if kind == "beam":
        K = rng.choice([1, 2, 3, 4, 4, 5, 8, 8, 12, 16, 32])
        return dict(kind=kind, B=_log(rng, 1, 32), T=_log(rng, 30, 400), E=rng.choice([1, 2, 2]), V=_log(rng, 200, 2000), K=K, dtype=dtype,
                    phrases=_log(rng, 20, 300), plants=10, merge=rng.random() < 0.5, prune=rng.choice([-1.0, 10.0]))
    if kind == "chunk":
        slots = _log(rng, 1, 512)
        n_dur = rng.choice([0, 0, 5, 5, 3])
        return dict(kind=kind, slots=slots, chunk=rng.choice([2, 4, 8, 8, 13, 16]), S=rng.choice([1, 2, 3, 3]), V=_log(rng, 200, 3000), n_dur=n_dur,
                    dtype=dtype, phrases=_log(rng, 20, 500), new=max(1, slots // 100), every=1 if slots >= 64 else 5)
    return dict(kind=kind, slots=_log(rng, 2, 128), chunk=rng.choice([4, 8, 8, 12]), E=rng.choice([1, 2, 2]), V=_log(rng, 200, 2000),
                K=rng.choice([2, 4, 4, 8, 16, 32]), dtype=dtype, phrases=_log(rng, 20, 400), new=1)


# ------------------------------------------------------------------------------------------------ inputs

def _flat(phrases):
    """A list of token lists as the (tokens, offsets) arrays a server holds."""
    offs = np.zeros(len(phrases) + 1, dtype=np.int64)
    offs[1:] = np.cumsum([len(p) for p in phrases])
    return np.fromiter((t for p in phrases for t in p), dtype=np.int32, count=int(offs[-1])), offs


def _join(a, b):
    return np.concatenate([a[0], b[0]]), np.concatenate([a[1], b[1][1:] + a[1][-1]])


def _workload(c, seed):
    return W.get_workload(2, seed=int(seed), V=c["V"], n_phrases=c["phrases"], len_lo=c.get("len_lo", 1), len_hi=c.get("len_hi", 6))


def _normals(shape, dtype, g):
    return torch.empty(shape, dtype=torch.bfloat16 if dtype == "bf16" else torch.float32, device="cuda").normal_(generator=g)


def _logits(shape, V, dtype, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    x = _normals(shape, dtype, g)
    x[..., V] += W.BLANK_BIAS
    return x


def _plant(x, V, plants, T, rng, spell):
    """Writes `plants` spelled phrases per stream into rows (t, 0) of x [B, T, S, W]: the token's logit becomes the row's
    largest other one less a margin of U[0, 1.5]; the blank of row (t, 1) gets a further +3."""
    B, S = x.shape[0], x.shape[2]
    plants = min(plants, T // 4)
    if plants <= 0:
        return
    seg = T // plants
    bs, ts, ks = [], [], []
    for b in range(B):
        for i in range(plants):
            toks = spell(b)[:seg]
            t0 = i * seg + int(rng.integers(0, max(1, seg - len(toks) + 1)))
            bs += [b] * len(toks)
            ts += range(t0, t0 + len(toks))
            ks += toks
    b, t, k = (torch.tensor(v, device="cuda") for v in (bs, ts, ks))
    margin = torch.from_numpy(rng.uniform(0.0, 1.5, len(ks)).astype(np.float32)).cuda()
    for lo in range(0, len(ks), 4096):
        s = slice(lo, lo + 4096)
        rows = x[b[s], t[s], 0, : V + 1].float()
        rows.scatter_(1, k[s, None], -math.inf)
        x[b[s], t[s], 0, k[s]] = (rows.max(1).values - margin[s]).to(x.dtype)
    if S > 1:
        x[b, t, 1, V] += W.BLANK_BIAS


def _token_speller(w, lists, rng, near_miss):
    v = w.vocab

    def spell(b):
        p = lists[b][int(rng.integers(0, len(lists[b])))]
        mode = int(rng.integers(0, 3))         # as listed (lower), upper, title
        toks = [v.recase(t, 1 if mode == 1 else 2 if mode == 2 and i == 0 else 0) for i, t in enumerate(p)]
        if near_miss and len(toks) > 1 and rng.random() < 1.0 / 3:     # a few leading tokens, then something else
            keep = int(rng.integers(1, min(3, len(toks) - 1) + 1))
            toks = toks[:keep] + [v.token_of(int(rng.integers(0, v.n_classes)))]
        return toks
    return spell


def _arena(n, phrases, text=False):
    per = (1 << 20) if text else 65536 + max(900 * phrases, int(min(2.6e6, 5 * phrases ** 2)) + 500 * phrases)
    return n * per + (8 << 20)


def _out(B, n, dev="cuda", durs=False, cursors=False):
    """The result tensors, which a decoder allocates once and passes in again."""
    o = dict(tokens=torch.zeros((B, n), dtype=torch.int32, device=dev), frames=torch.zeros((B, n), dtype=torch.int32, device=dev),
             counts=torch.zeros(B, dtype=torch.int32, device=dev), scores=torch.zeros(B, device=dev),
             states=torch.zeros(B, dtype=torch.int32, device=dev))
    if durs:
        o["durs"] = torch.zeros((B, n), dtype=torch.int32, device=dev)
    if cursors:
        o["cursors"] = torch.zeros(B, dtype=torch.int32, device=dev)
    return o


def _prepare_greedy(c, seed):
    rng = np.random.default_rng([int(seed), 101])
    B, T, S = c["B"], c["T"], c["S"]
    if c["lists"] == "text":
        merged = max(20, int((c["V"] - 52) / 1.73))
        pieces = W.make_piece_vocab(int(seed), letters=26, merged=merged, max_len=5)
        V = len(pieces)
        lists = [W.draw_string_phrases(int(seed) * 1000 + b, pieces, c["phrases"], 1, 4) for b in range(B)]
        cc, _ = tb.tb_piece_classes(pieces)
        graphs = [tb.tb_graph_compile_variative(p, pieces, tau=1.0) for p in lists]

        def spell(b):
            return W.random_spelling(rng, lists[b][int(rng.integers(0, len(lists[b])))], pieces)
        arena = _arena(B, c["phrases"], text=True)
    else:
        w = _workload(c, seed)
        V, cc = c["V"], w.vocab.case_class
        n_of = [c["phrases"] if c["kind"] == "greedy" else int(rng.integers(max(1, c["phrases"] // 10), c["phrases"] + 1)) for _ in range(B)]
        lists = [W.draw_phrases(w, np.random.default_rng([int(seed), 1, b]), n_of[b]) for b in range(B)]
        flat = [_flat(p) for p in lists]
        if c["shared"]:
            extra = _flat(W.draw_phrases(w, np.random.default_rng([int(seed), 2]), c["shared"]))
            flat = [_join(f, extra) for f in flat]
        graphs = None if c["kind"] == "fresh" else [tb.tb_graph_compile(f, V, case_class=cc) for f in flat]
        spell = _token_speller(w, lists, rng, bool(c["shared"]))
        arena = _arena(B, c["phrases"] + c["shared"]) * (2 if c["kind"] == "fresh" else 1)
    batch = tb.tb_batch_create(V, cc, B, arena_bytes=arena)
    if c["log_softmax"]:
        tb.tb_batch_set_flags(batch, tb.TB_FLAG_LOG_SOFTMAX)
    x = _logits((B, T, S, V + 1), V, c["dtype"], seed)
    _plant(x, V, c["plants"], T, rng, spell)
    lengths = torch.from_numpy(rng.integers((T + 1) // 2, T + 1, size=B).astype(np.int32)).cuda() if c["ragged"] else None
    s = dict(kind=c["kind"], batch=batch, logits=x, lengths=lengths, out=_out(B, T * S))
    if c["kind"] == "fresh":
        s.update(flat=flat, V=V, case_class=cc, slots=list(range(B)))
    else:
        tb.tb_batch_bind_streams(batch, list(range(B)), graphs)
    return s


def _prepare_beam(c, seed):
    rng = np.random.default_rng([int(seed), 102])
    w = _workload(c, seed)
    B, T, E, V, K = c["B"], c["T"], c["E"], c["V"], c["K"]
    lists = [W.draw_phrases(w, np.random.default_rng([int(seed), 1, b]), c["phrases"]) for b in range(B)]
    batch = tb.tb_batch_create(V, w.vocab.case_class, B, max_beam=K, max_tree_steps=T * E, arena_bytes=_arena(B, c["phrases"]))
    tb.tb_batch_bind_streams(batch, list(range(B)), [tb.tb_graph_compile(_flat(p), V, case_class=w.vocab.case_class) for p in lists])
    tb.tb_batch_set_beam_prune(batch, c["prune"])
    x = _logits((B, T, E, V + 1), V, c["dtype"], seed)
    _plant(x, V, c["plants"], T, rng, _token_speller(w, lists, rng, False))
    s = dict(kind="beam", batch=batch, logits=x, merge=c["merge"], T=T, **_beam_arrays(B, K))
    s.update(scores0=s["scores"].clone(), states0=s["states"].clone())
    return s


def _beam_arrays(B, K):
    scores = torch.full((B, K), -math.inf, device="cuda")
    states = torch.full((B, K), -1, dtype=torch.int32, device="cuda")
    scores[:, 0], states[:, 0] = 0.0, 0
    return dict(scores=scores, states=states, live=torch.zeros((B, K), dtype=torch.uint8, device="cuda"),
                parent=torch.zeros((B, K), dtype=torch.int32, device="cuda"), token=torch.zeros((B, K), dtype=torch.int32, device="cuda"))


def _prepare_stream(c, seed):
    """A session under way: every slot bound, the chunks' logits on the device, graphs for the streams to come compiled."""
    rng = np.random.default_rng([int(seed), 103])
    w = _workload(c, seed)
    n, V, beam = c["slots"], c["V"], c["kind"] == "beam_chunk"
    rows, width = (c["E"], V + 1) if beam else (c["S"], V + 1 + c["n_dur"])
    kw = dict(max_beam=c["K"], max_tree_steps=3000) if beam else {}
    batch = tb.tb_batch_create(V, w.vocab.case_class, n, arena_bytes=2 * _arena(n, c["phrases"]), **kw)
    lo = max(1, c["phrases"] // 10)
    graphs = []
    for b in range(n + 32):
        p = W.draw_phrases(w, np.random.default_rng([int(seed), 1, b]), int(rng.integers(lo, c["phrases"] + 1)))
        graphs.append(tb.tb_graph_compile(_flat(p), V, case_class=w.vocab.case_class))
    tb.tb_batch_bind_streams(batch, list(range(n)), graphs[:n])
    x = _logits((ROTATION, n, c["chunk"], rows, width), V, c["dtype"], seed)
    s = dict(kind=c["kind"], batch=batch, chunks=list(x.unbind(0)), graphs=graphs, slots=n, new=c["new"], at=0)
    if beam:
        tb.tb_batch_set_beam_prune(batch, 10.0)
        s.update(_beam_arrays(n, c["K"]), K=c["K"], ended=[], n_frames=torch.full((n,), c["chunk"], dtype=torch.int32, device="cuda"),
                 found=(torch.zeros((c["new"], c["K"], 256), dtype=torch.int32, device="cuda"), torch.zeros((c["new"], c["K"]), dtype=torch.int32, device="cuda")))
        tb.tb_beam_start_slots(batch, None, s["scores"], s["states"], s["live"])
    else:
        s.update(n_dur=c["n_dur"], every=c["every"], out=_out(n, c["chunk"] * c["S"], durs=True, cursors=True),
                 valid=torch.full((n,), ENDLESS, dtype=torch.int32, device="cuda"))
    return s


def prepare(case, seed):
    kind = case["kind"]
    return (_prepare_beam if kind == "beam" else _prepare_stream if kind in ("chunk", "beam_chunk") else _prepare_greedy)(case, seed)


# ------------------------------------------------------------------------------------------------ passes

def run(s):
    batch, kind = s["batch"], s["kind"]
    if kind == "greedy":
        return tb.tb_greedy_decode(batch, s["logits"], lengths=s["lengths"], out=s["out"])
    if kind == "fresh":
        graphs = [tb.tb_graph_compile(f, s["V"], case_class=s["case_class"]) for f in s["flat"]]
        tb.tb_batch_bind_streams(batch, s["slots"], graphs)
        return tb.tb_greedy_decode(batch, s["logits"], lengths=s["lengths"], out=s["out"])
    scores, states, live = (s.get(k) for k in ("scores", "states", "live"))
    if kind == "beam":
        scores.copy_(s["scores0"])
        states.copy_(s["states0"])
        tb.tb_beam_reset(batch)
        tb.tb_beam_frames(batch, s["logits"], s["merge"], scores, states, live, s["parent"], s["token"])
        tb.tb_apply_final_weights(batch, scores, states)
        tokens, lens = tb.tb_beam_backtrace(batch, scores.shape[0], scores.shape[1], s["T"])
        return dict(scores=scores, states=states, live=live, parent=s["parent"], token=s["token"], tokens=tokens, lens=lens)
    at = s["at"]
    s["at"] = at + 1
    n, new = s["slots"], s["new"]
    x = s["chunks"][at % len(s["chunks"])]
    if kind == "chunk":
        binds = []
        if at % s["every"] == 0:
            first = (at // s["every"]) * new
            binds = [(first + i) % n for i in range(new)]
        graphs = [s["graphs"][(at * new + i) % len(s["graphs"])] for i in range(len(binds))]
        return tb.tb_stream_chunk_binds(batch, binds, graphs, x, s["n_dur"], s["valid"], out=s["out"])
    if s["ended"]:                                       # new streams on the slots whose streams ended with the last chunk
        tb.tb_batch_bind_streams(batch, s["ended"], [s["graphs"][(at * new + i) % len(s["graphs"])] for i in range(new)])
        tb.tb_beam_start_slots(batch, s["ended"], scores, states, live)
    tb.tb_beam_chunk(batch, x, True, s["n_frames"], scores, states, live, s["parent"], s["token"])
    s["ended"] = ended = [(at * new + i) % n for i in range(new)]
    tb.tb_apply_final_weights_slots(batch, ended, scores, states)
    tokens, lens = tb.tb_beam_backtrace_slot_list(batch, ended, s["K"], 256, out=s["found"])
    return dict(scores=scores, states=states, live=live, parent=s["parent"], token=s["token"], tokens=tokens, lens=lens)


def work(case):
    """Bytes: the rows of logits that a row-by-row decode visits (about 1.5 per frame where a frame has more than one: a
    blank row each, and half the frames a token; TDT skips about half the frames), what it emits, and the lists' tokens
    where they are compiled in the pass.  A beam visits every row.  Operations: two per logit and hypothesis."""
    c = case
    size = 2 if c["dtype"] == "bf16" else 4
    if c["kind"] in ("greedy", "fresh"):
        frames = c["B"] * c["T"] * (0.75 if c["ragged"] else 1.0)
        rows, width, K = frames * (1.5 if c["S"] > 1 else 1.0), c["V"] + 1, 1
        out = 8 * 0.6 * frames + 12 * c["B"] + (c["B"] * c["phrases"] * 4 * 2 if c["kind"] == "fresh" else 0)
    elif c["kind"] == "beam":
        rows, width, K = c["B"] * c["T"] * c["E"], c["V"] + 1, c["K"]
        out = c["B"] * K * (4.0 * c["T"] + 25)
    elif c["kind"] == "chunk":
        frames = c["slots"] * c["chunk"]
        rows, width, K = frames * (0.8 if c["n_dur"] else 1.5 if c["S"] > 1 else 1.0), c["V"] + 1 + c["n_dur"], 1
        out = 12 * 0.6 * frames + 20 * c["slots"]
    else:
        rows, width, K = c["slots"] * c["chunk"] * c["E"], c["V"] + 1, c["K"]
        out = c["slots"] * K * 17.0 + 1024.0 * K * c["new"]
    return {"bytes": rows * width * size + out, "flops": 2.0 * rows * width * K}


def tolerance(case):
    """Tokens, frames and graph states are whole numbers and the same; scores are float32 sums in a stated order, the
    normalised ones with a float32 normaliser per row."""
    if case.get("log_softmax"):
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    return {"rel": 1e-6, "max": 1e-5, "differ": 0.0}
