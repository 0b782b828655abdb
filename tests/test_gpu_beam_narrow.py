"""Parity of narrow beams (steps by one warp) with the CPU oracle where that warp's layout has its edges: lists at and around
what a lane has at hand, vocabularies at the line to the team's steps, step counts around the groups that rows are brought in,
every width, ties, and more steps than its step numbers count."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2608_21343_b200 import workloads as W
from helpers import SCORE_TOL, make_batch, oracle_graph
from test_gpu_beam_stream import run_beam_frames

pytestmark = pytest.mark.gpu


def _hub_lists(V, sizes, rng):
    """Per stream: one first token followed by `size` different second tokens, some of those by a third."""
    lists = []
    for n in sizes:
        hub, *rest = rng.permutation(V)[: n + 1].tolist()
        lists.append([[hub, t] for t in rest] + [[hub, t, rest[0]] for t in rest[: n // 3]] + [[rest[0]]])
    return lists


def _check(tb, w, x, dtype, K, lists, prune=None, **kw):
    data = dict(logits=W.to_storage(x, dtype), phrases=lists)
    batch, _ = make_batch(tb, w, lists, max_beam=K, max_tree_steps=x.shape[1] * x.shape[2])
    if prune is not None:
        tb.tb_batch_set_beam_prune(batch, prune)
    out = run_beam_frames(tb, w, data, K, lists, batch, **kw)
    tol = SCORE_TOL * max(1.0, x.shape[1] * x.shape[2] / 1000)      # (float32 sums of the same terms in the same order)
    for i in range(len(lists)):
        ref = O.beam_decode(oracle_graph(w, lists[i]), data["logits"][i], K, prune_delta=-1.0 if prune is None else prune, **kw)
        assert np.array_equal(out["states"][i], ref["states"]) and np.array_equal(out["lens"][i], ref["lens"]), i
        for k in range(K):
            assert np.array_equal(out["tokens"][i, k, :ref["lens"][k]], ref["tokens"][k]), (i, k)
        fin = np.isfinite(ref["scores"])
        assert np.array_equal(np.isfinite(out["scores"][i]), fin)
        assert np.all(np.abs(out["scores"][i][fin] - ref["scores"][fin]) <= tol)


def _logits(rng, B, T, E, V, lists, coarse):
    x = rng.standard_normal((B, T, E, V + 1)).astype(np.float32)
    x[..., V] += 3.0
    for b, p in enumerate(lists):
        x[b, ::2, 0, p[0][0]] += 5.0                          # the hub is entered again and again
        x[b, 1::2, 0, p[-1][0]] += 2.0
    return np.round(x * 4) / 4 if coarse else x


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 8])
@pytest.mark.parametrize("V,dtype", [(63, "bf16"), (64, "f32"), (65, "bf16"), (300, "bf16"), (2046, "f32"), (2046, "bf16")])
@pytest.mark.parametrize("coarse", [False, True])
def test_lists_around_what_a_lane_holds(tb, K, V, dtype, coarse):
    rng = np.random.default_rng([K, V, coarse])
    sizes = [n for n in (1, 7, 8, 9, 16, 17, 32, 33, 63, 64, 65, 130, 257) if n < V - 1]
    lists = _hub_lists(V, sizes, rng)
    x = _logits(rng, len(sizes), 17, 2, V, lists, coarse)
    w = W.get_workload(4, B=len(sizes), T=17, V=V, S=2, K=K, dtype=dtype)
    w.vocab.case_class[:] = np.arange(V)
    _check(tb, w, x, dtype, K, lists, merge=bool(K & 1))


@pytest.mark.parametrize("K", [2, 4, 8])
@pytest.mark.parametrize("T,E", [(1, 1), (1, 2), (1, 3), (4, 1), (5, 1), (2, 2), (7, 1), (4, 2), (3, 3), (33, 1)])
def test_step_counts_around_the_groups(tb, K, T, E):
    rng = np.random.default_rng([K, T, E])
    lists = _hub_lists(200, [5, 40, 12], rng)
    x = _logits(rng, 3, T, E, 200, lists, False)
    w = W.get_workload(4, B=3, T=T, V=200, S=E, K=K, dtype="bf16")
    w.vocab.case_class[:] = np.arange(200)
    lists[1] = None
    _check(tb, w, x, "bf16", K, lists, merge=T % 2 == 0, prune=2.0 if T > 3 else None)


@pytest.mark.parametrize("K", [3, 8])
def test_more_steps_than_the_step_numbers_count(tb, K):
    rng = np.random.default_rng(K)
    lists = _hub_lists(70, [20, 35], rng)
    x = _logits(rng, 2, 4200, 1, 70, lists, True)
    w = W.get_workload(4, B=2, T=4200, V=70, S=1, K=K, dtype="f32")
    w.vocab.case_class[:] = np.arange(70)
    _check(tb, w, x, "f32", K, lists, merge=True)
