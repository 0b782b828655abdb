"""Parity of the steps that look at whole rows with the CPU oracle: a batch that asks for them, lists that are walked (in every stream, or beside
resolved ones and none), and rows whose picks come from few threads of the block."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2608_21343_b200 import workloads as W
from helpers import SCORE_TOL, make_batch, oracle_graph
from test_gpu_beam_narrow import _hub_lists, _logits
from test_gpu_beam_stream import run_beam_frames

pytestmark = pytest.mark.gpu


def _walked_list(V, rng, n=530):
    """States whose lists come to more entries than are laid out: n of them end in the state that lists n tokens."""
    hub, *rest = rng.permutation(V)[:2 * n + 1].tolist()
    return [[hub, t] for t in rest[:n]] + [[t, hub] for t in rest[n:]]


def _check(tb, x, dtype, K, lists, flags=0, prune=-1.0):
    B, T, E, Wd = x.shape
    w = W.get_workload(4, B=B, T=T, V=Wd - 1, S=E, K=K, dtype=dtype)
    w.vocab.case_class[:] = np.arange(Wd - 1)
    data = dict(logits=W.to_storage(x, dtype), phrases=lists)
    batch, _ = make_batch(tb, w, lists, max_beam=K, max_tree_steps=T * E)
    tb.tb_batch_set_flags(batch, flags)
    tb.tb_batch_set_beam_prune(batch, prune)
    out = run_beam_frames(tb, w, data, K, lists, batch, merge=True)
    for i in range(B):
        ref = O.beam_decode(oracle_graph(w, lists[i]), data["logits"][i], K, prune_delta=prune, merge=True)
        assert np.array_equal(out["states"][i], ref["states"]) and np.array_equal(out["lens"][i], ref["lens"]), i
        for k in range(K):
            assert np.array_equal(out["tokens"][i, k, :ref["lens"][k]], ref["tokens"][k]), (i, k)
        fin = np.isfinite(ref["scores"])
        assert np.array_equal(np.isfinite(out["scores"][i]), fin)
        assert np.all(np.abs(out["scores"][i][fin] - ref["scores"][fin]) <= SCORE_TOL)


@pytest.mark.parametrize("K", [1, 5, 9, 32])
@pytest.mark.parametrize("V,dtype", [(3, "f32"), (31, "bf16"), (544, "f32"), (1089, "bf16"), (2500, "bf16")])
@pytest.mark.parametrize("step", [0.0, 0.25, 2.0])              # every value alike; many ties; few, with most picks from a few tokens
def test_picks_of_few_threads(tb, K, V, dtype, step):
    if K * (V + 1) * 4 > 150 * 1024:
        K = 9
    rng = np.random.default_rng([K, V])
    lists = [None] + _hub_lists(V, [1, min(20, V - 2)], rng)
    x = _logits(rng, 3, 12, 2, V, lists[1:] + lists[1:2], False)
    x = np.round(x / step) * step if step else np.zeros_like(x)
    x[:, 8:, :, V // 2:V] -= 6.0
    _check(tb, x.astype(np.float32), dtype, K, lists, flags=tb.TB_FLAG_BEAM_WHOLE_ROWS, prune=4.0 if step else -1.0)


@pytest.mark.parametrize("K", [1, 4, 12, 32])
@pytest.mark.parametrize("mixed", [False, True])
def test_walked_lists(tb, K, mixed):
    V = 1100
    rng = np.random.default_rng(K)
    lists = [_walked_list(V, rng), _walked_list(V, rng)] + ([None] + _hub_lists(V, [40], rng) if mixed else [])
    x = _logits(rng, len(lists), 14, 2, V, [p or [[0]] for p in lists], False)
    _check(tb, x, "bf16", K, lists)
