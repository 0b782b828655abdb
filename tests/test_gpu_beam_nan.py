"""Rows with logits that are no numbers: a beam of any width goes on to the end of the call, within its arrays, and the other streams of the batch are
decoded as without them."""
import numpy as np
import pytest

from paper_2608_21343_b200 import workloads as W
from helpers import make_batch
from test_gpu_beam_narrow import _hub_lists, _logits
from test_gpu_beam_stream import run_beam_frames

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [1, 3, 4, 8, 9, 16, 32])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_other_streams_are_as_without(tb, K, dtype):
    V, T, E = 200, 24, 2
    rng = np.random.default_rng(K)
    lists = _hub_lists(V, [20, 35, 9], rng)
    x = _logits(rng, 3, T, E, V, lists, False)
    w = W.get_workload(4, B=3, T=T, V=V, S=E, K=K, dtype=dtype)
    w.vocab.case_class[:] = np.arange(V)
    outs = []
    for bad in (False, True):
        if bad:
            x[1, 5, 0, lists[1][0][0]] = np.nan                  # a listed token, another one, the blank, a whole row
            x[1, 9, 1, 3] = -np.float32(np.nan)
            x[1, 12, 0, V] = np.nan
            x[1, 15, 1, :] = np.nan
        batch, _ = make_batch(tb, w, lists, max_beam=K, max_tree_steps=T * E)
        outs.append(run_beam_frames(tb, w, dict(logits=W.to_storage(x, dtype), phrases=lists), K, lists, batch, merge=True))
    clean, dirty = outs
    for name in ("scores", "states", "lens"):
        assert np.array_equal(clean[name][[0, 2]], dirty[name][[0, 2]]), name
    for i in (0, 2):
        for k in range(K):
            assert np.array_equal(clean["tokens"][i, k, :clean["lens"][i, k]], dirty["tokens"][i, k, :clean["lens"][i, k]])
    assert dirty["lens"].min() >= 0 and dirty["lens"].max() <= T * E


# (K = 32 of V = 40, where the team's steps begin: once every place holds such a value, each kind of step has its own order for ties among them)
@pytest.mark.parametrize("V,dtype,K", [(V, d, K) for V, d in ((40, "bf16"), (200, "f32"), (301, "bf16")) for K in (1, 4, 12, 32) if (V, K) != (40, 32)])
def test_a_token_is_treated_alike_wherever_its_row_begins(tb, V, dtype, K):
    """Tokens whose logits are no numbers, at every distance from the row's aligned pieces (V + 1 elements a row): as the steps that look at whole rows have it."""
    T, E = 40, 2
    rng = np.random.default_rng([K, V])
    lists = _hub_lists(V, [9, 20, 15], rng)
    x = _logits(rng, 3, T, E, V, lists, False)
    for b in range(3):
        for t in range(3 + b, T, 7 if b else T):                 # (one row of the first stream)
            for v in rng.choice(V, size=1 + t % 3, replace=False):
                x[b, t, t % E, v] = np.nan if t & 1 else -np.float32(np.nan)
    w = W.get_workload(4, B=3, T=T, V=V, S=E, K=K, dtype=dtype)
    w.vocab.case_class[:] = np.arange(V)
    outs = []
    for flags in (0, tb.TB_FLAG_BEAM_WHOLE_ROWS):
        batch, _ = make_batch(tb, w, lists, max_beam=K, max_tree_steps=T * E)
        tb.tb_batch_set_flags(batch, flags)
        outs.append(run_beam_frames(tb, w, dict(logits=W.to_storage(x, dtype), phrases=lists), K, lists, batch, merge=True))
    few, whole = outs
    for name in ("scores", "states", "lens", "last"):
        assert np.array_equal(few[name], whole[name], equal_nan=name == "scores"), name
    for i in range(3):
        for k in range(K):
            assert np.array_equal(few["tokens"][i, k, :few["lens"][i, k]], whole["tokens"][i, k, :whole["lens"][i, k]])
