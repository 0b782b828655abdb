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
