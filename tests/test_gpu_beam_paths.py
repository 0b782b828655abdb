"""Which kind of step takes a beam's steps (tb_batch_beam_steps): the comparisons with the oracle hold whichever does, so they would not notice one that is never
taken."""
import numpy as np
import pytest

from paper_2608_21343_b200 import workloads as W
from helpers import make_batch
from test_gpu_beam_narrow import _hub_lists, _logits
from test_gpu_beam_stream import run_beam_frames
from test_gpu_beam_whole import _walked_list

pytestmark = pytest.mark.gpu


def _steps(tb, x, dtype, K, lists, flags=0, prune=-1.0):
    B, T, E, Wd = x.shape
    w = W.get_workload(4, B=B, T=T, V=Wd - 1, S=E, K=K, dtype=dtype)
    w.vocab.case_class[:] = np.arange(Wd - 1)
    batch, _ = make_batch(tb, w, lists, max_beam=K, max_tree_steps=T * E)
    tb.tb_batch_set_flags(batch, flags)
    tb.tb_batch_set_beam_prune(batch, prune)
    assert tb.tb_batch_beam_steps(batch) == dict(warps=0, team=0, block=0)
    run_beam_frames(tb, w, dict(logits=W.to_storage(x, dtype), phrases=lists), K, lists, batch, merge=True)
    n = tb.tb_batch_beam_steps(batch)
    assert sum(n.values()) == B * T * E
    return {k: v / (B * T * E) for k, v in n.items()}


@pytest.mark.parametrize("K", [1, 4, 5, 8, 9, 16, 17, 32])
@pytest.mark.parametrize("V,dtype", [(64, "f32"), (300, "bf16"), (1100, "bf16")])
def test_ordinary_rows_go_by_a_warp_or_a_crew(tb, K, V, dtype):
    rng = np.random.default_rng([K, V])
    lists = [None] + _hub_lists(V, [9, 40], rng)
    assert _steps(tb, _logits(rng, 3, 100, 2, V, lists[1:] + lists[1:2], False), dtype, K, lists)["warps"] > 0.95


@pytest.mark.parametrize("K", [1, 4, 8, 12])
def test_rows_of_few_finite_tokens_too(tb, K):
    rng = np.random.default_rng(K)
    lists = _hub_lists(300, [9, 40], rng)
    x = _logits(rng, 2, 100, 2, 300, lists, False)
    x[..., :300][rng.random(x[..., :300].shape).argsort(-1).argsort(-1) >= 14] = -np.inf
    assert _steps(tb, x, "bf16", K, lists)["warps"] > 0.95


@pytest.mark.parametrize("K", [1, 8, 16])
def test_what_goes_by_the_block(tb, K):
    rng = np.random.default_rng(K)
    x = _logits(rng, 2, 10, 2, 2500, [[[1]]] * 2, False)
    assert _steps(tb, x, "bf16", K, _hub_lists(2500, [9, 40], rng))["block"] == 1.0             # more tokens than lists are laid out for
    x = np.ascontiguousarray(x[..., :1101])
    lists = _hub_lists(1100, [9, 40], rng)
    assert _steps(tb, x, "bf16", K, lists, flags=tb.TB_FLAG_BEAM_WHOLE_ROWS)["block"] == 1.0
    assert _steps(tb, x, "bf16", K, [_walked_list(1100, rng), _walked_list(1100, rng)])["block"] == 1.0
    assert _steps(tb, x, "bf16", K, [_walked_list(1100, rng), lists[0]])["block"] == pytest.approx(0.5, abs=0.05)


@pytest.mark.parametrize("K", [9, 17, 24, 32])
@pytest.mark.parametrize("prune", [0.0, 1.0])
def test_frames_that_begin_with_one_hypothesis_go_by_a_crew(tb, K, prune):
    rng = np.random.default_rng(K)
    lists = [None] + _hub_lists(300, [9, 40], rng)
    x = _logits(rng, 3, 100, 1, 300, lists[1:] + lists[1:2], False)
    x[..., 300] += 5.0
    assert _steps(tb, x, "bf16", K, lists, prune=prune)["warps"] > 0.95


def test_new_streams_of_wide_beams_go_by_a_crew(tb):
    rng = np.random.default_rng(3)
    lists = [None] + _hub_lists(300, [9, 40], rng)
    assert _steps(tb, _logits(rng, 3, 1, 2, 300, lists[1:] + lists[1:2], False), "bf16", 32, lists)["warps"] == 1.0
