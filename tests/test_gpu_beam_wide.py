"""Parity of wide beams (steps by a crew of warps, four hypotheses each) with the CPU oracle where the crew's layout has its edges: widths
around the warps' shares, lists at and around what a lane has at hand, vocabularies at the line to the team's steps and where room ends,
step counts around the groups that rows are brought in, ties, few finite values, and more steps than its step numbers count."""
import numpy as np
import pytest

from paper_2608_21343_b200 import workloads as W
from test_gpu_beam_narrow import _check, _hub_lists, _logits

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [9, 12, 13, 16, 17, 31, 32])
@pytest.mark.parametrize("V,dtype", [(63, "bf16"), (64, "f32"), (300, "bf16"), (1100, "bf16"), (1100, "f32")])
@pytest.mark.parametrize("coarse", [False, True])
def test_widths_and_lists(tb, K, V, dtype, coarse):
    rng = np.random.default_rng([K, V, coarse])
    sizes = [n for n in (1, 8, 16, 17, 32, 33, 63, 65, 130) if n < V - 1]
    lists = _hub_lists(V, sizes, rng)
    x = _logits(rng, len(sizes), 13, 2, V, lists, coarse)
    w = W.get_workload(4, B=len(sizes), T=13, V=V, S=2, K=K, dtype=dtype)
    w.vocab.case_class[:] = np.arange(V)
    _check(tb, w, x, dtype, K, lists, merge=bool(K & 1))


@pytest.mark.parametrize("K", [10, 32])
@pytest.mark.parametrize("T,E", [(1, 1), (1, 2), (1, 3), (4, 1), (5, 1), (7, 1), (4, 2), (3, 3), (33, 1)])
def test_step_counts_around_the_groups(tb, K, T, E):
    rng = np.random.default_rng([K, T, E])
    lists = _hub_lists(200, [5, 40, 12], rng)
    x = _logits(rng, 3, T, E, 200, lists, False)
    w = W.get_workload(4, B=3, T=T, V=200, S=E, K=K, dtype="bf16")
    w.vocab.case_class[:] = np.arange(200)
    lists[1] = None
    _check(tb, w, x, "bf16", K, lists, merge=T % 2 == 0, prune=2.0 if T > 3 else None)


@pytest.mark.parametrize("K", [11, 32])
def test_few_finite_values(tb, K):
    rng = np.random.default_rng(K)
    lists = _hub_lists(100, [20, 35], rng)
    x = _logits(rng, 2, 40, 2, 100, lists, True)
    x[:, 8:16][rng.random(x[:, 8:16].shape) < 0.97] = -np.inf      # a few tokens a row
    x[:, 16:, :, :100][rng.random(x[:, 16:, :, :100].shape) < 0.8] = -np.inf
    x[:, :, :, 100] = np.maximum(x[:, :, :, 100], 0)
    w = W.get_workload(4, B=2, T=40, V=100, S=2, K=K, dtype="f32")
    w.vocab.case_class[:] = np.arange(100)
    _check(tb, w, x, "f32", K, lists, merge=True, prune=6.0)


def test_more_steps_than_the_step_numbers_count(tb):
    rng = np.random.default_rng(9)
    lists = _hub_lists(70, [20, 35], rng)
    x = _logits(rng, 2, 4200, 1, 70, lists, True)
    w = W.get_workload(4, B=2, T=4200, V=70, S=1, K=9, dtype="f32")
    w.vocab.case_class[:] = np.arange(70)
    _check(tb, w, x, "f32", 9, lists, merge=True)


@pytest.mark.parametrize("K", [9, 17, 25, 32])
@pytest.mark.parametrize("V,dtype", [(64, "bf16"), (300, "f32"), (1100, "bf16")])
@pytest.mark.parametrize("prune,coarse", [(0.0, False), (0.0, True), (0.5, False), (1.0, True)])
def test_frames_of_few_hypotheses(tb, K, V, dtype, prune, coarse):
    """One hypothesis, or a few, with most of a step's picks: lists around a warp's share of a second look (64 entries), rows of few finite tokens, and rows without."""
    rng = np.random.default_rng([K, V, coarse])
    sizes = [n for n in (1, 17, 62, 63, 66, 130, 260) if n < V - 1]
    lists = _hub_lists(V, sizes, rng)
    x = _logits(rng, len(sizes), 24, 1, V, lists, coarse)
    x[:, 1::3, :, V] += 6.0
    x[:, 4::5, :, :V][rng.random(x[:, 4::5, :, :V].shape) < 0.8] = -np.inf
    w = W.get_workload(4, B=len(sizes), T=24, V=V, S=1, K=K, dtype=dtype)
    w.vocab.case_class[:] = np.arange(V)
    _check(tb, w, x, dtype, K, lists, merge=True, prune=prune)


def test_more_equal_candidates_than_a_second_look_ranks(tb):
    rng = np.random.default_rng(4)
    lists = _hub_lists(1100, [500, 511, 640, 900], rng)
    x = np.zeros((4, 12, 1, 1101), np.float32)
    for b, p in enumerate(lists):
        x[b, ::2, 0, p[0][0]] = 9.0                           # the hub, and then every listed token alike
    w = W.get_workload(4, B=4, T=12, V=1100, S=1, K=32, dtype="f32")
    w.vocab.case_class[:] = np.arange(1100)
    _check(tb, w, x, "f32", 32, lists, merge=True, prune=0.0)
