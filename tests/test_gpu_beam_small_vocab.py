"""Parity of beam steps over small vocabularies with the CPU oracle: fewer tokens than a step looks at or has places, on both sides of the line between the
team's steps and a crew's."""
import numpy as np
import pytest

from paper_2608_21343_b200 import workloads as W
from test_gpu_beam_narrow import _check
from test_gpu_beam_paths import _steps

pytestmark = pytest.mark.gpu


def _inputs(K, V, E, coarse):
    rng = np.random.default_rng([K, V, E])
    lists = [[[int(t) for t in rng.integers(0, V, size=n)] for n in (1, 2, 3, 3)] for _ in range(3)]
    lists[1] = None
    x = rng.standard_normal((3, 30, E, V + 1)).astype(np.float32)
    x[..., V] += 1.0
    x[2, 5::4, :, :V // 2] = -np.inf
    return np.round(x * 2) / 2 if coarse else x, lists


@pytest.mark.parametrize("K", [1, 4, 8, 9, 17, 32])
@pytest.mark.parametrize("V,dtype", [(1, "f32"), (2, "bf16"), (7, "f32"), (9, "bf16"), (15, "f32"), (16, "bf16"), (17, "f32"), (28, "bf16"), (45, "f32")])
@pytest.mark.parametrize("E,coarse", [(1, False), (2, True)])
def test_against_the_oracle(tb, K, V, dtype, E, coarse):
    x, lists = _inputs(K, V, E, coarse)
    w = W.get_workload(4, B=3, T=30, V=V, S=E, K=K, dtype=dtype, n_plants=0)
    w.vocab.case_class[:] = np.arange(V)
    _check(tb, w, x, dtype, K, lists, merge=True, prune=None if coarse else 4.0)


@pytest.mark.parametrize("K,V,who", [(8, 16, "warps"), (9, 15, "team"), (9, 28, "warps"), (32, 15, "team"), (32, 63, "warps")])
def test_who_takes_the_steps(tb, K, V, who):
    x, lists = _inputs(K, V, 2, False)
    assert _steps(tb, x[:2], "f32", K, lists[:2])[who] > 0.9
