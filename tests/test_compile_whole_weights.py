"""Lists without token weights take short cuts in the compiler (suffix sums from the suffix state, class bits before a look at a state's arcs): the
graph and its device records are those of the same list with every weight spelled out as 1, and of the oracle's compiler."""
import os

import numpy as np
import pytest

from oracle import oracle as O
from test_library_host import ARRAYS


def _lists(kind, rng):
    if kind == "deep":                                          # chains of hundreds of suffix states
        return 40, [[3] * 255, [3, 4] * 120, [4, 3, 3], [3, 3, 4]]
    if kind == "fan":                                           # classes that share a bit, in states of more than sixteen arcs
        return 1000, [[7, v] for v in range(0, 1000, 3)] + [[9, 7, v] for v in range(64)] + [[9, 7, v, 7, v + 64] for v in range(0, 640, 64)]
    V = int(rng.integers(2, 300))
    return V, [rng.integers(0, min(V, 9), size=rng.integers(1, 8)).tolist() for _ in range(300)]


@pytest.mark.parametrize("kind", ["deep", "fan", 0, 1, 2, 3])
def test_graph_is_the_same_as_with_weights_of_one(tb, tmp_path, kind):
    V, lists = _lists(kind, np.random.default_rng(kind if isinstance(kind, int) else 9))
    files = []
    for name, weights in (("none", None), ("ones", [[1.0] * len(p) for p in lists])):
        g = tb.tb_graph_compile(lists, V, token_weights=weights, lam=1.25)
        tb.tb_graph_save(g, str(tmp_path / name))
        files.append(open(os.path.join(tmp_path, name), "rb").read())
        view, ref = g.view(), O.Graph(lists, V, lam=1.25)
        for a in ARRAYS:
            assert np.array_equal(view[a], getattr(ref, a)), (name, a)
    assert files[0] == files[1]
