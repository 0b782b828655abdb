"""Parity of lists that are walked along the suffix chain (graphs too large for resolved lists) with the CPU oracle, for chain states whose entries are
around what the walk asks for at once (four groups of 32), and lists around what a row's lanes ask for at once."""
import numpy as np
import pytest

from paper_2608_21343_b200 import workloads as W
from test_gpu_rows import _check, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("S", [1, 3])
def test_chain_states_of_many_entries(tb, S, dtype):
    sizes = [1, 31, 32, 33, 64, 127, 128, 129, 160, 255, 256, 257, 300]
    V = 700
    w, data = _inputs(5, len(sizes), 260, S, V, dtype, n_phrases=200, n_shared=2600, len_lo=3, len_hi=10)
    rng = np.random.default_rng(S)
    lists = []
    for i, (p, n) in enumerate(zip(data["phrases"], sizes)):
        hub, lead, *rest = rng.permutation(V)[: n + 2].tolist()
        lists.append(list(p) + [[hub, t] for t in rest] + [[lead, hub, rest[0]], [lead, hub, rest[-1], hub]])
        x = data["logits"] if dtype == "f32" else W.bf16_bits_to_f32(data["logits"])
        x[i, ::4, 0, lead] += 5.0                               # lead, hub: the hub's list is a suffix state's
        x[i, 1::4, 0, hub] += 6.0
        data["logits"] = W.to_storage(x, dtype)
    _check(tb, w, data, lists=lists, what="fan-out")
