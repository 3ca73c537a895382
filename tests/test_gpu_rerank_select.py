"""The selection of the best nodes at the edges of its groups, its candidate list and its budget, against the CPU oracle."""
import numpy as np
import pytest

from harness import GpuSelection, dev, host
from oracle import ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,D,m", [
    (1, 1, 1), (4, 3, 36), (4, 3, 128),     # everything is wanted
    (10, 6, 1), (10, 6, 64), (10, 6, 65), (10, 6, 128),  # groups of four threads, of two
    (16, 3, 60), (16, 5, 64),               # 528 nodes: two per thread; 1040
    (32, 4, 100), (31, 5, 128),             # 3104, 3875: more nodes than the candidate list
])
@pytest.mark.parametrize("values", ["normal", "ties", "equal", "masked"])
def test_selection_of_any_tree(k, D, m, values):
    B, N = 2, ref.n_nodes(k, D)
    rng = np.random.default_rng(N + m)
    parent = np.full((B, N), -1, np.int32)
    for i in range(k, N):  # children of k nodes of the level before
        level = (i - k) // (k * k)
        lo, n = (0, k) if level == 0 else (k + (level - 1) * k * k, k * k)
        parent[:, i] = lo + (i - k) % (k * k) // k * (n // k)
    value = np.zeros((B, N))
    step = -rng.random((B, N))
    if values == "ties":
        step = np.round(step * 4) / 4
    elif values == "equal":
        step[:] = 0.0
    elif values == "masked":
        step[rng.random((B, N)) < 0.9] = -np.inf
    for i in range(N):
        p = parent[:, i]
        value[:, i] = step[:, i] + np.where(p >= 0, value[np.arange(B), np.maximum(p, 0)], 0.0)
    token = rng.integers(0, 1000, (B, N)).astype(np.int32)
    want = ref.rerank(token, parent, value, k, D, m)
    got = GpuSelection(dev(token), dev(parent), dev(value), B, k, D, m)
    assert int(got.status.item()) == want.status == 0
    assert (host(got.index) == want.index).all() and (host(got.parent) == want.parent).all()
    assert (host(got.n_sel) == want.n_sel).all()
