"""Expansion with a cluster per row at the edges of its slices and of its rule, against the CPU oracle."""
import numpy as np
import pytest

import paper_2406_16858_b200 as e2
from harness import GpuTree, dev, host
from oracle import ref

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,k,D,B", [
    (33, 32, 2, 1),          # one block whose warps are mostly empty
    (1024, 1, 4, 2), (1028, 3, 3, 2),
    (4096, 10, 3, 1), (4097, 10, 3, 3),    # one block of 16 tokens per thread, and one token more (unaligned rows)
    (32768, 10, 2, 16),      # 160 rows of the longest slices that still go this way
    (131072, 10, 2, 2), (131071, 4, 2, 1),  # the largest vocabulary the registers hold
    (131076, 4, 2, 1),       # one that they do not
    (16388, 8, 3, 17),       # 136 rows
])
@pytest.mark.parametrize("values", ["normal", "ties", "masked"])
def test_rows_at_slice_edges(V, k, D, B, values):
    rng = np.random.default_rng(V + k)
    draft = (2.0 * rng.standard_normal((B, ref.n_draft_rows(k, D), V))).astype(np.float32)
    if values == "ties":  # few distinct logits: more candidates than a block ranks, ties to the lower token
        draft = np.round(draft / 3) * np.float32(3)
    elif values == "masked":  # most tokens excluded
        draft[rng.random(draft.shape) < 0.97] = -np.inf
        draft[..., :: max(1, V // (2 * k))] = rng.standard_normal(draft[..., :: max(1, V // (2 * k))].shape)
    want = ref.build_tree(draft, V, k, D)
    got = GpuTree(B, V, k, D).expand_all(dev(draft))
    assert int(got.status.item()) == want.status == 0
    finite = np.isfinite(want.value)
    assert (host(got.token) == want.token).all()
    assert (np.isfinite(host(got.value)) == finite).all()
    assert np.abs(host(got.value)[finite] - want.value[finite]).max() <= 1e-5 * np.abs(want.value[finite]).max()
    if values == "normal":  # (tied values may be ranked either way: their sums round differently)
        assert (host(got.parent) == want.parent).all()
        assert (host(got.frontier) == want.frontier).all()


def test_a_nan_or_a_row_of_minus_inf_raises_the_status():
    V, k, D = 32000, 10, 1
    for bad in (np.nan, np.inf, -np.inf):
        draft = np.zeros((1, 1, V), np.float32)
        draft[0, 0] = bad if bad == -np.inf else draft[0, 0]
        draft[0, 0, 31000] = bad
        got = GpuTree(1, V, k, D).expand_all(dev(draft))
        assert int(got.status.item()) & e2.STATUS_NONFINITE_LOGIT


@pytest.mark.parametrize("V,k,D,B", [
    (33, 4, 2, 1), (4097, 10, 3, 3), (20000, 10, 2, 2), (131071, 4, 2, 1),  # rows held by a cluster
    (131076, 4, 2, 1), (70004, 5, 2, 32),  # tiles: one per block, and streamed
])
@pytest.mark.parametrize("kind", ["run", "scattered", "flat", "one_huge"])
def test_tokens_masked_with_the_lowest_float(V, k, D, B, kind):
    """Masks often are the lowest number a float holds: whole threads, warps and blocks of such tokens weigh nothing."""
    rng = np.random.default_rng(V + k)
    lowest = np.finfo(np.float32).min
    draft = (2.0 * rng.standard_normal((B, ref.n_draft_rows(k, D), V))).astype(np.float32)
    if kind == "run":  # a run of tokens stays
        at = int(rng.integers(0, V - 4 * k))
        draft[..., :at] = draft[..., at + 4 * k:] = lowest
    elif kind == "scattered":  # of the others some are at -inf
        draft[rng.random(draft.shape) < 0.8] = lowest
        draft[rng.random(draft.shape) < 0.3] = -np.inf
        draft[..., :: max(1, V // (2 * k))] = rng.standard_normal(draft[..., :: max(1, V // (2 * k))].shape)
    elif kind == "flat":  # nothing but the mask
        draft[:] = lowest
    else:
        draft[..., V // 2] = -lowest
    want = ref.build_tree(draft, V, k, D)
    got = GpuTree(B, V, k, D).expand_all(dev(draft))
    assert int(got.status.item()) == want.status == 0
    assert (host(got.token) == want.token).all()
    assert np.abs(host(got.value) - want.value).max() <= 1e-5 * np.abs(want.value).max()
    assert (host(got.frontier) == want.frontier).all()


def test_a_nan_among_excluded_tokens_raises_the_status():
    """Also where every other token of the warps around it is at -inf, or masked."""
    for V, B in ((32000, 1), (131076, 1), (70004, 32)):
        for rest in (-np.inf, np.finfo(np.float32).min):
            draft = np.full((B, 1, V), rest, np.float32)
            draft[:, 0, :8] = 1.0
            draft[B - 1, 0, V - 5000:V - 1000] = np.nan
            got = GpuTree(B, V, 4, 1).expand_all(dev(draft))
            assert int(got.status.item()) & e2.STATUS_NONFINITE_LOGIT
