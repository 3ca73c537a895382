"""The one-launch acceptance walk at the edges of its slices, against the CPU oracle."""
import numpy as np
import pytest

import paper_2406_16858_b200 as e2
from harness import gpu_accept
from oracle import ref
from test_gpu_accept import _compare, _pipeline
from workloads import generators as gen
from workloads import get_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,B", [
    (32, 1),          # most of the only block's warps hold nothing
    (2048, 2), (2049, 2),        # one block with the shortest slice, and one token more (unaligned rows)
    (16384, 40), (16388, 40),    # more sequences than clusters: longest slice, one block or two
    (131072, 1), (131071, 1),    # the largest vocabulary the registers hold
    (131076, 1),                 # one that they do not
])
def test_walk_at_slice_edges(V, B):
    cfg = get_config("tiny", V=V, B=B, k=4, D=3, m=16)
    draft, sel, target, ua, ub = _pipeline(cfg, 11)
    _compare(cfg, draft, sel, target, ua, ub, 1.0)
    _compare(cfg, draft, sel, target, ua, ub, 0.7, point_mass=True)


@pytest.mark.parametrize("V,B,temperature,shift", [
    (33, 8, 1.0, -300.0),      # warps beyond the vocabulary have no maximum of their own
    (2052, 8, 1.0, -300.0),    # the second block holds four tokens
    (28676, 4, 0.05, -20.0),   # the last block does
])
def test_logits_far_below_zero(V, B, temperature, shift):
    """A softmax does not see an offset of its logits, however far below zero it takes them all."""
    cfg = get_config("tiny", V=V, B=B, k=4, D=3, m=16)
    draft, sel, target, ua, ub = _pipeline(cfg, 12)
    target, draft = target + np.float32(shift), draft + np.float32(shift)
    _compare(cfg, draft, sel, target, ua, ub, temperature)
    _compare(cfg, draft, sel, target, ua, ub, temperature, point_mass=True)


@pytest.mark.parametrize("V,B", [(33, 8), (2052, 8), (32000, 4), (131071, 2)])
@pytest.mark.parametrize("kind", ["masked", "mostly_masked", "flat", "one_huge", "far_below", "far_above"])
def test_logits_of_any_size(V, B, kind):
    """Rows whose tokens are excluded by the lowest number a float holds, whole warps of them, and rows far from zero."""
    cfg = get_config("tiny", V=V, B=B, k=4, D=3, m=16)
    rng = np.random.default_rng(V)
    lowest, highest = np.finfo(np.float32).min, np.finfo(np.float32).max
    at = int(rng.integers(0, V - 8))
    out = rng.random(V) < 0.9  # tokens excluded in every row
    out[at:at + 8] = False
    if kind == "masked":  # a run of tokens and a few others stay
        out[:] = True
        out[at:at + 8 + V // 50] = False
        out[rng.integers(0, V, 8)] = False

    def change(rows):
        if kind == "one_huge":
            rows[..., at] = highest
        elif kind.startswith("far"):  # steps of 1 to 4 between neighbouring numbers
            rows[:] = np.round(rows) * 4 + np.float32((-1 if kind == "far_below" else 1) * 2.0 ** 24)
        elif kind == "flat":  # nothing but the mask: every token is as likely as any other (to the oracle, of logits 0)
            rows[:] = 0.0
        else:
            rows[..., out] = lowest
        return rows

    draft = change(gen.draft_rows(cfg, 14))
    tree = ref.build_tree(draft, V, cfg.k, cfg.D)
    sel = ref.rerank(tree.token, tree.parent, tree.value, cfg.k, cfg.D, cfg.m)
    target = change(gen.target_rows(cfg, 14, draft, tree.parent, sel.index))
    ua, ub = gen.uniforms(cfg, 14)
    on_device = (lambda rows: np.full_like(rows, lowest)) if kind == "flat" else None
    for temperature in (1.0, 1.5):
        for point_mass in (False, True):
            _compare(cfg, draft, sel, target, ua, ub, temperature, point_mass=point_mass, on_device=on_device)


@pytest.mark.parametrize("V", [1004, 131076])  # the walk, and the two launches
@pytest.mark.parametrize("index", [10 ** 6, -1, 2 ** 31 - 1])
def test_a_selection_outside_the_tree_is_reported(V, index):
    """A child's candidate index says which draft row proposed it; one that is no node of the tree raises the status,
    and the other sequences are not touched by it."""
    cfg = get_config("tiny", V=V, B=3, k=4, D=3, m=16)
    draft, sel, target, ua, ub = _pipeline(cfg, 15)
    want = ref.accept(target, draft, sel, V, cfg.k, cfg.D, cfg.m, 1.0, ua, ub)
    bad = sel.index.copy()
    bad[1, :2] = index
    alen, apath, _, st = gpu_accept(target, draft, bad, sel.parent, sel.token, sel.n_sel, V, cfg.k, cfg.D, cfg.m, 1.0, ua, ub)
    assert st == e2.STATUS_BAD_TREE
    assert 0 <= alen[1] <= cfg.D and (apath[1] < cfg.m).all()
    for b in (0, 2):
        assert want.margins[b, 0] > 1e-6
        assert alen[b] == want.acc_len[b] and (apath[b] == want.acc_path[b]).all()


@pytest.mark.parametrize("V,B", [(1004, 8), (1001, 8), (32000, 1), (131076, 2)])
@pytest.mark.parametrize("point_mass", [False, True])
@pytest.mark.parametrize("temperature", [0.0, 1.0])
def test_bad_logits_on_the_walk_raise_the_status(V, B, point_mass, temperature):
    """NaN, +inf and a row of -inf, in a row that the walk reaches (a target row or the draft row of its children): the
    status, as the oracle has it.  A row that no walk reaches may be reported or not, and changes nothing else."""
    cfg = get_config("tiny", V=V, B=B, k=4, D=3, m=16)
    draft, sel, target, ua, ub = _pipeline(cfg, 16)
    args = (sel.index, sel.parent, sel.token, sel.n_sel, V, cfg.k, cfg.D, cfg.m, temperature, ua, ub)
    with_draft = temperature > 0 and not point_mass
    good = gpu_accept(target, draft if with_draft else None, *args)
    assert good[3] == 0
    b = B - 1
    stop = int(good[1][b, good[0][b] - 1]) if good[0][b] else -1  # the node where the walk ends
    off = next(x for x in range(cfg.m) if (sel.parent[b] == x).any() and x not in good[1][b])  # expanded, not on the walk

    def status(rows, b, row, bad):
        kept = rows[b, row].copy()
        if bad == "row":
            rows[b, row] = -np.inf
        else:
            rows[b, row, V - 3] = bad
        got = gpu_accept(target, draft if with_draft else None, *args)
        want = ref.accept(target, draft if with_draft else None, sel, V, cfg.k, cfg.D, cfg.m, temperature, ua, ub)
        rows[b, row] = kept
        return got, want

    kinds = [np.nan] if temperature == 0 else [np.nan, np.inf, "row"]  # (an arg-max needs no finite values)
    for bad in kinds:
        for rows, row in [(target, 0), (target, stop + 1)] + ([(draft, 0)] if with_draft else []):
            got, want = status(rows, b, row, bad)
            assert want.status == ref.ST_NONFINITE_LOGIT and got[3] == e2.STATUS_NONFINITE_LOGIT, (bad, row)
        got, want = status(target, b, off + 1, bad)
        assert want.status == 0 and got[3] in (0, e2.STATUS_NONFINITE_LOGIT)
        if temperature > 0 and V <= 131072:
            assert got[3] == 0
        for mine, was in zip(got[:3], good[:3]):
            assert (mine == was).all()


@pytest.mark.parametrize("V,B", [(1004, 40), (1001, 40), (32000, 8), (131076, 3)])
@pytest.mark.parametrize("lead", [14.0, 18.0, 40.0])
def test_a_proposal_that_one_child_nearly_fills(V, B, lead):
    """Behind a first child with all but a little of the draft's mass the second is tested against its share of what is
    left, which one minus the first child's probability does not say in 32 bits."""
    cfg = get_config("tiny", V=V, B=B, k=4, D=3, m=16)
    rng = np.random.default_rng(V)
    base = (2.0 * rng.standard_normal((B, ref.n_draft_rows(cfg.k, cfg.D), V))).astype(np.float32)
    base[..., :4] += 9.0  # four likely tokens
    draft = base.copy()
    np.put_along_axis(draft, draft.argmax(-1)[..., None], draft.max(-1, keepdims=True) + np.float32(lead), -1)
    tree = ref.build_tree(draft, V, cfg.k, cfg.D)
    sel = ref.rerank(tree.token, tree.parent, tree.value, cfg.k, cfg.D, cfg.m)
    target = gen.target_rows(cfg, 3, base, tree.parent, sel.index)
    ua, ub = gen.uniforms(cfg, 3)
    _, want = _compare(cfg, draft, sel, target, ua, ub, 1.0)
    tested = np.isfinite(want.accept_prob).sum(axis=1)
    assert (tested > want.acc_len + 1).any()  # a second child was tested at some node
