"""The one-launch acceptance walk at the edges of its slices, against the CPU oracle."""
import numpy as np
import pytest

from test_gpu_accept import _compare, _pipeline
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
