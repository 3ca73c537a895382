"""The launch that finishes a step from the LM head's partial results: few parts, and more equal keys than it lists."""
import numpy as np
import pytest
import torch

import paper_2406_16858_b200 as e2
from harness import DEV, host, make_ws, new_status

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,V,k,equal", [(1, 16, 16, False), (2, 130, 4, False), (3, 20000, 16, False), (1, 300, 1, False),
                                         (2, 20000, 16, True), (9, 20000, 16, True)])
def test_step_from_partial_results(B, V, k, equal):
    H, D = 64, 3
    N = k + (D - 1) * k * k
    g = torch.Generator(device=DEV).manual_seed(V + k)
    weight = torch.randn((V, H), generator=g, device=DEV).to(torch.bfloat16)
    trees = []
    for fused in (True, False):
        token, parent = (torch.zeros((B, N), dtype=torch.int32, device=DEV) for _ in range(2))
        value = torch.zeros((B, N), dtype=torch.float64, device=DEV)
        frontier, status = torch.zeros((B, k), dtype=torch.int32, device=DEV), new_status()
        ws = make_ws(max(e2.workspace_bytes(op, B=B, V=V, k=k, D=D) for op in (e2.OP_EXPAND, e2.OP_LM_HEAD_EXPAND)))
        g.manual_seed(7)
        for s in range(D):
            n = k if s else 1
            hidden = torch.randn((B * n, H), generator=g, device=DEV).to(torch.bfloat16)
            if equal:
                hidden.zero_()  # every logit is 0: ties go to the lowest tokens
            if fused:
                e2.lm_head_expand(hidden, weight, H, B, V, k, D, s, token, parent, value, frontier, ws, status)
            else:
                logits = torch.zeros((B * n, V), device=DEV)
                e2.lm_head(hidden, weight, B * n, H, V, logits, status)
                e2.expand(logits, n * V, B, V, k, D, s, token, parent, value, frontier, ws, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        trees.append([host(t) for t in (token, parent, frontier, value)])
    (t0, p0, f0, v0), (t1, p1, f1, v1) = trees
    assert (t0 == t1).all() and (p0 == p1).all() and (f0 == f1).all()
    assert np.abs(v0 - v1).max() <= 1e-5 * np.abs(v1).max()
