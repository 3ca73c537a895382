"""Compaction with a block per sequence and over the whole device, either side of the line between them."""
import numpy as np
import pytest
import torch

import paper_2406_16858_b200 as e2
from harness import DEV, dev, host, new_status

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n_layers,Hkv,d,D", [
    (1, 0, 4, 64, 3),       # lengths only
    (1, 1, 1, 8, 1),        # one segment
    (3, 1, 4, 64, 16),      # one block, the deepest tree
    (2, 8, 4, 72, 6),       # 576 segments: the second of most threads is missing
    (33, 4, 8, 128, 6), (2, 4, 8, 136, 6),  # 1024 segments, and 1088
    (32, 32, 8, 128, 6),
])
def test_rows_and_lengths(B, n_layers, Hkv, d, D):
    m = 20
    rng = np.random.default_rng(B * 100 + n_layers)
    kv_len = rng.integers(0, 9, B).astype(np.int32)
    kv_off = (np.arange(B) * 40).astype(np.int64)
    acc_len = rng.integers(0, D + 1, B).astype(np.int32)
    acc_len[0] = D
    path = np.full((B, D), -1, np.int32)
    for b in range(B):
        path[b, :acc_len[b]] = np.sort(rng.choice(m, acc_len[b], replace=False))
    bad = B - 1 if B > 1 else None
    if bad is not None:
        acc_len[bad], path[bad, 0] = 1, m  # outside the tree: reported, left alone
    caches = [[torch.randint(-30000, 30000, (B * 40, Hkv, d), dtype=torch.int16, device=DEV) for _ in range(n_layers)] for _ in range(2)]
    want = [[host(t).copy() for t in c] for c in caches]
    new_len = kv_len.copy()
    for b in range(B):
        if b == bad:
            continue
        new_len[b] += acc_len[b]
        at = kv_off[b] + kv_len[b]
        for c in want:
            for t in c:
                t[at:at + acc_len[b]] = t[at + path[b, :acc_len[b]]]
    ptrs = [torch.tensor([t.data_ptr() for t in c] or [0], dtype=torch.int64, device=DEV) for c in caches]
    lens, status = dev(kv_len), new_status()
    e2.kv_compact(ptrs[0], ptrs[1], n_layers, dev(kv_off), lens, dev(path), dev(acc_len), B, m, D, Hkv, d, status)
    torch.cuda.synchronize()
    assert int(status.item()) == (e2.STATUS_BAD_TREE if bad is not None else 0)
    assert (host(lens) == new_len).all()
    for got, exp in zip(caches, want):
        for g, e in zip(got, exp):
            assert (host(g) == e).all()
