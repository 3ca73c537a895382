"""Calls of different sizes from several threads at once, each on its own stream: a kernel's shared-memory limit is one
setting of the process, so that every launch has to stay within what any other one sets."""
import threading

import pytest
import torch

import paper_2406_16858_b200 as e2
from harness import DEV, make_ws, new_status

pytestmark = pytest.mark.gpu


def _rerank(k, D):
    N, m = k + (D - 1) * k * k, 60
    ints = dict(dtype=torch.int32, device=DEV)
    parent = torch.tensor([-1 if i < k else (i - k) // k for i in range(N)], **ints).repeat(2, 1).contiguous()
    token, value = torch.zeros((2, N), **ints), -torch.arange(N, dtype=torch.float64, device=DEV).repeat(2, 1).contiguous()
    out = [torch.zeros((2, m), **ints) for _ in range(4)] + [torch.zeros(2, **ints)]
    return lambda st: e2.rerank(token, parent, value, 2, k, D, m, *out, st), lambda: out[0]


def _attention(B, Hq, Hkv, longest):
    m, d = 60, 128
    lens = [longest] + [100] * (B - 1)
    off = [sum(lens[:i]) + i * m for i in range(B)]
    rows = sum(lens) + B * m
    q, kc, vc = (torch.randn(s, device=DEV).to(torch.bfloat16) for s in ((B, m, Hq, d), (rows, Hkv, d), (rows, Hkv, d)))
    kv_off, kv_len = torch.tensor(off, dtype=torch.int64, device=DEV), torch.tensor(lens, dtype=torch.int32, device=DEV)
    mask = torch.ones((B, m, 1), dtype=torch.int64, device=DEV)
    ws = make_ws(e2.workspace_bytes(e2.OP_TREE_ATTENTION, B=B, m=m, Hq=Hq, Hkv=Hkv, d=d, max_kv_len=longest))
    out = torch.zeros_like(q)
    return (lambda st: e2.tree_attention(q, kc, vc, rows, kv_off, kv_len, mask, B, m, Hq, Hkv, d, longest, 0.1, out, None, ws, st),
            lambda: out)


def _lm_head(B):
    k, D, H, V = 10, 1, 64, 2000
    rows = B  # the first step: one feature row per sequence
    hidden, weight = (torch.randn(s, device=DEV).to(torch.bfloat16) for s in ((rows, H), (V, H)))
    ints = dict(dtype=torch.int32, device=DEV)
    tree = (torch.zeros((B, k), **ints), torch.zeros((B, k), **ints), torch.zeros((B, k), dtype=torch.float64, device=DEV),
            torch.zeros((B, k), **ints), make_ws(e2.workspace_bytes(e2.OP_LM_HEAD_EXPAND, B=B, V=V, k=k, D=D)))
    return lambda st: e2.lm_head_expand(hidden, weight, H, B, V, k, D, 0, *tree, st), lambda: tree[0]


def _accept(V):
    k, D, m = 2, 1, 2
    ints = dict(dtype=torch.int32, device=DEV)
    target, draft = torch.randn((1, m + 1, V), device=DEV), torch.randn((1, 1, V), device=DEV)
    sel = (torch.tensor([[0, 1]], **ints), torch.tensor([[-1, -1]], **ints), torch.tensor([[3, V - 2]], **ints), torch.tensor([2], **ints))
    u, ub = torch.full((1, m), 0.5, device=DEV), torch.full((1,), 0.5, device=DEV)
    out = (torch.zeros(1, **ints), torch.zeros((1, D), **ints), torch.zeros(1, **ints))
    ws = make_ws(e2.workspace_bytes(e2.OP_ACCEPT, B=1, V=V, k=k, D=D, m=m))
    return (lambda st: e2.accept(target, (m + 1) * V, draft, V, *sel, 1, V, k, D, m, 1.0, u, ub, *out, ws, st), lambda: out[2])


@pytest.mark.parametrize("make,sizes", [
    (_rerank, [(16, 8), (32, 4)]),
    (_attention, [(8, 32, 8, 16384), (1, 8, 2, 12000)]),  # block pairs, served longest first and not
    (_lm_head, [(160,), (256,)]),
    (_accept, [(131076,), (180000,)]),                    # the two launches
])
def test_calls_of_different_sizes_at_once(make, sizes):
    calls = [make(*s) for s in sizes]
    for call, _ in calls:
        call(new_status())
    torch.cuda.synchronize()
    want = [get().clone() for _, get in calls]
    start, errors = threading.Barrier(len(calls)), []

    def work(i):
        stream, st = torch.cuda.Stream(), new_status()
        try:
            start.wait()
            with torch.cuda.stream(stream):
                for _ in range(400):
                    calls[i][0](st)
            stream.synchronize()
            assert int(st.item()) == 0
        except Exception as e:  # a thread's own would go unseen
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for (_, get), w in zip(calls, want):
        assert torch.equal(get(), w)
