"""What the framework is timed on: the work that a serving loop has it do, through its public entry points.

Kinds of case
  cycle       one whole draft-and-verify cycle of B sequences (``cycle.enqueue_cycle``): D expansions, the
              selection with mask and position ids, one tree attention per layer, acceptance, compaction.
              ``graph``: captured once and replayed, as a server with fixed shapes does; otherwise every
              call is made from Python, as in a first integration or where shapes change all the time.
  tree        drafting alone: the expansions and the selection of one cycle, logits at hand.
  head        drafting from features: the LM head in front of every expansion, as two calls for few rows
              and as the fused call from 100 rows on.
  verify      the attention of a verification pass alone, a call per layer.
  draft_attn  the draft layer's attention while the tree grows: m = k, 2k, ... (D-1)k tokens.
  accept      the acceptance of one cycle alone, with the draft rows or with the candidates as proposal.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2406_16858_b200 as e2
from paper_2406_16858_b200.cycle import CycleBuffers, CycleShape, enqueue_cycle

DEV = "cuda:0"


def _cycle(name, B, V, k, D, m, layers, Hq, Hkv, d, kv_lo, kv_hi, temperature, graph):
    return {"name": name, "kind": "cycle", "B": B, "V": V, "k": k, "D": D, "m": m, "layers": layers, "Hq": Hq,
            "Hkv": Hkv, "d": d, "kv_lo": kv_lo, "kv_hi": kv_hi, "temperature": temperature, "graph": graph}


def listed():
    return [
        # the smallest call there is: a toy model driven from Python, where launches and host time count
        _cycle("cycle_tiny_eager", 1, 1000, 4, 3, 16, 1, 4, 4, 64, 128, 128, 0.0, False),
        # one user at a time, greedy, a 7B model with plain multi-head attention and a short prompt
        _cycle("cycle_vicuna7b", 1, 32000, 10, 6, 60, 32, 32, 32, 128, 1024, 1024, 0.0, True),
        # one user at a time, sampling, an 8B model with grouped heads and a large vocabulary
        _cycle("cycle_llama3_8b", 1, 128256, 10, 6, 60, 32, 32, 8, 128, 4096, 4096, 1.0, True),
        # the same for a 70B model: many layers, eight query heads per KV head, a long prompt
        _cycle("cycle_llama2_70b", 1, 32000, 10, 6, 60, 80, 64, 8, 128, 8192, 8192, 1.0, True),
        # a server's batches: prompts of very different lengths
        _cycle("cycle_batch8", 8, 128256, 10, 6, 60, 32, 32, 8, 128, 512, 16384, 1.0, True),
        _cycle("cycle_batch32", 32, 128256, 10, 6, 60, 32, 32, 8, 128, 512, 16384, 1.0, True),
        # drafting with a vocabulary that a padding token made odd: no row but the first is 16-byte aligned
        {"name": "tree_odd_vocab", "kind": "tree", "B": 4, "V": 32001, "k": 10, "D": 6, "m": 60},
        # drafting through the LM head: one user, and a batch whose rows go through the fused call
        {"name": "head_one", "kind": "head", "B": 1, "V": 128256, "H": 4096, "k": 10, "D": 6},
        {"name": "head_batch16", "kind": "head", "B": 16, "V": 128256, "H": 4096, "k": 10, "D": 6},
        # a few ragged sequences, 40 heads without grouping, another budget of tokens, the sums asked for
        {"name": "verify_mha40", "kind": "verify", "B": 3, "m": 50, "Hq": 40, "Hkv": 40, "d": 128, "kv_lo": 701,
         "kv_hi": 3001, "layers": 8, "lse": True},
        # the draft layer's growing tree behind a long prompt
        {"name": "draft_attn_long", "kind": "draft_attn", "B": 1, "k": 10, "D": 6, "Hq": 32, "Hkv": 8, "d": 128,
         "kv_lo": 12345, "kv_hi": 12345},
        # sampling's acceptance for a batch
        {"name": "accept_batch16", "kind": "accept", "B": 16, "V": 128256, "k": 10, "D": 6, "m": 60,
         "temperature": 1.0, "draft_rows": True},
    ]


# ---- drawn cases -----------------------------------------------------------------------------------
def _log(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def _vocab(rng):
    """Vocabularies of trained models are a few distinct sizes; any other size comes from added tokens."""
    V = rng.choice((32000, 32000, 128256, 128256, _log(rng, 1000, 130000)))
    return V + rng.choice((0, 0, 0, 1, 2, 4, 8))


def _tree_shape(rng):
    k = rng.choice((10, 10, 10, 4, 8, rng.randint(2, 16)))
    D = rng.choice((6, 6, rng.randint(3, 8)))
    N = k + (D - 1) * k * k
    return {"k": k, "D": D, "m": min(N, rng.choice((60, 60, 50, 48, rng.randint(16, 64))))}


def _heads(rng):
    """Query heads, KV heads, head size."""
    return dict(zip(("Hq", "Hkv", "d"), rng.choice(((32, 32, 128), (32, 8, 128), (32, 8, 128), (64, 8, 128), (40, 40, 128),
                                                     (28, 4, 128), (16, 8, 64), (32, 8, 64), (24, 8, 128)))))


def _lengths(rng, B):
    if B == 1 or rng.random() < 0.3:
        L = _log(rng, 128, 16384)
        return {"kv_lo": L, "kv_hi": L}
    lo = _log(rng, 128, 2048)
    return {"kv_lo": lo, "kv_hi": _log(rng, lo, 16384)}


def draw(rng: random.Random):
    most = {x: max(work(c)[x] for c in listed()) for x in ("bytes", "flops")}
    while True:
        kind = rng.choice(("cycle", "cycle", "cycle", "cycle", "tree", "head", "verify", "draft_attn", "accept"))
        c = {"kind": kind}
        if kind == "cycle":
            B = _log(rng, 1, 32)
            c.update(B=B, V=_vocab(rng), **_tree_shape(rng), layers=_log(rng, 2, 80), **_heads(rng), **_lengths(rng, B),
                     temperature=rng.choice((0.0, 1.0, 1.0, 0.7)), graph=rng.random() < 0.75)
        elif kind == "tree":
            c.update(B=_log(rng, 1, 64), V=_vocab(rng), **_tree_shape(rng))
        elif kind == "head":
            s = _tree_shape(rng)
            c.update(B=_log(rng, 1, 32), V=_vocab(rng), H=64 * rng.randint(16, 80), k=s["k"], D=s["D"])
        elif kind == "verify":
            B = _log(rng, 1, 32)
            c.update(B=B, m=rng.choice((60, 50, 48, rng.randint(8, 100))), **_heads(rng), **_lengths(rng, B),
                     layers=rng.randint(1, 12), lse=rng.random() < 0.3)
        elif kind == "draft_attn":
            s, B = _tree_shape(rng), _log(rng, 1, 8)
            if (s["D"] - 1) * s["k"] > 128:
                continue
            c.update(B=B, k=s["k"], D=s["D"], **_heads(rng), **_lengths(rng, B))
        else:
            temperature = rng.choice((0.0, 1.0, 1.0, 0.7))
            c.update(B=_log(rng, 1, 32), V=_vocab(rng), **_tree_shape(rng), temperature=temperature,
                     draft_rows=temperature > 0 and rng.random() < 0.8)
        if all(work(c)[x] <= most[x] for x in most):
            return c


# ---- inputs ----------------------------------------------------------------------------------------
def _kv_lengths(case):
    """The lengths' quantiles, so that every seed has the same work; which sequence gets which is the seed's."""
    B, lo, hi = case["B"], case["kv_lo"], case["kv_hi"]
    return [round(lo * (hi / lo) ** ((i + 0.5) / B)) if hi > lo else lo for i in range(B)]


def _placed(case, seed, m):
    """Lengths in the seed's order and the packed cache: (kv_len, kv_off, rows, longest)."""
    lens = _kv_lengths(case)
    random.Random(seed).shuffle(lens)
    off = [0]
    for n in lens[:-1]:
        off.append(off[-1] + n + m)
    return (torch.tensor(lens, dtype=torch.int32, device=DEV), torch.tensor(off, dtype=torch.int64, device=DEV),
            off[-1] + lens[-1] + m, max(lens))


def _logit_rows(g, B, rows, V):
    """Half of the contexts are easy: one token holds most of the mass (0.8 of it in the middle); in the
    others a likely token stands out little from a wide field."""
    z = torch.randn((B, rows, V), generator=g, device=DEV).mul_(2.0)
    easy = torch.rand((B, rows, 1), generator=g, device=DEV) < 0.5
    sure = math.log(V) + 3.4 + torch.randn((B, rows, 1), generator=g, device=DEV)
    at = torch.randint(0, V, (B, rows, 1), generator=g, device=DEV)
    return z.scatter_(2, at, torch.where(easy, sure, z.gather(2, at) + 2.0))


def _target_rows(g, draft, buf):
    """The target model's rows follow the draft rows of the same contexts, with noise; nodes that were not
    expanded have rows of their own."""
    s = buf.shape
    first = torch.tensor([s.k + (t - 1) * s.k * s.k + j * s.k for t in range(1, s.D) for j in range(s.k)], device=DEV)
    row_of = torch.full((s.B, s.N), -1, dtype=torch.int64, device=DEV)
    rows = torch.arange(1, s.R, device=DEV).expand(s.B, -1)
    row_of.scatter_(1, buf.tree_parent[:, first].long(), rows)
    src = row_of.gather(1, buf.sel_index.clamp(min=0).long())
    src = torch.cat([torch.zeros((s.B, 1), dtype=torch.int64, device=DEV), src], 1)
    out = _logit_rows(g, s.B, s.m + 1, s.V)
    for b in range(s.B):
        out[b] = torch.where(src[b, :, None] >= 0, draft[b, src[b].clamp(min=0)], out[b])
    return out.add_(torch.randn(out.shape, generator=g, device=DEV), alpha=0.5)


def _bf16(g, *shape):
    return torch.empty(shape, dtype=torch.bfloat16, device=DEV).normal_(generator=g)


def _buffers(case, longest=0):
    return CycleBuffers(CycleShape(case["B"], case["V"], case["k"], case["D"], case["m"], case.get("layers", 1), case.get("Hq", 1),
                                   case.get("Hkv", 1), case.get("d", 128), longest, case.get("temperature", 0.0)), DEV)


def _grown_masks(case, seed, m, level):
    """Mask bits of a random tree: every token of a level hangs on a random one of the level before."""
    r = random.Random(seed + 1)
    B = case["B"]
    parent = [[-1 if i < level else r.randrange((i // level - 1) * level, i // level * level) for i in range(m)] for _ in range(B)]
    depth = [[i // level for i in range(m)] for _ in range(B)]
    ints = dict(dtype=torch.int32, device=DEV)
    bits = torch.zeros((B, m, (m + 63) // 64), dtype=torch.int64, device=DEV)
    e2.tree_mask(torch.tensor(parent, **ints), torch.tensor(depth, **ints), torch.full((B,), m, **ints), torch.zeros(B, **ints),
                 B, m, bits, None, torch.zeros((B, m), **ints), torch.zeros(1, **ints))
    return bits


def _workspace(op, **sizes):
    ws = torch.empty(max(256, e2.workspace_bytes(op, **sizes)), dtype=torch.uint8, device=DEV)
    e2.workspace_init(ws)
    return ws


def prepare(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return {"cycle": _prepare_cycle, "tree": _prepare_tree, "head": _prepare_head, "verify": _prepare_verify,
            "draft_attn": _prepare_draft_attn, "accept": _prepare_accept}[case["kind"]](case, seed, g)


def _prepare_cycle(case, seed, g):
    B, m, n = case["B"], case["m"], case["layers"]
    kv_len0, kv_off, rows, longest = _placed(case, seed, m)
    buf = _buffers(case, longest)
    draft = _logit_rows(g, B, buf.shape.R, case["V"])
    buf.expand_all(draft)
    buf.rerank_and_mask(kv_len0)
    k_all, v_all = (_bf16(g, n, rows, case["Hkv"], case["d"]) for _ in range(2))
    q_all = _bf16(g, n, B, m, case["Hq"], case["d"])
    st = {"case": case, "buf": buf, "draft": draft, "target": _target_rows(g, draft, buf),
          "u_accept": torch.rand((B, m), generator=g, device=DEV), "u_bonus": torch.rand(B, generator=g, device=DEV),
          "k_all": k_all, "v_all": v_all, "out_all": torch.zeros_like(q_all), "q": list(q_all.unbind(0)),
          "k": list(k_all.unbind(0)), "v": list(v_all.unbind(0)), "kv_off": kv_off, "kv_len0": kv_len0, "kv_len": kv_len0.clone(),
          "scale": 1.0 / math.sqrt(case["d"])}
    st["out"] = list(st["out_all"].unbind(0))
    for name in ("k", "v"):
        st[name + "_ptrs"] = torch.tensor([t.data_ptr() for t in st[name]], dtype=torch.int64, device=DEV)
    if case["graph"]:
        _cycle_calls(st)  # the first call of a kernel loads it, which a capture cannot hold
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            _cycle_calls(st)
        st["graph"] = graph
    return st


def _cycle_calls(st):
    st["kv_len"].copy_(st["kv_len0"])  # every pass starts behind the same prefix
    enqueue_cycle(st["buf"], st["draft"], st["target"], st["u_accept"], st["u_bonus"], st["q"], st["k"], st["v"], st["out"],
                  st["k_ptrs"], st["v_ptrs"], st["kv_off"], st["kv_len"], st["scale"])


def _prepare_tree(case, seed, g):
    buf = _buffers(case)
    return {"case": case, "buf": buf, "draft": _logit_rows(g, case["B"], buf.shape.R, case["V"]),
            "kv_len": torch.randint(128, 4096, (case["B"],), generator=g, device=DEV, dtype=torch.int32)}


def _prepare_head(case, seed, g):
    B, V, H, k, D = (case[x] for x in ("B", "V", "H", "k", "D"))
    N = k + (D - 1) * k * k
    ints = dict(dtype=torch.int32, device=DEV)
    return {"case": case, "features": [_bf16(g, B, 1 if s == 0 else k, H) for s in range(D)],
            "weight": _bf16(g, V, H).mul_(2.0 / math.sqrt(H)), "logits": torch.empty((B * k, V), device=DEV),
            "token": torch.zeros((B, N), **ints), "parent": torch.zeros((B, N), **ints),
            "value": torch.zeros((B, N), dtype=torch.float64, device=DEV), "frontier": torch.zeros((B, k), **ints),
            "status": torch.zeros(1, **ints),
            "ws": _workspace(e2.OP_LM_HEAD_EXPAND if B * k >= 100 else e2.OP_EXPAND, B=B, V=V, k=k, D=D)}


def _prepare_verify(case, seed, g):
    B, m, Hq, Hkv, d, n = (case[x] for x in ("B", "m", "Hq", "Hkv", "d", "layers"))
    kv_len, kv_off, rows, longest = _placed(case, seed, m)
    out = torch.zeros((n, B, m, Hq, d), dtype=torch.bfloat16, device=DEV)
    lse = torch.zeros((n, B, Hq, m), device=DEV) if case["lse"] else None
    return {"case": case, "kv_len": kv_len, "kv_off": kv_off, "rows": rows, "longest": longest, "q": list(_bf16(g, n, B, m, Hq, d).unbind(0)),
            "k": list(_bf16(g, n, rows, Hkv, d).unbind(0)), "v": list(_bf16(g, n, rows, Hkv, d).unbind(0)), "out_all": out, "lse_all": lse,
            "out": list(out.unbind(0)), "lse": list(lse.unbind(0)) if lse is not None else [None] * n,
            "mask": _grown_masks(case, seed, m, 8), "status": torch.zeros(1, dtype=torch.int32, device=DEV),
            "ws": _workspace(e2.OP_TREE_ATTENTION, B=B, m=m, Hq=Hq, Hkv=Hkv, d=d, max_kv_len=longest)}


def _prepare_draft_attn(case, seed, g):
    B, k, D, Hq, Hkv, d = (case[x] for x in ("B", "k", "D", "Hq", "Hkv", "d"))
    kv_len, kv_off, rows, longest = _placed(case, seed, (D - 1) * k)
    ms = [s * k for s in range(1, D)]
    q = [_bf16(g, B, m, Hq, d) for m in ms]
    need = max(e2.workspace_bytes(e2.OP_TREE_ATTENTION, B=B, m=m, Hq=Hq, Hkv=Hkv, d=d, max_kv_len=longest) for m in ms)
    ws = torch.empty(max(256, need), dtype=torch.uint8, device=DEV)
    e2.workspace_init(ws)
    return {"case": case, "kv_len": kv_len, "kv_off": kv_off, "rows": rows, "longest": longest, "ms": ms, "q": q,
            "out": [torch.zeros_like(x) for x in q], "k": _bf16(g, rows, Hkv, d), "v": _bf16(g, rows, Hkv, d),
            "mask": [_grown_masks(case, seed, m, k) for m in ms], "status": torch.zeros(1, dtype=torch.int32, device=DEV), "ws": ws}


def _prepare_accept(case, seed, g):
    B, m = case["B"], case["m"]
    buf = _buffers(case)
    draft = _logit_rows(g, B, buf.shape.R, case["V"])
    buf.expand_all(draft)
    buf.rerank_and_mask(torch.zeros(B, dtype=torch.int32, device=DEV))
    return {"case": case, "buf": buf, "target": _target_rows(g, draft, buf), "draft": draft if case["draft_rows"] else None,
            "u_accept": torch.rand((B, m), generator=g, device=DEV), "u_bonus": torch.rand(B, generator=g, device=DEV)}


# ---- one pass --------------------------------------------------------------------------------------
def run(state):
    return {"cycle": _run_cycle, "tree": _run_tree, "head": _run_head, "verify": _run_verify, "draft_attn": _run_draft_attn,
            "accept": _run_accept}[state["case"]["kind"]](state)


def _tree_of(buf):
    return {"token": buf.tree_token, "parent": buf.tree_parent, "value": buf.tree_value, "frontier": buf.frontier,
            "sel_index": buf.sel_index, "sel_parent": buf.sel_parent, "sel_token": buf.sel_token, "sel_depth": buf.sel_depth,
            "n_sel": buf.n_sel, "mask": buf.mask_bits, "pos": buf.pos_ids, "status": buf.status}


def _accepted(buf):
    return {"acc_len": buf.acc_len, "acc_path": buf.acc_path, "bonus": buf.bonus_token, "status": buf.status}


def _run_cycle(st):
    if "graph" in st:
        st["graph"].replay()
    else:
        _cycle_calls(st)
    return {"tree": _tree_of(st["buf"]), "accepted": _accepted(st["buf"]), "out": st["out_all"], "k": st["k_all"], "v": st["v_all"],
            "kv_len": st["kv_len"]}


def _run_tree(st):
    st["buf"].expand_all(st["draft"])
    st["buf"].rerank_and_mask(st["kv_len"])
    return _tree_of(st["buf"])


def _run_head(st):
    c = st["case"]
    B, V, H, k, D = (c[x] for x in ("B", "V", "H", "k", "D"))
    tree = (st["token"], st["parent"], st["value"], st["frontier"], st["ws"], st["status"])
    for s in range(D):
        n = 1 if s == 0 else k
        if B * k >= 100:
            e2.lm_head_expand(st["features"][s], st["weight"], H, B, V, k, D, s, *tree)
        else:
            e2.lm_head(st["features"][s], st["weight"], B * n, H, V, st["logits"], st["status"])
            e2.expand(st["logits"], n * V, B, V, k, D, s, *tree)
    return {x: st[x] for x in ("token", "parent", "value", "frontier", "status")}


def _run_verify(st):
    c = st["case"]
    for q, k, v, out, lse in zip(st["q"], st["k"], st["v"], st["out"], st["lse"]):
        e2.tree_attention(q, k, v, st["rows"], st["kv_off"], st["kv_len"], st["mask"], c["B"], c["m"], c["Hq"], c["Hkv"], c["d"],
                          st["longest"], 1.0 / math.sqrt(c["d"]), out, lse, st["ws"], st["status"])
    return {"out": st["out_all"], "lse": st["lse_all"], "status": st["status"]}


def _run_draft_attn(st):
    c = st["case"]
    for m, q, out, mask in zip(st["ms"], st["q"], st["out"], st["mask"]):
        e2.tree_attention(q, st["k"], st["v"], st["rows"], st["kv_off"], st["kv_len"], mask, c["B"], m, c["Hq"], c["Hkv"], c["d"],
                          st["longest"], 1.0 / math.sqrt(c["d"]), out, None, st["ws"], st["status"])
    return {"out": st["out"], "status": st["status"]}


def _run_accept(st):
    st["buf"].accept(st["target"], st["draft"], st["u_accept"], st["u_bonus"])
    return _accepted(st["buf"])


# ---- what a pass cannot do without, and how close another implementation comes ---------------------
def _attention_work(case, m):
    keys = [n + m for n in _kv_lengths(case)]
    B, Hq, Hkv, d = (case[x] for x in ("B", "Hq", "Hkv", "d"))
    return 4.0 * sum(keys) * Hkv * d + 4.0 * B * m * Hq * d, 4.0 * sum(keys) * m * Hq * d


def work(case):
    """Logits, features, weights, keys, values and queries read once, outputs written once.  Of the target's
    rows those on one root-to-leaf walk count, and the draft rows there: more no acceptance needs."""
    kind, B, D, k = case["kind"], case["B"], case.get("D", 0), case.get("k", 0)
    N, R = k + (D - 1) * k * k, 1 + (D - 1) * k
    V = case.get("V", 0)
    total, flops = 0.0, 0.0
    if kind in ("cycle", "tree"):
        total += B * (4.0 * R * V + 16.0 * N + 28.0 * case["m"])
        flops += 2.0 * B * R * V
    if kind in ("cycle", "accept"):
        rows = D + 1 + (D if kind == "accept" and case["draft_rows"] else 0)
        total += 4.0 * B * rows * V
        flops += 2.0 * B * rows * V
    if kind in ("cycle", "verify"):
        b, f = _attention_work(case, case["m"])
        total, flops = total + case["layers"] * b, flops + case["layers"] * f
    if kind == "draft_attn":
        for s in range(1, D):
            b, f = _attention_work(case, s * k)
            total, flops = total + b, flops + f
    if kind == "head":
        total += D * 2.0 * V * case["H"] + 2.0 * B * R * case["H"] + 16.0 * B * N
        flops += 2.0 * B * R * V * case["H"]
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """Node values are 64-bit sums of logarithms of 32-bit sums.  Attention is bf16 with 32-bit sums; the sums
    it can return share its limit.  A whole value may differ where two values tie or a draw falls on a step."""
    if case["kind"] in ("cycle", "verify", "draft_attn"):
        return {"rel": 1e-2, "differ": 0.005}
    return {"rel": 1e-5, "differ": 0.005}
