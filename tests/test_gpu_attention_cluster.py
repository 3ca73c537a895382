"""Attention launches whose blocks combine their rows inside a thread-block cluster, and those that put a whole
sequence on one block, at the edges of their plan, against the CPU oracle."""
import numpy as np
import pytest

import paper_2406_16858_b200 as e2
from test_gpu_attention import _compare, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,Hq,Hkv,d,lens", [
    (60, 8, 2, 128, [1000]),            # two row blocks of 120 rows per KV head
    (60, 2, 2, 128, [2000, 0]),         # the second sequence has one tile for a whole cluster
    (33, 3, 1, 64, [700, 650, 128]),    # 99 rows (odd share), query rows copied by hand, fewer tiles than blocks
    (1, 4, 4, 128, [5000]),             # one row: most blocks of a cluster combine nothing
    (128, 8, 1, 128, [3000]),           # eight row blocks
    (16, 4, 4, 64, [112, 113]),         # exactly one tile of 128 keys, and one key more
    (60, 16, 2, 128, [196, 452]),       # four tiles on one block
    (40, 20, 20, 128, [1300, 2600]),    # as many groups as clusters of a few blocks
])
def test_cluster_and_single_block_launches(m, Hq, Hkv, d, lens):
    B = len(lens)
    assert e2.tree_attention_launches(B, m, Hq, Hkv, d, max(lens)) == 1
    q, kc, vc, off, kl, bits = _inputs(77, B, m, Hq, Hkv, d, lens)
    rng = np.random.default_rng(5)
    n = 400
    samples = np.stack([rng.integers(0, B, n), rng.integers(0, Hq, n), rng.integers(0, m, n)], axis=1).astype(np.int32)
    _compare(q, kc, vc, off, kl, bits, 1.0 / np.sqrt(d), samples=samples)


@pytest.mark.parametrize("kv_len", [11254, 11255])
def test_long_sequences_of_few_heads_are_split(kv_len):
    """Either side of the line from which a cluster per KV head would leave too much of the device idle."""
    m, Hq, Hkv, d = 10, 8, 2, 128
    if kv_len > 11254:
        assert e2.tree_attention_launches(1, m, Hq, Hkv, d, kv_len) == 2
    q, kc, vc, off, kl, bits = _inputs(78, 1, m, Hq, Hkv, d, [kv_len])
    rng = np.random.default_rng(6)
    samples = np.stack([np.zeros(200, int), rng.integers(0, Hq, 200), rng.integers(0, m, 200)], axis=1).astype(np.int32)
    _compare(q, kc, vc, off, kl, bits, 1.0 / np.sqrt(d), samples=samples)
