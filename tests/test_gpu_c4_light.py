"""Light anchors of the 4-cycle enumeration (csrc/tg_c4_light.cu) at the edges of
their classes: anchors whose walk cost lies just below, at and above each
table's bound, in global totals and per-edge rows, against the oracles.

K_{2,b} with a path on every leaf has two anchors of walk cost about 2 b: the far
end of each is met b times, the largest count a table can hold for its cost."""
import numpy as np
import pytest

import oracle
import paper_1901_10026_gb300 as tg
from oracle import o2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_10026_gb300 import build
    build.build()
    oracle.build()
    o2.build()


def _k2b(b, L):
    """Nodes 0 and 1 joined to b middles; middle q also has a leaf for even q."""
    mid = np.arange(2, 2 + b, dtype=np.int32)
    leaf = np.arange(2 + b, 2 + b + (b + 1) // 2, dtype=np.int32)
    src = np.concatenate([np.zeros(b, np.int32), np.ones(b, np.int32), mid[::2]])
    dst = np.concatenate([mid, mid, leaf])
    n = 2 + b + leaf.size
    return n, src, dst, (np.arange(n) * 7 % 5 % L).astype(np.uint8)


# walk cost of node 0: 3 per even middle, 2 per odd one
@pytest.mark.parametrize("b", [2, 31, 203, 204, 205, 206, 818, 819, 820, 3275, 3276, 3277, 3278])
@pytest.mark.parametrize("L", [1, 5])
def test_class_bounds(b, L):
    n, src, dst, types = _k2b(b, L)
    g = tg.tg_build_csr(n, src, dst, types, L)
    assert np.array_equal(tg.tg_count_global(g, 4), o2.global_counts(n, src, dst, types, L, 4))
    og = oracle.OracleGraph(n, src, dst, types, L)
    rows = tg.tg_count_per_edge(g, 4, tg.TG_ORBIT)
    e = np.unique(np.concatenate([np.arange(min(g.M, 40)), np.arange(max(0, g.M - 40), g.M)]))
    want = og.per_edge(4, "orbit", edges=e)
    assert np.array_equal(rows[e], want)
