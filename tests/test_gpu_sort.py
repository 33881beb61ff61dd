"""The radix sort behind the CSR builder (csrc/tg_prim.cu) at the sizes where it
changes kernels or tiles: graphs whose number of raw pairs, edges or directed
entries lies at a single CTA's capacity (12,288 keys) or a tile's (4,096), with
repeated pairs, one hub (equal digits), and ids that need one more digit."""
import numpy as np
import pytest

import oracle
import paper_1901_10026_gb300 as tg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_10026_gb300 import build
    build.build()
    oracle.build()


def _check(n, src, dst, L=3):
    types = (np.arange(n) * 7 % 11 % L).astype(np.uint8)
    g = tg.tg_build_csr(n, src, dst, types, L)
    lo, hi = np.minimum(src, dst).astype(np.int64), np.maximum(src, dst).astype(np.int64)
    key = np.unique((lo * n + hi)[lo != hi])
    u, v = tg.tg_edge_list(g)
    assert g.M == key.size
    assert np.array_equal(u, key // n) and np.array_equal(v, key % n)
    # every row sum of the 3-node counts: 2-node entry count and wedges per edge
    rows = tg.tg_count_per_edge(g, 3)
    deg = np.bincount(np.concatenate([u, v]), minlength=n)
    assert np.array_equal(rows.sum(1).astype(np.int64),
                          deg[u] + deg[v] - 2 - rows[:, L:].sum(1).astype(np.int64))


@pytest.mark.parametrize("n", [200, 257, 70000])
@pytest.mark.parametrize("m", [1, 2, 4095, 4096, 4097, 6143, 6145, 12287, 12288, 12289, 40000])
def test_random_pairs(n, m):
    g = np.random.default_rng([n, m])
    _check(n, g.integers(0, n, m).astype(np.int32), g.integers(0, n, m).astype(np.int32))


def test_hub_and_repeats():
    g = np.random.default_rng(3)
    n, m = 30000, 50000
    src = np.where(g.random(m) < 0.7, 17, g.integers(0, n, m)).astype(np.int32)
    dst = g.integers(0, 40, m).astype(np.int32) * 700
    _check(n, src, dst)


@pytest.mark.parametrize("L", [1, 3, 16])
@pytest.mark.parametrize("top", [1, 2, 15, 16, 17, 32, 33, 63, 64, 65, 66])
def test_lists_around_the_degree_bound(top, L):
    """Lists sorted by themselves (no node beyond 64 neighbours) and by the radix sort:
    a node of `top` neighbours among random pairs of low degree, against the lists'
    own counts; 31 to 33 edges of equal lower ends in a row among them."""
    g = np.random.default_rng([top, L])
    n = 500
    src = np.concatenate([np.full(top, 3), g.integers(100, n, 300)]).astype(np.int32)
    dst = np.concatenate([np.arange(top) + 5, g.integers(100, n, 300)]).astype(np.int32)
    _check(n, src, dst, L)
    types = (np.arange(n) * 7 % 11 % L).astype(np.uint8)
    want = oracle.OracleGraph(n, src, dst, types, L).per_edge(4, "orbit")
    got = tg.tg_count_per_edge(tg.tg_build_csr(n, src, dst, types, L), 4, tg.TG_ORBIT)
    assert np.array_equal(got, want)
