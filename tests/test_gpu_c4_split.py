"""Every 4-cycle anchor split over the grid (``unroll = 4``): more anchors than one CTA
sorts and more than a wave holds, against the default classes and O1; and the launches
that the waves of many cheap anchors take."""
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


@pytest.fixture
def split_all():
    tg.tg_set_tune(unroll=4)
    yield
    tg.tg_set_tune(reset=True)


def _graph(n, m, hub, L):
    """Random pairs, and a hub beyond the 16-bit counters' degree when hub >= 2^16."""
    r = np.random.default_rng([n, hub])
    other = r.permutation(np.arange(1, n))[:hub]
    src = np.concatenate([r.integers(0, n, m), np.zeros(other.size, int)]).astype(np.int32)
    dst = np.concatenate([r.integers(0, n, m), other]).astype(np.int32)
    return n, src, dst, r.integers(0, L, n).astype(np.uint8), L


@pytest.mark.parametrize("n,m,hub,L", [(4000, 20000, 0, 3), (12000, 50000, 300, 5), (15000, 70000, 500, 9),
                                       (70000, 150000, 66000, 2)])
def test_many_split_anchors(n, m, hub, L, split_all):
    G = _graph(n, m, hub, L)
    g = tg.tg_build_csr(*G)
    split = tg.tg_count_global(g, 4), tg.tg_count_per_edge(g, 4, tg.TG_ORBIT)
    tg.tg_set_tune(reset=True)
    assert np.array_equal(split[0], tg.tg_count_global(g, 4))
    assert np.array_equal(split[1], tg.tg_count_per_edge(g, 4, tg.TG_ORBIT))
    e = np.unique(np.random.default_rng(1).integers(0, g.M, 50))
    assert np.array_equal(split[1][e], oracle.OracleGraph(*G).per_edge(4, "orbit", edges=e))


def test_cheap_anchors_take_few_waves(split_all):
    """Rows of a cycle: 40,000 anchors of one member each."""
    n = 40000
    v = np.arange(n, dtype=np.int32)
    g = tg.tg_build_csr(n, v, ((v + 1) % n).astype(np.int32), np.zeros(n, np.uint8), 1)
    tg.tg_count_per_edge(g, 4)
    before = tg.tg_launch_count()
    rows = tg.tg_count_per_edge(g, 4)
    assert tg.tg_launch_count() - before < 300  # 128 anchors a wave: above 900
    # two nodes off either end; induced 4-paths: the edge in the middle once, at an end twice
    assert np.array_equal(rows, np.tile(np.array([2, 0, 3, 0, 0, 0, 0, 0], np.uint64), (n, 1)))
