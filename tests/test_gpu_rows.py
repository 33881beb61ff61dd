"""Per-edge rows from k_cyc_rows (csrc/tg_edges.cu): T sums of edges whose larger
end has up to 256 neighbours and beyond, type counts around the kernel's register
classes, 32- and 64-bit terms (hubs of 8,192 and 8,193 neighbours), batches of edges,
k = 3, against the fused kernel and the per-edge oracle."""
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
    yield
    tg.tg_set_tune(reset=True)


def _hub_graph(deg, L, seed=3):
    """Hub 0 with `deg` neighbours; 90 of them form a sparse random graph with 40 others."""
    r = np.random.default_rng(seed)
    n = deg + 41
    a, b = np.triu_indices(90, 1)
    keep = r.random(a.shape[0]) < 0.3
    x, y = np.meshgrid(np.arange(1, 91), np.arange(deg + 1, n), indexing="ij")
    k2 = r.random(x.shape) < 0.2
    src = np.concatenate([np.zeros(deg, np.int64), a[keep] + 1, x[k2]]).astype(np.int32)
    dst = np.concatenate([np.arange(1, deg + 1), b[keep] + 1, y[k2]]).astype(np.int32)
    return n, src, dst, r.integers(0, L, n).astype(np.uint8)


@pytest.mark.parametrize("L", [1, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("deg", [95, 256, 257, 8192, 8193])
def test_rows_against_fused_and_oracle(deg, L):
    n, src, dst, types = _hub_graph(deg, L)
    g = tg.tg_build_csr(n, src, dst, types, L)
    og = oracle.OracleGraph(n, src, dst, types, L)
    e = np.unique(np.random.default_rng(5).integers(0, g.M, 40))
    for k, level, name in ((4, tg.TG_ORBIT, "orbit"), (4, tg.TG_GRAPHLET, "graphlet"),
                           (3, tg.TG_GRAPHLET, "graphlet")):
        tg.tg_set_tune(kernel=tg.TG_KERNEL_CYCLES, edge_pass=tg.TG_EDGE_PASS_FUSED)
        want = tg.tg_count_per_edge(g, k, level)
        for tune in ({}, dict(edge_batch=64, grid_limit=3)):
            tg.tg_set_tune(kernel=tg.TG_KERNEL_CYCLES, **tune)
            got = tg.tg_count_per_edge(g, k, level)
            bad = np.argwhere(got != want)
            assert bad.shape[0] == 0, (k, level, tune, bad[:5])
        assert np.array_equal(got[e], og.per_edge(k, name, edges=e))
    tg.tg_set_tune(reset=True)


def _star_of_types(deg, L):
    """A node with `deg` neighbours spread over L types, joined in a ring."""
    ring = np.arange(1, deg + 1)
    src = np.concatenate([np.zeros(deg, np.int64), ring[:-1]]).astype(np.int32)
    dst = np.concatenate([ring, ring[1:]]).astype(np.int32)
    return deg + 1, src, dst, (np.arange(deg + 1) * 7 % 11 % L).astype(np.uint8)


@pytest.mark.parametrize("L", [1, 2, 3, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("deg", [3, 31, 63, 64, 65, 300])
def test_node_sums_around_the_degree_bound(deg, L):
    """Theta and D by lane groups up to 64 neighbours, by warps beyond (global and rows)."""
    n, src, dst, types = _star_of_types(deg, L)
    g = tg.tg_build_csr(n, src, dst, types, L)
    og = oracle.OracleGraph(n, src, dst, types, L)
    tg.tg_set_tune(kernel=tg.TG_KERNEL_CYCLES)
    rows = tg.tg_count_per_edge(g, 4, tg.TG_ORBIT)
    assert np.array_equal(rows, og.per_edge(4, "orbit"))
    assert np.array_equal(tg.tg_count_global(g, 4), o2.global_counts(n, src, dst, types, L, 4))
    tg.tg_set_tune(reset=True)
