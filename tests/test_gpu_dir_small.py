"""Global directed triads on both sides of the rule between the two ways to count them
(csrc/tg_directed.cu): edge by edge for small graphs, from totals for larger ones,
against the directed oracle, bit-exact; and the launches of the small graphs' way."""
import numpy as np
import pytest

import paper_1901_10026_gb300 as tg
from oracle import odir
from paper_1901_10026_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_10026_gb300 import build
    build.build()
    odir.build()


def _hub(n, m, hub, L, seed):
    """Random arcs, and a hub with `hub` neighbours in all three states."""
    r = np.random.default_rng(seed)
    other = r.permutation(np.arange(1, n))[:hub]
    out, back = other[r.random(hub) < 0.6], other
    src = np.concatenate([r.integers(0, n, m), np.zeros(out.size, int), back])
    dst = np.concatenate([r.integers(0, n, m), out, np.zeros(back.size, int)])
    return synth.TypedEdgeList(n, src.astype(np.int32), dst.astype(np.int32),
                               r.integers(0, L, n).astype(np.uint8), L, f"hub{hub}")


def _check(G):
    g = tg.tg_build_csr(G.n, G.src, G.dst, G.types, G.L, directed=True)
    _, want = odir.counts_of(G)
    assert np.array_equal(tg.tg_count_directed_global(g), want)


@pytest.mark.parametrize("L,m", [(1, 60), (8, 150_000), (8, 185_000), (8, 200_000), (9, 200_000), (9, 330_000),
                                 (16, 300_000)])
def test_around_the_rule(L, m):
    _check(_hub(40_000, m, 300, L, m + L))


@pytest.mark.parametrize("hub,L", [(1, 4), (240, 1), (256, 4), (257, 4), (2100, 5), (256, 8), (257, 8), (2100, 8),
                                   (257, 9), (2100, 16)])
def test_totals_with_hubs(hub, L):
    """Units of a node of at most 256 neighbours and above, hubs beyond the one-warp
    degree bound and every bound of the type templates, in graphs counted from totals."""
    _check(_hub(60_000, 230_000 if L <= 8 else 345_000, hub, L, hub + L))


@pytest.mark.parametrize("hub", [1, 300])
def test_small_graphs_take_few_launches(hub):
    G = _hub(500, 3000, hub, 3, 7)
    g = tg.tg_build_csr(G.n, G.src, G.dst, G.types, 3, directed=True)
    tg.tg_count_directed_global(g)
    before = tg.tg_launch_count()
    tg.tg_count_directed_global(g)
    assert tg.tg_launch_count() - before <= 3  # degrees, edges, division
