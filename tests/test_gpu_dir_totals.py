"""Global directed counts from totals (csrc/tg_directed.cu) at the edges of their
kernels, against the directed oracles, bit-exact: units of a node of at most 256
neighbours and above, hubs above the one-warp degree bound, every bound of the
type templates; edges whose staged neighbourhood has 128 members and more."""
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


@pytest.mark.parametrize("L", [1, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("hub", [1, 240, 256, 257, 2100])
def test_triads(hub, L):
    G = _hub(2400, 9000, hub, L, hub + L)
    g = tg.tg_build_csr(G.n, G.src, G.dst, G.types, L, directed=True)
    _, want = odir.counts_of(G)
    assert np.array_equal(tg.tg_count_directed_global(g), want)


@pytest.mark.parametrize("hub,L", [(100, 1), (126, 2), (127, 2), (128, 3), (129, 2), (131, 5), (150, 2)])
def test_tetrads(hub, L):
    G = _hub(260, 500, hub, L, hub + L)
    g = tg.tg_build_csr(G.n, G.src, G.dst, G.types, L, directed=True)
    _, want = odir.counts4_of(G, rows=False)
    assert np.array_equal(tg.tg_count_directed4_global(g), want)
