"""Whole-graph sums from node and edge totals (csrc/tg_sums.cu) against the
second oracle, bit-exact, at the edges of its tiles: 1, 31, 32, 33 edges (a
warp's chunk), around one CTA's 256, every bound of the type templates
(L = 4 | 5, 8 | 9, 16), isolated nodes, a hub above the one-thread degree."""
import numpy as np
import pytest

import paper_1901_10026_gb300 as tg
from oracle import o2
from paper_1901_10026_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_10026_gb300 import build
    build.build()
    o2.build()


@pytest.mark.parametrize("L", [1, 2, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("n,m", [(3, 1), (40, 31), (40, 32), (40, 33), (70, 255), (70, 257), (300, 4000)])
def test_totals_at_tile_edges(n, m, L):
    G = synth.er_exact(n, m, L, seed=3)
    src, dst = G.src.copy(), G.dst.copy()
    if m > 200:  # a hub over nodes 0..: more than 64 neighbours
        src = np.concatenate([src, np.zeros(n - 1, np.int32)])
        dst = np.concatenate([dst, np.arange(1, n, dtype=np.int32)])
    iso = n + 5  # isolated nodes at the end
    types = np.concatenate([G.types, np.zeros(5, np.uint8)])
    g = tg.tg_build_csr(iso, src, dst, types, L)
    for k in (3, 4):
        want = o2.global_counts(iso, src, dst, types, L, k)
        assert np.array_equal(tg.tg_count_global(g, k), want), k
