"""Global directed triads of a graph with more ids than the shared-memory map of a hub's
neighbours covers (911,424 at L = 1): the hubs' triangles lie on nodes of the smallest
degrees, whose ids come last, so every one of them is found by a search."""
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


@pytest.mark.parametrize("L", [1, 2])
def test_triangles_beyond_the_map(L):
    r = np.random.default_rng(L)
    n, ring = 1_200_000, 20_000
    first = n - ring  # the ring's nodes: two ring edges, one or two to the hubs 0 and 1
    x = first + np.arange(ring)
    src = [r.integers(0, first, 4_800_000), np.where(r.random(ring) < 0.5, 0, x), x, np.full(ring // 3, 1)]
    dst = [r.integers(0, first, 4_800_000), np.where(src[1] == 0, x, 0), np.roll(x, 1), x[: ring // 3]]
    back = r.permutation(ring)[: ring // 4]
    src.append(np.roll(x, 1)[back])
    dst.append(x[back])
    G = synth.TypedEdgeList(n, np.concatenate(src).astype(np.int32), np.concatenate(dst).astype(np.int32),
                            r.integers(0, L, n).astype(np.uint8), L, "ring")
    g = tg.tg_build_csr(G.n, G.src, G.dst, G.types, L, directed=True)
    assert g.n_nonisolated > 1_100_000 and g.max_degree >= ring
    _, want = odir.counts_of(G)
    assert np.array_equal(tg.tg_count_directed_global(g), want)
