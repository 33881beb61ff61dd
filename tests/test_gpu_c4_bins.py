"""Binned 4-cycle waves (csrc/tg_cycles.cu, k_c4_bin_*) against the second oracle:
every row width of the far-end table (L = 1, 2 | 3, 4 | 5..8, and the list form
above 8), 16-bit and 32-bit counts (hubs of 65,535 and 65,536 neighbours), types
that fill less than a window, several windows per type, one type holding no node
and isolated nodes among the ids."""
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


@pytest.fixture(autouse=True)
def _all_binned():
    tg.tg_set_tune(c4_bin_fill=1)  # every costly anchor goes to the binned waves
    yield
    tg.tg_set_tune(reset=True)


def _check(n, src, dst, types, L):
    g = tg.tg_build_csr(n, src.astype(np.int32), dst.astype(np.int32), types, L)
    want = o2.global_counts(n, src.astype(np.int32), dst.astype(np.int32), types, L, 4)
    assert np.array_equal(tg.tg_count_global(g, 4), want)


@pytest.mark.parametrize("L", [1, 2, 3, 4, 5, 6, 8, 9, 16])
@pytest.mark.parametrize("n", [900, 20000])
def test_row_widths(n, L):
    r = np.random.default_rng([n, L])
    m = 4 * n
    src, dst = [r.integers(0, n, m)], [r.integers(0, n, m)]
    for h in range(6):  # hubs over a random part of the nodes
        part = r.permutation(n)[: n // 2]
        src.append(np.full(part.size, 11 * h))
        dst.append(part)
    types = r.integers(0, L, n + 40).astype(np.uint8)
    if L > 2:
        types[types == 1] = 2  # a type without nodes
    _check(n + 40, np.concatenate(src), np.concatenate(dst), types, L)


@pytest.mark.parametrize("b", [65535, 65536])
@pytest.mark.parametrize("L", [2, 4, 8])
def test_count_widths(b, L):
    r = np.random.default_rng([b, L])
    n = b + 2
    mid = np.arange(2, n)
    src = np.concatenate([np.zeros(b), np.ones(b // 2), r.integers(2, n, 30000)])
    dst = np.concatenate([mid, mid[: b // 2], r.integers(2, n, 30000)])
    _check(n, src, dst, r.integers(0, L, n).astype(np.uint8), L)


@pytest.mark.parametrize("y", [254, 255, 256, 257, 511])
@pytest.mark.parametrize("x", [257, 129])
@pytest.mark.parametrize("L", [5, 8])
def test_full_tables(x, y, L):
    """K_{x,y} with leaves on the x side, so that every x is an anchor whose x - 1
    far ends all have y middles of one type: sums of 255^2 over a whole block of
    far ends, the largest a block of byte-sized counts takes, and one more."""
    a, b = np.meshgrid(np.arange(x), x + np.arange(y), indexing="ij")
    leaves = x + y + np.arange(x * 300)
    src = np.concatenate([a.ravel(), np.repeat(np.arange(x), 300)])
    dst = np.concatenate([b.ravel(), leaves])
    n = x + y + leaves.size
    types = np.zeros(n, np.uint8)
    types[x + y:] = L - 1
    types[x: x + y: 7] = 1 if y == 511 else 0
    _check(n, src, dst, types, L)
