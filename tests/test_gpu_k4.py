"""4-cliques from bitmaps of the up lists (csrc/tg_k4.cu) at the edges of their
classes, in global totals and per-edge rows, and the per-edge 4-cycle waves
(k_c4_wedges), against the oracles and closed forms.

The lowest node of a clique of m nodes has an up list of m - 1 entries.  For
lists beyond shared memory, complete bipartite graphs with a few edges inside
one side: every node of the other side has that side as its up list."""
from math import comb

import numpy as np
import pytest

import oracle
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
    oracle.build()
    o2.build()


def _check(n, src, dst, types, L, sample=60):
    g = tg.tg_build_csr(n, src, dst, types, L)
    assert np.array_equal(tg.tg_count_global(g, 4), o2.global_counts(n, src, dst, types, L, 4))
    rows = tg.tg_count_per_edge(g, 4, tg.TG_ORBIT)
    e = np.unique(np.random.default_rng(5).integers(0, g.M, sample))
    want = oracle.OracleGraph(n, src, dst, types, L).per_edge(4, "orbit", edges=e)
    bad = np.argwhere(rows[e] != want)
    assert bad.shape[0] == 0, bad[:5]


@pytest.mark.parametrize("L", [1, 3, 8, 16])
@pytest.mark.parametrize("m", [4, 33, 34, 65, 161, 162])
def test_cliques_at_class_bounds(m, L):
    u, v = np.triu_indices(m, 1)
    _check(m, u.astype(np.int32), v.astype(np.int32), (np.arange(m) * 5 % 7 % L).astype(np.uint8), L)


@pytest.mark.parametrize("n,p,L", [(60, 0.7, 4), (420, 0.5, 9), (700, 0.9, 5), (560, 0.99, 16)])
def test_dense_random(n, p, L):
    g = synth.rng(4, n, L)
    u, v = synth.erdos_renyi(n, p, g)
    _check(n, u, v, synth.uniform_types(n, L, g), L, sample=25)


def _bipartite(m, inner):
    """K_{m,m} (sides 0..m-1 and m..2m-1) with the first `inner` nodes a clique."""
    a, b = np.meshgrid(np.arange(m), np.arange(m, 2 * m), indexing="ij")
    u, v = np.triu_indices(inner, 1)
    return (2 * m, np.concatenate([a.ravel(), u]).astype(np.int32),
            np.concatenate([b.ravel(), v]).astype(np.int32))


@pytest.mark.parametrize("m", [2100, 4110])  # rows of 66 words; lists beyond every row
def test_long_up_lists(m):
    inner = 9
    n, src, dst = _bipartite(m, inner)
    g = tg.tg_build_csr(n, src, dst, np.zeros(n, np.uint8), 1)
    got = tg.tg_count_global(g, 4)
    assert got[-1] == m * comb(inner, 3) + comb(inner, 4)
    if m > 3000:
        return
    import torch
    rows = torch.zeros((g.M, tg.tg_slots(1, 4, tg.TG_ORBIT)), dtype=torch.int64, device="cuda")
    tg.tg_count_per_edge(g, 4, tg.TG_ORBIT, rows)
    u, v = tg.tg_edge_list(g)
    k4 = rows[:, -1].cpu().numpy()
    want = np.where(v < m, comb(inner - 2, 2) + m * (inner - 2),
                    np.where(u < inner, comb(inner - 1, 2), 0))
    assert np.array_equal(k4, want)


@pytest.mark.parametrize("L", [1, 5, 9])
def test_hub_rows(L):
    """Costly anchors in per-edge mode: hubs over a random graph, lists on both
    sides of the whole-warp bound."""
    g = synth.rng(6, L)
    n = 3000
    u, v = synth.erdos_renyi(n, 0.01, g)
    hubs = [np.stack([np.full(900, h), g.integers(0, n, 900)]) for h in (3, 5, 8, 13)]
    src = np.concatenate([u] + [h[0] for h in hubs]).astype(np.int32)
    dst = np.concatenate([v] + [h[1] for h in hubs]).astype(np.int32)
    _check(n, src, dst, synth.uniform_types(n, L, g), L)


@pytest.mark.parametrize("L", [1, 5, 16])
@pytest.mark.parametrize("low", [3, 4, 7, 8, 31, 32])
def test_short_lists_of_members_with_long_lists(low, L):
    """Lowest nodes of `low` members whose own up lists have 200 to 231 entries: the
    members' lists are searched, not scanned, for even and odd numbers of members."""
    core = 232
    u, v = np.triu_indices(core, 1)
    r = np.random.default_rng(low)
    keep = r.random(u.shape[0]) < 0.97
    src, dst = [u[keep]], [v[keep]]
    for x in range(core, core + 40):
        m = r.choice(core, low, replace=False)
        src.append(np.full(low, x))
        dst.append(m)
    n = core + 40
    src = np.concatenate(src).astype(np.int32)
    dst = np.concatenate(dst).astype(np.int32)
    _check(n, src, dst, r.integers(0, L, n).astype(np.uint8), L, sample=20)


@pytest.mark.parametrize("m", [1000, 1984])  # rows of up to 62 words, beyond shared memory
def test_rows_in_global_memory(m):
    inner = 7
    n, src, dst = _bipartite(m, inner)
    g = tg.tg_build_csr(n, src, dst, np.zeros(n, np.uint8), 1)
    assert tg.tg_count_global(g, 4)[-1] == m * comb(inner, 3) + comb(inner, 4)
