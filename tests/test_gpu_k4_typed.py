"""The widest 4-clique kernels (csrc/tg_k4.cu) with several types: rows in global memory of
one, two and four words a lane, whose words are padded type by type, and up lists beyond
every row, in global totals and per edge.

K_{m,m} with a random graph G on some nodes of one side: every node of the other side
has that side as its up list, and the 4-cliques are the triangles of G with each node of
the other side, and those of G."""
from itertools import combinations

import numpy as np
import pytest

import paper_1901_10026_gb300 as tg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1901_10026_gb300 import build
    build.build()


def _graph(m, L, seed):
    """(n, src, dst, types), the nodes of G and its adjacency; types interleaved."""
    r = np.random.default_rng(seed)
    a, b = np.meshgrid(np.arange(m), np.arange(m, 2 * m), indexing="ij")
    nodes = np.sort(r.permutation(m)[:40])
    u, v = np.triu_indices(nodes.size, 1)
    keep = r.random(u.size) < 0.5
    adj = np.zeros((nodes.size, nodes.size), bool)
    adj[u[keep], v[keep]] = adj[v[keep], u[keep]] = True
    src = np.concatenate([a.ravel(), nodes[u[keep]]]).astype(np.int32)
    dst = np.concatenate([b.ravel(), nodes[v[keep]]]).astype(np.int32)
    return (2 * m, src, dst, r.integers(0, L, 2 * m).astype(np.uint8)), nodes, adj


def _cliques(adj, k):
    return [c for c in combinations(range(adj.shape[0]), k) if all(adj[x, y] for x, y in combinations(c, 2))]


def _pair(L, a, b):
    a, b = min(a, b), max(a, b)
    return a * L - a * (a - 1) // 2 + (b - a)


@pytest.mark.parametrize("m,L", [(1000, 5), (1000, 16), (1984, 3), (1500, 16), (2100, 2), (2100, 5), (2100, 16),
                                 (3500, 16), (4110, 2)])
def test_typed_cliques(m, L):
    import torch
    G, nodes, adj = _graph(m, L, m + L)
    t = G[3].astype(int)
    tn = t[nodes]  # types of G's nodes
    other = np.bincount(t[m:], minlength=L)  # of the other side
    tri, quad = _cliques(adj, 3), _cliques(adj, 4)
    want = np.zeros(tg.tg_config_count(L, 4), np.uint64)
    for x, y, z in tri:
        for b in range(L):
            want[tg.tg_config_rank(sorted([tn[x], tn[y], tn[z], b]))] += np.uint64(other[b])
    for q in quad:
        want[tg.tg_config_rank(sorted(tn[list(q)]))] += np.uint64(1)
    g = tg.tg_build_csr(*G, L)
    got = tg.tg_count_global(g, 4)
    assert np.array_equal(got[-want.size:], want)
    # per edge: the 4-cliques by the types of the other two nodes, the last columns of a row
    P = L * (L + 1) // 2
    rows = torch.zeros((g.M, tg.tg_slots(L, 4)), dtype=torch.int64, device="cuda")
    tg.tg_count_per_edge(g, 4, tg.TG_GRAPHLET, rows)
    k4 = rows[:, -P:].cpu().numpy()
    del rows
    u, v = tg.tg_edge_list(g)
    edge = {(int(x), int(y)): e for e, (x, y) in enumerate(zip(u, v)) if y < m}
    exp = np.zeros((g.M, P), np.int64)
    for x, y, z in tri:
        for p, q, r in ((x, y, z), (x, z, y), (y, z, x)):
            e = edge[int(nodes[p]), int(nodes[q])]
            for b in range(L):
                exp[e, _pair(L, tn[r], b)] += other[b]
    for c in quad:
        for p, q in combinations(c, 2):
            r, s = [x for x in c if x not in (p, q)]
            exp[edge[int(nodes[p]), int(nodes[q])], _pair(L, tn[r], tn[s])] += 1
    per = np.zeros((m, P), np.int64)  # of an edge to the other side, by its end in G
    for x, y, z in tri:
        for p, q, r in ((x, y, z), (y, x, z), (z, x, y)):
            per[nodes[p], _pair(L, tn[q], tn[r])] += 1
    across = v >= m
    exp[across] = per[u[across]]
    assert np.array_equal(k4, exp)
