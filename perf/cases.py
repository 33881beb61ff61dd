"""Performance cases of the typed-graphlet library, through its Python entry points.

Every case draws its graph from a seed with torch or numpy generators, in the
families the library is used on: Erdos-Renyi, Chung-Lu (exponent 2.1) and
R-MAT graphs with uniform or Zipf node types, undirected and directed.  Inputs
that a program holds on the device are made there; the serving case takes host
arrays, as its requests come from outside.

Kinds of a case:
  count     raw edge draws on the device -> ``tg_build_csr`` + ``tg_count_global``
            (a new graph counted once: the benchmark's step)
  rows      ``tg_count_per_edge`` of a resident graph into a device tensor with
            room for a row per raw pair
  directed  ``tg_count_directed_global`` of a resident directed graph
  directed4 ``tg_count_directed4_global`` of a resident directed graph
  batch     one run of a ``Batch`` plan over many small resident graphs
  serve     a burst of requests through a ``Server``, every result awaited
"""
from __future__ import annotations

import math
from itertools import product

import numpy as np
import torch

import paper_1901_10026_gb300 as tg

# Scratch the library keeps mapped between calls, as a counting or serving
# loop sets it (the benchmark's default).
RETAIN_BYTES = 64 << 30


def listed():
    return [
        # The smallest call: ER-1000 (p = 0.01), the parity graph of the tests;
        # launches and synchronisations count.
        dict(name="count_er_1k", kind="count", family="er", n=1000, m=5000, L=3, zipf=0.0, k=4),
        # The number-of-types sweep's graph without hubs (100K nodes, 1M edges).
        dict(name="count_er_100k", kind="count", family="er", n=100_000, m=1_000_000, L=5,
             zipf=0.0, k=4),
        # One member of a type-permutation null model (Chung-Lu, 100K nodes,
        # 1M edges, L = 5 Zipf types): the same count over many medium graphs.
        dict(name="count_cl_100k", kind="count", family="cl", n=100_000, m=1_200_000, L=5,
             zipf=1.2, k=4),
        # CL-1M: a skewed graph of 8M edges, the second benchmark workload.
        dict(name="count_cl_1m", kind="count", family="cl", n=1_000_000, m=9_720_000, L=5,
             zipf=1.2, k=4),
        # R-MAT, the headline family (edge factor 16, L = 8), at the largest
        # scale whose step stays within a second or so.
        dict(name="count_rmat_21", kind="count", family="rmat", n=1 << 21, m=16 << 21, L=8,
             zipf=0.0, k=4),
        # 3-node graphlets only, on the largest graph of the scalability
        # series (ER, 1M nodes, average degree 10).
        dict(name="count3_er_1m", kind="count", family="er", n=1_000_000, m=5_000_000, L=3,
             zipf=0.0, k=3),
        # Per-edge graphlet rows of a skewed graph: features of every edge for
        # a downstream model.
        dict(name="rows_cl_125k", kind="rows", family="cl", n=125_000, m=1_200_000, L=5,
             zipf=1.2, k=4, level="graphlet"),
        # Per-edge orbit rows, many types (L = 8), a graph without hubs.
        dict(name="orbits_er_30k", kind="rows", family="er", n=30_000, m=240_000, L=8, zipf=0.0,
             k=4, level="orbit"),
        # Directed typed triads of a skewed digraph.
        dict(name="directed_rmat_20", kind="directed", family="rmat", n=1 << 20, m=16 << 20, L=8,
             zipf=0.0),
        # Directed typed 4-node graphlets (199 classes) with reciprocal arcs.
        dict(name="directed4_er_20k", kind="directed4", family="er_arcs", n=20_000, m=120_000,
             L=2, zipf=0.0, recip=0.3),
        # A batch of small graphs of mixed sizes and type counts, per-edge rows.
        dict(name="batch_400", kind="batch", graphs=400, n_lo=20, n_hi=5000),
        # A saturated server: requests of 1e3 to 2e6 edges, L = 6.
        dict(name="serve_48", kind="serve", requests=48, m_lo=1000, m_hi=2_000_000, L=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count"] * 5 + ["rows", "rows", "directed", "directed4", "batch", "serve"])
    if kind == "count":
        family = rng.choice(["er", "cl", "rmat"])
        k = rng.choice([4, 4, 4, 3])
        if family == "rmat":
            n = 1 << rng.randint(12, 20)
            return dict(kind=kind, family=family, n=n, m=int(n * rng.uniform(8, 16)),
                        L=rng.randint(2, 9), zipf=0.0, k=k)
        n = _log_int(rng, 100, 1_000_000)
        deg = rng.uniform(4, 18) if n > 1000 else rng.uniform(4, 12)
        return dict(kind=kind, family=family, n=n, m=int(n * deg / 2), L=rng.randint(1, 9),
                    zipf=rng.choice([0.0, 1.2]), k=k)
    if kind == "rows":
        level = rng.choice(["graphlet", "orbit"])
        n = _log_int(rng, 500, 60_000)
        return dict(kind=kind, family=rng.choice(["er", "cl"]), n=n,
                    m=int(n * rng.uniform(4, 9)), L=rng.randint(1, 8),
                    zipf=rng.choice([0.0, 1.2]), k=rng.choice([3, 4, 4]), level=level)
    if kind == "directed":
        if rng.random() < 0.5:
            n = 1 << rng.randint(12, 19)
            return dict(kind=kind, family="rmat", n=n, m=int(n * rng.uniform(8, 16)),
                        L=rng.randint(1, 8), zipf=0.0)
        n = _log_int(rng, 500, 500_000)
        return dict(kind=kind, family="er_arcs", n=n, m=int(n * rng.uniform(3, 9)),
                    L=rng.randint(1, 8), zipf=0.0, recip=round(rng.uniform(0, 0.5), 3))
    if kind == "directed4":
        n = _log_int(rng, 200, 18_000)
        return dict(kind=kind, family="er_arcs", n=n, m=int(n * rng.uniform(3, 6)),
                    L=rng.randint(1, 3), zipf=0.0, recip=round(rng.uniform(0, 0.4), 3))
    if kind == "batch":
        return dict(kind=kind, graphs=rng.randint(20, 380), n_lo=20, n_hi=_log_int(rng, 500, 5000))
    return dict(kind=kind, requests=rng.randint(8, 44), m_lo=1000,
                m_hi=_log_int(rng, 20_000, 2_000_000), L=rng.randint(2, 6))


# ------------------------------------------------------------------- inputs --
# Graphs of up to this many draws are made on the host (the same values on
# every machine), larger ones on the device.
HOST_DRAWS = 200_000


def _generator(seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(seed)
    return g


def _types(n, L, zipf, g):
    """Node types: uniform, or P(t) proportional to (t + 1)^-zipf."""
    p = torch.arange(1, L + 1, dtype=torch.float64, device=g.device) ** -zipf
    cdf = torch.cumsum(p, 0) / p.sum()
    x = torch.rand(n, dtype=torch.float64, generator=g, device=g.device)
    return torch.searchsorted(cdf, x, right=True).clamp_(max=L - 1).to(torch.uint8)


def _edges(case, g):
    """Raw draws (loops and repeats included) as two int32 tensors."""
    n, m, dev = case["n"], case["m"], g.device
    if case["family"] in ("er", "er_arcs"):
        src = torch.randint(0, n, (m,), generator=g, device=dev, dtype=torch.int32)
        dst = torch.randint(0, n, (m,), generator=g, device=dev, dtype=torch.int32)
        if case["family"] == "er_arcs":  # each arc's reverse with probability recip
            back = torch.rand(m, generator=g, device=dev) < case["recip"]
            src, dst = torch.cat([src, dst[back]]), torch.cat([dst, src[back]])
        return src, dst
    if case["family"] == "cl":  # endpoints i.i.d. proportional to (v + 1)^(-1 / (2.1 - 1))
        w = torch.arange(1, n + 1, dtype=torch.float64, device=dev) ** (-1.0 / 1.1)
        cdf = torch.cumsum(w, 0)
        cdf /= cdf[-1].clone()
        return tuple(
            torch.searchsorted(cdf, torch.rand(m, dtype=torch.float64, generator=g, device=dev),
                               right=True).clamp_(max=n - 1).to(torch.int32) for _ in range(2))
    # R-MAT: one quadrant choice (0.57, 0.19, 0.19, 0.05) per level, no noise
    src = torch.zeros(m, dtype=torch.int32, device=dev)
    dst = torch.zeros(m, dtype=torch.int32, device=dev)
    for _ in range(n.bit_length() - 1):
        x = torch.rand(m, generator=g, device=dev)
        src = 2 * src + (x >= 0.76)
        dst = 2 * dst + (((x >= 0.57) & (x < 0.76)) | (x >= 0.95))
    return src.to(torch.int32), dst.to(torch.int32)


def _graph(case, seed, device=None):
    """(n, src, dst, types, L) of a case, on the GPU unless another device is named."""
    small = case["m"] <= HOST_DRAWS
    g = _generator(seed, "cpu" if small else "cuda")
    src, dst = _edges(case, g)
    types = _types(case["n"], case["L"], case["zipf"], g)
    device = device or "cuda"
    return case["n"], src.to(device), dst.to(device), types.to(device), case["L"]


def _batch_sizes(case):
    """(n, raw pairs, L) of a batch's graphs: n log-uniform, average degree 4 to 32,
    L uniform in 2..8."""
    r = np.random.Generator(np.random.Philox(np.random.SeedSequence([31, case["graphs"]])))
    sizes = []
    for _ in range(case["graphs"]):
        n = int(math.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]))))
        deg = min(float(r.uniform(4.0, 32.0)), (n - 1) / 2.0)
        sizes.append((n, max(1, int(round(n * deg / 2.0))), int(r.integers(2, 9))))
    return sizes


def _batch_graphs(case, seed):
    """The graphs of a batch: half ER, half Chung-Lu."""
    r = np.random.Generator(np.random.Philox(np.random.SeedSequence([33, seed])))
    for i, (n, m, L) in enumerate(_batch_sizes(case)):
        if i % 2 == 0:
            src, dst = (r.integers(0, n, m).astype(np.int32) for _ in range(2))
        else:
            cdf = np.cumsum((np.arange(n) + 1.0) ** (-1.0 / float(r.uniform(1.0, 1.8))))
            src, dst = (np.minimum(np.searchsorted(cdf, r.random(m) * cdf[-1], side="right"),
                                   n - 1).astype(np.int32) for _ in range(2))
        yield n, src, dst, r.integers(0, L, n).astype(np.uint8), L


def _requests(case, seed):
    """Chung-Lu request graphs in host memory, draws log-uniform, average degree 16."""
    r = np.random.Generator(np.random.Philox(np.random.SeedSequence([37, seed])))
    reqs = []
    for q in range(case["requests"]):
        m = int(math.exp(r.uniform(math.log(case["m_lo"]), math.log(case["m_hi"]))))
        c = dict(family="cl", n=max(16, m // 8), m=m, L=case["L"], zipf=0.0)
        n, src, dst, types, L = _graph(c, (seed * 1009 + q) % (1 << 31), "cpu")
        reqs.append((n, src.numpy(), dst.numpy(), types.numpy(), L))
    return reqs


# -------------------------------------------------------------------- state --
def prepare(case, seed):
    tg.tg_set_memory_retention(RETAIN_BYTES)
    kind = case["kind"]
    if kind == "batch":
        graphs = [tg.tg_build_csr(*G) for G in _batch_graphs(case, seed)]
        sizes = [m * tg.tg_slots(L, 4, tg.TG_GRAPHLET) for _, m, L in _batch_sizes(case)]
        rows = torch.zeros(sum(sizes), dtype=torch.int64, device="cuda")
        outs = list(rows.split(sizes))
        return dict(case=case, rows=rows,
                    plan=tg.Batch(graphs, 4, tg.TG_BATCH_PER_EDGE_GRAPHLET, outs))
    if kind == "serve":
        return dict(case=case, requests=_requests(case, seed),
                    server=tg.Server(slots=4, batch_max=32, batch_edges=20000))
    G = _graph(case, seed)
    if kind == "count":
        return dict(case=case, graph=G)
    g = tg.tg_build_csr(*G, directed=kind.startswith("directed"))
    state = dict(case=case, graph=g)
    if kind == "rows":
        level = tg.TG_ORBIT if case["level"] == "orbit" else tg.TG_GRAPHLET
        state["level"] = level
        state["rows"] = torch.zeros((case["m"], tg.tg_slots(g.L, case["k"], level)),
                                    dtype=torch.int64, device="cuda")
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "count":
        g = tg.tg_build_csr(*state["graph"])
        out = tg.tg_count_global(g, case["k"])
        g.close()
        return out
    if kind == "rows":
        return tg.tg_count_per_edge(state["graph"], case["k"], state["level"], state["rows"])
    if kind == "directed":
        return tg.tg_count_directed_global(state["graph"])
    if kind == "directed4":
        return tg.tg_count_directed4_global(state["graph"])
    if kind == "batch":
        state["plan"].run()
        return state["rows"]
    server = state["server"]
    tickets = [server.submit(*req) for req in state["requests"]]
    return np.concatenate([server.wait(t)[0] for t in tickets])


# --------------------------------------------------------------------- work --
def _slots(case, L):
    P = L * (L + 1) // 2
    if case.get("k", 4) == 3:
        return 2 * L
    return 2 * L + (10 if case.get("level") == "orbit" else 6) * P


def work(case):
    """Bytes: the raw pairs (8 B) or a resident graph's adjacency (one packed
    4 B entry per direction of a pair) and the node types read once, the
    outputs written once.  Operations: one per pair read (the enumeration
    behind a count depends on the graph's structure and is left out)."""
    kind = case["kind"]
    if kind == "batch":
        sizes = _batch_sizes(case)
        return {"bytes": sum(n + m * (8 + 8 * _slots(case, L)) for n, m, L in sizes),
                "flops": sum(m for _, m, _ in sizes)}
    if kind == "serve":
        lo, hi = case["m_lo"], case["m_hi"]
        m = case["requests"] * (hi - lo) / math.log(hi / lo)
        return {"bytes": 8 * m + m / 8, "flops": m}
    n, m, L = case["n"], case["m"], case["L"]
    if case["family"] == "er_arcs":
        m = int(m * (1 + case["recip"]))
    out = 8 * 6 * math.comb(L + 3, 4)
    if kind == "rows":
        out = 8 * m * _slots(case, L)
    elif kind == "directed":
        out = 8 * 13 * math.comb(L + 2, 3)
    elif kind == "directed4":
        out = 8 * 199 * math.comb(L + 3, 4)
    return {"bytes": 8 * m + n + out, "flops": m}


# -------------------------------------------------------------------- exact --
def _rank(types):
    """Colex rank of a type multiset."""
    return sum(math.comb(c + q, q + 1) for q, c in enumerate(sorted(types)))


def exact(case, seed):
    """Global counts of a small graph from dense typed adjacency products:
    non-induced copies of every pattern per type multiset, then the
    containment inversion."""
    if case["kind"] != "count" or case["n"] > 1500 or case["m"] > HOST_DRAWS:
        return None
    n, src, dst, types, L = (x.numpy() if hasattr(x, "numpy") else x
                             for x in _graph(case, seed, "cpu"))
    A = np.zeros((n, n))
    A[src, dst] = A[dst, src] = 1.0
    np.fill_diagonal(A, 0.0)
    ty = types.astype(np.int64)
    H = np.eye(L)[ty]                    # n x L type indicator
    d = A @ H                            # typed degrees
    W = np.stack([(A * H[:, t]) @ A for t in range(L)])  # W[t][x, y]: middles of type t
    u, v = np.nonzero(np.triu(A))
    tau = W[:, u, v].T                   # per edge, typed triangles
    by = [np.nonzero(ty == t)[0] for t in range(L)]

    def block(count, size):
        out = np.zeros(math.comb(L + size - 1, size))
        for key, value in count:
            out[_rank(key)] += value
        return out

    edge_of = {(a, b): np.nonzero((ty[u] == a) & (ty[v] == b))[0]
               for a, b in product(range(L), repeat=2)}
    edges = block((((a, b), float(e.size)) for (a, b), e in edge_of.items()), 2)
    tri = block((((a, b, c), tau[e, c].sum() / 3) for (a, b), e in edge_of.items()
                 for c in range(L)), 3)
    p3 = block((((t, a, b), (d[by[t], a] * (d[by[t], b] - (a == b))).sum() / 2)
                for t, a, b in product(range(L), repeat=3)), 3)
    blocks = [edges, p3 - 3 * tri, tri]
    if case["k"] == 4:
        eye = np.eye(L)
        s4 = block((((t, a, b, c), (d[by[t], a] * (d[by[t], b] - eye[a, b]) *
                                    (d[by[t], c] - eye[a, c] - eye[b, c])).sum() / 6)
                    for t, a, b, c in product(range(L), repeat=4)), 4)
        p4 = block((((a, b, c, f), ((d[u[e], c] - eye[b, c]) * (d[v[e], f] - eye[a, f]) -
                                    (c == f) * tau[e, c]).sum())
                    for (a, b), e in edge_of.items() for c, f in product(range(L), repeat=2)), 4)
        dia = block((((a, b, c, f), (tau[e, c] * (tau[e, f] - eye[c, f])).sum() / 2)
                     for (a, b), e in edge_of.items() for c, f in product(range(L), repeat=2)), 4)
        at = np.zeros((n, L, L))         # ordered typed triangles at a node
        for c in range(L):
            for x, y in ((u, v), (v, u)):
                np.add.at(at, (x, ty[y], c), tau[:, c])
        tt = block((((t, a, b, c), (at[by[t], a, b] * (d[by[t], c] - eye[a, c] - eye[b, c])).sum() / 2)
                    for t, a, b, c in product(range(L), repeat=4)), 4)
        off = 1.0 - np.eye(n)
        c4 = []
        for a, b in product(range(L), repeat=2):
            sel = np.ix_(by[a], by[b])
            for c, f in product(range(L), repeat=2):
                w = W[c][sel] * off[sel]
                c4.append(((a, b, c, f), (w * (W[f][sel] - (c == f))).sum() / 8))
        c4 = block(c4, 4)
        k4 = []
        for e in range(u.size):
            T = np.nonzero(A[u[e]] * A[v[e]])[0]
            if T.size > 1:
                q = H[T].T @ A[np.ix_(T, T)] @ H[T]
                k4 += [((ty[u[e]], ty[v[e]], a, b), q[a, b] / 12)
                       for a, b in zip(*np.nonzero(q))]
        k4 = block(k4, 4)
        dia = dia - 6 * k4
        tt = tt - 4 * dia - 12 * k4
        c4 = c4 - dia - 3 * k4
        s4 = s4 - tt - 2 * dia - 4 * k4
        p4 = p4 - 2 * tt - 4 * c4 - 6 * dia - 12 * k4
        blocks += [p4, s4, c4, tt, dia, k4]
    return np.rint(np.concatenate(blocks)).astype(np.int64).view(np.uint64)
