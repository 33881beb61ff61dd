"""The checks between the totals of a whole-graph count (csrc/tg_sums.cu): totals counted
on the host from the definitions pass and give the library's sums; one entry off by one
sets the error that a count reports as TG_EINTERNAL."""
import ctypes

import numpy as np
import pytest

import paper_1901_10026_gb300 as tg
from tests import internals

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    internals.load()


def _graph(kind, L):
    r = np.random.default_rng(L)
    n = 14 if kind == "clique" else 45
    u, v = np.triu_indices(n, 1)
    if kind == "random":
        keep = r.random(u.size) < 0.3
        u, v = u[keep], v[keep]
    types = (np.arange(n) % L).astype(np.uint8)
    return tg.tg_build_csr(n, u.astype(np.int32), v.astype(np.int32), types, L)


def _totals(g, k, mistake, at=0, type_=0):
    hist = np.zeros(tg.tg_global_len(g.L, k), np.uint64)
    err = ctypes.c_uint(0)
    r = internals.load().tgi_sum_totals(g.handle, k, mistake, ctypes.c_int64(at), type_,
                                        hist.ctypes.data_as(ctypes.c_void_p), ctypes.byref(err))
    assert r == 0
    return hist, err.value


@pytest.mark.parametrize("L", [1, 2, 4, 5, 8, 9, 16])
@pytest.mark.parametrize("k", [3, 4])
@pytest.mark.parametrize("kind", ["random", "clique"])
def test_right_totals_pass(kind, k, L):
    g = _graph(kind, L)
    hist, err = _totals(g, k, 0)
    assert err == 0
    assert np.array_equal(hist, tg.tg_count_range(g, k, 0, g.M))
    assert np.array_equal(hist, tg.tg_count_shard(g, k, 0, 1))


@pytest.mark.parametrize("L", [1, 2, 5, 8, 9, 16])
@pytest.mark.parametrize("mistake", [1, 2, 3, 4])
def test_wrong_edge_and_node_totals(mistake, L):
    g = _graph("random", L)
    r = np.random.default_rng(mistake)
    for _ in range(6):
        _, err = _totals(g, 4, mistake, int(r.integers(0, g.M)), int(r.integers(0, L)))
        assert err != 0


@pytest.mark.parametrize("L", [1, 2, 5, 9])
@pytest.mark.parametrize("mistake", [5, 7, 8])
def test_wrong_enumerations(mistake, L):
    """In a clique every 4-cycle lies in a 4-clique: one less, or a clique more or less,
    leaves a negative number of induced 4-cycles or diamonds."""
    g = _graph("clique", L)
    for at in range(tg.tg_config_count(L, 4)):
        _, err = _totals(g, 4, mistake, at)
        assert err != 0


@pytest.mark.parametrize("L", [1, 4])
def test_wrong_triangles_of_three_nodes(L):
    """k = 3 in a clique: more triangles than 3-paths."""
    _, err = _totals(_graph("clique", L), 3, 1, 5, L - 1)
    assert err != 0
