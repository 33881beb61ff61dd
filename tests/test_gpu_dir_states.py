"""Global directed triads of a graph whose adjacency entries lost their direction: every
entry carries an arc, so a count that meets one without reports an internal error, by
both ways of counting, and counts right again once the graph is built anew."""
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


def _graph(n, m, hub, L):
    r = np.random.default_rng(m)
    other = r.permutation(np.arange(1, n))[:hub]
    src = np.concatenate([r.integers(0, n, m), np.zeros(hub, int)]).astype(np.int32)
    dst = np.concatenate([r.integers(0, n, m), other]).astype(np.int32)
    return tg.tg_build_csr(n, src, dst, r.integers(0, L, n).astype(np.uint8), L, directed=True)


@pytest.mark.parametrize("n,m,hub,L", [(500, 3000, 100, 3), (60_000, 240_000, 200, 4), (60_000, 240_000, 900, 4),
                                       (60_000, 350_000, 900, 9)])
@pytest.mark.parametrize("where", ["hub", "last"])
def test_entry_without_a_state(n, m, hub, L, where):
    g = _graph(n, m, hub, L)
    want = tg.tg_count_directed_global(g)
    # the hub's first entries (its id is 0), or the last lists' entries
    first, count = (0, 8) if where == "hub" else (2 * g.M - 8, 8)
    err = internals.load().tgi_clear_states(g.handle, ctypes.c_int64(first), ctypes.c_int64(count))
    assert err == 0
    with pytest.raises(tg.TGError) as e:
        tg.tg_count_directed_global(g)
    assert e.value.status == tg.TG_EINTERNAL
    assert np.array_equal(tg.tg_count_directed_global(_graph(n, m, hub, L)), want)
