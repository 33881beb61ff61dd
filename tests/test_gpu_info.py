"""tg_graph_info's device_bytes: the CSR, and what the graph's counts add to it and keep."""
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


@pytest.mark.parametrize("n,m,L", [(50, 0, 2), (700, 4000, 3), (3000, 9000, 16)])
def test_device_bytes_follow_the_counts(n, m, L):
    r = np.random.default_rng(m)
    g = tg.tg_build_csr(n, r.integers(0, n, m).astype(np.int32), r.integers(0, n, m).astype(np.int32),
                        r.integers(0, L, n).astype(np.uint8), L)
    built = g.info()["device_bytes"]
    assert built == 8 * (n + 1) + 4 * 4 * g.M + 4 * n * (L + 1) + n + 8 * g.M + 4 * n
    lists = built + 8 * (n + 1) + 4 * n * (L + 1) + 16 * g.M
    for k in (3, 4, 4):
        tg.tg_count_global(g, k)
        assert g.info()["device_bytes"] == g.device_bytes == lists
    tg.tg_count_shard(g, 4, 0, 2)
    assert g.device_bytes == lists + 4 * g.M
    tg.tg_work_model(g)
    last = lists + 4 * g.M + (8 * n if g.M else 0)  # without edges the model needs no sums
    assert tg.tg_graph_info(g)["device_bytes"] == last
    g.close()
    assert g.device_bytes == last
