"""The radix sort (csrc/tg_prim.cu) when tiles do not wait for the tiles before them: with
no idle look, one, or the library's number, a tile that is late is counted by the tile
that needs it, and keys and values come out as a stable sort has them."""
import ctypes

import numpy as np
import pytest

from tests import internals

pytestmark = pytest.mark.gpu
LOOKS = 1 << 18  # the library's


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    internals.load()


@pytest.mark.parametrize("looks", [-1, 0, 1, LOOKS])
@pytest.mark.parametrize("values", [False, True])
@pytest.mark.parametrize("n,bits", [(12288, 20), (12289, 20), (16384, 8), (16385, 37), (200_001, 17),
                                    (60_000, 64), (1_000_003, 30)])
def test_late_tiles(n, bits, values, looks):
    r = np.random.default_rng(n)
    keys = r.integers(0, 1 << bits, n, dtype=np.uint64) if bits < 64 else \
        r.integers(0, 1 << 64, n, dtype=np.uint64)
    keys[: n // 3] &= np.uint64(0xff)  # many equal digits
    vals = np.arange(n, dtype=np.uint32)
    order = np.argsort(keys, kind="stable")
    got, gv = keys.copy(), vals.copy()
    assert internals.load().tgi_sort(ctypes.c_int64(n), bits, looks, got.ctypes.data_as(ctypes.c_void_p),
                                     gv.ctypes.data_as(ctypes.c_void_p) if values else None) == 0
    assert np.array_equal(got, keys[order])
    if values:
        assert np.array_equal(gv, vals[order])
