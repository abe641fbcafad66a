"""The weight-stacked exact-slice GEMM at the edges of its narrow tiles (16 and 32 columns, 128 rows, 16 values
of K a stage), against the oracle.  The 64-column tiles and the drains: test_gpu_dst_drains.py."""
import ctypes as C

import numpy as np
import pytest

from oracle import dst as odst
from paper_1005_0542_gb300 import lagwave as L

from gpu_util import make_ctx, dev, empty, host, plan, ptr

pytestmark = pytest.mark.gpu
RNG = np.random.default_rng(641)
TOL = 1e-14  # per row: float64 rounding of the result (2^-53) and of the oracle's K-term float64 sums


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    L.lag_destroy(c)


def _row_err(y, ref):
    sc = np.maximum(np.abs(ref).max(axis=-1, keepdims=True), 1e-300)
    return np.linalg.norm((y - ref) / sc, axis=-1) / np.linalg.norm(ref / sc, axis=-1)


# row lengths: ceil(n/2) around multiples of 16 and 64, short and long stage counts, and row counts around
# the 128-row tile
@pytest.mark.parametrize("nx", [16, 31, 33, 95, 127, 128, 129, 384, 385, 577, 768, 961, 1216, 1537, 1921, 2047, 2048])
@pytest.mark.parametrize("nz", [1, 127, 129])
def test_tile_edges(ctx, nx, nz):
    x = RNG.standard_normal((1, nz, nx)) * 10.0 ** RNG.uniform(-3, 3, (1, nz, nx))
    p = plan(ctx, nx, nz, 5.0, 5.0, 1.0, 1.0, 0.1)
    xd, yd = dev(x), empty(x.shape)
    L.check(L.lag_precond_dst(p, ptr(xd), ptr(yd), 1), ctx)
    assert L.lag_precond_status(p) == L.LAG_OK
    assert _row_err(host(yd), odst.dst_x(x)).max() < TOL
    L.lag_precond_destroy(p)


# rows whose digits are all equal and of one sign against the DCT's constant mode, and rows of the extreme
# values of a digit
@pytest.mark.parametrize("nz", [64, 1000, 2048])
@pytest.mark.parametrize("value", [1.0, -1.0, 1.0 - 2.0 ** -53, 0.5 + 0.5 / 255, -(0.5 + 2.0 ** -40)])
def test_extreme_sums(ctx, nz, value):
    nr = 130
    p = C.c_void_p()
    g = L.grid(nr, nz, 5.0, 5.0, cylindrical=True)
    L.check(L.lag_precond_create_sep(ctx, C.byref(g), 1.0, 1.0, 0.1, L.LAG_FP64, 0, C.byref(p)), ctx)
    x = np.full((1, nr, nz), value)
    x[0, 1::2] *= np.where(np.arange(nz) % 2, -1.0, 1.0)
    xd, yd, zd = dev(x), empty(x.shape), empty(x.shape)
    L.check(L.lag_precond_dst(p, ptr(xd), ptr(yd), 1), ctx)
    y = host(yd)
    # the constant rows are the mode q = 0 alone, sqrt(n) value; every row comes back from its modes
    want = np.zeros((nr // 2, nz))
    want[:, 0] = value * np.sqrt(nz)
    assert np.abs(y[0, 0::2] - want).max() < TOL * np.abs(want).max()
    L.check(L.lag_precond_dst_inverse(p, ptr(yd), ptr(zd), 1), ctx)
    assert _row_err(host(zd), x).max() < TOL
    L.lag_precond_destroy(p)
