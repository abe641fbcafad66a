"""The mode tile of general float32 tridiagonal solves: the default's half tile on few blocks, and an
explicit choice that runs as asked."""
import ctypes as C

import numpy as np
import pytest

from paper_1005_0542_gb300 import lagwave as L

from gpu_util import make_ctx, dev, host, ptr

pytestmark = pytest.mark.gpu
RNG = np.random.default_rng(652)


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    L.lag_destroy(c)


def _layered(ctx, nx, nz, prec=L.LAG_MIXED):
    rows = np.concatenate([RNG.uniform(2e9, 4e9, 2 * nz), RNG.uniform(1e7, 2e7, nz)])
    ax, az, d = (np.ascontiguousarray(v) for v in rows.reshape(3, nz))
    p = C.c_void_p()
    g = L.grid(nx, nz, 5.0, 4.0)
    (_, pa), (_, pz), (_, pd) = L.f64(ax), L.f64(az), L.f64(d)
    L.check(L.lag_precond_create_layered(ctx, C.byref(g), pa, pz, pd, prec, 0, C.byref(p)), ctx)
    return p


def _solve(ctx, p, r):
    rd, zd = dev(r), dev(np.zeros_like(r))
    L.check(L.lag_precond_tridiag_f32(p, ptr(rd), ptr(zd), r.shape[0]), ctx)
    return host(zd)


# the one partition of two rows that the register kernel takes, ragged last tiles, the longest partitions.
# Each tile runs one mode's sums in the same order, contraction apart: partition length x 2^-24 < 1e-5
@pytest.mark.parametrize("nx,nz", [(17, 2), (39, 64), (100, 1000), (300, 2000)])
def test_explicit_tile_runs_as_asked(ctx, nx, nz):
    p = _layered(ctx, nx, nz)
    many = 1000
    assert L.lag_precond_tri_modes(p, 1) == 8 and L.lag_precond_tri_modes(p, many) == 16
    r = RNG.standard_normal((1, nz, nx)).astype(np.float32)
    ref = _solve(ctx, p, r)
    mt = C.c_int()
    for want in (16, 8):
        L.check(L.lag_precond_set_layout(p, 0, want), ctx)
        L.check(L.lag_precond_info(p, None, None, C.byref(mt)), ctx)
        assert mt.value == want
        for nrhs in (1, many):
            assert L.lag_precond_tri_modes(p, nrhs) == want
        assert np.linalg.norm(_solve(ctx, p, r) - ref) <= 1e-5 * np.linalg.norm(ref)
    L.check(L.lag_precond_set_layout(p, 0, 0), ctx)
    assert L.lag_precond_tri_modes(p, 1) == 8 and L.lag_precond_tri_modes(p, many) == 16
    L.lag_precond_destroy(p)


def test_autotuned_tile_is_the_tile_that_runs(ctx):
    p = _layered(ctx, 96, 128)
    out = [C.c_int() for _ in range(3)]
    ms = C.c_double()
    L.check(L.lag_precond_autotune(p, 1, *map(C.byref, out), C.byref(ms)), ctx)
    assert L.lag_precond_tri_modes(p, 1) == L.lag_precond_tri_modes(p, 1000) == out[1].value
    L.lag_precond_destroy(p)


def test_tiles_of_other_plans_are_the_plan_s(ctx):
    p = _layered(ctx, 96, 128, L.LAG_FP64)
    assert L.lag_precond_tri_modes(p, 1) == L.lag_precond_tri_modes(p, 1000) == 4
    assert L.lag_precond_tri_modes(p, 0) == L.LAG_EINVAL and L.lag_precond_tri_modes(None, 1) == L.LAG_EINVAL
    L.lag_precond_destroy(p)
    p = _layered(ctx, 96, 1, L.LAG_MIXED)  # a single row: the shared-memory kernel's tile
    mt = C.c_int()
    L.check(L.lag_precond_info(p, None, None, C.byref(mt)), ctx)
    assert L.lag_precond_tri_modes(p, 1) == mt.value
    L.lag_precond_destroy(p)
