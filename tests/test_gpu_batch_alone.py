"""A right-hand side's result is the same, bit for bit, alone and in a batch: no sum and no choice of kernel
that enters it depends on how many others run with it."""
import ctypes as C

import numpy as np
import pytest

from paper_1005_0542_gb300 import lagwave as L

from gpu_util import make_ctx, dev, empty, host, ptr

pytestmark = pytest.mark.gpu
H, D = 200.0, 5.0


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    L.lag_destroy(c)


def _precond(ctx, g, prec, plan, nx, nz, mid, rng):
    p = C.c_void_p()
    if plan == "layered":
        n = nx if g.cylindrical else nz
        rows = [np.ascontiguousarray(v * rng.uniform(0.9, 1.1, n)) for v in mid]
        (_, pa), (_, pz), (_, pd) = (L.f64(v) for v in rows)
        L.check(L.lag_precond_create_layered(ctx, C.byref(g), pa, pz, pd, prec, 0, C.byref(p)), ctx)
    else:
        L.check(L.lag_precond_create_sep(ctx, C.byref(g), *mid, prec, 0, C.byref(p)), ctx)
    return p


def _grid(kind, nx, nz):
    return L.grid(nx, nz, D, D, cylindrical=True) if kind == "cyl" else L.grid(nx, nz, D, D, kind == "surface")


# acoustic systems around every rule on the tiles and blocks of a batch
@pytest.mark.parametrize("prec", [L.LAG_FP64, L.LAG_MIXED])
@pytest.mark.parametrize("kind,plan,nx,nz,nrhs",
                         [("cart", "const", 63, 40, 20), ("cart", "const", 200, 150, 16), ("surface", "layered", 333, 257, 17),
                          ("cart", "const", 640, 500, 6), ("cart", "const", 1500, 700, 2), ("cyl", "const", 100, 130, 24),
                          ("cyl", "layered", 513, 300, 5)])
def test_acoustic_solve(ctx, prec, kind, plan, nx, nz, nrhs):
    rng = np.random.default_rng(nx + nrhs)
    g = _grid(kind, nx, nz)
    shape = (nx, nz) if kind == "cyl" else (nz, nx)
    c = rng.uniform(2000, 3000, shape)
    rho = 310 * c ** 0.25
    m = C.c_void_p()
    (_, pc), (_, pr) = L.f64(c), L.f64(rho)
    L.check(L.lag_medium_create_acoustic(ctx, C.byref(g), pc, pr, H, C.byref(m)), ctx)
    mid = (C.c_double * 3)()
    L.check(L.lag_medium_midranges(m, mid))
    p = _precond(ctx, g, prec, plan, nx, nz, (mid[0], mid[0], mid[1] * H * H / 4), rng)
    b = dev(rng.standard_normal((nrhs, *shape)) * 10.0 ** rng.uniform(-6, 6, (nrhs, 1, 1)))
    x, one = empty(b.shape), empty(shape)
    s = L.solver(tol=1e-10, prec=prec)

    def solve(bd, xd, n):
        its, res = (C.c_int * n)(), (C.c_double * n)()
        L.check(L.lag_solve_system(m, p, None, ptr(bd), ptr(xd), n, C.byref(s), its, res), ctx)
        return list(its)

    its, xh = solve(b, x, nrhs), host(x)
    for i in sorted({0, 1, nrhs - 1}):
        assert solve(b[i], one, 1) == [its[i]]
        assert np.array_equal(host(one), xh[i]), i
    L.lag_precond_destroy(p)
    L.lag_medium_destroy(m)


# elastic systems (flexible GMRES on the mixed path): grids whose batch takes the larger operator tiles
@pytest.mark.parametrize("nx,nz,nrhs", [(70, 50, 3), (300, 200, 8), (900, 500, 2)])
def test_elastic_solve(ctx, nx, nz, nrhs):
    rng = np.random.default_rng(nx + nrhs)
    g, h, d = L.grid(nx, nz, 2.5, 2.5), 300.0, 2.5
    vp = rng.uniform(2800, 3200, (nz, nx))
    rho, vs = 310 * vp ** 0.25, vp / 1.73
    m = C.c_void_p()
    (_, pc), (_, pv), (_, pr) = L.f64(vp), L.f64(vs), L.f64(rho)
    L.check(L.lag_medium_create_elastic(ctx, C.byref(g), pc, pv, pr, h, C.byref(m)), ctx)
    mid = (C.c_double * 3)()
    L.check(L.lag_medium_midranges(m, mid))
    w = mid[2] * h * h / 4
    ps = []
    for ax, az in ((mid[0], mid[1]), (mid[1], mid[0])):
        p = C.c_void_p()
        L.check(L.lag_precond_create_sep(ctx, C.byref(g), ax, az, w, L.LAG_MIXED, 0, C.byref(p)), ctx)
        ps.append(p)
    b = dev(rng.standard_normal((nrhs, 2, nz, nx)) * 10.0 ** rng.uniform(-3, 3, (nrhs, 1, 1, 1)))
    x, one = empty(b.shape), empty((2, nz, nx))
    s = L.solver(tol=1e-9, prec=L.LAG_MIXED)

    def solve(bd, xd, n):
        its, res = (C.c_int * n)(), (C.c_double * n)()
        L.check(L.lag_solve_system(m, ps[0], ps[1], ptr(bd), ptr(xd), n, C.byref(s), its, res), ctx)
        return list(its)

    its, xh = solve(b, x, nrhs), host(x)
    for i in sorted({0, nrhs - 1}):
        assert solve(b[i], one, 1) == [its[i]]
        assert np.array_equal(host(one), xh[i]), i
    for p in ps:
        L.lag_precond_destroy(p)
    L.lag_medium_destroy(m)
