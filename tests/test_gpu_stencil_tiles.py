"""The direction update + stencil kernel (ragged tiles, batches, systems that stop at different iterations):
the recursive residual of the solve must be the true one, formed by the oracle's operator.  Also the update
that packs the next operand, the elastic operator's larger tiles and other fused passes."""
import ctypes as C

import numpy as np
import pytest

from oracle import cyl, fd, krylov
from paper_1005_0542_gb300 import lagwave as L

from gpu_util import make_ctx, dev, empty, host, medium, plan, ptr

pytestmark = pytest.mark.gpu
RNG = np.random.default_rng(4021)


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    L.lag_destroy(c)


# one and several right-hand sides, partial tiles in both directions, narrow grids, more tiles than blocks
@pytest.mark.parametrize("nx,nz,nrhs", [(1021, 1013, 1), (130, 517, 10), (65, 1000, 8), (193, 353, 17), (40, 2600, 7)])
def test_residual_is_true(ctx, nx, nz, nrhs):
    h, d, tol = 200.0, 5.0, 1e-11
    c = RNG.uniform(1800, 2600, (nz, nx))
    rho = 310 * c ** 0.25
    m = medium(ctx, nx, nz, d, d, c, rho, h)
    mid = (C.c_double * 3)()
    L.check(L.lag_medium_midranges(m, mid))
    p = plan(ctx, nx, nz, d, d, mid[0], mid[0], mid[1] * h * h / 4)
    b = RNG.standard_normal((nrhs, nz, nx)) * 10.0 ** RNG.uniform(-4, 4, (nrhs, 1, 1))
    b[nrhs // 2, :, : nx // 2] = 0.0     # another right-hand side, another iteration count
    bd, xd = dev(b), empty(b.shape)
    its, res = (C.c_int * nrhs)(), (C.c_double * nrhs)()
    s = L.solver(tol=tol)
    L.check(L.lag_solve_system(m, p, None, ptr(bd), ptr(xd), nrhs, C.byref(s), its, res), ctx)
    kap = fd.kappa_from_velocity(c, rho)
    x = host(xd)
    for i in range(nrhs):
        r = b[i] - fd.apply_A(x[i], kap, rho, h, d, d)
        # tol plus the rounding of ~50 float64 iterations
        assert np.linalg.norm(r) / np.linalg.norm(b[i]) < 2 * tol
    L.lag_precond_destroy(p)
    L.lag_medium_destroy(m)


# the residual update that also packs the next forward transform's operand: odd and even rows, a middle
# element, rows shorter than a K tile, padding rows of the last 128-row tile, more rows than blocks,
# systems of different sizes and iteration counts, both operand formats, residuals far from 1
@pytest.mark.parametrize("prec", [L.LAG_FP64, L.LAG_MIXED])
@pytest.mark.parametrize("nx,nz,nrhs", [(16, 5, 1), (63, 40, 3), (129, 130, 2), (2047, 33, 2), (24, 1500, 2)])
def test_packed_update(ctx, nx, nz, nrhs, prec):
    h, d, tol = 200.0, 5.0, 1e-11
    c = RNG.uniform(1800, 2600, (nz, nx))
    rho = 310 * c ** 0.25
    m = medium(ctx, nx, nz, d, d, c, rho, h)
    mid = (C.c_double * 3)()
    L.check(L.lag_medium_midranges(m, mid))
    p = plan(ctx, nx, nz, d, d, mid[0], mid[0], mid[1] * h * h / 4, prec=prec)
    assert L.lag_precond_uses_tensor_cores(p) == 1
    b = RNG.standard_normal((nrhs, nz, nx)) * (10.0 ** np.linspace(-60, 60, nrhs))[:, None, None]
    b[-1, :, nx // 3:] = 0.0
    bd, xd = dev(b), empty(b.shape)
    its, res = (C.c_int * nrhs)(), (C.c_double * nrhs)()
    s = L.solver(tol=tol, prec=prec)
    kap = fd.kappa_from_velocity(c, rho)
    for _ in range(2):     # the second solve runs as a graph where the stream allows it
        L.check(L.lag_solve_system(m, p, None, ptr(bd), ptr(xd), nrhs, C.byref(s), its, res), ctx)
        x = host(xd)
        for i in range(nrhs):
            r = b[i] - fd.apply_A(x[i], kap, rho, h, d, d)
            assert np.linalg.norm(r) / np.linalg.norm(b[i]) < 2 * tol
    L.lag_precond_destroy(p)
    L.lag_medium_destroy(m)


# the elastic operator on its 64 x 16 tiles (456 or more of them): ragged in both directions, a width
# below one tile, several right-hand sides
@pytest.mark.parametrize("nx,nz,nrhs", [(1000, 517, 1), (130, 333, 8), (65, 17, 230), (37, 1030, 9)])
def test_elastic_operator(ctx, nx, nz, nrhs):
    h, dx, dz = 300.0, 2.5, 3.5
    vp = RNG.uniform(2000, 5000, (nz, nx))
    vs, rho = vp / 1.73, RNG.uniform(1800, 2600, (nz, nx))
    m = medium(ctx, nx, nz, dx, dz, vp, rho, h, vs=vs)
    p = RNG.standard_normal((nrhs, 2, nz, nx))
    pd, qd = dev(p), empty(p.shape)
    L.check(L.lag_apply_operator(m, ptr(pd), ptr(qd), nrhs), ctx)
    mu = rho * vs * vs
    lam = rho * (vp * vp - 2 * vs * vs)
    q = host(qd)
    for i in range(nrhs):
        ref = np.stack(fd.apply_C(p[i, 0], p[i, 1], lam, mu, rho, h, dx, dz))
        assert np.abs(q[i] - ref).max() < 1e-14 * np.abs(ref).max()  # some 30 roundings of 1.1e-16 a node
    L.lag_medium_destroy(m)


# the DCT-II's last pass that also forms (r, z) and beta: an odd length's middle value, more rows than
# blocks, several right-hand sides of which one stops first; a wrong beta costs iterations, so the count
# is the oracle's up to the rounding that moves the last residual across the tolerance
@pytest.mark.parametrize("nr,nz,nrhs", [(20, 16, 1), (33, 257, 3), (1300, 17, 2)])
def test_cylindrical_beta(ctx, nr, nz, nrhs):
    hr, hz, h, tol = 5.0, 4.0, 300.0, 1e-10
    c = RNG.uniform(1800, 2600, (nr, nz))
    rho = 310 * c ** 0.25
    kap = fd.kappa_from_velocity(c, rho)
    kt, dt = cyl.precond_params(kap, rho, h)
    g = L.grid(nr, nz, hr, hz, cylindrical=True)
    m, p = C.c_void_p(), C.c_void_p()
    (c_, pc), (r_, pr) = L.f64(c), L.f64(rho)
    L.check(L.lag_medium_create_acoustic(ctx, C.byref(g), pc, pr, h, C.byref(m)), ctx)
    L.check(L.lag_precond_create_sep(ctx, C.byref(g), kt, kt, dt, L.LAG_FP64, 0, C.byref(p)), ctx)
    b = RNG.standard_normal((nrhs, nr, nz)) * (10.0 ** np.linspace(-6, 6, nrhs))[:, None, None]
    b[-1, nr // 3:] = 0.0
    bd, xd = dev(b), empty(b.shape)
    its, res = (C.c_int * nrhs)(), (C.c_double * nrhs)()
    s = L.solver(tol=tol)
    L.check(L.lag_solve_system(m, p, None, ptr(bd), ptr(xd), nrhs, C.byref(s), its, res), ctx)
    a1, a2, w = cyl.coefficients(kap, rho, hr, hz, h)
    x = host(xd)
    for i in range(nrhs):
        A = lambda v: cyl.apply_A(v.reshape(nr, nz), a1, a2, w, hr, hz).ravel()
        B = lambda v: cyl.apply_inverse(v.reshape(nr, nz), hr, hz, kt, dt).ravel()
        _, n, _ = krylov.pcg(A, B, b[i].ravel(), tol)
        assert abs(its[i] - n) <= 1
        assert np.linalg.norm(b[i].ravel() - A(x[i].ravel())) / np.linalg.norm(b[i]) < 2 * tol
    L.lag_precond_destroy(p)
    L.lag_medium_destroy(m)


# whole-medium extremes from the rows' own: one row, one column, more rows than threads; whichever row
# holds them
@pytest.mark.parametrize("nx,nz", [(1, 1), (37, 1), (1, 300), (5, 256), (3, 1025)])
def test_midranges(ctx, nx, nz):
    for row in (0, nz // 2, nz - 1):
        c, rho = RNG.uniform(2000, 3000, (nz, nx)), RNG.uniform(1000, 2000, (nz, nx))
        rho[row, nx - 1], rho[nz - 1 - row, 0] = 2500.0, 500.0 if nx * nz > 1 else 2500.0
        m = medium(ctx, nx, nz, 5.0, 5.0, c, rho, 200.0)
        mid = (C.c_double * 3)()
        L.check(L.lag_medium_midranges(m, mid))
        assert mid[1] == 0.5 * (rho.min() + rho.max())
        L.lag_medium_destroy(m)


# the mixed solve that writes the inverse transform's operand: planes that start on multiples of the
# partition length (constant addresses) and planes that do not, over m-tile borders, short last
# partitions; plane by plane against the same field alone, whose plane starts at 0.  Same operands and
# float32 sums of at most 100 terms in another order: 100 x 2^-24 < 1e-5
@pytest.mark.parametrize("nx,nz,nrhs", [(40, 64, 5), (200, 96, 4), (33, 130, 3), (64, 257, 3), (17, 1000, 2)])
def test_packed_tridiagonal(ctx, nx, nz, nrhs):
    p = plan(ctx, nx, nz, 5.0, 4.0, 3e9, 3e9, 1e7, prec=L.LAG_MIXED)
    assert L.lag_precond_uses_tensor_cores(p) == 1
    r = RNG.standard_normal((nrhs, nz, nx))
    rd, zd = dev(r), empty(r.shape)
    L.check(L.lag_precond_apply(p, ptr(rd), ptr(zd), nrhs), ctx)
    z = host(zd)
    for i in range(nrhs):
        one, zo = dev(r[i:i + 1]), empty((1, nz, nx))
        L.check(L.lag_precond_apply(p, ptr(one), ptr(zo), 1), ctx)
        ref = host(zo)[0]
        assert np.linalg.norm(z[i] - ref) / np.linalg.norm(ref) < 1e-5
    L.lag_precond_destroy(p)


# general float32 systems: the half mode tile of small launches (ragged last tile, one partition, 64-row
# partitions) against the full tile that a larger batch takes; float32 sums in the same order per mode,
# contraction apart: partition length x 2^-24 < 1e-5
@pytest.mark.parametrize("nx,nz", [(17, 40), (100, 1), (39, 1000), (300, 2000)])
def test_general_systems_on_few_blocks(ctx, nx, nz):
    rows = np.concatenate([RNG.uniform(2e9, 4e9, 2 * nz), RNG.uniform(1e7, 2e7, nz)])
    ax, az, d = (np.ascontiguousarray(v) for v in rows.reshape(3, nz))
    p = C.c_void_p()
    g = L.grid(nx, nz, 5.0, 4.0)
    (_, pa), (_, pz), (_, pd) = L.f64(ax), L.f64(az), L.f64(d)
    L.check(L.lag_precond_create_layered(ctx, C.byref(g), pa, pz, pd, L.LAG_MIXED, 0, C.byref(p)), ctx)
    nrhs = 160 // (2 * ((nx + 15) // 16)) + 1
    r = RNG.standard_normal((nrhs, nz, nx)).astype(np.float32)
    rd, zd = dev(r), dev(np.zeros_like(r))
    L.check(L.lag_precond_tridiag_f32(p, ptr(rd), ptr(zd), nrhs), ctx)
    one, zo = dev(r[-1:]), dev(np.zeros_like(r[-1:]))
    L.check(L.lag_precond_tridiag_f32(p, ptr(one), ptr(zo), 1), ctx)
    a, b = host(zd)[-1], host(zo)[0]
    assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(a)
    L.lag_precond_destroy(p)
