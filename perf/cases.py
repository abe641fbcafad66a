"""Performance cases of the library: what its users have it do, through the C ABI's Python binding.

A case is a dict of plain values.  ``kind`` names the entry point:

* ``apply``  lag_precond_apply: the Laplace preconditioner z = B^-1 r alone (Sec. 2.4 of the paper);
* ``solve``  lag_solve_system: one Laguerre harmonic of ``nrhs`` sources, preconditioned CG (acoustic)
             or flexible GMRES(20) (elastic) to 1e-10, plans and media kept between calls;
* ``shot``   lag_solve_acoustic: a whole shot from host arrays to receiver traces in one call.

``prec`` is the preconditioner's precision (``fp64`` or ``mixed``), ``plan`` its coefficients (``const``:
whole-medium midranges; ``layered``: midranges per row, on cylindrical grids per radius), ``grid`` is
``cart``, ``surface`` (Cartesian with a free surface on top) or ``cyl`` (the axisymmetric (r, z) problem,
nx radii, nz depths), ``medium`` is ``acoustic`` or ``elastic``.

``exact`` restates every case in float64 with torch alone: the separable operators are inverted by
FFTs along the transformed axis and a symmetric eigendecomposition along the other one, the
variable-coefficient systems by conjugate gradients driven to rounding.
"""
import ctypes as C
import functools
import math

import numpy as np
import torch

from paper_1005_0542_gb300 import lagwave as L

F64 = torch.float64
TOL = 1e-10            # the workload's solver tolerance
SHOT_TOL = 1e-12       # whole shots: later harmonics build on earlier ones


def _case(name, kind, nx, nz, nrhs=1, prec="fp64", plan="const", grid="cart", medium="acoustic", n_harm=0):
    c = dict(kind=kind, nx=nx, nz=nz, nrhs=nrhs, prec=prec, plan=plan, grid=grid, medium=medium, n_harm=n_harm)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the preconditioner alone: its smallest calls (a small model in an interactive program,
        # launches and latency), the float64 inner step of one production source, a batch of
        # right-hand sides, and a ragged layered model under a free surface
        _case("apply_small", "apply", 63, 40),
        _case("apply_one_field", "apply", 2048, 1024),
        _case("apply_batch", "apply", 1024, 1024, nrhs=256),
        _case("apply_ragged_layered", "apply", 1403, 611, nrhs=5, plan="layered", grid="surface"),
        # one harmonic of one production source: the float64 reference path, the layered
        # preconditioner on a ragged model, the mixed path
        _case("solve_fp64", "solve", 2048, 1024),
        _case("solve_fp64_layered", "solve", 1501, 701, nrhs=3, plan="layered", grid="surface"),
        _case("solve_mixed", "solve", 2048, 1024, prec="mixed"),
        # a batch of sources on one medium (survey processing), mixed path
        _case("solve_mixed_batch", "solve", 2048, 1024, nrhs=32, prec="mixed"),
        # elastic sources on a Cartesian grid, mixed path
        _case("solve_elastic_mixed", "solve", 2048, 1024, nrhs=4, prec="mixed", medium="elastic"),
        # the paper's axisymmetric problem: acoustic in float64, elastic on the mixed path
        _case("solve_cyl_fp64", "solve", 1000, 1024, grid="cyl"),
        _case("solve_cyl_elastic", "solve", 768, 512, prec="mixed", grid="cyl", medium="elastic"),
        # a whole small shot in one call, set-up included: 64 harmonics of a two-layer model
        _case("shot_two_layer", "shot", 128, 128, n_harm=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["apply", "solve", "elastic", "cyl", "cyl_elastic", "shot"], [4, 6, 1, 2, 1, 1])[0]
    if kind == "shot":
        return _case("", "shot", rng.randint(64, 160), rng.randint(64, 160), n_harm=rng.randint(24, 64))
    if kind == "apply":
        nx, nz = _log_int(rng, 40, 2100), _log_int(rng, 24, 1100)
        most = min(256, max(1, (1 << 28) // (nx * nz)))
        grid = rng.choice(["cart", "cart", "surface", "cyl"])
        if grid == "cyl":
            nx, nz = min(nx, 1100), min(nz, 1100)
        return _case("", "apply", nx, nz, nrhs=_log_int(rng, 1, most), plan=rng.choice(["const", "layered"]), grid=grid)
    if kind == "elastic":
        nx, nz = _log_int(rng, 150, 2048), _log_int(rng, 120, 1024)
        most = min(16, max(1, (1 << 23) // (nx * nz)))
        return _case("", "solve", nx, nz, nrhs=rng.randint(1, most), prec="mixed", plan=rng.choice(["const", "layered"]),
                     medium="elastic")
    if kind == "cyl":
        return _case("", "solve", _log_int(rng, 100, 1024), _log_int(rng, 100, 1024), nrhs=rng.randint(1, 3),
                     prec=rng.choice(["fp64", "mixed"]), plan=rng.choice(["const", "layered"]), grid="cyl")
    if kind == "cyl_elastic":
        return _case("", "solve", _log_int(rng, 100, 800), _log_int(rng, 100, 640), prec="mixed", grid="cyl",
                     medium="elastic")
    nx, nz = _log_int(rng, 100, 2100), _log_int(rng, 80, 1100)
    prec = rng.choice(["fp64", "mixed"])
    most = max(1, (1 << (22 if prec == "fp64" else 25)) // (nx * nz))
    return _case("", "solve", nx, nz, nrhs=_log_int(rng, 1, min(48, most)), prec=prec,
                 plan=rng.choice(["const", "layered"]), grid=rng.choice(["cart", "surface"]))


def work(case):
    """Bytes: every input read once, every output written once.  Flops: transforms counted as fast
    ones (2.5 n log2 2n a row and direction), 9 a point for the tridiagonal solves, 30 (acoustic) or
    120 (elastic) a point for the rest of an iteration, at the iteration counts such media need."""
    nx, nz, nc = case["nx"], case["nz"], 2 if case["medium"] == "elastic" else 1
    n = nx if case["grid"] != "cyl" else nz
    pts = float(nx) * nz * nc * case["nrhs"]
    prec = pts * (2 * 2.5 * math.log2(2.0 * n) + 9.0)
    if case["kind"] == "apply":
        return {"bytes": 16.0 * pts, "flops": prec}
    its = 8 if case["plan"] == "layered" else 30
    step = prec + pts * (120.0 if nc == 2 else 30.0)
    if case["kind"] == "shot":
        return {"bytes": 16.0 * nx * nz, "flops": case["n_harm"] * its * step}
    return {"bytes": 16.0 * pts + 16.0 * nx * nz * (1 + nc), "flops": its * step}


# ---------------------------------------------------------------------------- inputs
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


class _Inputs:
    """Everything of a case that is drawn from the seed: medium, spacing, right-hand sides."""


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=g.device, dtype=F64)


def _medium(g, case):
    """20 layers along the depth, c ~ U(1500, 4500) m/s times (1 + 2.5 % noise, clipped at 5 %), the
    density from c; elastic: Vs = Vp / 1.73.  [nz][nx], on cylindrical grids [nx][nz]."""
    nx, nz = case["nx"], case["nz"]
    layer = _uniform(g, 1500.0, 4500.0, 20)
    rows = layer[(torch.arange(nz, device=g.device) * 20) // nz]
    eps = (0.025 * torch.randn(nz, nx, generator=g, device=g.device, dtype=F64)).clamp_(-0.05, 0.05)
    c = rows[:, None] * (1.0 + eps)
    if case["grid"] == "cyl":
        c = c.t().contiguous()
    return c, 310.0 * c ** 0.25, (c / 1.73 if case["medium"] == "elastic" else None)


def _history(g, n0, n1):
    """A smooth field as the history sums hold: wave packets of a few wavelengths."""
    y, x = torch.arange(n0, device=g.device, dtype=F64)[:, None], torch.arange(n1, device=g.device, dtype=F64)[None, :]
    out = torch.zeros(n0, n1, device=g.device, dtype=F64)
    for a, y0, x0, w, ky, kx, ph in _uniform(g, 0.0, 1.0, 6, 7).tolist():
        s = 4.0 + 0.08 * min(n0, n1) * (0.5 + w)
        out += (0.5 + a) * torch.exp(-((y - y0 * n0) ** 2 + (x - x0 * n1) ** 2) / (2 * s * s)) * torch.cos(
            (2 * math.pi / 24.0) * ((ky - 0.5) * y + (kx - 0.5) * x) + 2 * math.pi * ph)
    return out


def _inputs(case, seed):
    g = torch.Generator(device=_device())
    g.manual_seed(1005 + int(seed))
    nx, nz, nrhs = case["nx"], case["nz"], case["nrhs"]
    cyl, elastic = case["grid"] == "cyl", case["medium"] == "elastic"
    s = _Inputs()
    s.n0, s.n1 = (nx, nz) if cyl else (nz, nx)   # rows, row length of the fields
    if case["kind"] == "shot":
        v = _uniform(g, 0.9, 1.1, 3).tolist()
        s.h, s.alpha, s.d = 200.0, 9, 10.0
        s.c = torch.full((nz, nx), 2000.0 * v[0], dtype=F64, device=g.device)
        s.rho = torch.full((nz, nx), 1000.0 * v[1], dtype=F64, device=g.device)
        s.c[nz // 2:] *= 1.5
        s.rho[nz // 2:] *= 2.0
        s.f0 = 30.0 * v[2]
        s.t0 = 2.5 / s.f0
        s.src = (int(torch.randint(nx // 3, 2 * nx // 3, (1,), generator=g, device=g.device)), 16)
        s.rcv = [(i, 16) for i in range(nx // 32, nx, max(1, nx // 16))][:16]
        s.t = np.linspace(0.002, 0.6, 300)
        return s
    s.h, s.d = (300.0, 2.5) if elastic else (200.0, 5.0)
    s.c, s.rho, s.vs = _medium(g, case)
    if case["kind"] == "apply":
        s.r = torch.randn(nrhs, s.n0, s.n1, generator=g, device=g.device, dtype=F64)
        return s
    # one harmonic's right-hand sides: a point source near the surface and the history term
    # -rho h^2 c_m S, each source at its own place (cylindrical: on the axis, weighted by r)
    w = s.rho * (s.h * s.h)
    if cyl:
        w = w * ((torch.arange(nx, device=g.device, dtype=F64) + 0.5) * s.d)[:, None]
    depth = min(2 if elastic else 16, nz - 1)
    nc = 2 if elastic else 1
    b = torch.zeros(nrhs, nc, s.n0, s.n1, dtype=F64, device=g.device)
    for k in range(nrhs):
        for comp in range(nc):
            b[k, comp] = -w * _history(g, s.n0, s.n1)
        amp = float(b[k].abs().max()) * 20.0
        ix = 0 if cyl else int(round((k + 0.5) * nx / nrhs)) % nx
        b[k, nc - 1, ix if cyl else depth, depth if cyl else ix] += amp * float(_uniform(g, 0.5, 1.5, 1))
    s.b = b if elastic else b[:, 0].contiguous()
    return s


def _midranges(s, case):
    """[coefficient rows]: kappa, rho (acoustic) or lambda+2mu, mu, rho (elastic): midranges over the
    whole medium (scalars) or over each row of the fields."""
    if case["medium"] == "elastic":
        mu = s.rho * s.vs * s.vs
        f = [s.rho * s.c * s.c, mu, s.rho]
    else:
        f = [s.rho * s.c * s.c, s.rho]
    if case["plan"] == "layered":
        return [(0.5 * (v.amin(1) + v.amax(1))).cpu().numpy() for v in f]
    return [0.5 * float(v.min() + v.max()) for v in f]


# ---------------------------------------------------------------------------- the library's side
@functools.lru_cache(maxsize=None)
def _ctx():
    return L.create(0)   # one context, on a stream of its own, for the whole program


def _ptr(t):
    return C.c_void_p(t.data_ptr())


class _State:
    """Plans, media and buffers that a program keeps between its calls."""

    def __init__(self):
        self.plans, self.medium = [], None

    def __del__(self):
        for p in self.plans:
            L.lag_precond_destroy(p)
        if self.medium is not None:
            L.lag_medium_destroy(self.medium)


def _grid(case, d):
    return L.grid(case["nx"], case["nz"], d, d, case["grid"] != "cart", case["grid"] == "cyl")


def _plan(ctx, g, prec, ax, az, d, hoop=None):
    p = C.c_void_p()
    if isinstance(ax, np.ndarray):
        keep = [L.f64(v) for v in (ax, az, d)]
        L.check(L.lag_precond_create_layered(ctx, C.byref(g), *(k[1] for k in keep), prec, 0, C.byref(p)), ctx)
    elif hoop is not None:
        L.check(L.lag_precond_create_cyl(ctx, C.byref(g), ax, az, d, hoop, prec, 0, C.byref(p)), ctx)
    else:
        L.check(L.lag_precond_create_sep(ctx, C.byref(g), ax, az, d, prec, 0, C.byref(p)), ctx)
    return p


def prepare(case, seed):
    s, st, ctx = _inputs(case, seed), _State(), _ctx()
    st.case, st.ctx = case, ctx
    g = _grid(case, s.d)
    prec = L.LAG_FP64 if case["prec"] == "fp64" else L.LAG_MIXED
    if case["kind"] == "shot":
        st.grid, st.lag = g, L.laguerre(s.h, s.alpha, case["n_harm"])
        st.solver, st.wavelet = L.solver(tol=SHOT_TOL, prec=prec), L.wavelet(s.f0, s.t0)
        st.c, st.rho, st.t = L.f64(s.c.cpu().numpy()), L.f64(s.rho.cpu().numpy()), L.f64(s.t)
        st.src, st.rcv, st.nrcv = L.points([s.src]), L.points(s.rcv), len(s.rcv)
        st.traces = np.zeros((1, st.nrcv, s.t.size))
        return st
    mid = _midranges(s, case)
    q = s.h * s.h / 4.0
    if case["medium"] == "elastic":
        p2m, mu, rho = mid
        hoop = (p2m, 0.0) if case["grid"] == "cyl" else (None, None)
        st.plans = [_plan(ctx, g, prec, p2m, mu, rho * q, hoop[0]), _plan(ctx, g, prec, mu, p2m, rho * q, hoop[1])]
    else:
        st.plans = [_plan(ctx, g, prec, mid[0], mid[0], mid[1] * q)]
    if case["kind"] == "apply":
        st.r, st.z = s.r, torch.empty_like(s.r)
    else:
        st.medium = C.c_void_p()
        c, rho = L.f64(s.c.cpu().numpy()), L.f64(s.rho.cpu().numpy())
        if case["medium"] == "elastic":
            vs = L.f64(s.vs.cpu().numpy())
            rc = L.lag_medium_create_elastic(ctx, C.byref(g), c[1], vs[1], rho[1], s.h, C.byref(st.medium))
        else:
            rc = L.lag_medium_create_acoustic(ctx, C.byref(g), c[1], rho[1], s.h, C.byref(st.medium))
        L.check(rc, ctx)
        st.solver = L.solver(tol=TOL, max_iter=2000, restart_k=20, prec=prec)
        st.b, st.x = s.b, torch.empty_like(s.b)
    if torch.cuda.is_available():
        torch.cuda.synchronize()   # torch's stream made the inputs, the library reads them on its own
    return st


def run(st):
    ctx, case = st.ctx, st.case
    if case["kind"] == "apply":
        L.check(L.lag_precond_apply(st.plans[0], _ptr(st.r), _ptr(st.z), case["nrhs"]), ctx)
        return st.z
    if case["kind"] == "shot":
        L.check(L.lag_solve_acoustic(ctx, C.byref(st.grid), st.c[1], st.rho[1], C.byref(st.lag), C.byref(st.solver),
                                     C.byref(st.wavelet), 1, st.src, st.nrcv, st.rcv, st.t[0].size, st.t[1],
                                     st.traces.ctypes.data_as(L.PD), None), ctx)
        return st.traces
    L.check(L.lag_solve_system(st.medium, st.plans[0], st.plans[1] if len(st.plans) > 1 else None, _ptr(st.b),
                               _ptr(st.x), case["nrhs"], C.byref(st.solver), None, None), ctx)
    return st.x


# ---------------------------------------------------------------------------- plain float64
def _dst(x):
    """Orthonormal DST-I along the last axis (its own inverse), by an FFT of the odd extension."""
    n = x.shape[-1]
    z = torch.zeros(*x.shape[:-1], 1, dtype=F64, device=x.device)
    return -torch.fft.rfft(torch.cat([z, x, z, -x.flip(-1)], -1)).imag[..., 1:n + 1] * (0.5 * math.sqrt(2.0 / (n + 1)))


def _dct(x, inverse=False):
    """Orthonormal DCT-II along the last axis, or its inverse, by an FFT of the even extension."""
    n = x.shape[-1]
    q = torch.arange(n, dtype=F64, device=x.device)
    scale = torch.full((n,), math.sqrt(2.0 / n), dtype=F64, device=x.device)
    scale[0] = math.sqrt(1.0 / n)
    if not inverse:
        f = torch.fft.rfft(torch.cat([x, x.flip(-1)], -1))[..., :n]
        return (f * torch.exp(-0.5j * math.pi / n * q)).real * (0.5 * scale)
    u = x * scale   # sum_q u_q cos(pi q (k + 1/2) / n)
    f = torch.zeros(*x.shape[:-1], n + 1, dtype=torch.complex128, device=x.device)
    f[..., :n] = u * torch.exp(0.5j * math.pi / n * q)
    f[..., 0] *= 2.0
    return torch.fft.irfft(f, n=2 * n)[..., :n] * n


class _Separable:
    """B^-1 for B = T + lambda_j diag(w): rows i of T are (-zf_i, zf_i + zf_{i+1} + dd_i, -zf_{i+1})."""

    def __init__(self, case, n0, n1, d, ax, az, dd, hoop=0.0):
        dev = _device()
        self.cyl = case["grid"] == "cyl"
        i = np.arange(n0)
        ax, az, dd = (np.broadcast_to(np.asarray(v, dtype=np.float64), (n0,)) for v in (ax, az, dd))
        zf, a = np.zeros(n0 + 1), (ax if self.cyl else az)
        zf[1:n0], zf[n0] = 0.5 * (a[:-1] + a[1:]), a[-1]
        if self.cyl:
            r = (i + 0.5) * d
            zf = zf * np.arange(n0 + 1) / d
            w, dd = r * az, r * dd + hoop / r
        else:
            zf[0] = 0.0 if case["grid"] == "surface" else a[0]
            zf, w = zf / (d * d), ax
        j = torch.arange(n1, dtype=F64, device=dev)
        ang = math.pi * j / (2 * n1) if self.cyl else math.pi * (j + 1) / (2 * (n1 + 1))
        lam = 4.0 / (d * d) * torch.sin(ang) ** 2
        self.flat = case["grid"] == "cart" and np.ptp(w) == 0 and np.ptp(a) == 0 and np.ptp(dd) == 0
        if self.flat:   # constant coefficients between Dirichlet ends: a sine transform along z as well
            k = torch.arange(n0, dtype=F64, device=dev)
            mz = 4.0 * a[0] / (d * d) * torch.sin(math.pi * (k + 1) / (2 * (n0 + 1))) ** 2
            self.den = mz[:, None] + w[0] * lam[None, :] + dd[0]
            return
        sw = 1.0 / np.sqrt(w)
        m = np.diag((zf[:-1] + zf[1:] + dd) * sw * sw)
        off = -zf[1:n0] * sw[:-1] * sw[1:]
        m[i[:-1], i[1:]] = off
        m[i[1:], i[:-1]] = off
        e, v = np.linalg.eigh(m)
        self.v = torch.from_numpy(v * sw[:, None]).to(dev)
        self.den = torch.from_numpy(e).to(dev)[:, None] + lam[None, :]

    def __call__(self, r):
        y = _dct(r) if self.cyl else _dst(r)
        if self.flat:
            y = _dst((_dst(y.transpose(-1, -2)).transpose(-1, -2) / self.den).transpose(-1, -2)).transpose(-1, -2)
        else:
            y = torch.matmul(self.v, torch.matmul(self.v.t(), y) / self.den)
        return _dct(y, inverse=True) if self.cyl else _dst(y)


def _faces(f, dim, lo_zero=False, hi_zero=False):
    """Means of neighbouring nodes along dim; the end faces repeat their node or are zero."""
    a, b = f.narrow(dim, 0, f.shape[dim] - 1), f.narrow(dim, 1, f.shape[dim] - 1)
    lo, hi = f.narrow(dim, 0, 1), f.narrow(dim, f.shape[dim] - 1, 1)
    return torch.cat([lo * (0.0 if lo_zero else 1.0), 0.5 * (a + b), hi * (0.0 if hi_zero else 1.0)], dim)


def _diffusion(face, p, dim, d):
    """-d/dx (face dp/dx) with p = 0 beyond both ends."""
    z = torch.zeros_like(p.narrow(dim, 0, 1))
    q = torch.cat([z, p, z], dim)
    f = face * (q.narrow(dim, 1, q.shape[dim] - 1) - q.narrow(dim, 0, q.shape[dim] - 1))
    return -(f.narrow(dim, 1, f.shape[dim] - 1) - f.narrow(dim, 0, f.shape[dim] - 1)) / (d * d)


def _acoustic(s, case):
    kap, mass = s.rho * s.c * s.c, s.rho * (s.h * s.h / 4.0)
    if case["grid"] == "cyl":   # the equation times r: rows are the radii
        rb = (torch.arange(s.n0 + 1, dtype=F64, device=kap.device) * s.d)[:, None]
        r = rb[:-1] + 0.5 * s.d
        f0, f1, mass = _faces(kap, 0) * rb, _faces(kap, 1, True, True) * r, mass * r
    else:
        f0, f1 = _faces(kap, 0, lo_zero=case["grid"] == "surface"), _faces(kap, 1)
    return lambda p: _diffusion(f0, p, -2, s.d) + _diffusion(f1, p, -1, s.d) + mass * p


def _elastic(s):
    mu = s.rho * s.vs * s.vs
    lam = s.rho * s.c * s.c - 2.0 * mu
    p2m, mass = lam + 2.0 * mu, s.rho * (s.h * s.h / 4.0)
    px, mx, pz, mz = _faces(p2m, 1), _faces(mu, 1), _faces(p2m, 0), _faces(mu, 0)

    def cd(f, dim):   # centred difference, zero beyond the ends
        z = torch.zeros_like(f.narrow(dim, 0, 1))
        q = torch.cat([z, f, z], dim)
        return (q.narrow(dim, 2, f.shape[dim]) - q.narrow(dim, 0, f.shape[dim])) / (2.0 * s.d)

    def op(v):
        u, w = v[:, 0], v[:, 1]
        qu = _diffusion(px, u, -1, s.d) + _diffusion(mz, u, -2, s.d) + mass * u \
            - cd(lam * cd(w, -2), -1) - cd(mu * cd(w, -1), -2)
        qw = _diffusion(mx, w, -1, s.d) + _diffusion(pz, w, -2, s.d) + mass * w \
            - cd(mu * cd(u, -2), -1) - cd(lam * cd(u, -1), -2)
        return torch.stack([qu, qw], 1)
    return op


def _elastic_cyl(s):
    """The gradient of the discrete strain energy of the axisymmetric problem."""
    mu = s.rho * s.vs * s.vs
    lam = s.rho * s.c * s.c - 2.0 * mu
    d, nr = s.d, s.n0
    r = ((torch.arange(nr, dtype=F64, device=mu.device) + 0.5) * d)[:, None]
    rb = ((torch.arange(nr, dtype=F64, device=mu.device) + 1.0) * d)[:, None]
    rg = torch.cat([r, r[-1:] + d])

    def rf(f):
        return torch.cat([0.5 * (f[:-1] + f[1:]), f[-1:]])

    def zf(f):
        return 0.5 * (f[..., :-1] + f[..., 1:])
    lr, mr, pr = rf(lam), rf(mu), rf(lam + 2 * mu)
    lz, mz, pz = zf(lam), zf(mu), zf(lam + 2 * mu)
    lc, mc = zf(lr), zf(mr)
    mass = s.rho * r * (s.h * s.h / 4.0)

    def energy(v):
        q, u = v[:, 0], v[:, 1]
        g = torch.zeros_like(q[:, :1])
        qg, ug = torch.cat([q, g], 1), torch.cat([u, g], 1)
        qr, ur = (qg[:, 1:] - qg[:, :-1]) / d, (ug[:, 1:] - ug[:, :-1]) / d
        qz, uz = (q[..., 1:] - q[..., :-1]) / d, (u[..., 1:] - u[..., :-1]) / d
        tt = q / r
        ttr = 0.5 * ((qg / rg)[:, 1:] + (qg / rg)[:, :-1])
        e = (rb * (pr * qr * qr + mr * ur * ur + 2 * lr * qr * ttr)).sum()
        e = e + (r * (pz * uz * uz + mz * qz * qz + 2 * lz * uz * zf(tt))).sum()
        e = e + (r * (lam + 2 * mu) * tt * tt).sum()
        uzg, qzg = torch.cat([uz, g[..., 1:]], 1), torch.cat([qz, g[..., 1:]], 1)
        uzc, qzc = 0.5 * (uzg[:, 1:] + uzg[:, :-1]), 0.5 * (qzg[:, 1:] + qzg[:, :-1])
        e = e + (rb * (2 * lc * zf(qr) * uzc + 2 * mc * qzc * zf(ur))).sum()
        return 0.5 * (e + (mass * (q * q + u * u)).sum())

    def op(v):
        with torch.enable_grad():
            x = v.detach().requires_grad_(True)
            return torch.autograd.grad(energy(x), x)[0]
    return op


def _cg(op, inv, b, most=400):
    """Preconditioned CG on every right-hand side at once, driven to rounding."""
    def dot(x, y):
        return (x * y).flatten(1).sum(1).view(-1, *([1] * (b.dim() - 1)))
    x, r = torch.zeros_like(b), b.clone()
    z = inv(r)
    p, rz, bb = z.clone(), dot(r, z), dot(b, b)
    for _ in range(most):
        q = op(p)
        a = rz / dot(p, q)
        x += a * p
        r -= a * q
        if float((dot(r, r) / bb).max()) < 1e-28:
            break
        z = inv(r)
        new = dot(r, z)
        p = z + (new / rz) * p
        rz = new
    return x


def _inverse(s, case, mid):
    q = s.h * s.h / 4.0
    if case["medium"] != "elastic":
        return _Separable(case, s.n0, s.n1, s.d, mid[0], mid[0], mid[1] * q)
    p2m, mu, rho = mid
    b1 = _Separable(case, s.n0, s.n1, s.d, p2m, mu, rho * q, hoop=p2m if case["grid"] == "cyl" else 0.0)
    b2 = _Separable(case, s.n0, s.n1, s.d, mu, p2m, rho * q)
    return lambda r: torch.stack([b1(r[:, 0]), b2(r[:, 1])], 1)


def _laguerre(n, alpha, x):
    """sqrt(m!/(m+alpha)!) e^{-x/2} L_m^alpha(x), m < n."""
    out = np.zeros((n, x.size))
    cur, prev = np.exp(-0.5 * x - 0.5 * math.lgamma(alpha + 1.0)), np.zeros_like(x)
    for m in range(n):
        out[m] = cur
        cur, prev = ((2 * m + alpha + 1 - x) * cur - math.sqrt(m * (m + alpha)) * prev) / math.sqrt(
            (m + 1) * (m + alpha + 1)), cur
    return out


def _exact_shot(case, s):
    n, h = case["n_harm"], s.h
    t_end, panels = s.t0 + 4.0 / s.f0, 400
    gx, gw = np.polynomial.legendre.leggauss(16)
    edges = np.linspace(0.0, t_end, panels + 1)
    half = 0.5 * (edges[1:] - edges[:-1])[:, None]
    t = (half * gx + 0.5 * (edges[1:] + edges[:-1])[:, None]).ravel()
    a2 = (math.pi * s.f0 * (t - s.t0)) ** 2
    fm = math.sqrt(h) * (_laguerre(n, s.alpha, h * t) * ((half * gw).ravel() * (1.0 - 2.0 * a2) * np.exp(-a2))).sum(1)
    table = math.sqrt(h) * (h * s.t) ** s.alpha * _laguerre(n, s.alpha, h * s.t)
    op, inv = _acoustic(s, case), _inverse(s, case, _midranges(s, case))
    S, T = torch.zeros_like(s.c)[None], torch.zeros_like(s.c)[None]
    rec = np.zeros((n, len(s.rcv)))
    ix, iz = [p[0] for p in s.rcv], [p[1] for p in s.rcv]
    for m in range(n):
        lc = 0.5 * (math.lgamma(m + 1.0) - math.lgamma(m + s.alpha + 1.0))
        b = -math.exp(lc) * (s.rho * (h * h)) * S
        b[0, s.src[1], s.src[0]] += fm[m] / (s.d * s.d)
        x = _cg(op, inv, b)
        T = T + math.exp(-lc) * x
        S = S + T
        rec[m] = x[0, iz, ix].cpu().numpy()
    return (rec.T @ table)[None]


def exact(case, seed):
    s = _inputs(case, seed)
    if case["kind"] == "shot":
        return _exact_shot(case, s)
    if case["kind"] == "apply":
        inv = _inverse(s, case, _midranges(s, case))
        out = torch.empty_like(s.r)
        for k in range(0, case["nrhs"], 16):
            out[k:k + 16] = inv(s.r[k:k + 16])
        return out
    inv = _inverse(s, case, _midranges(s, dict(case, plan="const")))
    if case["medium"] != "elastic":
        op = _acoustic(s, case)
    else:
        op = _elastic_cyl(s) if case["grid"] == "cyl" else _elastic(s)
    out = torch.empty_like(s.b)
    for k in range(0, case["nrhs"], 8):
        out[k:k + 8] = _cg(op, inv, s.b[k:k + 8])
    return out
