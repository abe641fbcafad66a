"""Opt-in GEMM variants of the exact-slice transform: what a plan holds for them, and when."""
import numpy as np
import pytest

from oracle import dst as odst
from paper_1005_0542_gb300 import lagwave as L

from gpu_util import make_ctx, dev, empty, host, plan, ptr, rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    L.lag_destroy(c)


@pytest.mark.parametrize("name,value", [("LAGWAVE_OZ_PAIR", "1"), ("LAGWAVE_OZ_CLUSTER", "2x2"), ("LAGWAVE_OZ_SK", "1")])
def test_operands_come_with_the_plan(ctx, monkeypatch, name, value):
    nx, nz = 2000, 600
    x = np.random.default_rng(7).standard_normal((1, nz, nx))
    xd, yd = dev(x), empty(x.shape)
    monkeypatch.setenv(name, value)
    p = plan(ctx, nx, nz, 5.0, 5.0, 1.0, 1.0, 0.1)
    monkeypatch.delenv(name)
    L.check(L.lag_precond_dst(p, ptr(xd), ptr(yd), 1), ctx)  # the apply scratch
    held = L.lag_bytes_in_use(ctx)
    monkeypatch.setenv(name, value)
    assert L.lag_precond_dst_gemm(p, 1) > L.LAG_GEMM_SLICE_TILES
    L.check(L.lag_precond_dst(p, ptr(xd), ptr(yd), 1), ctx)
    assert L.lag_bytes_in_use(ctx) == held
    assert L.lag_precond_status(p) == L.LAG_OK
    assert rel(host(yd), odst.dst_x(x)) < 1e-14
    L.lag_precond_destroy(p)


def test_operands_of_a_variant_chosen_later(ctx, monkeypatch):
    nx, nz = 700, 130
    x = np.random.default_rng(8).standard_normal((1, nz, nx))
    xd, yd = dev(x), empty(x.shape)
    p = plan(ctx, nx, nz, 5.0, 5.0, 1.0, 1.0, 0.1)
    L.check(L.lag_precond_dst(p, ptr(xd), ptr(yd), 1), ctx)
    held = L.lag_bytes_in_use(ctx)
    L.check(L.lag_precond_dst(p, ptr(xd), ptr(yd), 1), ctx)
    assert L.lag_bytes_in_use(ctx) == held
    monkeypatch.setenv("LAGWAVE_OZ_PAIR", "1")
    L.check(L.lag_precond_dst(p, ptr(xd), ptr(yd), 1), ctx)
    assert L.lag_bytes_in_use(ctx) > held
    assert rel(host(yd), odst.dst_x(x)) < 1e-14
    L.lag_precond_destroy(p)
