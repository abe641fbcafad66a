"""The weight-stacked exact-slice GEMM on each of its tile widths: rows built from the operand's own digits,
whose sums leave FP32's whole numbers unless every drain takes place, and the 64-column tiles over every
stage count at which a drain falls on, just before or just after a tile's end."""
import ctypes as C

import numpy as np
import pytest

from oracle import dst as odst
from paper_1005_0542_gb300 import lagwave as L

from gpu_util import make_ctx, dev, empty, host, plan, ptr, torch

TOL = 1e-14  # of a row's largest value: float64 rounding of the result and of the oracle's K-term float64 sums
NS = 7       # base-256 digits of an operand


def digits(T):
    """Balanced base-256 digits of integers |T| <= 2^55, most significant first: T = sum d_i 256^(6 - i)."""
    T, out = T.astype(object), []
    for i in range(NS - 1, -1, -1):
        d = ((T + 128) % 256) - 128 if i else T
        out.append(d.astype(np.int64))
        T = (T - d) // 256
    return np.array(out[::-1])


def operand(n, mode):
    """Digits of column `mode` of the DST matrix (first floor(n / 2) rows) and the exponent of the expansion."""
    _, e = np.frexp(np.sqrt(2.0 / (n + 1)))
    k = np.arange(1, n // 2 + 1, dtype=np.int64)
    s = np.sqrt(2.0 / (n + 1)) * np.sin(np.pi * ((k * (mode + 1)) % (2 * (n + 1))).astype(np.float64) / (n + 1))
    return digits(np.rint(np.ldexp(s, 55 - int(e))).astype(np.int64)), int(e)


def row_for(n, mode, weight):
    """A row whose digits have one sign with the operand's in every product of `weight` and are odd and as large
    as they may be.  Only the first half of the row is filled, so both parities' folds are these values;
    the leading digit (at most 64 after the fold's headroom) enters weight 4 and sets the row's exponent
    elsewhere at one element."""
    b, _ = operand(n, mode)
    a = np.zeros((NS, n // 2), dtype=np.int64)
    for i in range(1 if weight == 4 else 2, weight):
        a[i - 1] = (63 if i == 1 else 127) * np.where(b[weight - i - 1] < 0, -1, 1)
    if weight != 4:
        a[:, n // 5] = 0
        a[0, n // 5] = 63
    x = np.zeros(n)
    # T = sum a_i 256^(7 - i) with x = T 2^(e - 55); the row's exponent e is 1 (largest |x| in [1/2, 1))
    T = sum(a[i].astype(object) * 256 ** (NS - 1 - i) for i in range(NS))
    x[:n // 2] = [np.ldexp(float(t), 1 - 55) for t in T]
    assert all(int(np.ldexp(v, 54)) == t for v, t in zip(x[:n // 2], T)) and 0.5 <= np.abs(x).max() < 1.0
    return x, a


def undrained(n, mode, a, weight):
    """Error that one accumulator of `weight` makes when FP32 sums the whole column, a K step of 16 and a
    product at a time, in units of the result."""
    b, eb = operand(n, mode)
    acc, exact = np.float32(0.0), 0
    for k in range(0, n // 2, 16):
        for i in range(1, weight):
            part = int((a[i - 1, k:k + 16] * b[weight - i - 1, k:k + 16]).sum())
            exact += part
            acc = np.float32(acc + np.float32(part))
    return abs(float(acc) - exact) * 2.0 ** (1 + eb + 2 - 8 * weight), abs(exact)


CASES = [(2048, 4), (2048, 5), (2048, 6), (2047, 6), (1216, 6)]


def rows_of(n, weight):
    modes = [0, 1, n // 7, 2 * n // 5, n - 2, n - 1]
    return modes, [row_for(n, m, weight) for m in modes]


# the rows do what they are for: without a drain at least one of them loses more than twice the tolerance, so
# that the transform, itself within the tolerance, could not pass
@pytest.mark.parametrize("n,weight", CASES)
def test_rows_need_their_drains(n, weight):
    S = odst.dst_matrix(n)
    modes, rows = rows_of(n, weight)
    lost = [undrained(n, m, a, weight) for m, (_, a) in zip(modes, rows)]
    assert any(total > 2 ** 24 and err > 2 * TOL * np.abs(x @ S).max() for (err, total), (x, _) in zip(lost, rows))


@pytest.fixture(scope="module")
def ctx():
    c = make_ctx()
    yield c
    L.lag_destroy(c)


def _up(a, b):
    return -(-a // b)


def tile_width(n, rows):
    """Columns of the tiles that a transform takes: the narrowest that run in one wave of the SMs."""
    sms = torch().cuda.get_device_properties(0).multi_processor_count
    for w in (16, 32):
        if _up(rows, 128) * (_up(_up(n, 2), w) + _up(n // 2, w)) <= sms:
            return w
    return 64


def transform(ctx, x):
    p = plan(ctx, x.shape[2], x.shape[1], 5.0, 5.0, 1.0, 1.0, 0.1)
    xd, yd = dev(x), empty(x.shape)
    L.check(L.lag_precond_dst(p, ptr(xd), ptr(yd), x.shape[0]), ctx)
    assert L.lag_precond_status(p) == L.LAG_OK
    L.lag_precond_destroy(p)
    return host(yd)


# the rows at both ends of a transform of every width; 64 columns with a second tile for some CTAs
@pytest.mark.gpu
@pytest.mark.parametrize("width", [16, 32, 64])
@pytest.mark.parametrize("n,weight", CASES)
def test_drains(ctx, n, weight, width):
    nz = {16: 100, 32: 300 if n < 2000 else 200, 64: 1300}[width]
    assert tile_width(n, nz) == width
    _, rows = rows_of(n, weight)
    x = np.random.default_rng(n + weight).standard_normal((1, nz, n))
    for i, (row, _) in enumerate(rows):
        x[0, i] = x[0, nz - 1 - i] = row
    y, ref = transform(ctx, x)[0], odst.dst_x(x)[0]
    assert (np.abs(y - ref).max(axis=1) <= TOL * np.abs(ref).max(axis=1)).all()


# 64-column tiles: stage counts up to, at and past every drain (12, 20, 24, 36, 40, 48, 60) and the largest,
# with full and ragged last stages, one row in the last row tile
@pytest.mark.gpu
@pytest.mark.parametrize("nk", [11, 12, 13, 20, 21, 24, 25, 36, 37, 40, 41, 48, 49, 60, 61, 64])
@pytest.mark.parametrize("short", [0, 1, 31])
def test_stage_counts(ctx, nk, short):
    n = 32 * nk - short
    assert _up(_up(n, 2), 16) == nk
    sms = torch().cuda.get_device_properties(0).multi_processor_count
    nz = 128 * (sms // (2 * _up(n // 2, 32)) + 1) + 1
    assert tile_width(n, nz) == 64
    rng = np.random.default_rng(n)
    x = rng.standard_normal((1, nz, n)) * 10.0 ** rng.uniform(-3, 3, (1, nz, n))
    y, ref = transform(ctx, x)[0], odst.dst_x(x)[0]
    assert (np.abs(y - ref).max(axis=1) <= TOL * np.abs(ref).max(axis=1)).all()


# weights 7 and 8 are summed in FP32 past its whole numbers here: every width adds their products in the same
# order, so a row's transform is the same bit for bit on each
@pytest.mark.gpu
@pytest.mark.parametrize("n", [2048, 2047, 1600])
@pytest.mark.parametrize("weight", [7, 8])
def test_same_bits_on_every_width(ctx, n, weight):
    _, rows = rows_of(n, weight)
    x = np.array([[r for r, _ in rows]])
    y = {}
    for copies in (1, 30, 220):
        w = tile_width(n, copies * len(rows))
        y[w] = transform(ctx, np.repeat(x, copies, axis=0))
    assert sorted(y) == [16, 32, 64]
    for w in y:
        assert (y[w] == y[16][0]).all(), w
