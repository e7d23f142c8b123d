"""The reciprocals of the factorization's diagonal blocks against 1 / d.

A supernode of 20 columns whose first pivot is d and whose first column is one
below it has L(i, 0) = 1 * (1 / d) to the last bit.  The real reciprocal is one
third-order step from a seed of relative error e <= 2^-19: e^3 = 2^-57 beside
the last rounding, 0.5 + 2^-57 2^53 = 0.5625 units in the last place at most,
and the division itself outside the exponents 64 .. 1982.  The complex one is
conj(d) / |d|^2: roundings of the sum (2), of its reciprocal (1.125) and of the
product (1), each 2^-53 of the result, and a unit of the larger part is at least
that: 4.2 units.  Outside its exponents it is scaled first, with 11 roundings."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

S = 20


def _first_columns(native, d):
    """fl(1 / d_b) of block b, for each entry of d."""
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    m = d.size
    colptr = np.concatenate([[0], np.cumsum(np.tile(np.arange(S, 0, -1), m))]).astype(np.int64)
    rowind = np.concatenate([np.arange(b * S + j, (b + 1) * S) for b in range(m) for j in range(S)]).astype(np.int32)
    values = np.zeros((m, S * (S + 1) // 2), d.dtype)
    values[:, 0] = d
    values[:, 1:S] = 1.0
    values[:, S:] = 1.0
    p = synth.Problem("pivots", m * S, colptr, rowind, values.ravel(), np.arange(m * S),
                      {"kind": "fundamental", "cap": S, "fill": 0.0}, {"hermitian": False})
    ctx = SelInvContext.from_problem(p)
    assert ctx.nsuper == m
    L, D = ctx.factor(torch.from_numpy(p.values).cuda())
    torch.cuda.synchronize()
    assert np.array_equal(D.cpu().numpy().reshape(m, S)[:, 0], d, equal_nan=True)
    got = L.cpu().numpy().reshape(m, S, S)[:, 0, 1:]         # column 0, rows 1..
    assert np.array_equal(got, np.repeat(got[:, :1], S - 1, axis=1), equal_nan=True)
    return got[:, 0]


def _mantissas(rng, n):
    edge = np.array([1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.5, 4.0 / 3.0])
    return rng.choice([-1.0, 1.0], n) * np.concatenate([edge, rng.uniform(1.0, 2.0, n - edge.size)])


@pytest.mark.parametrize("lo,hi", [(-40, 40), (-1022, 1023), (-962, -954), (956, 964)])
def test_real(native, cuda_device, lo, hi):
    rng = np.random.default_rng(hi - lo)
    n = 3000
    d = np.ldexp(_mantissas(rng, n), rng.integers(lo, hi + 1, n))
    got = _first_columns(native, d)
    want = np.longdouble(1.0) / d.astype(np.longdouble)
    ulp = np.abs(got.astype(np.longdouble) - want) / np.spacing(np.abs(1.0 / d))
    assert float(ulp.max()) <= 0.5625 + 1e-3


def test_real_specials(native, cuda_device):
    d = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -1e-310, 2.0 ** -1024, 3e-309, 2.0 ** -1022, 1.7976931348623157e308])
    with np.errstate(all="ignore"):
        assert np.array_equal(_first_columns(native, d), 1.0 / d, equal_nan=True)


@pytest.mark.parametrize("lo,hi,units", [(-40, 40, 4.2), (-395, 395, 4.2), (-403, -396, 11.0), (396, 403, 11.0), (-500, 500, 11.0)])
def test_complex(native, cuda_device, lo, hi, units):
    rng = np.random.default_rng(abs(hi))
    n = 2000
    e = rng.integers(lo, hi + 1, n)
    other = np.ldexp(_mantissas(rng, n), -rng.integers(0, 60, n))
    re, im = _mantissas(rng, n), other
    swap = rng.random(n) < 0.5
    d = np.ldexp(np.where(swap, im, re), e) + 1j * np.ldexp(np.where(swap, re, im), e)
    got = _first_columns(native, d)
    x, y = d.real.astype(np.longdouble), d.imag.astype(np.longdouble)
    x, y = np.ldexp(x, -e), np.ldexp(y, -e)
    want = np.ldexp(x / (x * x + y * y), -e), np.ldexp(-y / (x * x + y * y), -e)
    unit = np.spacing(np.maximum(np.abs(want[0]), np.abs(want[1])).astype(np.float64))
    for part, w in ((got.real, want[0]), (got.imag, want[1])):
        assert float((np.abs(part.astype(np.longdouble) - w) / unit).max()) <= units
