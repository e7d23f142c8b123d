"""selinv_dinv_noalloc on blocks with pivots and entries at the ends of the
range: Dinv(i, j) = sum over k >= max(i, j) of X(k, i) / D_k X(k, j) with
X = L^{-1}, every term as IEEE arithmetic gives it and no other term."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _call(native, L, D):
    import torch
    s = D.size
    out = torch.full((s, s), float("nan"), dtype=torch.float64, device="cuda")
    native.selinv_dinv_noalloc(s, torch.from_numpy(np.ascontiguousarray(L.T)).cuda(), s, torch.from_numpy(D).cuda(), out, s)
    torch.cuda.synchronize()
    return out.cpu().numpy().T


def _reference(L, D):
    """In the order of the definition, in 64 bits."""
    s = D.size
    X = np.eye(s)
    with np.errstate(all="ignore"):
        for i in range(s):
            for k in range(i):
                X[i, :k + 1] -= L[i, k] * X[k, :k + 1]
        out = np.zeros((s, s))
        for k in range(s):
            out[:k + 1, :k + 1] += np.outer(X[k, :k + 1] / D[k], X[k, :k + 1])
    return out


def _block(s, seed):
    """Unit lower, its entries small enough that X stays of their size: 2^-53 of
    a term in each of at most 3 s operations, 128 * 3 * 2^-53 = 5e-14."""
    rng = np.random.default_rng(seed)
    return np.tril(rng.standard_normal((s, s)) / s, -1) + np.eye(s), rng.uniform(0.5, 2.0, s) * rng.choice([-1, 1], s)


def _agree(got, want):
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(np.isinf(got), np.isinf(want))
    ok = np.isfinite(want)
    assert np.abs(got[ok] - want[ok]).max() <= 1e-13 * np.abs(want[ok]).max()


@pytest.mark.parametrize("bad", [0.0, -0.0, np.inf, np.nan])
@pytest.mark.parametrize("s,k", [(1, 0), (16, 3), (17, 16), (33, 20), (96, 40), (128, 100), (128, 127)])
def test_a_pivot_reaches_its_own_terms_only(native, cuda_device, s, k, bad):
    L, D = _block(s, s + k)
    D[k] = bad
    want = _reference(L, D)
    if np.isfinite(want).any():
        _agree(_call(native, L, D), want)
    else:
        assert np.array_equal(np.isnan(_call(native, L, D)), np.isnan(want))


def test_terms_are_quotients(native, cuda_device):
    """With D_0 infinite, Dinv(0, 0) of a 2 x 2 block is the one term
    (X / D_1) X: bit for bit a division and a product, also where 1 / D_1
    overflows."""
    rng = np.random.default_rng(1)
    tiny = 5e-324 * 2.0 ** 49
    mantissa = lambda n: rng.choice([-1.0, 1.0], n) * rng.uniform(1.0, 2.0, n)     # noqa: E731
    l = [mantissa(1500), np.ldexp(mantissa(200), rng.integers(-410, -390, 200)), np.ldexp(mantissa(200), rng.integers(390, 410, 200)),
         [1e-5, -3e-7, 1e-8, 0.0]]
    d = [mantissa(1500), np.ldexp(mantissa(200), rng.integers(-410, -390, 200)), np.ldexp(mantissa(200), rng.integers(390, 410, 200)),
         [tiny, -tiny, tiny / 3, 2.0]]
    for l, d in zip(np.concatenate(l), np.concatenate(d)):
        got = _call(native, np.array([[1.0, 0.0], [l, 1.0]]), np.array([np.inf, d]))
        with np.errstate(all="ignore"):
            assert got[0, 0] == (-l / d) * -l


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("s,i,j", [(2, 1, 0), (17, 9, 4), (33, 32, 0), (40, 36, 34), (96, 50, 10), (96, 95, 62), (128, 127, 126), (128, 65, 64)])
def test_an_entry_of_l_reaches_its_own_columns_only(native, cuda_device, s, i, j, bad):
    """L(i, j) is in the columns of X up to j; those after it never meet it,
    although they share a warp with column j."""
    L, D = _block(s, 7 * s + j)
    L[i, j] = bad
    _agree(_call(native, L, D), _reference(L, D))
