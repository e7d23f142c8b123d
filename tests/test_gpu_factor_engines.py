"""The factorization's real updates on the tensor cores and in FP64 FMA: matrices
that are neither definite nor diagonally dominant, whose L grows, and the
options that choose between the two.

Tolerance: with S_ii = sum_k L_ik^2 |D_k|, an entry of A - L D L^T is a sum of
at most n rounded products.  FMA: 2^-53 of each product and of each partial
sum, together at most 2 n 2^-53 sqrt(S_ii S_jj) by Cauchy-Schwarz.  Tensor
cores: the factors of a product rounded by 2^-55 and 2^-54 of the largest entry
of their row of L sqrt(|D|), at most sqrt(S_ii), and digit pairs below 2^-59
dropped: less than 2^-53 sqrt(S_ii S_jj) a product, and the FP64 additions as
before."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _indefinite(n, seed, pivot, sparse):
    """A dense symmetric Gaussian matrix; every fifth pivot is `pivot` times the
    others (L grows by its inverse), and a part of the rows has no entry in
    those columns, so that large and small rows meet in one product."""
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((n, n))
    a = (a + a.T) / 2
    small = np.arange(0, n // 2, 5)
    a[small, small] *= pivot
    if sparse:
        rows = np.arange(1, n, 2)
        for j in small:
            a[rows[rows > j], j] = a[j, rows[rows > j]] = 0.0
    colptr = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    rowind = np.concatenate([np.arange(j, n) for j in range(n)]).astype(np.int32)
    values = np.concatenate([a[j:, j] for j in range(n)])
    return a, synth.Problem("indefinite", n, colptr, rowind, values, np.arange(n), {"kind": "fundamental", "cap": 64, "fill": 0.0},
                            {"hermitian": False})


def _factor(p, cap, **opts):
    """L as a dense matrix, D."""
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    p.supernodes = {"kind": "fundamental", "cap": cap, "fill": 0.0}
    ctx = SelInvContext.from_problem(p)
    ctx.set_options(**opts)
    L, D = ctx.factor(torch.from_numpy(p.values).cuda())
    torch.cuda.synchronize()
    assert ctx.status() == 0
    a, x, l = ctx.analysis, L.cpu().numpy(), np.zeros((p.n, p.n))
    at = 0
    for K in range(a["nsuper"]):
        c0, c1 = a["super_ptr"][K], a["super_ptr"][K + 1]
        rows = a["rows"][a["rowptr"][K]:a["rowptr"][K + 1]]
        l[rows, c0:c1] = x[at:at + rows.size * (c1 - c0)].reshape(c1 - c0, rows.size).T
        at += rows.size * (c1 - c0)
    return l, D.cpu().numpy()


def _backward_error(a, l, d):
    """Largest |A - L D L^T|_ij / sqrt(S_ii S_jj), in units of n 2^-53."""
    hi = np.longdouble
    e = np.abs(a.astype(hi) - (l.astype(hi) * d.astype(hi)) @ l.astype(hi).T)
    s = np.sqrt((l.astype(hi) ** 2 * np.abs(d.astype(hi))).sum(axis=1))
    return float((e / np.outer(s, s)).max()) / (a.shape[0] * 2.0 ** -53)


@pytest.mark.parametrize("sparse", [False, True])
@pytest.mark.parametrize("pivot", [1.0, 1e-4, 1e-9])
@pytest.mark.parametrize("cap", [17, 40, 64, 128])
def test_indefinite_matrices_with_growth(native, cuda_device, cap, pivot, sparse):
    a, p = _indefinite(290, 11, pivot, sparse)
    for fast in (1, 0):
        l, d = _factor(p, cap, fast_contraction=fast)
        if pivot < 1:
            assert np.abs(l).max() > 0.01 / pivot        # it did grow
        assert _backward_error(a, l, d) <= 2.0


@pytest.mark.parametrize("cap,ozm,same", [(40, 41, True), (40, 40, False), (64, 128, True), (16, 1, True)])
def test_engine_follows_oz_min_s(native, cuda_device, cap, ozm, same):
    _, p = _indefinite(290, 12, 1.0, False)
    l0, d0 = _factor(p, cap, fast_contraction=0)
    l1, d1 = _factor(p, cap, oz_min_s=ozm)
    assert (np.array_equal(l0, l1) and np.array_equal(d0, d1)) == same
