"""The adjoints over trees of every shape: chains (every level in the last
group), forests of one level (every level in the first), trees with both, and
widths around the edges of the 8, 16 and 32-entry tiles of their products.

Tolerance: diagonally dominant matrices; each entry passes through five
products of at most 300 terms: 5 * 300 * 2^-53 = 2e-13 of the largest, and
1e-11 leaves room for the oracle's own errors and the growth by D^{-1}."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _positions(sym, p):
    off, sp = sym.panel_offsets(), sym.super_ptr
    owner = np.repeat(np.arange(sym.nsuper), np.diff(sp))
    cols = np.repeat(np.arange(p.n), np.diff(p.colptr))
    at = []
    for i, j in zip(p.rowind, cols):
        K = owner[j]
        R = sym.rows[sym.rowptr[K]:sym.rowptr[K + 1]]
        at.append(off[K] + (j - sp[K]) * R.size + np.searchsorted(R, i))
    return np.array(at, np.int64)


def _forest(count, size):
    """`count` dense diagonal blocks of `size` columns: one level of `count` supernodes."""
    rng = np.random.default_rng(size)
    colptr, rows, vals = [0], [], []
    for b in range(count):
        g = rng.standard_normal((size, size))
        a = (g + g.T) / 2
        np.fill_diagonal(a, np.abs(a).sum(axis=1) + 1.0)
        for j in range(size):
            rows.append(np.arange(b * size + j, (b + 1) * size))
            vals.append(a[j:, j])
            colptr.append(colptr[-1] + size - j)
    return synth.Problem(f"forest{count}x{size}", count * size, np.array(colptr, np.int64),
                         np.concatenate(rows).astype(np.int32), np.concatenate(vals), np.arange(count * size),
                         dict(synth.problems.RELAXED_128), {"hermitian": False})


def _dense(n, cap):
    return synth.random_sparse_spd(n, 1.0, n, supernodes={"kind": "fundamental", "cap": cap, "fill": 0.0})


@pytest.mark.parametrize("ozm", [8, 16])
@pytest.mark.parametrize("make", [lambda: synth.tridiagonal(40), lambda: _forest(1, 33), lambda: _forest(20, 17),
                                  lambda: _dense(70, 7), lambda: _dense(90, 9), lambda: _dense(140, 31),
                                  lambda: _dense(200, 33), lambda: _dense(260, 65), lambda: _dense(300, 127),
                                  lambda: synth.laplacian_3d(10, 4), lambda: synth.tridiagonal(300, nd=True)])
def test_adjoint_trees(native, cuda_device, make, ozm):
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    p = make()
    sym = oracle.symbolic_for(p)
    L, D = oracle.ldlt(p, sym)
    Z = oracle.selinv(sym, L, D)
    low = oracle.lower_mask(sym)
    W = np.where(low, np.random.default_rng(3).standard_normal(low.size), 0.0)
    Lb0, Db0 = oracle.selinv_adjoint(sym, L, D, Z, W)
    Ab0 = oracle.ldlt_adjoint(sym, L, D, Lb0, Db0)[_positions(sym, p)]
    ctx = SelInvContext.from_problem(p)
    ctx.attach_matrix()
    ctx.set_options(oz_min_s=ozm)
    t = lambda x: torch.from_numpy(np.ascontiguousarray(x)).cuda()
    Lt, Dt, Zt, Wt = t(L), t(D), t(Z), t(W)
    r, c, _ = oracle.panel_entries(sym)
    strict = r > c
    for _ in range(3):      # issued, captured, replayed
        Lb, Db = torch.full_like(Lt, float("nan")), torch.full_like(Dt, float("nan"))
        native.selinv_adjoint(ctx.plan, native.SELINV_F64, Lt, Dt, Zt, Wt, Lb, Db)
        Av = torch.full((p.values.size,), float("nan"), dtype=torch.float64, device="cuda")
        native.selinv_factor_adjoint(ctx.plan, native.SELINV_F64, Lt, Dt, t(Lb0), t(Db0), Av)
        torch.cuda.synchronize()
        assert ctx.status() == 0
        for got, want in ((np.where(strict, Lb.cpu().numpy(), 0), np.where(strict, Lb0, 0)),
                          (Db.cpu().numpy(), Db0), (Av.cpu().numpy(), Ab0)):
            assert np.abs(got - want).max() <= 1e-11 * np.abs(want).max()
