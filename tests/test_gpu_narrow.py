"""Narrow supernodes (one CTA or cluster each) at the edges: widths 1 to 16 and
the first past them, C from empty through the sizes at which the cluster
grows to the largest that fits, levels of one to many supernodes, each value
type and the LU form, with the tensor cores kept off these widths.

Tolerance: diagonally dominant matrices, FP64 products of at most 260 terms:
300 2^-53 = 3e-14 normwise; 1e-12 leaves room for the oracle's own."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _selinv(p, **opts):
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    ctx = SelInvContext.from_problem(p)
    ctx.set_options(oz_min_s=128, **opts)
    sym = oracle.symbolic_for(p)
    L0, D0 = oracle.ldlt(p, sym)
    L, D = torch.from_numpy(L0).cuda(), torch.from_numpy(D0).cuda()
    Z0 = oracle.selinv(sym, L0, D0, hermitian=p.hermitian)
    for _ in range(3):      # issued, captured, replayed
        Z = torch.full_like(L, float("nan"))
        ctx.selinv(L, D, out=Z)
        torch.cuda.synchronize()
        assert ctx.status() == 0
        assert oracle.block_errors(sym, Z.cpu().numpy(), Z0).max() <= 1e-12


@pytest.mark.parametrize("kind", ["f64", "c128", "c128h"])
@pytest.mark.parametrize("cap,n", [(1, 1), (1, 2), (1, 40), (2, 35), (3, 66), (5, 70), (7, 38), (8, 72), (8, 105), (11, 43),
                                   (15, 79), (16, 16), (16, 17), (16, 96), (16, 144), (17, 60)])
def test_narrow_widths(native, cuda_device, cap, n, kind):
    make = synth.random_sparse_hpd if kind == "c128h" else synth.random_sparse_spd
    kw = {"complex_values": True} if kind == "c128" else {}
    _selinv(make(n, 1.0, n, supernodes={"kind": "fundamental", "cap": cap, "fill": 0.0}, **kw),
            debug_checks=4)


@pytest.mark.parametrize("make", [lambda: synth.laplacian_2d(23, 19), lambda: synth.laplacian_3d(9, 4),
                                  lambda: synth.magnetic_laplacian_3d(8, 4), lambda: synth.tridiagonal(500, nd=True),
                                  lambda: synth.random_sparse_spd(200, 0.02, 8, complex_values=True)])
def test_narrow_levels(native, cuda_device, make):
    _selinv(make())
    _selinv(make(), symmetrize=0)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("cap,n", [(1, 33), (4, 30), (8, 70), (13, 50), (16, 75), (16, 110)])
def test_narrow_lu(native, cuda_device, cap, n, cplx):
    import torch
    p = synth.random_sparse_nonsym(n, 1.0, n, complex_values=cplx,
                                   supernodes={"kind": "fundamental", "cap": cap, "fill": 0.0})
    sym = oracle.symbolic_for(p)
    L, Ut = oracle.lu(p, sym)
    Zl0, Zu0 = oracle.selinv_lu(sym, L, Ut)
    plan = native.selinv_symbolic(sym.n, sym.nsuper, sym.super_ptr, sym.sparent, sym.rowptr, sym.rows)
    Lt, Ut_t = torch.from_numpy(L).cuda(), torch.from_numpy(Ut).cuda()
    Zl, Zu = torch.full_like(Lt, float("nan")), torch.full_like(Lt, float("nan"))
    native.selinv_numeric_lu(plan, native.SELINV_C128 if cplx else native.SELINV_F64, Lt, Ut_t, Zl, Zu)
    torch.cuda.synchronize()
    assert native.selinv_status(plan) == 0
    low = oracle.lower_mask(sym)
    assert oracle.block_errors(sym, Zl.cpu().numpy(), Zl0).max() <= 1e-12
    assert oracle.block_errors(sym, np.where(low, Zu.cpu().numpy(), 0), np.where(low, Zu0, 0)).max() <= 1e-12


# more supernodes in a level than SMs: small CTAs on the packed triangle
@pytest.mark.parametrize("make", [lambda: synth.laplacian_2d(63, 19), lambda: synth.laplacian_3d(14, 4),
                                  lambda: synth.magnetic_laplacian_3d(13, 4)])
def test_narrow_long_levels(native, cuda_device, make):
    _selinv(make())
