"""FP64 tiles of the level schedule at their edges: widths around 16 and 32
columns, C around 16-, 32- and 64-row tiles and cluster splits, every value
type with the tensor cores off, the LU form, and mixed trees whose tensor-core
supernodes gather from supernodes that ran on the tiles (their column bounds).

Tolerance: diagonally dominant matrices, products of at most 600 terms:
600 2^-53 = 7e-14 normwise; 1e-12 leaves room for the oracle's own.  The mixed
trees keep the suite's 1e-10."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _selinv(p, tol, **opts):
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    ctx = SelInvContext.from_problem(p)
    ctx.set_options(**opts)
    sym = oracle.symbolic_for(p)
    L0, D0 = oracle.ldlt(p, sym)
    L, D = torch.from_numpy(L0).cuda(), torch.from_numpy(D0).cuda()
    Z0 = oracle.selinv(sym, L0, D0, hermitian=p.hermitian)
    for _ in range(2):
        Z = torch.full_like(L, float("nan"))
        ctx.selinv(L, D, out=Z)
        torch.cuda.synchronize()
        assert ctx.status() == 0
        assert oracle.block_errors(sym, Z.cpu().numpy(), Z0).max() <= tol


@pytest.mark.parametrize("kind", ["f64", "c128", "c128h"])
@pytest.mark.parametrize("cap,n", [(17, 48), (17, 49), (31, 63), (32, 96), (33, 98), (48, 48), (64, 161), (100, 230), (128, 400), (17, 560)])
def test_wide(native, cuda_device, cap, n, kind):
    make = synth.random_sparse_hpd if kind == "c128h" else synth.random_sparse_spd
    kw = {"complex_values": True} if kind == "c128" else {}
    _selinv(make(n, 1.0, n, supernodes={"kind": "fundamental", "cap": cap, "fill": 0.0}, **kw), 1e-12,
            fast_contraction=0, debug_checks=4)


@pytest.mark.parametrize("make,low", [(lambda: synth.laplacian_3d(14, 4), 33), (lambda: synth.laplacian_3d(14, 4), 65),
                                      (lambda: synth.dft_sheet(side=8, nbasis=16), 33),
                                      (lambda: synth.magnetic_laplacian_3d(11, 4), 33)])
def test_mixed_with_tensor_cores(native, cuda_device, make, low):
    _selinv(make(), 1e-10, oz_min_s=low)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("cap,n", [(17, 34), (32, 97), (33, 200), (90, 181), (128, 300), (20, 540)])
def test_lu(native, cuda_device, cap, n, cplx):
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
