"""Inverses of diagonal blocks at the edges of the column-wise kernels: widths
around one block of 8 and of 32 columns up to the widest supernode, real,
complex symmetric, Hermitian and the LU form, and the allocation-free entry
point with leading dimensions above s.

Tolerance: diagonally dominant blocks (condition number below 3), so the
explicit inverse is good to a few s 2^-53 < 1e-13 normwise; 1e-12."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["f64", "c128", "c128h"])
@pytest.mark.parametrize("width", [33, 40, 63, 64, 65, 95, 97, 121, 128])
def test_selinv_widths(native, cuda_device, width, kind):
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    make = synth.random_sparse_hpd if kind == "c128h" else synth.random_sparse_spd
    kw = {"complex_values": True} if kind == "c128" else {}
    p = make(2 * width + 3, 1.0, width, supernodes={"kind": "fundamental", "cap": width, "fill": 0.0}, **kw)
    ctx = SelInvContext.from_problem(p)
    sym = oracle.symbolic_for(p)
    L0, D0 = oracle.ldlt(p, sym)
    Z = ctx.selinv(torch.from_numpy(L0).cuda(), torch.from_numpy(D0).cuda())
    torch.cuda.synchronize()
    assert ctx.status() == 0
    assert oracle.block_errors(sym, Z.cpu().numpy(), oracle.selinv(sym, L0, D0, hermitian=kind == "c128h")).max() <= 1e-12


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("width", [33, 64, 65, 121, 128])
def test_lu_widths(native, cuda_device, width, cplx):
    import torch
    p = synth.random_sparse_nonsym(2 * width + 3, 1.0, width, complex_values=cplx,
                                   supernodes={"kind": "fundamental", "cap": width, "fill": 0.0})
    sym = oracle.symbolic_for(p)
    L, Ut = oracle.lu(p, sym)
    Zl0, Zu0 = oracle.selinv_lu(sym, L, Ut)
    plan = native.selinv_symbolic(sym.n, sym.nsuper, sym.super_ptr, sym.sparent, sym.rowptr, sym.rows)
    Lt, Ut_t = torch.from_numpy(L).cuda(), torch.from_numpy(Ut).cuda()
    Zl, Zu = torch.empty_like(Lt), torch.empty_like(Lt)
    native.selinv_numeric_lu(plan, native.SELINV_C128 if cplx else native.SELINV_F64, Lt, Ut_t, Zl, Zu)
    torch.cuda.synchronize()
    assert native.selinv_status(plan) == 0
    low = oracle.lower_mask(sym)
    assert oracle.block_errors(sym, Zl.cpu().numpy(), Zl0).max() <= 1e-12
    assert oracle.block_errors(sym, np.where(low, Zu.cpu().numpy(), 0), np.where(low, Zu0, 0)).max() <= 1e-12


@pytest.mark.parametrize("s", [1, 2, 7, 8, 9, 15, 16, 17, 31, 32, 33, 64, 65, 96, 127, 128])
def test_noalloc_widths(native, cuda_device, s):
    import torch
    rng = np.random.default_rng(s)
    g = rng.standard_normal((s, s))
    a = g @ g.T / s + np.eye(s)
    c = np.linalg.cholesky(a)
    L, D = c / np.diag(c), np.diag(c) ** 2
    ld, ldo = s + 3, s + 1
    host = np.full((s, ld), np.nan)                  # column-major: row j holds column j
    host[:, :s] = np.where(np.tri(s, k=-1), L, np.nan).T   # the diagonal and what lies above are not read
    out = torch.full((s, ldo), -7.0, dtype=torch.float64, device="cuda")
    for _ in range(2):
        native.selinv_dinv_noalloc(s, torch.from_numpy(host).cuda(), ld, torch.from_numpy(D).cuda(), out, ldo)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    ref = np.linalg.inv(a)
    assert np.linalg.norm(got[:, :s] - ref) <= 1e-12 * np.linalg.norm(ref)
    assert np.all(got[:, s:] == -7.0)                # nothing past the block's rows


# complex Lhat on the tensor cores: the widths around its narrowest, one and
# two 128-row tiles of the 2s output rows, odd remainders of the 16-step k,
# C of one to several 64-row tiles, and values spread over decades by rows.
# The digits carry 54 bits below a row's largest entry and the dropped pairs
# 2^-61 of it, so Lhat errs by s 2^-54 of row times column maxima: 1e-12
# normwise with room.
@pytest.mark.parametrize("kind", ["c128", "c128h"])
@pytest.mark.parametrize("width,n", [(16, 90), (17, 81), (18, 82), (31, 96), (32, 97), (33, 290), (63, 128), (64, 200), (65, 194), (127, 300)])
def test_complex_lhat_widths(native, cuda_device, width, n, kind):
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    make = synth.random_sparse_hpd if kind == "c128h" else synth.random_sparse_spd
    kw = {"complex_values": True} if kind == "c128" else {}
    p = make(n, 1.0, n, supernodes={"kind": "fundamental", "cap": width, "fill": 0.0}, **kw)
    ctx = SelInvContext.from_problem(p)
    ctx.set_options(oz_min_s=1)
    sym = oracle.symbolic_for(p)
    L0, D0 = oracle.ldlt(p, sym)
    Z = ctx.selinv(torch.from_numpy(L0).cuda(), torch.from_numpy(D0).cuda())
    torch.cuda.synchronize()
    assert ctx.status() == 0
    assert oracle.block_errors(sym, Z.cpu().numpy(), oracle.selinv(sym, L0, D0, hermitian=kind == "c128h")).max() <= 1e-12
