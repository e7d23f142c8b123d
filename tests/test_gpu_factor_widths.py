"""The factorization's kernels at the edges of their ranges: supernode widths
around the narrow kernel's limit, the 8-column panels and the 32-column
blocks, and levels with few to many diagonal blocks (clusters of 8 to 1 CTAs).

Tolerance: the matrices are diagonally dominant, so the entries of L are at
most 1 and an entry's error is a sum of at most n = 300 rounded products,
n 2^-53 = 3e-14 of the largest; 1e-12 leaves room for the oracle's own."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _blocks(count, size, kind, seed):
    """`count` dense diagonal blocks of `size` columns."""
    rng = np.random.default_rng(seed)
    colptr, rows, vals = [0], [], []
    for b in range(count):
        g = rng.standard_normal((size, size)) + (1j * rng.standard_normal((size, size)) if kind != "f64" else 0)
        a = (g + (g.conj().T if kind == "c128h" else g.T)) / 2
        np.fill_diagonal(a, np.abs(a).sum(axis=1) + 1.0)
        for j in range(size):
            rows.append(np.arange(b * size + j, (b + 1) * size))
            vals.append(a[j:, j])
            colptr.append(colptr[-1] + size - j)
    return synth.Problem(f"blocks{count}x{size}", count * size, np.array(colptr, np.int64),
                         np.concatenate(rows).astype(np.int32), np.concatenate(vals), np.arange(count * size),
                         dict(synth.problems.RELAXED_128), {"hermitian": kind == "c128h"})


def _check(p):
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    ctx = SelInvContext.from_problem(p)
    sym = oracle.symbolic_for(p)
    L0, D0 = oracle.ldlt(p, sym)
    L, D = ctx.factor(torch.from_numpy(p.values).cuda())
    torch.cuda.synchronize()
    assert ctx.status() == 0
    r, c, _ = oracle.panel_entries(sym)
    Lg = L.cpu().numpy()
    assert np.abs(D.cpu().numpy() - D0).max() <= 1e-12 * np.abs(D0).max()
    assert np.abs(np.where(r > c, Lg - L0, 0)).max() <= 1e-12
    assert np.all(Lg[r == c] == 1) and np.all(Lg[r < c] == 0)


@pytest.mark.parametrize("kind", ["f64", "c128", "c128h"])
@pytest.mark.parametrize("width", [1, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 65, 100, 127, 128])
def test_widths(native, cuda_device, width, kind):
    p = _blocks(1, 2 * width + 5, kind, width)
    p.supernodes = {"kind": "fundamental", "cap": width, "fill": 0.0}
    _check(p)


@pytest.mark.parametrize("count,size", [(1, 40), (19, 40), (20, 40), (39, 33), (77, 40), (160, 33)])
def test_levels_of_many_blocks(native, cuda_device, count, size):
    _check(_blocks(count, size, "f64", count))
    if count in (1, 160):
        _check(_blocks(count, size, "c128", count))


# the update matrix on the tensor cores: C from just below its shortest, one
# and several 128 x 64 tiles, remainders of the 16-column steps
@pytest.mark.parametrize("cap,n", [(17, 112), (17, 113), (17, 114), (24, 153), (32, 160), (33, 290), (128, 256), (128, 449)])
def test_update_on_tensor_cores(native, cuda_device, cap, n):
    p = _blocks(1, n, "f64", n)
    p.supernodes = {"kind": "fundamental", "cap": cap, "fill": 0.0}
    _check(p)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_nonfinite_entry_reaches_a_pivot(native, cuda_device, bad):
    """A non-finite entry below the diagonal blocks is reported by a later
    pivot, through the digit planes as through FP64 products."""
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    p = _blocks(1, 300, "f64", 3)
    p.supernodes = {"kind": "fundamental", "cap": 64, "fill": 0.0}
    ctx = SelInvContext.from_problem(p)
    v = p.values.copy()
    v[int(p.colptr[5]) + 200] = bad
    for fast in (1, 0):
        ctx.set_options(fast_contraction=fast)
        ctx.factor(torch.from_numpy(v).cuda())
        torch.cuda.synchronize()
        assert ctx.status() == native.SELINV_ERR_ZERO_PIVOT


@pytest.mark.parametrize("cap", [17, 64, 128])
def test_badly_scaled_matrix(native, cuda_device, cap):
    """S A S with S over six decades: D spans twelve within a supernode, rows
    of L as many the other way.  Row p of L times sqrt(D), over S_p, is of even
    size (at most 1), and its error the unscaled factorization's: 1e-12."""
    import torch
    from paper_1604_02528_gb300.api import SelInvContext
    p = synth.symmetric_scaling(_blocks(1, 300, "f64", 5), 12.0, 7)
    p.supernodes = {"kind": "fundamental", "cap": cap, "fill": 0.0}
    ctx = SelInvContext.from_problem(p)
    sym = oracle.symbolic_for(p)
    L0, D0 = oracle.ldlt(p, sym)
    L, D = ctx.factor(torch.from_numpy(p.values).cuda())
    torch.cuda.synchronize()
    assert ctx.status() == 0
    r, c, _ = oracle.panel_entries(sym)
    scale = np.sqrt(np.abs(D0))[c] / np.sqrt(p.values[p.diag_positions()])[r]
    assert np.abs(np.where(r > c, (L.cpu().numpy() - L0) * scale, 0)).max() <= 1e-12
    assert np.abs(D.cpu().numpy() / D0 - 1).max() <= 1e-12


# row tiles of 4 to 64 rows: groups of four, two and one row per warp, and ragged last tiles
@pytest.mark.parametrize("kind", ["f64", "c128h"])
@pytest.mark.parametrize("count,size,cap", [(6, 101, 34), (10, 143, 50), (16, 167, 33), (16, 230, 96), (24, 167, 33), (30, 201, 70)])
def test_row_tiles(native, cuda_device, count, size, cap, kind):
    p = _blocks(count, size, kind, size)
    p.supernodes = {"kind": "fundamental", "cap": cap, "fill": 0.0}
    _check(p)
