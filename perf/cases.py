"""Performance cases: what a user of the library has it do, through its public calls.

A case is a dict of plain values.  ``call`` names the path, ``sites`` the
lattice ("40x40x40"), ``matrix`` the values put on it and ``dtype`` the element
type; the remaining keys are the path's own.  Matrices are lattices in
nested-dissection order, as in the workloads of ``bench.py``:

  laplacian  5- / 7-point Laplacian, diagonal 2d + U(0,1) (2D: + 0.1 more);
             complex types: minus a pole shift z = E + i eta
  magnetic   the same with hopping exp(i theta) on the edges (Hermitian)
  diffusion  edge conductances exp(0.5 N(0,1)), Dirichlet ghost edges
  sheet      dense ``basis`` x ``basis`` blocks within 2.5 lattice units,
             H - z S as an atomic-orbital calculation has it (complex symmetric)

``listed()`` holds the cases, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` what a program has in hand before the call,
``run(state)`` one pass, ``work(case)`` the bytes and operations that the path
cannot do without and ``exact(case, seed)`` the outputs from dense 64-bit
linear algebra.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1604_02528_gb300 import _native as N
from paper_1604_02528_gb300.api import SelInvContext, pole_sum
from paper_1604_02528_gb300.autograd import SelInv

DTYPES = {"f64": N.SELINV_F64, "c128": N.SELINV_C128, "c128h": N.SELINV_C128H}
# the supernode rules of the workloads: 2D grids and sheets, 3D grids
FUNDAMENTAL, RELAXED = ("fundamental", 64, 0.0), ("relaxed", 128, 0.10)
SHEET_CUTOFF = 2.5
# dense 64-bit inverses up to this size (real; a complex one costs four times as much)
EXACT_N = 17000


def listed():
    return [
        # One diagonal block inverted inside a caller's own loop: the smallest call.
        {"name": "block_96", "call": "block", "s": 96, "dtype": "f64"},
        # A small planar mesh, where launches and the tree's depth count.
        {"name": "selinv_2d", "call": "selinv", "matrix": "laplacian", "sites": "63x63", "dtype": "f64"},
        # The headline workload, with the options that the autotuner settles on for it.
        {"name": "selinv_3d", "call": "selinv", "matrix": "laplacian", "sites": "40x40x40", "dtype": "f64",
         "oz_min_s": 8, "split_min_steps": 8},
        # An electronic-structure matrix at one pole: complex symmetric, dense blocks.
        {"name": "selinv_sheet", "call": "selinv", "matrix": "sheet", "sites": "32x32", "basis": 16, "dtype": "c128"},
        # A magnetic-field Hamiltonian: complex Hermitian, ragged box.
        {"name": "selinv_hermitian", "call": "selinv", "matrix": "magnetic", "sites": "20x21x19", "dtype": "c128h"},
        # Pole shifts of one pattern and two unrelated real meshes in one call.
        {"name": "batched", "call": "batched", "matrix": "laplacian", "sites": "18x19x17", "dtype": "c128", "poles": 6,
         "extra_2d": 100, "extra_3d": 13},
        # A pole expansion from the matrices on: factor, invert and sum the diagonal, pole after pole.
        {"name": "poles", "call": "poles", "matrix": "laplacian", "sites": "16x17x15", "dtype": "c128", "poles": 4},
        # The factorization in front of every inversion, at the headline workload's size.
        {"name": "factor_3d", "call": "factor", "matrix": "laplacian", "sites": "40x40x40", "dtype": "f64"},
        # A training step on conductances: factor, invert, and both adjoints behind autograd.
        {"name": "train_3d", "call": "train", "matrix": "diffusion", "sites": "24x24x24", "dtype": "f64"},
        # Factors of a nonsymmetric matrix (convection on a mesh) from an external LU.
        {"name": "lu_3d", "call": "lu", "matrix": "diffusion", "sites": "22x20x21", "dtype": "f64"},
        # Host buffers in and out: a solver on the host that hands its factors over.
        {"name": "host_3d", "call": "host", "matrix": "laplacian", "sites": "24x25x23", "dtype": "f64"},
        # Only the diagonal of one corner of the mesh (an eighth of the unknowns).
        {"name": "subset_3d", "call": "subset", "matrix": "laplacian", "sites": "24x22x26", "dtype": "f64", "part": 8},
    ]


def draw(rng):
    """A case of the listed ones' ranges: the same calls, sizes from a handful
    of unknowns to the listed ones, every side drawn by itself."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi, d=3):
        base = log_int(lo, hi)
        return "x".join(str(max(2, min(hi, int(round(base * rng.uniform(0.85, 1.15)))))) for _ in range(d))

    kind = rng.choice(["block", "selinv_2d", "selinv_3d", "sheet", "hermitian", "batched", "poles", "factor",
                       "factor_c", "train", "lu", "host", "subset"])
    if kind == "block":
        return {"call": "block", "s": rng.randint(1, 128), "dtype": "f64"}
    if kind == "selinv_2d":
        return {"call": "selinv", "matrix": "laplacian", "sites": box(10, 245, 2), "dtype": "f64"}
    if kind == "selinv_3d":
        return {"call": "selinv", "matrix": "laplacian", "sites": box(5, 40), "dtype": rng.choice(["f64", "f64", "c128"]),
                "oz_min_s": rng.choice([8, 16]), "split_min_steps": rng.choice([8, 16])}
    if kind == "sheet":
        return {"call": "selinv", "matrix": "sheet", "sites": box(5, 30, 2), "basis": rng.choice([4, 9, 13, 16]), "dtype": "c128"}
    if kind == "hermitian":
        return {"call": "selinv", "matrix": "magnetic", "sites": box(5, 22), "dtype": "c128h"}
    if kind == "batched":
        return {"call": "batched", "matrix": "laplacian", "sites": box(5, 18), "dtype": "c128", "poles": rng.randint(2, 8),
                "extra_2d": log_int(12, 100), "extra_3d": log_int(4, 13)}
    if kind == "poles":
        return {"call": "poles", "matrix": "laplacian", "sites": box(5, 16), "dtype": "c128", "poles": rng.randint(2, 5)}
    if kind == "factor":
        return {"call": "factor", "matrix": rng.choice(["laplacian", "diffusion"]), "sites": box(6, 38), "dtype": "f64"}
    if kind == "factor_c":
        matrix = rng.choice(["laplacian", "magnetic"])
        return {"call": "factor", "matrix": matrix, "sites": box(5, 22), "dtype": "c128h" if matrix == "magnetic" else "c128"}
    if kind == "train":
        return {"call": "train", "matrix": "diffusion", "sites": box(5, 24), "dtype": "f64"}
    if kind == "lu":
        return {"call": "lu", "matrix": "diffusion", "sites": box(5, 21), "dtype": "f64"}
    if kind == "host":
        return {"call": "host", "matrix": "laplacian", "sites": box(5, 30), "dtype": "f64"}
    return {"call": "subset", "matrix": "laplacian", "sites": box(6, 30), "dtype": "f64", "part": rng.choice([3, 8, 16])}


# ---------------------------------------------------------------------------
# matrices
# ---------------------------------------------------------------------------
class Pattern:
    """A lattice's lower CSC pattern in nested-dissection order.  Entry k is
    (rowind[k], cols[k]); dist[k] the distance of its two sites."""

    def __init__(self, sites, reach, basis, leaf):
        order = _dissection(sites, int(reach), leaf)
        m = order.size
        inverse = np.empty(m, dtype=np.int64)
        inverse[order] = np.arange(m)
        xyz = np.stack(np.unravel_index(np.arange(m), sites[::-1])[::-1], axis=1)   # x fastest
        r = int(reach)
        shifts = [d for d in np.ndindex(*([2 * r + 1] * len(sites)))]
        rows, cols, dist = [], [], []
        for d in shifts:
            d = np.array(d) - r
            norm = math.sqrt(float((d * d).sum()))
            if norm > reach:
                continue
            to = xyz + d
            ok = ((to >= 0) & (to < np.array(sites))).all(axis=1)
            a = inverse[np.nonzero(ok)[0]]
            b = inverse[(to[ok] * np.cumprod([1] + list(sites[:-1]))).sum(axis=1)]
            keep = b >= a
            rows.append(b[keep])
            cols.append(a[keep])
            dist.append(np.full(int(keep.sum()), norm))
        rows, cols, dist = np.concatenate(rows), np.concatenate(cols), np.concatenate(dist)
        # every site pair becomes a dense basis x basis block (its lower half on the diagonal)
        i, j = np.divmod(np.arange(basis * basis), basis)
        rows = (rows[:, None] * basis + i).ravel()
        cols = (cols[:, None] * basis + j).ravel()
        dist = np.repeat(dist, basis * basis)
        low = rows >= cols
        rows, cols, dist = rows[low], cols[low], dist[low]
        by = np.lexsort((rows, cols))
        self.sites, self.n = sites, m * basis
        self.rowind, self.cols, self.dist = rows[by].astype(np.int32), cols[by].astype(np.int32), dist[by]
        self.colptr = np.concatenate([[0], np.cumsum(np.bincount(cols, minlength=self.n))]).astype(np.int64)
        self.diag = self.colptr[:-1]            # the diagonal comes first in its column
        self.rule = RELAXED if len(sites) == 3 else FUNDAMENTAL
        # ghost edges of a site: the lattice faces that it lies on (Dirichlet boundary)
        faces = sum(((xyz[:, d] == 0).astype(int) + (xyz[:, d] == sites[d] - 1)) for d in range(len(sites)))
        self.faces = faces[order]


def _dissection(sites, width, leaf):
    """Nested dissection of a box: halves along the longest side, the
    separator (``width`` planes) last; boxes of at most ``leaf`` sites as they lie."""
    strides = np.cumprod([1] + list(sites[:-1]))
    out = []

    def box(lo, hi):
        grids = np.meshgrid(*[np.arange(a, b) * s for a, b, s in zip(lo, hi, strides)][::-1], indexing="ij")
        return sum(grids).ravel()

    def cut(lo, hi):
        sides = [b - a for a, b in zip(lo, hi)]
        if min(sides) <= 0:
            return
        if math.prod(sides) <= leaf or max(sides) < width + 2:
            out.append(box(lo, hi))
            return
        d = sides.index(max(sides))
        mid = lo[d] + (sides[d] - width + 1) // 2
        put = lambda v, x: v[:d] + [x] + v[d + 1:]   # noqa: E731
        cut(lo, put(hi, mid))
        cut(put(lo, mid + width), hi)
        out.append(box(put(lo, mid), put(hi, mid + width)))

    cut([0] * len(sites), list(sites))
    return np.concatenate(out)


def _sites(text):
    return tuple(int(x) for x in text.split("x"))


@functools.lru_cache(maxsize=24)
def _pattern(matrix, sites, basis=1):
    if matrix == "sheet":
        return Pattern(_sites(sites), SHEET_CUTOFF, basis, 4)
    return Pattern(_sites(sites), 1.0, 1, 32)


def _pattern_of(case):
    return _pattern(case["matrix"], case["sites"], case.get("basis", 1))


def _values(p, matrix, dtype, rng):
    """One matrix's stored lower values on pattern ``p``."""
    nnz, off = p.rowind.size, p.rowind != p.cols
    if matrix == "diffusion":
        theta = np.where(off, np.exp(0.5 * rng.standard_normal(nnz)), 0.0)
        v = -theta
        diag = np.bincount(p.cols, theta, p.n) + np.bincount(p.rowind, theta, p.n)
        v[p.diag] = diag + p.faces * np.exp(0.5 * rng.standard_normal(p.n))
    elif matrix == "sheet":
        z = complex(-0.2, 0.05)
        decay = np.exp(-p.dist)
        per_row = np.bincount(p.rowind, minlength=p.n) + np.bincount(p.cols, minlength=p.n)
        v = rng.standard_normal(nnz) * decay - z * 0.1 * rng.standard_normal(nnz) * decay / per_row[p.cols]
        v[p.diag] = rng.standard_normal(p.n) - z * 1.1
    else:
        v = np.where(off, -1.0, 0.0)
        if matrix == "magnetic":
            v = v * np.exp(0.5j * np.pi * rng.uniform(-1.0, 1.0, nnz))
        v[p.diag] = 2.0 * len(p.sites) + rng.uniform(0.0, 1.0, p.n) + (0.1 if len(p.sites) == 2 else 0.0)
        if dtype == "c128":
            v = v - np.where(off, 0.0, _shift(rng))
    return v.astype(np.float64 if dtype == "f64" else np.complex128)


def _shift(rng):
    """A pole of a pole expansion: E ~ U(-1,1), eta log-uniform in 1e-3 .. 1e-1."""
    return complex(rng.uniform(-1.0, 1.0), 10.0 ** rng.uniform(-3.0, -1.0))


def _matrices(case, seed):
    """(pattern, values, dtype) of every matrix that a pass takes, in order."""
    rng = np.random.default_rng(seed)
    p, dtype = _pattern_of(case), case["dtype"]
    got = [(p, _values(p, case["matrix"], dtype, rng), dtype) for _ in range(case.get("poles", 2 if case["call"] == "lu" else 1))]
    if "extra_2d" in case:
        for side, d in ((case["extra_2d"], 2), (case["extra_3d"], 3)):
            q = _pattern("laplacian", "x".join([str(side)] * d))
            got.append((q, _values(q, "laplacian", "f64", rng), "f64"))
    return got


def _weights(count, seed):
    rng = np.random.default_rng([seed, 1])
    return rng.standard_normal(count) + 1j * rng.standard_normal(count)


def _block(case, seed):
    rng = np.random.default_rng(seed)
    g = rng.standard_normal((case["s"], case["s"]))
    return torch.from_numpy(g @ g.T / case["s"] + np.eye(case["s"]))


def _picked(case, n):
    return np.arange(max(1, n // case["part"]))


# ---------------------------------------------------------------------------
# the passes
# ---------------------------------------------------------------------------
def _context(p, dtype, options=None):
    kind, cap, fill = p.rule
    ctx = SelInvContext(p.n, p.colptr, p.rowind, kind, cap, fill, hermitian=dtype == "c128h")
    if options:
        ctx.set_options(**options)
    return ctx


def _panel_columns(ctx):
    """Column of every panel element, and the places of the diagonal ones."""
    a = ctx.analysis
    width, rows = np.diff(a["super_ptr"]).astype(np.int64), np.diff(a["rowptr"])
    start = np.concatenate([[0], np.cumsum(width * rows)[:-1]])
    column = np.arange(ctx.n)
    of = np.repeat(np.arange(width.size), width)
    inside = column - a["super_ptr"][of]
    return np.repeat(column, rows[of]), start[of] + inside * (rows[of] + 1)


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["call"] == "block":
        s = case["s"]
        c = torch.linalg.cholesky(_block(case, seed))
        d = c.diagonal()
        column_major = (c / d).T.contiguous().to(dev)
        return {"call": "block", "s": s, "L": column_major, "D": (d * d).to(dev),
                "out": torch.empty(s, s, dtype=torch.float64, device=dev)}
    options = {k: case[k] for k in ("oz_min_s", "split_min_steps") if k in case}
    every, ctxs = _matrices(case, seed), {}
    for p, _, dtype in every:
        if id(p) not in ctxs:
            ctxs[id(p)] = _context(p, dtype, options)
    ctx = ctxs[id(every[0][0])]
    A = [torch.from_numpy(v).to(dev) for _, v, _ in every]
    state = {"call": case["call"], "ctx": ctx, "A": A}
    if case["call"] == "train":
        nnz = ctx.nnz
        state["W"] = torch.from_numpy(np.random.default_rng([seed, 1]).standard_normal(nnz)).to(dev)
        return state
    if case["call"] in ("factor", "poles"):
        dt = DTYPES[case["dtype"]]
        ctx.attach_matrix()
        state["L"], state["D"] = ctx.empty_panels(dt), torch.empty(ctx.n, dtype=A[0].dtype, device=dev)
        if case["call"] == "poles":
            state["Z"] = [ctx.empty_panels(dt) for _ in A]
            state["pos"] = torch.from_numpy(ctx.select(np.arange(ctx.n), np.arange(ctx.n))).to(dev)
            state["weights"] = _weights(len(A), seed)
        return state
    factors = [ctxs[id(p)].factor(a) for (p, _, _), a in zip(every, A)]
    del state["A"]
    if case["call"] == "lu":
        # L of one matrix and (D L^T) of another: the factors of a nonsymmetric matrix
        column, diagonal = (torch.from_numpy(x).to(dev) for x in _panel_columns(ctx))
        ut, d = factors[1]
        ut = ut * d[column]
        ut[diagonal] = d
        state |= {"L": factors[0][0], "Ut": ut, "Zl": torch.empty_like(ut), "Zu": torch.empty_like(ut)}
    elif case["call"] == "host":
        state["host"] = [x.cpu().pin_memory() for x in factors[0]]
        state["out"] = torch.empty(ctx.nnz, dtype=torch.float64).pin_memory()
    elif case["call"] == "batched":
        state["plans"] = [ctxs[id(p)].plan for p, _, _ in every]
        state["dtypes"] = [DTYPES[t] for _, _, t in every]
        state["ctxs"] = list(ctxs.values())
        state["L"], state["D"] = [f[0] for f in factors], [f[1] for f in factors]
        state["Z"] = [torch.empty_like(x) for x in state["L"]]
    else:
        state["L"], state["D"] = factors[0]
        state["Z"] = torch.empty_like(factors[0][0])
        if case["call"] == "subset":
            cols = _picked(case, ctx.n)
            ctx.select(cols, cols)
            state["out"] = torch.empty(cols.size, dtype=torch.float64, device=dev)
    return state


def run(state):
    call, ctx = state["call"], state.get("ctx")
    if call == "block":
        N.selinv_dinv_noalloc(state["s"], state["L"], state["s"], state["D"], state["out"], state["s"])
        return state["out"]
    if call == "selinv":
        return ctx.selinv(state["L"], state["D"], out=state["Z"])
    if call == "factor":
        return ctx.factor(state["A"][0], state["L"], state["D"])
    if call == "train":
        values = state["A"][0].detach().requires_grad_(True)
        Z = SelInv.apply(ctx, values)
        (grad,) = torch.autograd.grad(Z, values, state["W"])
        return Z.detach(), grad
    if call == "poles":
        for a, z in zip(state["A"], state["Z"]):
            ctx.factor(a, state["L"], state["D"])
            ctx.selinv(state["L"], state["D"], out=z)
        return {"sum": pole_sum(state["Z"], state["weights"], state["pos"]), "Z": state["Z"]}
    if call == "batched":
        N.selinv_numeric_batched(state["plans"], state["dtypes"], state["L"], state["D"], state["Z"])
        return state["Z"]
    if call == "lu":
        N.selinv_numeric_lu(ctx.plan, N.SELINV_F64, state["L"], state["Ut"], state["Zl"], state["Zu"])
        return state["Zl"], state["Zu"]
    if call == "host":
        return ctx.selinv_host(state["host"][0], state["host"][1], out=state["out"])
    ctx.selinv(state["L"], state["D"], out=state["Z"])      # subset
    return ctx.gather(state["Z"], out=state["out"])


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _counts(matrix, sites, basis):
    """s and c of every supernode, and its parent."""
    p = _pattern(matrix, sites, basis)
    kind, cap, fill = p.rule
    a = N.selinv_analyse(p.n, p.colptr, p.rowind, {"fundamental": 0, "relaxed": 1}[kind], cap, fill)
    s = np.diff(a["super_ptr"]).astype(np.float64)
    return s, np.diff(a["rowptr"]) - s, a["sparent"], a["super_ptr"]


def work(case):
    if case["call"] == "block":
        s = case["s"]
        return {"bytes": 8.0 * (s * (s + 1) / 2 + s + s * s), "flops": 2.0 * s ** 3 / 3}
    call, real = case["call"], case["dtype"] == "f64"
    w, x = (8.0, 1.0) if real else (16.0, 4.0)
    p = _pattern_of(case)
    s, c, parent, start = _counts(case["matrix"], case["sites"], case.get("basis", 1))
    if call == "subset":        # the picked columns' supernodes and their ancestors
        need = np.zeros(s.size, dtype=bool)
        need[: np.searchsorted(start, _picked(case, p.n)[-1], side="right")] = True
        for k in range(s.size):
            if need[k] and parent[k] >= 0:
                need[parent[k]] = True
        s, c = s[need], c[need]
    panels = float((s * (s + c)).sum())
    invert = float((2 * c * c * s + 2 * c * s * s + c * s * s + s ** 3).sum())
    factor = float((c * c * s + c * s * s + s ** 3 / 3).sum())
    inverting = {"bytes": w * (2 * panels + p.n), "flops": x * invert}
    factoring = {"bytes": w * (p.rowind.size + panels + p.n), "flops": x * factor}
    if call == "factor":
        return factoring
    if call == "lu":            # both factors in, both halves of the inverse out
        return {"bytes": 2 * inverting["bytes"], "flops": 2 * inverting["flops"]}
    if call == "subset":
        return {"bytes": w * (panels + p.n + _picked(case, p.n).size), "flops": invert}
    if call == "train":         # forward, then each product once for either of its factors
        return {"bytes": w * (2 * p.rowind.size + 2 * panels), "flops": 3 * (factor + invert)}
    if call == "poles":         # values in, inverses and their sum out
        return {"bytes": case["poles"] * w * (p.rowind.size + panels) + w * p.n,
                "flops": case["poles"] * x * (factor + invert)}
    if call == "batched":
        total = {k: case["poles"] * v for k, v in inverting.items()}
        for side, d in ((case["extra_2d"], 2), (case["extra_3d"], 3)):
            more = work({"call": "selinv", "matrix": "laplacian", "sites": "x".join([str(side)] * d), "dtype": "f64"})
            total = {k: total[k] + more[k] for k in total}
        return total
    return inverting


# ---------------------------------------------------------------------------
# the outputs in 64 bits, from dense linear algebra
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=8)
def _panel_index(matrix, sites, basis):
    """(row, column) of every panel element: column structures by merging the
    children's, supernodes by the workload's rule."""
    p = _pattern(matrix, sites, basis)
    kind, cap, fill = p.rule
    n, below = p.n, []
    children = [[] for _ in range(n)]
    for j in range(n):
        parts = [p.rowind[p.colptr[j] + 1: p.colptr[j + 1]]] + [below[k] for k in children[j]]
        rows = np.unique(np.concatenate(parts)) if len(parts) > 1 else parts[0]
        below.append(rows[rows > j])
        if below[j].size:
            children[below[j][0]].append(j)
    size = np.array([b.size + 1 for b in below])
    groups = []                                  # fundamental supernodes: [first, end)
    for j in range(n):
        joins = (groups and j > 0 and below[j - 1].size and below[j - 1][0] == j and len(children[j]) == 1
                 and size[j] == size[j - 1] - 1 and j - groups[-1][0] < cap)
        if joins:
            groups[-1][1] = j + 1
        else:
            groups.append([j, j + 1])
    if kind == "relaxed":
        merged = [groups[0]]
        for g in groups[1:]:
            h = merged[-1]
            top = below[h[1] - 1]
            s, c = g[1] - h[0], size[g[0]] - (g[1] - g[0])
            stored = s * (s + 1) // 2 + s * c
            zeros = stored - size[h[0]: g[1]].sum()
            if top.size and g[0] <= top[0] < g[1] and s <= cap and zeros <= fill * stored:
                merged[-1] = [h[0], g[1]]
            else:
                merged.append(g)
        groups = merged
    row, col = [], []
    for a, b in groups:
        rows = np.concatenate([np.arange(a, b), below[b - 1]])
        row.append(np.tile(rows, b - a))
        col.append(np.repeat(np.arange(a, b), rows.size))
    return tuple(torch.from_numpy(np.concatenate(x).astype(np.int64)).cuda() for x in (row, col))


def _dense(p, v, hermitian=False):
    a = torch.zeros(p.n, p.n, dtype=torch.float64 if v.dtype == np.float64 else torch.complex128, device="cuda")
    r, c = torch.from_numpy(p.rowind.astype(np.int64)).cuda(), torch.from_numpy(p.cols.astype(np.int64)).cuda()
    x = torch.from_numpy(v).cuda()
    a[c, r] = x.conj() if hermitian else x
    a[r, c] = x
    return a


def _inverse(a):
    """A dense inverse; positive definite real matrices by their Cholesky factor."""
    if a.is_complex():
        return torch.linalg.inv(a)
    return torch.cholesky_inverse(torch.linalg.cholesky(a))


def _unit_factor(a):
    c = torch.linalg.cholesky(a)
    d = c.diagonal().clone()
    c /= d.conj()[None, :]
    return c, (d * d)


def exact(case, seed):
    if case["call"] == "block":
        return _inverse(_block(case, seed).cuda())
    p = _pattern_of(case)
    cost = p.n * (1.0 if case["dtype"] == "f64" else 4.0 ** (1 / 3)) * case.get("poles", 1) ** (1 / 3)
    if cost > EXACT_N:
        return None
    every = _matrices(case, seed)
    row, col = _panel_index(case["matrix"], case["sites"], case.get("basis", 1))
    v = every[0][1]
    if case["call"] == "factor":
        if case["dtype"] == "c128":      # no dense unpivoted complex symmetric factorization to compare with
            return None
        L, D = _unit_factor(_dense(p, v, hermitian=case["dtype"] == "c128h"))
        return torch.where(row >= col, L[row, col], torch.zeros((), dtype=L.dtype, device=L.device)), D
    if case["call"] == "lu":
        L, _ = _unit_factor(_dense(p, v))
        U, d = _unit_factor(_dense(p, every[1][1]))
        half = torch.linalg.solve_triangular(L, torch.eye(p.n, dtype=L.dtype, device=L.device), upper=False, unitriangular=True)
        half /= d[:, None]
        del L
        Z = torch.linalg.solve_triangular(U.T, half, upper=True, unitriangular=True)
        return Z[row, col], Z[col, row]
    if case["call"] == "train":
        Z = _inverse(_dense(p, v))
        W = torch.from_numpy(np.random.default_rng([seed, 1]).standard_normal(row.numel())).cuda()
        ZW = torch.sparse.mm(torch.sparse_coo_tensor(torch.stack([col, row]), W, (p.n, p.n)).coalesce(), Z).T  # Z W, Z symmetric
        r, c = (torch.from_numpy(x.astype(np.int64)).cuda() for x in (p.rowind, p.cols))
        M = lambda i, j: torch.cat([(ZW[a] * Z[b]).sum(1) for a, b in zip(i.split(4096), j.split(4096))])   # noqa: E731
        return Z[row, col], -torch.where(r == c, M(r, c), M(r, c) + M(c, r))
    if case["call"] == "subset":
        return _inverse(_dense(p, v)).diagonal()[torch.from_numpy(_picked(case, p.n)).cuda()]
    if case["call"] in ("poles", "batched"):
        Zs, total = [], 0.0
        weights = _weights(case["poles"], seed)
        for k, (q, u, _) in enumerate(every):
            if q.n > EXACT_N:
                Zs.append(None)
                continue
            at = (row, col) if k < case["poles"] else _panel_index("laplacian", "x".join(str(x) for x in q.sites), 1)
            Z = _inverse(_dense(q, u))
            Zs.append(Z[at])
            if case["call"] == "poles":
                total = total + complex(weights[k]) * Z.diagonal()
        return {"sum": total, "Z": Zs} if case["call"] == "poles" else Zs
    Z = _inverse(_dense(p, v, hermitian=case["dtype"] == "c128h"))
    return Z[row, col]
