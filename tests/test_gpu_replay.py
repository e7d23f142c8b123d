"""Calls that are repeated: issued, captured and replayed level loops give the
oracle's values in every pass, on the default stream and on others, inside a
graph of the caller, and across changes of type, options and buffers.

Tolerances: diagonally dominant matrices of at most 800 unknowns; an entry
passes through at most 5 products of at most 300 terms, 5 * 300 * 2^-53 = 2e-13
of the largest (normwise); 1e-11 leaves room for the oracle's own errors and
the growth by D^{-1}, 1e-12 where there is one such product."""
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


class Training:
    """Factorization, inversion and both adjoints of one FP64 pattern."""

    def __init__(self, p):
        from paper_1604_02528_gb300.api import SelInvContext
        self.p, self.sym, self.ctx = p, oracle.symbolic_for(p), SelInvContext.from_problem(p)
        self.ctx.attach_matrix()
        self.strict = (lambda rc: rc[0] > rc[1])(oracle.panel_entries(self.sym))
        self.low, self.at = oracle.lower_mask(self.sym), _positions(self.sym, p)

    def values(self, seed):
        """The matrix with another (larger) diagonal, and weights of a loss."""
        rng = np.random.default_rng(seed)
        v = self.p.values.copy()
        v[self.p.diag_positions()] *= 1.0 + rng.random(self.p.n)
        return v, np.where(self.low, rng.standard_normal(self.low.size), 0.0)

    def want(self, v, W):
        q = self.p.with_values(v)
        L, D = oracle.ldlt(q, self.sym)
        Z = oracle.selinv(self.sym, L, D)
        Lb, Db = oracle.selinv_adjoint(self.sym, L, D, Z, W)
        return L, D, Z, Lb, Db, oracle.ldlt_adjoint(self.sym, L, D, Lb, Db)[self.at]

    def buffers(self):
        import torch
        nan = lambda n: torch.full((n,), float("nan"), dtype=torch.float64, device="cuda")   # noqa: E731
        nnz, n, m = self.ctx.nnz, self.p.n, self.p.values.size
        return {"A": nan(m), "W": nan(nnz), "L": nan(nnz), "D": nan(n), "Z": nan(nnz), "Lb": nan(nnz), "Db": nan(n), "Ab": nan(m)}

    def parts(self, native, b, stream=None):
        """The calls of a step: factorization, inversion, adjoints."""
        f64, plan = native.SELINV_F64, self.ctx.plan

        def adjoints():
            native.selinv_adjoint(plan, f64, b["L"], b["D"], b["Z"], b["W"], b["Lb"], b["Db"], stream)
            native.selinv_factor_adjoint(plan, f64, b["L"], b["D"], b["Lb"], b["Db"], b["Ab"], stream)
        return [lambda: self.ctx.factor(b["A"], b["L"], b["D"], stream),
                lambda: self.ctx.selinv(b["L"], b["D"], b["Z"], stream), adjoints]

    def step(self, native, b, stream=None):
        for call in self.parts(native, b, stream):
            call()

    def check(self, b, want):
        import torch
        torch.cuda.synchronize()
        assert self.ctx.status() == 0
        L, D, Z, Lb, Db, Ab = want
        for name, w, mask in (("L", L, self.strict), ("D", D, None), ("Z", Z, self.low), ("Lb", Lb, self.strict), ("Db", Db, None),
                              ("Ab", Ab, None)):
            g = b[name].cpu().numpy()
            if mask is not None:
                g, w = np.where(mask, g, 0), np.where(mask, w, 0)
            assert np.abs(g - w).max() <= 1e-11 * np.abs(w).max(), name


MAKE = {"mesh": lambda: synth.laplacian_3d(9, 4), "dense": lambda: synth.random_sparse_spd(260, 1.0, 5, supernodes={
    "kind": "fundamental", "cap": 64, "fill": 0.0}), "chain": lambda: synth.tridiagonal(300, nd=True)}


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("make", list(MAKE))
def test_graph_of_the_caller(native, cuda_device, make, use_graph):
    """A step captured into the caller's graphs (with use_graph 1 all but the
    inversion, which is then a graph launch itself), replayed with other values
    after calls with other buffers."""
    import torch
    t = Training(MAKE[make]())
    t.ctx.set_options(use_graph=use_graph)
    b, other = t.buffers(), t.buffers()
    v, W = t.values(0)
    b["A"].copy_(torch.from_numpy(v))
    b["W"].copy_(torch.from_numpy(W))
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        for _ in range(2):                      # workspaces, lists and graphs exist before the capture
            t.step(native, b)
    side.synchronize()
    replay = []
    for k, call in enumerate(t.parts(native, b)):
        if k == 1 and use_graph:
            replay.append(call)
            continue
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side, capture_error_mode="thread_local"):
            call()
        replay.append(graph.replay)
    for seed in (1, 2, 3):
        v, W = t.values(seed)
        other["A"].copy_(torch.from_numpy(v))
        other["W"].copy_(torch.from_numpy(W))
        t.step(native, other)                   # the plan's descriptors now name these buffers
        t.check(other, t.want(v, W))
        v, W = t.values(10 + seed)
        b["A"].copy_(torch.from_numpy(v))
        b["W"].copy_(torch.from_numpy(W))
        for name in ("Z", "Lb", "Db", "Ab"):
            b[name].fill_(float("nan"))
        torch.cuda.synchronize()
        for call in replay:
            call()
        t.check(b, t.want(v, W))


@pytest.mark.parametrize("stream", [False, True])
@pytest.mark.parametrize("make", list(MAKE))
def test_training_step(native, cuda_device, make, stream):
    """Issued, captured, replayed, and then on buffers of its own in every pass."""
    import torch
    t = Training(MAKE[make]())
    st = torch.cuda.Stream() if stream else None
    kept = t.buffers()
    for k in range(5):
        b = kept if k < 3 else t.buffers()
        v, W = t.values(k)
        for name in b:
            b[name].fill_(float("nan"))
        b["A"].copy_(torch.from_numpy(v))
        b["W"].copy_(torch.from_numpy(W))
        torch.cuda.synchronize()
        t.step(native, b, st)
        t.check(b, t.want(v, W))


def _dense(n, cap, kind, seed):
    """One dense diagonally dominant matrix in supernodes of `cap` columns."""
    rng = np.random.default_rng(seed)
    g = rng.standard_normal((n, n)) + (1j * rng.standard_normal((n, n)) if kind != "f64" else 0)
    a = (g + (g.conj().T if kind == "c128h" else g.T)) / 2
    np.fill_diagonal(a, np.abs(a).sum(axis=1) + 1.0)
    colptr = np.concatenate([[0], np.cumsum(np.arange(n, 0, -1))]).astype(np.int64)
    rowind = np.concatenate([np.arange(j, n) for j in range(n)]).astype(np.int32)
    return synth.Problem("dense", n, colptr, rowind, np.concatenate([a[j:, j] for j in range(n)]), np.arange(n),
                         {"kind": "fundamental", "cap": cap, "fill": 0.0}, {"hermitian": kind == "c128h"})


class Pattern:
    """One plan for matrices of any type and values on a dense pattern."""

    def __init__(self, native, n, cap):
        from paper_1604_02528_gb300.api import SelInvContext
        self.native, self.n, self.cap = native, n, cap
        p = _dense(n, cap, "f64", 0)
        self.sym, self.ctx = oracle.symbolic_for(p), SelInvContext.from_problem(p)
        self.ctx.attach_matrix()
        r, c, _ = oracle.panel_entries(self.sym)
        self.lower, self.diag = r > c, r == c

    def check(self, kind, seed, stream=None, keep=None):
        """Factorization and inversion of one matrix, on fresh buffers or on `keep`."""
        import torch
        N = self.native
        p = _dense(self.n, self.cap, kind, seed)
        L0, D0 = oracle.ldlt(p, self.sym)
        Z0 = oracle.selinv(self.sym, L0, D0, hermitian=p.hermitian)
        new = lambda m: torch.full((m,), float("nan"), dtype=torch.from_numpy(L0).dtype, device="cuda")   # noqa: E731
        L, D, Z = keep if keep else (new(self.ctx.nnz), new(self.n), new(self.ctx.nnz))
        for x in (L, D, Z):
            x.fill_(float("nan"))
        A, dt = torch.from_numpy(p.values).cuda(), {"f64": N.SELINV_F64, "c128": N.SELINV_C128, "c128h": N.SELINV_C128H}[kind]
        torch.cuda.synchronize()
        N.selinv_factor(self.ctx.plan, dt, A, L, D, stream)
        N.selinv_numeric(self.ctx.plan, dt, L, D, Z, stream)
        torch.cuda.synchronize()
        assert self.ctx.status() == 0
        Lg = L.cpu().numpy()
        assert np.abs(D.cpu().numpy() - D0).max() <= 1e-12 * np.abs(D0).max()
        assert np.abs(np.where(self.lower, Lg - L0, 0)).max() <= 1e-12
        assert np.all(Lg[self.diag] == 1) and np.all(Lg[~self.lower & ~self.diag] == 0)
        assert oracle.block_errors(self.sym, Z.cpu().numpy(), Z0).max() <= 1e-11
        return L, D, Z


# narrow and wide kernels, one and several blocks of 32 columns, the shortest C
# of the tensor-core update and several tiles of it
@pytest.mark.parametrize("stream", [False, True])
@pytest.mark.parametrize("kind", ["f64", "c128", "c128h"])
@pytest.mark.parametrize("cap,n", [(9, 30), (16, 60), (17, 113), (33, 180), (65, 150), (128, 290)])
def test_factor_and_inverse(native, cuda_device, cap, n, kind, stream):
    import torch
    t, st, keep = Pattern(native, n, cap), torch.cuda.Stream() if stream else None, None
    for k in range(4):
        keep = t.check(kind, 10 * n + k, st, keep if k < 3 else None)


def test_types_alternate_on_one_plan(native, cuda_device):
    """Real, complex symmetric and Hermitian values, each issued, captured and
    replayed between the others; the workspace is widened on the way."""
    t = Pattern(native, 200, 40)
    for k, kind in enumerate(["f64"] * 3 + ["c128"] * 3 + ["c128h"] * 2 + ["c128", "f64", "c128h", "f64", "c128"]):
        t.check(kind, k)


@pytest.mark.parametrize("stream", [False, True])
def test_options_change_between_replays(native, cuda_device, stream):
    import torch
    t, st = Pattern(native, 290, 64), torch.cuda.Stream() if stream else None
    bits = {}
    for k, (fast, ozm, graph) in enumerate([(1, 16, 1), (0, 16, 1), (1, 16, 1), (1, 65, 1), (1, 16, 0), (2, 16, 1), (1, 16, 1)]):
        t.ctx.set_options(fast_contraction=fast, oz_min_s=ozm, use_graph=graph)
        keep = None
        for _ in range(3):
            keep = t.check("f64", 5, st, keep)
            L = keep[0].cpu().numpy()
            engine = "tensor" if fast == 1 and ozm <= 64 else "fma"
            assert np.array_equal(bits.setdefault(engine, L), L)      # the engine decides, and nothing else
    assert not np.array_equal(bits["tensor"], bits["fma"])


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("cap,n", [(8, 50), (16, 110), (33, 120), (64, 200), (128, 300)])
def test_lu_form(native, cuda_device, cap, n, cplx):
    import torch
    p = synth.random_sparse_nonsym(n, 1.0, n, complex_values=cplx, supernodes={"kind": "fundamental", "cap": cap, "fill": 0.0})
    sym = oracle.symbolic_for(p)
    L, Ut = oracle.lu(p, sym)
    Zl0, Zu0 = oracle.selinv_lu(sym, L, Ut)
    low = oracle.lower_mask(sym)
    plan = native.selinv_symbolic(sym.n, sym.nsuper, sym.super_ptr, sym.sparent, sym.rowptr, sym.rows)
    Lt, Ut_t = torch.from_numpy(L).cuda(), torch.from_numpy(Ut).cuda()
    Zl, Zu = torch.empty_like(Lt), torch.empty_like(Lt)
    for _ in range(3):
        Zl.fill_(float("nan"))
        Zu.fill_(float("nan"))
        native.selinv_numeric_lu(plan, native.SELINV_C128 if cplx else native.SELINV_F64, Lt, Ut_t, Zl, Zu)
        torch.cuda.synchronize()
        assert native.selinv_status(plan) == 0
        assert oracle.block_errors(sym, Zl.cpu().numpy(), Zl0).max() <= 1e-12
        assert oracle.block_errors(sym, np.where(low, Zu.cpu().numpy(), 0), np.where(low, Zu0, 0)).max() <= 1e-12
