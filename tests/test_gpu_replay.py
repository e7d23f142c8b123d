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
