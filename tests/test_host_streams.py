"""What the host side issues, without a GPU: the library runs on a CUDA runtime
that executes nothing and logs launches, their order over streams and the
addresses that they are given (fake_cudart.cpp)."""
import json
import os
import subprocess
import sys

import pytest

import oracle
import synth

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes as ct, json, os, sys
sys.path.insert(0, {root!r})
import numpy as np
import synth
from paper_1604_02528_gb300 import _native as N
LIB, RT = N.LIB, ct.CDLL(None)
def mem(count):
    p = ct.c_void_p()
    assert RT.cudaMalloc(ct.byref(p), ct.c_size_t(16 * count)) == 0
    return p
class Ctx:
    def __init__(self, p, **opts):
        self.p, sn = p, p.supernodes
        a = N.selinv_analyse(p.n, p.colptr, p.rowind, 1 if sn["kind"] == "relaxed" else 0, sn["cap"], sn["fill"])
        o = N.selinv_default_opts()
        for k, v in opts.items():
            setattr(o, k, v)
        self.plan = N.selinv_symbolic(p.n, a["nsuper"], a["super_ptr"], a["sparent"], a["rowptr"], a["rows"], o)
        self.h, self.opts = self.plan.handle, o
        nnz = self.plan.nnz
        self.L, self.D, self.Z, self.Zu, self.Lb, self.Db = (mem(x) for x in (nnz, p.n, nnz, nnz, nnz, p.n))
        self.A = mem(p.colptr[-1])
        N.selinv_plan_set_matrix(self.plan, p.n, p.colptr, p.rowind)
    def set(self, **opts):
        for k, v in opts.items():
            setattr(self.opts, k, v)
        N.selinv_plan_set_opts(self.plan, self.opts)
    def selinv(self, dtype=0, stream=None):
        return LIB.selinv_numeric(self.h, dtype, self.L, self.D, self.Z, stream)
    def lu(self, dtype=0, stream=None):
        return LIB.selinv_numeric_lu(self.h, dtype, self.L, self.Lb, self.Z, self.Zu, stream)
    def factor(self, dtype=0, stream=None):
        return LIB.selinv_factor(self.h, dtype, self.A, self.L, self.D, stream)
    def adjoint(self, stream=None):
        return LIB.selinv_adjoint(self.h, 0, self.L, self.D, self.Z, self.Zu, self.Lb, self.Db, stream)
    def factor_adjoint(self, stream=None):
        return LIB.selinv_factor_adjoint(self.h, 0, self.L, self.D, self.Lb, self.Db, self.A, stream)
def batched(ctxs, dtypes):
    n = len(ctxs)
    arr = lambda xs: (ct.c_void_p * n)(*[x.value for x in xs])
    return LIB.selinv_numeric_batched(n, (ct.c_void_p * n)(*[c.h.value for c in ctxs]), (ct.c_int * n)(*dtypes),
                                      arr([c.L for c in ctxs]), arr([c.D for c in ctxs]), arr([c.Z for c in ctxs]), None)
def mark(name):      # a line of its own in the log
    with open(os.environ["FAKE_CUDART_LOG"], "a") as f:
        f.write("# " + name + "\\n")
"""


@pytest.fixture(scope="module")
def fake(native, tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-w", "-o", so, os.path.join(HERE, "fake_cudart.cpp"),
                    "-I" + os.path.join(cuda, "include"), "-I" + os.path.join(ROOT, "include"),
                    "-I" + os.path.join(ROOT, "paper_1604_02528_gb300", "csrc")], check=True)
    return so


def run(fake, tmp_path, script):
    """The log of a script: [(mark, [line, ...])] in order, and what it printed (JSON)."""
    log = str(tmp_path / "log")
    env = dict(os.environ, LD_PRELOAD=fake, FAKE_CUDART_LOG=log)
    r = subprocess.run([sys.executable, "-c", PRELUDE.format(root=ROOT) + script], env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    parts = [("", [])]
    for line in open(log):
        if line.startswith("# "):
            parts.append((line[2:].strip(), []))
        else:
            parts[-1][1].append(line.split())
    return parts, (json.loads(r.stdout) if r.stdout.strip() else None)


class Launch:
    def __init__(self, f):
        self.stream, self.index, self.stale, self.yacc, self.name = int(f[1]), int(f[2]), int(f[4]), int(f[5]), f[7]
        self.panels = [int(x) for x in f[6].split(",")[1:]]
        self.clock = [int(x) for x in f[3].split(",")]
        self.ks = {int(x) for x in f[8:]}

    def after(self, other):
        return other.stream < len(self.clock) and self.clock[other.stream] >= other.index


def launches(lines):
    return [Launch(f) for f in lines if f[0] == "L"]


def _ordered(sym, got):
    """Launches that touch one supernode come one after the other, and a
    traversal launch of a supernode after everything that touches its parent."""
    by = {}
    for x in got:
        for K in x.ks:
            for y in by.setdefault(K, []):
                assert x.after(y), (K, y.name, x.name)
            by[K].append(x)
    norm = ("k_linv", "k_dinv", "k_lhat", "k_fma_lhat", "digits", "k_selinv_tcw<false,_true", "k_selinv_tcw<true,_true")
    for K, own in by.items():
        J = int(sym.sparent[K])
        for x in own:
            if J >= 0 and not any(n in x.name for n in norm):
                for y in by[J]:
                    assert x.after(y), (K, J, y.name, x.name)
    return set(by)


# every branch, the side stream's phases, and a selection that needs the first
# of them only (the second then has no launch)
@pytest.mark.parametrize("picked", ["all", "top", "middle", "leaf"])
@pytest.mark.parametrize("make,dtype", [("laplacian_3d(12, 4)", 0), ("laplacian_2d(31, 19)", 0), ("magnetic_laplacian_3d(10, 4)", 2),
                                        ("random_sparse_spd(900, 0.002, 2, supernodes=synth.problems.RELAXED_128)", 0)])
def test_launches_of_dependent_supernodes_are_ordered(fake, tmp_path, make, dtype, picked):
    parts, active = run(fake, tmp_path, f"""
c = Ctx(synth.{make}, use_graph=0)
level, lptr, lst = (N.selinv_plan_get(c.plan, x) for x in ("level", "level_ptr", "level_list"))
a = N.selinv_analyse(c.p.n, c.p.colptr, c.p.rowind, 1 if c.p.supernodes["kind"] == "relaxed" else 0, c.p.supernodes["cap"], c.p.supernodes["fill"])
at = {{"top": np.searchsorted(lptr, 16, "right") - 2, "middle": np.searchsorted(lptr, 256, "right") - 2, "leaf": len(lptr) - 2}}.get({picked!r})
if at is not None:
    cols = a["super_ptr"][lst[lptr[at]:lptr[at + 1]]]
    N.selinv_plan_select(c.plan, cols, cols)
mark("run")
assert c.selinv({dtype}) == 0
print(json.dumps(N.selinv_plan_get(c.plan, "active").tolist()))
""")
    sym = oracle.symbolic_for(eval("synth." + make))
    assert _ordered(sym, launches(parts[-1][1])) == {K for K in range(sym.nsuper) if active[K]}


@pytest.mark.parametrize("call", ["c.selinv({0})", "batched([c], [{0}])"])
def test_real_sums_have_room_beside_a_complex_workspace(fake, tmp_path, call):
    """The mma.sync engine adds split contractions of real values into two
    words per panel entry, whatever type the plan's workspace was made for."""
    parts, nnz = run(fake, tmp_path, f"""
c = Ctx(synth.laplacian_3d(12, 4), use_graph=0)
assert {call.format(1)} == 0
c.set(fast_contraction=2)
mark("run")
assert {call.format(0)} == 0
print(c.plan.nnz)
""")
    got = [x.yacc for x in launches(parts[-1][1]) if "k_selinv_oz" in x.name]
    assert got and min(got) >= 16 * nnz


@pytest.mark.parametrize("first,widen", [("c.selinv(0)", "c.lu(1)"), ("c.lu(0)", "c.selinv(1)"), ("c.lu(0)", "c.selinv(2)"),
                                         ("batched([c, c], [0, 0])", "batched([c, c], [1, 0])")])
def test_schedules_follow_their_workspace(fake, tmp_path, first, widen):
    """A workspace made again for a wider type: a schedule kept from before
    must not run on the buffers that were given back."""
    parts, _ = run(fake, tmp_path, f"""
c = Ctx(synth.laplacian_3d(9, 4))
for call in ({first!r}, {first!r}, {widen!r}):
    assert eval(call) == 0
N.selinv_release_cached_memory()
mark("run")
assert eval({first!r}) == 0 and eval({first!r}) == 0
""")
    got = launches(parts[-1][1])
    assert got and not any(x.stale for x in got)


@pytest.mark.parametrize("dtype", [0, 1])
def test_batch_workspaces_fit_their_plans(fake, tmp_path, dtype):
    """An item's place in a batch is taken by a larger problem than before:
    its workspace has to grow (digit planes, panels, the exact sums)."""
    parts, sizes = run(fake, tmp_path, f"""
a, b, c = Ctx(synth.laplacian_3d(7, 4)), Ctx(synth.laplacian_3d(7, 4)), Ctx(synth.laplacian_3d(12, 4))
for x in (a, b, c):
    x.set(fast_contraction=2, use_graph=0)
assert batched([a, b], [{dtype}, {dtype}]) == 0
mark("run")
assert batched([a, c], [{dtype}, {dtype}]) == 0
mark("back")
assert batched([a, b], [{dtype}, {dtype}]) == 0
print([x.plan.nnz for x in (a, b, c)])
""")
    for lines, want in ((parts[-2][1], [sizes[0], sizes[2]]), (parts[-1][1], sizes[:2])):
        got = launches(lines)
        assert got and not any(x.stale for x in got)
        for x in got:
            for have, nnz in zip(x.panels, want):
                assert have >= (16 if dtype else 8) * nnz


def test_batch_of_a_plan_at_a_destroyed_plans_address(fake, tmp_path):
    """A batch is recognized by its plans: a new plan whose handle has the
    address of a destroyed one is another plan."""
    parts, same = run(fake, tmp_path, """
a, b = Ctx(synth.laplacian_3d(7, 4)), Ctx(synth.laplacian_3d(7, 4))
s = N.selinv_analyse(b.p.n, b.p.colptr, b.p.rowind, 1, b.p.supernodes["cap"], b.p.supernodes["fill"])
assert batched([a, b], [0, 0]) == 0
old = b.h.value
LIB.selinv_plan_destroy(b.plan.handle)
b.plan.handle = None
b.plan = N.selinv_symbolic(b.p.n, s["nsuper"], s["super_ptr"], s["sparent"], s["rowptr"], s["rows"], b.opts)
b.h = b.plan.handle
mark("run")
assert batched([a, b], [0, 0]) == 0
print(int(b.h.value == old))
""")
    got = launches(parts[-1][1])
    assert same and got and not any(x.stale for x in got)


def test_options_of_every_plan_reach_a_batch(fake, tmp_path):
    parts, _ = run(fake, tmp_path, """
a, b = Ctx(synth.laplacian_3d(12, 4), fast_contraction=0), Ctx(synth.laplacian_3d(12, 5))
assert batched([a, b], [0, 0]) == 0
b.set(fast_contraction=0)
mark("run")
assert batched([a, b], [0, 0]) == 0
""")
    tensor = [sum("k_selinv_tc" in x.name for x in launches(lines)) for _, lines in parts]
    assert tensor[0] > 0 and tensor[1] == 0


def test_options_reach_the_lu_form(fake, tmp_path):
    """debug_checks bit 2 sits in the descriptors of a kept schedule."""
    parts, _ = run(fake, tmp_path, """
c = Ctx(synth.laplacian_3d(7, 4))
for _ in range(3):
    assert c.lu() == 0
mark("replay")
assert c.lu() == 0
c.set(debug_checks=4)
mark("checked")
assert c.lu() == 0
""")
    assert not launches(parts[1][1])
    assert launches(parts[2][1])


LOOPS = ["c.factor()", "c.adjoint()", "c.factor_adjoint()"]


@pytest.mark.parametrize("call", ["c.selinv()", "c.lu()"] + LOOPS)
@pytest.mark.parametrize("stream", [None, 0x1000000])
def test_use_graph_0_keeps_every_call_off_graphs(fake, tmp_path, call, stream):
    parts, _ = run(fake, tmp_path, f"""
st = {stream}
c = Ctx(synth.laplacian_3d(9, 4))
for graph in (1, 0):
    c.set(use_graph=graph)
    for _ in range(3):
        mark(str(graph))
        assert {call.replace("()", "(stream=st)")} == 0
""")
    kinds = [{f[0] for f in lines} for _, lines in parts[1:]]
    assert "G" in kinds[2]                                   # replayed
    assert all(k == {"L"} for k in kinds[3:])


@pytest.mark.parametrize("call", LOOPS)
def test_a_new_spin_limit_reaches_every_loop(fake, tmp_path, call):
    """The bound of the device waits is an argument of the captured launches:
    a call after it has changed cannot replay them."""
    parts, _ = run(fake, tmp_path, f"""
c = Ctx(synth.laplacian_3d(9, 4))
for limit in (1 << 22, 1 << 23, (1 << 62) + 1):
    c.set(spin_limit=limit)
    for _ in range(3):
        mark(str(limit))
        assert {call} == 0
""")
    assert ["G" in [f[0] for f in lines] for _, lines in parts[1:]] == [False, True, True] * 3


@pytest.mark.parametrize("call", LOOPS)
def test_a_launch_that_fails_under_capture_is_reported(fake, tmp_path, call):
    """A kernel that cannot be launched must not drop out of the graph unnoticed."""
    _, rc = run(fake, tmp_path, f"""
c = Ctx(synth.laplacian_3d(9, 4))
assert {call} == 0
RT.fake_fail(3, 1 << 30)
rc = [{call}, {call}]
RT.fake_fail(3, 0)
print(rc + [{call}, {call}])
""")
    assert rc == [-7, -7, 0, 0]
@pytest.mark.parametrize("what", [1, 2])
@pytest.mark.parametrize("call", ["c.selinv()", "c.lu()", "batched([c], [0])"] + LOOPS)
def test_default_stream_runs_without_a_graph_where_none_can_be_made(fake, tmp_path, call, what):
    """No capture (1) or no instantiation (2): the launches themselves go out,
    once, and are counted."""
    parts, n = run(fake, tmp_path, f"""
c = Ctx(synth.laplacian_3d(9, 4))
count = []
for k in range(4):
    RT.fake_fail({what}, 1 if k == 1 else 0)
    before = LIB.selinv_launch_count()
    mark(str(k))
    assert {call} == 0
    count.append(LIB.selinv_launch_count() - before)
print(count)
""")
    want = [x.name for x in launches(parts[1][1])]
    lines = parts[2][1]                                       # the call that cannot capture
    kinds = [f[0] for f in lines]
    begin, end = kinds.index("B"), kinds.index("I") if what == 2 else kinds.index("B")
    names = lambda part: [x.name for x in launches(part)]     # noqa: E731
    assert names(lines[:begin]) + names(lines[end:]) == want and "G" not in kinds
    assert all("G" in [f[0] for f in p[1]] for p in parts[3:])
    assert len(set(n)) == 1




@pytest.mark.parametrize("stream", [None, 0x1000000])
def test_autotuner_times_replays_only(fake, tmp_path, stream):
    """What a candidate's timed runs contain is what later calls will do: no
    capture and no instantiation between the two events of a run."""
    parts, _ = run(fake, tmp_path, f"""
c = Ctx(synth.laplacian_3d(7, 4), autotune=1)
assert c.selinv(stream={stream}) == 0
""")
    kinds = [f[0] for f in parts[0][1]]
    timed, inside = 0, False
    for k in kinds:
        if k == "T":
            inside, timed = not inside, timed + 1
        assert not (inside and k in "BIL")
    assert timed >= 4 and not inside


def _syrk(lines):
    return set().union(*([set()] + [x.ks for x in launches(lines) if x.name.endswith("k_selinv_tcw<false,_false,_2>")]))


def test_factorization_keeps_the_callers_engine(fake, tmp_path):
    """What the autotuner settles on by timing the inversion must not change
    the arithmetic of the factorization."""
    parts, tuned = run(fake, tmp_path, """
out = []
for engine in (1, 0):
    c = Ctx(synth.laplacian_3d(12, 4), autotune=1, fast_contraction=engine, use_graph=0)
    mark("before")
    assert c.factor() == 0
    mark("tuning")
    RT.fake_slow(1 if engine else 0)
    assert c.selinv() == 0
    out.append(N.selinv_plan_get_opts(c.plan).fast_contraction)
    mark("after")
    assert c.factor() == 0
print(out)
""")
    on, off = (parts[1][1], parts[3][1]), (parts[4][1], parts[6][1])
    assert tuned == [2, 1]
    assert _syrk(on[0]) and _syrk(on[0]) == _syrk(on[1])
    assert not _syrk(off[0]) and not _syrk(off[1])


def test_factorization_follows_oz_min_s(fake, tmp_path):
    """Narrower supernodes than the caller's oz_min_s keep FP64 updates; the
    lists follow a later change, under replay too."""
    parts, _ = run(fake, tmp_path, """
c = Ctx(synth.laplacian_3d(12, 4))
for ozm in (16, 40, 128, 16):
    c.set(oz_min_s=ozm)
    for k in range(3):
        mark(str(ozm))
        assert c.factor() == 0
""")
    sym = oracle.symbolic_for(synth.laplacian_3d(12, 4))
    s = sym.super_ptr[1:] - sym.super_ptr[:-1]
    c = (sym.rowptr[1:] - sym.rowptr[:-1]) - s
    for i, ozm in enumerate((16, 40, 128, 16)):
        want = set((((s >= max(17, ozm)) & (c >= 96)).nonzero()[0]).tolist())
        first, second, third = (p[1] for p in parts[1 + 3 * i:4 + 3 * i])
        assert _syrk(first) == want and _syrk(second) == want            # issued, captured
        assert "G" in [f[0] for f in third] and not any("k_fupd" in x.name for x in launches(third))
        updated = lambda n: sum("k_fupd<" in x.name for x in launches(n))     # noqa: E731
        assert bool(updated(first)) and not any(x.stale for x in launches(first) + launches(second))


@pytest.mark.parametrize("call", LOOPS)
def test_a_captured_call_copies_nothing_from_the_stack(fake, tmp_path, call):
    """A copy node of a caller's graph reads its host source when the graph is
    launched, long after the call's descriptors have gone."""
    parts, _ = run(fake, tmp_path, f"""
c = Ctx(synth.laplacian_3d(9, 4))
st = 0x1000000
assert {call.replace("()", "(stream=st)")} == 0
RT.fake_capturing(ct.c_void_p(st))
mark("captured")
assert {call.replace("()", "(stream=st)")} == 0
""")
    kinds = [f[0] for f in parts[1][1]]
    assert "L" in kinds and "H" not in kinds and "G" not in kinds


@pytest.mark.parametrize("dtype", [0, 1])
@pytest.mark.parametrize("cap,n,ozm,schedule", [(1, 240, 128, 1), (16, 240, 128, 1), (16, 240, 8, 1), (40, 200, 16, 1), (16, 120, 16, 0)])
def test_bench_counts_the_kernels_supernodes(fake, tmp_path, cap, n, ozm, schedule, dtype):
    """bench.py's roofline divides the operations of a kernel's supernodes by its
    time: its classes are those of the launches."""
    import bench
    from paper_1604_02528_gb300 import _native as N
    parts, _ = run(fake, tmp_path, f"""
p = synth.random_sparse_spd({n}, 1.0, 1, supernodes={{"kind": "fundamental", "cap": {cap}, "fill": 0.0}})
c = Ctx(p, oz_min_s={ozm}, schedule={schedule}, use_graph=0)
mark("run")
assert c.selinv({dtype}) == 0
""")
    sym = oracle.symbolic_for(synth.random_sparse_spd(n, 1.0, 1, supernodes={"kind": "fundamental", "cap": cap, "fill": 0.0}))
    opts = N.selinv_default_opts()
    opts.oz_min_s, opts.schedule = ozm, schedule
    s = (sym.super_ptr[1:] - sym.super_ptr[:-1]).astype(float)
    c = (sym.rowptr[1:] - sym.rowptr[:-1]) - s
    oz, narrow = bench.kernel_classes(s, c, dtype != 0, opts)
    got = {"narrow": set(), "oz": set()}
    for x in launches(parts[-1][1]):
        if "k_selinv_narrow" in x.name:
            got["narrow"] |= x.ks
        if "k_selinv_tc" in x.name and "_true" not in x.name.split(",")[1:2]:
            got["oz"] |= x.ks
    assert got["narrow"] == set(narrow.nonzero()[0].tolist())
    assert got["oz"] == set((oz & (c > 0)).nonzero()[0].tolist())


def test_lu_form_follows_the_selection(fake, tmp_path):
    """Its schedule is built for the supernodes of the current selection."""
    parts, active = run(fake, tmp_path, """
c = Ctx(synth.laplacian_3d(9, 4), use_graph=0)
top = np.array([c.p.n - 1], np.int32)
out = []
for cols in (top[:0], top, top[:0]):
    N.selinv_plan_select(c.plan, cols, cols)
    mark("lu")
    assert c.lu() == 0
    out.append(N.selinv_plan_get(c.plan, "active").tolist())
print(json.dumps(out))
""")
    for (_, lines), a in zip(parts[1:], active):
        assert set().union(*(x.ks for x in launches(lines))) == {K for K, on in enumerate(a) if on}


CALLS_THAT_ALLOCATE = ["c.selinv()", "c.lu()", "c.factor()", "batched([c, c], [0, 1])"]


@pytest.mark.parametrize("call", CALLS_THAT_ALLOCATE)
def test_calls_after_a_failed_allocation(fake, tmp_path, call):
    """Whichever allocation of a first call fails, that call says so, and the
    next ones are complete."""
    parts, rc = run(fake, tmp_path, f"""
rc = []
for n in range(1, 41):
    c = None
    N.selinv_release_cached_memory()     # (every buffer of this call is an allocation)
    c = Ctx(synth.laplacian_3d(6, 4), use_graph=0)
    mark("first")
    RT.fake_fail(4, n)
    r = [{call}]
    RT.fake_fail(4, 0)
    for _ in range(2):
        mark("later")
        r.append({call})
    rc.append(r)
print(json.dumps(rc))
""")
    assert all(r[0] in (0, -6) and r[1:] == [0, 0] for r in rc) and [-6, 0, 0] in rc and [0, 0, 0] in rc
    later = [launches(lines) for name, lines in parts if name == "later"]
    assert len({tuple(x.name for x in got) for got in later}) == 1
    assert not any(x.stale for got in later for x in got)


def test_adjoint_lists_after_a_failed_allocation(fake, tmp_path):
    """Lists that could not be rebuilt for a new option are rebuilt by the next
    call, also under the old option: nothing is launched on freed or missing ones."""
    parts, rc = run(fake, tmp_path, """
rc = []
for n in range(1, 41):
    c = Ctx(synth.laplacian_3d(9, 4), use_graph=0)
    r = [c.adjoint()]
    mark("under 16")
    r.append(c.adjoint())
    c.set(oz_min_s=8)
    mark("fails")
    RT.fake_fail(4, n)
    r.append(c.adjoint())
    RT.fake_fail(4, 0)
    c.set(oz_min_s=16)
    mark("under 16")
    r.append(c.adjoint())
    mark("done")
    rc.append(r)
print(json.dumps(rc))
""")
    assert all(r[:2] == [0, 0] and r[2] in (0, -6) and r[3] == 0 for r in rc) and [0, 0, -6, 0] in rc
    same = [launches(lines) for name, lines in parts if name == "under 16"]
    assert len({tuple(x.name for x in got) for got in same}) == 1
    assert not any(x.stale for got in same for x in got)
