"""Host code of the library over a CUDA runtime without a GPU (tests/fake/cudart.cpp): the order of allocations,
streams, events and graph launches, and what a failing allocation leaves behind.

The library's own objects are linked with that runtime in place of NVIDIA's.  Kernels do nothing there, so nothing is
said about values; each test reads the log of the calls that the library made.
"""
import contextlib
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2412_01138_gb300 import inputs as I

HERE = os.path.dirname(os.path.abspath(__file__))


class Runtime:
    def __init__(self, path):
        from paper_2412_01138_gb300 import pe

        self.lib = pe.load_library(path)
        self.lib.fake_line.restype = C.c_char_p
        self.lib.fake_malloc.restype = C.c_void_p
        self.lib.fake_malloc.argtypes = [C.c_size_t]

    def clear(self):
        self.lib.fake_clear()

    def log(self):
        return [self.lib.fake_line(i).decode().split() for i in range(self.lib.fake_count())]

    @contextlib.contextmanager
    def allocation_fails(self, after):
        self.lib.fake_fail_in(after)
        try:
            yield
        finally:
            self.lib.fake_fail_in(-1)


@pytest.fixture(scope="module")
def linked(tmp_path_factory):
    from paper_2412_01138_gb300 import build

    build.build()
    out = tmp_path_factory.mktemp("fake")
    obj, lib = str(out / "cudart.o"), str(out / "libpe.so")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-I", include, "-c",
                    os.path.join(HERE, "fake", "cudart.cpp"), "-o", obj], check=True)
    objs = [os.path.join(build.OUT, f[:-3] + ".o") for f in sorted(os.listdir(build.CSRC)) if f.endswith(".cu")]
    # -Bsymbolic: a runtime that another package has loaded into the process does not take the calls
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", lib] + objs + [obj], check=True)
    return Runtime(lib)


@pytest.fixture
def rt(linked, monkeypatch):
    from paper_2412_01138_gb300 import pe

    monkeypatch.setattr(pe, "_lib", linked.lib)
    linked.clear()
    linked.lib.fake_set_device(0)
    return linked


def _prob(columns, n=(40, 33), N=4, M=16):
    """`columns` exponential terms: as many source columns."""
    box = ((0.0, 1.0),) * len(n)
    u0, _, _ = I.sin_mode(len(n), box, 0.05)
    facs = tuple(I.Factor(I.S_SIN, (3.0, 0.1)) for _ in n)
    f = tuple(I.Term(1.0, facs, I.T_EXP, (-0.1 * i, 0.0)) for i in range(columns))
    return I.Problem(len(n), n, box, 0.05, 0.0, 1.0, N, M, I.uniform_nodes(3), I.uniform_nodes(2), u0, f, 3, 1e-6)


def _with(s, prob):
    s.prob, s._f_struct = prob, None  # (the binding marshals its terms once)


def _solve(s, **kw):
    from paper_2412_01138_gb300 import pe

    try:
        s.solve(**kw)
    except pe.PEError as e:  # no kernel ran, so no residual was written
        assert e.status == pe.PE_ENOCONV


def _stale_launches(log):
    """Launches of graphs that were made before some device memory was freed."""
    made, last_free = {}, -1
    out = []
    for i, l in enumerate(log):
        if l[0] == "exec_new":
            made[l[1]] = i
        elif l[0] == "free":
            last_free = i
        elif l[0] == "exec_launch" and made[l[2]] < last_free:
            out.append(i)
    return out


@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
@pytest.mark.parametrize("between", ["set_problem", "solve", "out_of_memory"])
def test_loop_graph_does_not_outlive_the_weights_it_reads(rt, precision, between):
    """Few columns, a problem with more (whose weight tables are allocated anew), the first one again."""
    from paper_2412_01138_gb300 import pe

    few, more = _prob(5), _prob(9)
    with pe.Solver(few, precision=precision, device_loop=1) as s:
        _solve(s)
        _with(s, more)
        if between == "set_problem":
            s.set_problem()
        elif between == "solve":
            _solve(s)
        else:
            with rt.allocation_fails(1):  # the second of the two tables
                with pytest.raises(pe.PEError) as ei:
                    s.solve()
            assert ei.value.status == pe.PE_ENOMEM
        _with(s, few)
        _solve(s)
        log = rt.log()
    assert sum(l[0] == "exec_launch" for l in log) >= 2 and any(l[0] == "free" for l in log)
    assert not _stale_launches(log)


@pytest.mark.parametrize("columns", [3, 9, 14], ids=["fewer", "as_many", "more"])
def test_replayed_set_up_is_dropped_by_a_solve_from_host_memory(rt, columns):
    """device_loop = 2: the replayed set-up relies on the host state (terms, columns, weight tables) of its own problem;
    a solve in between with u0 in host memory, which runs its set-up directly, replaces that state."""
    from paper_2412_01138_gb300 import pe

    first, other = _prob(9), _prob(columns)
    host = np.zeros(first.ndof)

    def dev(s):  # u0 in (what this runtime takes for) device memory
        f = pe.pe_field(pe.PE_FIELD_NODAL, 0, None, u0)
        st = rt.lib.pe_solve(s.ctx, C.byref(f), C.byref(s._forcing()), 1e-6, None)
        assert st == pe.PE_ENOCONV

    u0 = rt.lib.fake_malloc(8 * first.ndof)
    with pe.Solver(first, device_loop=2) as s:
        dev(s)
        dev(s)  # captures the set-up and output phases
        held = {l[1] for l in rt.log() if l[0] == "exec_new"}
        assert len(held) == 3
        _with(s, other)
        rt.clear()
        _solve(s, u0_kind=pe.PE_FIELD_NODAL, nodal=host)
        dropped = {l[1] for l in rt.log() if l[0] == "exec_del"}
        _with(s, first)
        rt.clear()
        dev(s)
        launched = {l[2] for l in rt.log() if l[0] == "exec_launch"}
    assert len(dropped & held) >= 2 and not launched & dropped
    # the first problem's set-up ran directly again
    assert any(l[0] == "launch" and "time_tables" in l[2] for l in rt.log())


@pytest.mark.parametrize("precision,n", [(0, (208, 208)), (1, (160, 160))], ids=["fp64", "mixed"])
@pytest.mark.parametrize("D,T,rates", [(0.1, 4.0, (-0.5,)), (0.1, 4.0, (-1.0, 2.0, 0.0)), (1.0, 4.0, (5.0,)),
                                       (1.0, 4.0, (-0.5, -20.0)), (1.0, 4.0, (-40.0,)), (1e-4, 4.0, (-1e4,))])
def test_weights_are_tabulated_only_within_the_tables_reach(rt, precision, n, D, T, rates):
    """The table where every term persists, grows or decays little over a slice (here of length 1), the direct evaluation where
    the table's error, relative to the weight of some mode, could pass the form's rounding."""
    from paper_2412_01138_gb300 import pe

    prob = _prob(1, n=n, N=int(T))
    f = tuple(I.Term(1.0, prob.forcing[0].factors, I.T_EXP, (r, 0.0)) for r in rates)
    f += (I.Term(1.0, prob.forcing[0].factors, I.T_SIN, (30.0, 0.0)),)
    prob = I.Problem(2, n, prob.box, D, 0.0, T, prob.N, prob.M, prob.fine_nodes, prob.coarse_nodes, prob.u0, f, 3, 1e-6)
    with pe.Solver(prob, precision=precision) as s:
        rt.clear()
        s.set_problem()
        names = " ".join(l[2] for l in rt.log() if l[0] == "launch")
    decays = max(-min(rates), 0.0)  # over a slice
    limit = 1.84 if precision else 0.55
    assert ("response_weights" in names) == (decays < limit) and ("column_weights" in names) == (decays > limit)


def _batch_probs(count=3):
    return [_prob(3 + i, n=(17 + i, 9), N=3) for i in range(count)]


def _recorded(log, upto, event):
    return max(i for i in range(upto) if log[i][0] == "record" and log[i][2] == event)


@pytest.mark.parametrize("stream", [None, 1000007], ids=["default", "callers"])
def test_batch_times_run_forward(rt, stream):
    """Both ends of every reported time were recorded in order (the event of one was once recorded again to order the
    caller's stream)."""
    from paper_2412_01138_gb300 import pe

    with pe.BatchSolver(_batch_probs(), stream=stream) as b:
        rt.clear()
        b.solve(tol=1e-6)
        log = rt.log()
    pairs = [(i, l) for i, l in enumerate(log) if l[0] == "elapsed"]
    assert len(pairs) == 2
    for i, l in pairs:
        assert _recorded(log, i, l[1]) < _recorded(log, i, l[2])


@pytest.mark.parametrize("stream", [None, 1000007], ids=["default", "callers"])
@pytest.mark.parametrize("call", ["solve", "solution", "modal"])
def test_batch_works_after_the_callers_stream(rt, stream, call):
    """Whatever writes a buffer of the caller's runs on the caller's stream (the legacy default stream where none was
    given); the batch's own stream, which waits for nothing by itself, is ordered after it before a solve (which
    reads a network of the caller's)."""
    from paper_2412_01138_gb300 import pe

    with pe.BatchSolver(_batch_probs(), stream=stream) as b:
        b.solve(tol=1e-6)
        rt.clear()
        if call == "solve":
            b.solve(tol=1e-6)
        elif call == "solution":
            b.solution(1)
        else:
            b.modal(1, 0)
        log = rt.log()
    callers = str(stream or 0)
    for i, l in enumerate(log):
        if l[0] not in ("launch", "copy", "exec_launch") or l[1] in (callers, "0"):  # (0: copies that wait themselves)
            continue
        waited = {m[2] for m in log[:i] if m[0] == "wait" and m[1] == l[1]}
        assert any(m[0] == "record" and m[1] == callers and m[2] in waited for m in log[:i]), l
        assert call == "solve"
    if call != "solve":
        assert {l[1] for l in log if l[0] in ("launch", "copy")} == {callers} and ["sync", callers] in log


def test_two_threads_fetch_from_one_batch_one_after_the_other(rt):
    """A fetch transforms through the batch's scratch on the batch's stream and waits: until then no other fetch may
    enqueue anything."""
    import threading

    from paper_2412_01138_gb300 import pe

    probs = [_prob(3, n=(17, 9, 8), N=3) for _ in range(3)]
    with pe.BatchSolver(probs) as b:
        b.solve(tol=1e-6)
        b.solution(0)
        rt.clear()
        b.solution(0)
        one = [l[0] for l in rt.log()]
        rt.clear()
        rt.lib.fake_slow(200)  # microseconds a launch: the calls of two threads meet
        try:
            ts = [threading.Thread(target=lambda: [b.solution(i % 3) for i in range(20)]) for _ in range(4)]
            for t in ts:
                t.start()
            for t in ts:
                t.join()
        finally:
            rt.lib.fake_slow(0)
        log = [l[0] for l in rt.log()]
    assert log == one * 80


def test_autotune_without_room_for_the_results_changes_nothing(rt):
    from paper_2412_01138_gb300 import pe

    with pe.BatchSolver(_batch_probs()) as b:
        b.solve(tol=1e-6)
        rt.clear()
        with rt.allocation_fails(0):
            b.autotune(None)
        assert not any(l[0] in ("launch", "copy", "exec_launch") for l in rt.log())
        rt.clear()
        b.autotune(None)
        log = rt.log()
    # kept aside, timed, put back
    copies = [i for i, l in enumerate(log) if l[0] == "copy"]
    walks = [i for i, l in enumerate(log) if l[0] == "launch" and "b_walk" in l[2]]
    assert len(copies) == 6 and copies[2] < walks[0] and walks[-1] < copies[3]
    assert [l for l in log if l[0] == "malloc"][0][1] == [l for l in log if l[0] == "free"][0][1]


def test_tuning_files_of_another_kernel_are_not_taken(rt, tmp_path):
    """A tuning file from before the walk holds shapes that were timed on the per-substep kernel, keyed by device and
    signature alone: they are left in place and the walk is timed."""
    from paper_2412_01138_gb300 import pe

    cache = tmp_path / "tune.txt"
    with pe.BatchSolver(_batch_probs()) as b:
        b.autotune(str(cache))
    device, kernel, signature = cache.read_text().split()[0].split("|")
    cache.write_text(f"{device}|{signature} 256 2\n")
    with pe.BatchSolver(_batch_probs()) as b:
        rt.clear()
        b.autotune(str(cache))
        assert any("b_walk" in l[2] for l in rt.log() if l[0] == "launch")
        lines = cache.read_text().splitlines()
        assert len(lines) == 2 and lines[0] == f"{device}|{signature} 256 2"
        rt.clear()
        b.autotune(str(cache))  # the new line is taken
        assert not any(l[0] == "launch" for l in rt.log())


@pytest.mark.parametrize("call", ["set_problem", "solve"])
@pytest.mark.parametrize("fails", [0, 1, "general"])
def test_a_failing_set_up_leaves_nothing_running(rt, call, fails):
    """Grids large enough for set-up on three streams: where an allocation fails beside the transform of the caller's u0
    (a weight table, or the moving terms' stage tables), the call waits for the other streams before it returns."""
    from paper_2412_01138_gb300 import pe

    prob = _prob(5, n=(71, 65))
    kw = {}
    if fails == "general":
        hat = I.Term(1.0, (I.Factor(I.S_MOVING_HAT, (0.5, 0.2, 1.0, 0.1)), prob.forcing[0].factors[1]))
        prob = I.Problem(2, prob.n, prob.box, prob.D, 0.0, 1.0, prob.N, prob.M, prob.fine_nodes, prob.coarse_nodes, prob.u0,
                         prob.forcing + (hat,), 3, 1e-6)
        kw = {"forcing_path": pe.PE_FORCING_GENERAL}
    with pe.Solver(prob, **kw) as s:
        rt.clear()
        with rt.allocation_fails(0 if fails == "general" else fails):
            with pytest.raises(pe.PEError) as ei:
                getattr(s, call)(u0_kind=pe.PE_FIELD_NODAL, nodal=np.zeros(prob.ndof))
        assert ei.value.status == pe.PE_ENOMEM
        log = rt.log()
    main = "0"
    used = {l[1] for l in log if l[0] in ("launch", "copy")} - {main}
    assert len(used) == 2
    for stream in used:
        last = max(i for i, l in enumerate(log) if l[0] in ("launch", "copy") and l[1] == stream)
        assert ["sync", stream] in log[last:]


def test_shared_memory_limits_are_raised_on_every_device(rt):
    """Function attributes belong to a device: kernels that take more than 48 KB have them raised on each one, and never
    lowered where a call with less follows."""
    from paper_2412_01138_gb300 import pe

    def transforms():
        for f32, n in ((0, (7000,)), (1, (13000,)), (0, (255, 255, 9)), (0, (1023, 700)), (1, (255, 255, 3)), (1, (511, 511)),
                       (1, (511, 63, 500)), (1, (1023, 1023)), (0, (127, 127, 127)), (0, (511, 1023)), (0, (7000,))):
            size = int(np.prod(n)) * (4 if f32 else 8)
            a, b = rt.lib.fake_malloc(size), rt.lib.fake_malloc(size)
            fn = rt.lib.pe_dst_f32 if f32 else rt.lib.pe_dst
            assert fn(len(n), (C.c_int32 * len(n))(*n), a, b, None) == pe.PE_OK
        net = pe.MLP()
        x = np.zeros((64, 2), dtype=np.float32)
        net.train(x, x, epochs=1, batch=32)
        net.close()

    for device in (0, 1):
        rt.lib.fake_set_device(device)
        transforms()
    limit, big = {}, set()
    for l in rt.log():
        if l[0] == "attribute":
            limit[l[1], l[2]] = int(l[3])
        elif l[0] == "launch" and int(l[3]) > 48 * 1024:
            big.add((l[4], l[2]))
            assert limit.get((l[4], l[2]), 0) >= int(l[3]), l
    assert len({k for d, k in big}) >= 5 and len(big) == 2 * len({k for d, k in big})


@pytest.mark.parametrize("form,at_setup,by_refine", [("fp64", 2, 0), ("mixed", 0, 1), ("mixed_general", 2, 0),
                                                     ("mixed_cached", 1, 0), ("fp64_cached", 2, 0)])
def test_forced_parts_are_allocated_where_something_fills_them(rt, form, at_setup, by_refine):
    """Arrays of a value per mode and slice beside the iterate: the forced parts of the fine and the coarse step (cached: of
    the fine step, kept) where kernels store them; none in the mixed separable form until a refinement."""
    from paper_2412_01138_gb300 import pe

    prob = _prob(5, n=(37, 29), N=11)
    size = str(8 * prob.N * prob.ndof)
    kw = {"precision": int(form.startswith("mixed")), "cache_forced": form.endswith("cached")}
    if form.endswith("general"):
        kw["forcing_path"] = pe.PE_FORCING_GENERAL

    def count():
        return sum(l[0] == "malloc" and l[2] == size for l in rt.log())

    with pe.Solver(prob, **kw) as s:
        assert count() == at_setup
        s.set_problem()
        s.iterate()
        assert count() == at_setup
        s.refine()
        s.refine()
        assert count() == at_setup + by_refine


def test_loop_graph_is_kept_where_no_weights_were_given_back(rt):
    """The float64 weights of a mixed context's first refinement are one more table: the loop graph stays."""
    from paper_2412_01138_gb300 import pe

    with pe.Solver(_prob(5), precision=1, device_loop=1) as s:
        _solve(s)
        s.set_problem()
        s.refine()
        rt.clear()
        _solve(s)
        log = rt.log()
    assert any(l[0] == "exec_launch" for l in log) and not any(l[0] == "exec_new" for l in log)
