"""GPU: one context, several problems one after the other: what a solve leaves behind (graphs, tables, host state) must not
show in the next.  Every solve is compared bit for bit with a fresh context's.
"""
import numpy as np
import pytest

from paper_2412_01138_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pe():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_01138_gb300 import pe as _pe

    _pe.lib()
    return _pe


def _prob(columns, n=(71, 65), N=5, M=16):
    """`columns` source columns: one exponential, sinusoids for the rest."""
    box = ((0.0, 1.0),) * len(n)
    u0, f, _ = I.sin_mode(len(n), box, 0.05)
    rng = I.SplitMix64(columns)
    f = f[:columns % 2] + I.gaussian_bumps(rng, len(n), columns // 2)
    return I.Problem(len(n), n, box, 0.05, 0.0, 1.0, N, M, I.uniform_nodes(3), I.uniform_nodes(2), u0, f, 3, 1e-8)


def _with(s, prob):
    s.prob, s._f_struct = prob, None  # (the binding marshals its terms once)


def _state(s, info):
    return info["k"], info["history"], [s.modal(m) for m in range(s.prob.N + 1)], s.solution(s.prob.N)


def _same(a, b):
    assert a[0] == b[0] and a[1] == b[1]
    for m, (x, y) in enumerate(zip(a[2], b[2])):
        assert np.array_equal(x, y), m
    assert np.array_equal(a[3], b[3])


@pytest.mark.parametrize("loop", [1, 2])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_more_columns_between_two_solves(pe, precision, loop):
    """A problem with more source columns has the weight tables allocated anew: the loop graph of the solve before
    must not be launched again."""
    few, more = _prob(5), _prob(19)
    with pe.Solver(few, precision=precision) as s:
        want = _state(s, s.solve())
    with pe.Solver(few, precision=precision, device_loop=loop) as s:
        for _ in range(3):
            _same(_state(s, s.solve()), want)
        _with(s, more)
        s.set_problem()
        _with(s, few)
        for _ in range(3):
            _same(_state(s, s.solve()), want)


@pytest.mark.parametrize("columns", [3, 19], ids=["fewer", "more"])
@pytest.mark.parametrize("precision", [0, 1], ids=["fp64", "mixed"])
def test_host_u0_between_two_replays(pe, precision, columns):
    """device_loop = 2: a solve with initial data in host memory runs its set-up directly and so changes the host state
    that the replayed set-up of the problem before relies on (columns, terms, tables)."""
    import torch

    first, other = _prob(9), _prob(columns)
    u0 = np.random.default_rng(1).standard_normal(first.ndof)
    dev = torch.from_numpy(u0).cuda()

    def full(s, nodal):
        info = s.solve(u0_kind=pe.PE_FIELD_NODAL, nodal=nodal)
        s.refine()
        return _state(s, info)

    want = {}
    for name, prob, nodal in (("first", first, dev), ("other", other, u0)):
        with pe.Solver(prob, precision=precision) as s:
            want[name] = full(s, nodal)
    with pe.Solver(first, precision=precision, device_loop=2) as s:
        for _ in range(3):
            _same(full(s, dev), want["first"])
        _with(s, other)
        _same(full(s, u0), want["other"])
        _with(s, first)
        for _ in range(3):
            _same(full(s, dev), want["first"])


@pytest.mark.parametrize("n", [(63,), (40, 33), (120, 90)], ids=["line", "small", "large"])
def test_async_result_in_pageable_memory_is_there_on_return(pe, n):
    """pe_solve_async waits for a copy to pageable memory of any size; pe_solve_wait only reports."""
    prob = _prob(5, n=n)
    with pe.Solver(prob) as s:
        s.solve()
        want = s.solution(prob.N)
    with pe.Solver(prob, device_loop=1) as s:
        out = np.full(prob.ndof, np.nan)
        s.solve_async(out=out)
        got = out.copy()
        s.wait()
    assert np.array_equal(got, want) and np.array_equal(out, want)
