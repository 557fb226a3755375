"""GPU: moving terms of the general path where the per-axis evaluation can go wrong, against the oracle's full
element quadrature of f(t, x).

Cases: one to six stages (the kernel unrolls one to four), terms that move along the first, the last or every axis,
several of them beside fixed ones, none fixed, a periodic axis, more stage times than one chunk of slices
holds (65535), grids without an FFT form.  Bounds: the forms' own, 1e-12 (float64) and 1e-6 (mixed).
"""
import numpy as np
import pytest

from oracle import solver as osolver
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


def _rel(a, b, w):
    return float(np.sqrt(np.sum(w * (a - b) ** 2)) / np.sqrt(np.sum(w * b * b)))


def _hat(c0, amp, f, w=0.13):
    return I.Factor(I.S_MOVING_HAT, (c0, amp, f, w))


def _prob(n, axes, q, N=3, M=5, fixed=2, periodic=()):
    """One moving term per entry of `axes` (the axes it moves along) beside `fixed` bumps."""
    d = len(n)
    box = ((0.0, 1.0), (0.0, 1.2), (0.0, 0.9))[:d]
    u0, f, _ = I.sin_mode(d, box, 0.07)
    rng = I.SplitMix64(11)
    move = []
    for e, ax in enumerate(axes):
        facs = tuple(_hat(0.45, 0.2, 1.0 + 0.5 * e + a) if a in ax else I.Factor(I.S_GAUSS, (0.4, 0.2))
                     for a in range(d))
        move.append(I.Term(2.0 - e, facs, I.T_SIN if e % 2 else I.T_EXP, (3.0, 0.4) if e % 2 else (-0.8, 0.0)))
    forcing = (I.gaussian_bumps(rng, d, fixed) if fixed else ()) + tuple(move)
    return I.Problem(d, n, box, 0.07, 0.2, 0.9, N, M, I.uniform_nodes(q), I.draw_random_nodes(2, 9), u0, forcing, 3,
                     1e-12, None, "", (), periodic)


CASES = {"line_q1": _prob((37,), [(0,)], 1), "line_q6": _prob((63,), [(0,), (0,)], 6),
         "first_axis": _prob((21, 15), [(0,)], 2), "last_axis": _prob((21, 15), [(1,)], 4),
         "both_axes": _prob((14, 19), [(0, 1), (1,)], 3), "none_fixed": _prob((17, 12), [(0,), (0, 1)], 4, fixed=0),
         "box": _prob((7, 9, 8), [(0, 1, 2), (2,), (0, 2)], 2, M=3),
         "periodic": _prob((16, 11), [(0,), (1,)], 3, periodic=(True, False)),
         "chunks": _prob((9,), [(0,)], 8, N=129, M=64)}


@pytest.mark.parametrize("name", list(CASES))
def test_moving_terms_match_full_quadrature(pe, name):
    prob = CASES[name]
    sys_ = osolver.ModalSystem(prob, forcing_route="full")
    ref = osolver.sequential_fine(sys_)
    for prec, bound in ((pe.PE_FP64, 1e-12), (pe.PE_MIXED, 1e-6)):
        with pe.Solver(prob, precision=prec, forcing_path=pe.PE_FORCING_GENERAL) as s:
            s.solve(tol=1e-10)
            for m in range(1, prob.N + 1, max(1, prob.N // 9)):
                assert _rel(s.modal(m), ref[m], sys_.norm_w) <= bound, (prec, m)


@pytest.mark.parametrize("n,axes", [((37,), [(0,), (0,)]), ((17, 12), [(0,), (0, 1)])], ids=["line", "plane"])
def test_one_context_with_and_without_fixed_terms(pe, n, axes):
    """Problems with fixed terms, without, and with them again on one context give what a fresh context gives, bit for bit,
    and a float64 refinement of the one without reaches the oracle."""
    probs = [_prob(n, axes, 3), _prob(n, axes, 3, fixed=0), _prob(n, axes, 3)]
    with pe.Solver(probs[0], precision=pe.PE_MIXED, forcing_path=pe.PE_FORCING_GENERAL) as s:
        for prob in probs:
            s.prob, s._f_struct = prob, None  # (the binding marshals its terms once)
            s.set_problem()
            s.iterate()
            s.refine()
            s.refine()
            s.refine()
            with pe.Solver(prob, precision=pe.PE_MIXED, forcing_path=pe.PE_FORCING_GENERAL) as fresh:
                fresh.set_problem()
                fresh.iterate()
                fresh.refine()
                fresh.refine()
                fresh.refine()
                for m in range(prob.N + 1):
                    assert np.array_equal(s.modal(m), fresh.modal(m)), m
            sys_ = osolver.ModalSystem(prob, forcing_route="full")
            assert _rel(s.modal(prob.N), osolver.sequential_fine(sys_)[prob.N], sys_.norm_w) <= 1e-12
