"""GPU parity of the slice sums contracted over every substep (pe_contract.cuh) where they can go wrong.

The oracle takes every substep.  Cases: M with every kind of bit pattern (1, powers of two, odd, 2^k +- 1:
doublings with and without an added step); K from 1 to 64 columns (float32 rows of 4 .. 64, the
float64 kernel's exact counts); slice counts around the group of eight the walk prefetches and
beyond the slices staged at a time; mode counts around a CTA; exponentials that grow and decay over a slice by
more than the range of a double.  Bounds: the forms' own, 1e-12 (float64) and 1e-6 (mixed), in relative L2 at
every slice of every iterate.
"""
import math

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


def _terms(kinds, d, seed):
    rng = I.SplitMix64(seed)
    out = []
    for k in kinds:
        facs = tuple(I.Factor(I.S_SIN, (math.pi * (1 + int(3 * rng.uniform())), 0.0)) for _ in range(d))
        amp = 0.5 + rng.uniform()
        if k == "e":
            out.append(I.Term(amp, facs, I.T_EXP, (6.0 * rng.uniform() - 4.0, 0.0)))
        else:
            out.append(I.Term(amp, facs, I.T_SIN, (30.0 * rng.uniform(), 2.0 * math.pi * rng.uniform())))
    return tuple(out)


def _prob(n, N, M, kinds, seed=5, t0=0.1, T=0.8, forcing=None):
    d = len(n)
    box = ((0.0, 1.0),) * d
    u0, _, _ = I.sin_mode(d, box, 0.05)
    return I.Problem(d, n, box, 0.05, t0, T, N, M, I.draw_random_nodes(3, 7), I.uniform_nodes(2), u0,
                     _terms(kinds, d, seed) if forcing is None else forcing, 3, 1e-12)


CASES = [((33,), 3, 1, "e"), ((33,), 7, 2, "s"), ((64,), 8, 3, "es"), ((65,), 9, 5, "see"), ((31, 9), 16, 7, "ses"),
         ((31, 9), 17, 31, "s" * 8), ((20, 13), 5, 33, "e" * 5 + "s" * 4), ((9, 8, 7), 4, 64, "s" * 16),
         ((40,), 6, 97, "s" * 24 + "e"), ((16, 17), 2, 255, "e" * 32), ((24,), 100, 6, "s" * 32),
         ((200,), 700, 4, "se"), ((127, 191), 3, 12, "s" * 6 + "e")]


@pytest.mark.parametrize("n,N,M,kinds", CASES, ids=[f"{'x'.join(map(str, c[0]))}_N{c[1]}_M{c[2]}_{len(c[3])}" for c in CASES])
def test_every_iterate_matches_the_substeps(pe, n, N, M, kinds):
    prob = _prob(n, N, M, kinds)
    sys_ = osolver.ModalSystem(prob)
    ref = osolver.parareal(sys_, tol=0.0, k_max=2)
    for prec, bound in ((pe.PE_FP64, 1e-12), (pe.PE_MIXED, 1e-6)):
        with pe.Solver(prob, precision=prec) as s:
            s.set_problem()
            for k in range(3):
                if k:
                    s.iterate()
                for m in range(1, N + 1, max(1, N // 9)):
                    assert _rel(s.modal(m), ref.history[k][m], sys_.norm_w) <= bound, (prec, k, m)
            stepped = [s.modal(m) for m in range(0, N + 1, max(1, N // 9))]
        # the solve makes the coarse iterate inside its first iteration: the same iterates, bit for bit
        with pe.Solver(prob, precision=prec, max_iter=2) as s:
            try:
                s.solve(tol=0.0)
            except pe.PEError as e:
                assert e.status == pe.PE_ENOCONV
            for x, m in zip(stepped, range(0, N + 1, max(1, N // 9))):
                assert np.array_equal(s.modal(m), x), (prec, m)


@pytest.mark.parametrize("a,t0", [(600.0, -2.0), (-600.0, 0.0)], ids=["grows", "decays"])
def test_exponentials_beyond_the_range_of_a_slice(pe, a, t0):
    """e^{at} over one slice across which it changes by e^{1200} or e^{-1800}, beyond the range of a
    double: its value at the slice's other end is zero; the sums take it at the end where it is large."""
    facs = (I.Factor(I.S_SIN, (math.pi, 0.0)),)
    prob = _prob((33,), 1, 16, "", t0=t0, T=2.0 if a > 0 else 3.0,
                 forcing=(I.Term(1.0, facs, I.T_EXP, (a, 0.0)),) + _terms("s", 1, 3))
    sys_ = osolver.ModalSystem(prob)
    fine = osolver.sequential_fine(sys_)
    for prec, bound in ((pe.PE_FP64, 1e-12), (pe.PE_MIXED, 1e-6)):
        with pe.Solver(prob, precision=prec) as s:
            s.solve(tol=1e-6)
            for m in range(1, prob.N + 1):
                assert _rel(s.modal(m), fine[m], sys_.norm_w) <= bound, (prec, m)


def test_batched_walk_stages_slices_in_chunks(pe):
    """Problems of one batch with one to 39 columns and one to 210 slices (more than the walk stages at a
    time), mode counts that leave partial items, one problem that converges before the others."""
    probs = [_prob((130,), 210, 4, "s" * 19 + "e"), _prob((129, 3), 104, 3, "se"), _prob((5, 9), 1, 7, "e"),
             _prob((16, 8), 9, 33, "s" * 8), _prob((257,), 97, 2, "ss")]
    for prec, bound in ((pe.PE_FP64, 1e-12), (pe.PE_MIXED, 1e-6)):
        with pe.BatchSolver(probs, precision=prec) as b:
            b.solve(tol=1e-10)
            _, k = b.status()
            for i, p in enumerate(probs):
                sys_ = osolver.ModalSystem(p)
                fine = osolver.sequential_fine(sys_)
                assert k[i] == min(2, p.N)
                for m in range(0, p.N + 1, max(1, p.N // 9)):
                    assert _rel(b.modal(i, m), fine[m], sys_.norm_w) <= bound, (prec, i, m)


RESPONSE = {"plane": ((160, 131), 0.05, (), "s" * 5 + "e", 31), "box": ((30, 26, 27), 0.4, (), "sse", 8),
            "periodic": ((128, 150), 0.01, (True, True), "ses", 17), "line": ((16384,), 1.0, (), "se", 5),
            "thin": ((16, 2000), 3.0, (), "s" * 9, 64), "one_periodic": ((64, 300), 20.0, (True, False), "ees", 3)}


@pytest.mark.parametrize("name", list(RESPONSE))
def test_weights_from_the_response_table(pe, name):
    """Grids large enough for the tabulated weights: spectra of 3 to 30 octaves, the zero eigenvalue of an
    all-periodic grid (an interval of its own), stiff and slow modes; every mode of every slice against the
    oracle, in the norm of each form's bound and mode by mode against the largest."""
    n, D, periodic, kinds, M = RESPONSE[name]
    d = len(n)
    box = ((0.0, 1.0),) * d
    facs = tuple(I.Factor(I.S_GAUSS, (0.4, 0.02)) for _ in range(d))  # excites the whole spectrum
    forcing = tuple(I.Term(t.amp, facs, t.tkind, t.tp) for t in _terms(kinds, d, 3))
    prob = I.Problem(d, n, box, D, 0.1, 0.8, 3, M, I.uniform_nodes(4), I.uniform_nodes(2), (), forcing, 3, 1e-12, None, "",
                     (), periodic)
    sys_ = osolver.ModalSystem(prob)
    ref = osolver.parareal(sys_, tol=0.0, k_max=1)
    for prec, bound in ((pe.PE_FP64, 1e-12), (pe.PE_MIXED, 1e-6)):
        with pe.Solver(prob, precision=prec) as s:
            s.set_problem()
            s.iterate()
            for m in range(1, prob.N + 1):
                got, want = s.modal(m), ref.history[1][m]
                assert _rel(got, want, sys_.norm_w) <= bound, (prec, m)
                assert np.abs(got - want).max() <= bound * np.abs(want).max(), (prec, m)
