"""GPU: the two values of pe_options.fine_engine run the same kernels (the sums over the source columns), so what they
return is equal bit for bit; and the mixes of many random terms, up to 64 columns and 200 rad a unit of time, meet the mixed
form's own bound against the oracle's substeps, 1e-6 in relative L2 at every slice of two iterates (float32 rounding of
17 to 64 weights a mode that partly cancel; taken one by one, the substeps of such mixes were up to 1.5e-6 off).
"""
import numpy as np
import pytest

from oracle import solver as osolver
from paper_2412_01138_gb300 import inputs as I
from test_gpu_fine_tc import _rel, _term_mix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pe():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_01138_gb300 import pe as _pe

    _pe.lib()
    return _pe


# K = 1, 2, 28, 34, 40, 64, 61, 18 columns: float32 rows of 4, 28, 36, 40, 64 and 20, whole and padded
@pytest.mark.parametrize("kinds,M,N", [("e", 16, 21), ("s", 32, 9), ("esses" * 3 + "ss", 64, 7), ("esse" * 4 + "s" * 5, 96, 5),
                                       ("s" * 20, 48, 11), ("s" * 32, 128, 3), ("s" * 30 + "e", 32, 6), ("s" * 9, 32, 7)])
def test_stress_mixes(pe, kinds, M, N):
    box = ((0.0, 1.0), (0.0, 1.0))
    u0, _, _ = I.sin_mode(2, box, 0.05)
    prob = I.Problem(2, (47, 61), box, 0.05, 0.1, 0.6, N, M, I.draw_random_nodes(4, 78), I.uniform_nodes(2), u0,
                     _term_mix(kinds, len(kinds) + 3), 3, 1e-12)
    sys_ = osolver.ModalSystem(prob)
    ref = osolver.parareal(sys_, tol=0.0, k_max=2)
    out = {}
    for eng in (pe.PE_FINE_SIMT, pe.PE_FINE_TC):
        out[eng] = []
        with pe.Solver(prob, precision=pe.PE_MIXED, fine_engine=eng) as s:
            s.set_problem()
            for k in range(1, 3):
                s.iterate()
                out[eng] += [s.modal(m) for m in range(1, N + 1)]
    for x, y in zip(*out.values()):
        assert np.array_equal(x, y)
    want = [ref.history[k][m] for k in range(1, 3) for m in range(1, N + 1)]
    assert max(_rel(x, y, sys_.norm_w) for x, y in zip(out[pe.PE_FINE_TC], want)) <= 1e-6


def test_batch_engines_are_one(pe):
    probs = I.config4(count=8)
    out = []
    for eng in (pe.PE_FINE_SIMT, pe.PE_FINE_TC):
        with pe.BatchSolver(probs, precision=pe.PE_MIXED, fine_engine=eng) as b:
            b.solve(tol=1e-6)
            r, k = b.status()
            out.append([r, k] + [b.modal(i, m) for i, p in enumerate(probs) for m in (1, p.N)] +
                       [b.solution(i) for i in range(len(probs))])
    for x, y in zip(*out):
        assert np.array_equal(x, y)
