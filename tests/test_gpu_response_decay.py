"""GPU: sources that decay over a slice by many factors of e, on grids large enough for the tabulated weights
(pe_contract.cuh, "Response tables"), against the oracle's substeps.

The weight of e^{at}, a < 0, at a mode is of the size e^{-min(lam, -a) dT}, while the table's error is bounded in units
of the weight's size without that factor; the library therefore evaluates such a problem's weights mode by mode.  No initial
data and no other source, so that the whole solution decays; every slice of the fixed point.  Bounds: the forms' own,
1e-12 (float64) and 1e-6 (mixed), in relative L2.  The last cases are just inside the rule: their weights are
tabulated.
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


# D, T, N, rate; lam_min is about 20 D
DECAYS = [(1.0, 1.0, 2, -25.0), (1.0, 4.0, 4, -20.0), (1.0, 4.0, 4, -40.0), (1.0, 3.0, 2, -30.0), (1.0, 6.0, 2, -40.0),
          (0.05, 6.0, 2, -19.0), (3.0, 1.0, 2, -1000.0)]
NEAR = {0: [(1.0, 1.0, 2, -1.1), (3.0, 1.1, 2, -1.0)], 1: [(1.0, 4.0, 4, -1.8), (2.0, 0.5, 2, -7.0)]}
CASES = [(p, c) for p in (0, 1) for c in DECAYS + NEAR[p]]


@pytest.mark.parametrize("precision,case", CASES, ids=[f"{'mixed' if p else 'fp64'}_D{c[0]}_T{c[1]}_N{c[2]}_a{c[3]}"
                                                       for p, c in CASES])
def test_decaying_source(pe, precision, case):
    D, T, N, rate = case
    n = (160, 160) if precision else (208, 208)  # (more modes than eight per table node)
    facs = tuple(I.Factor(I.S_GAUSS, (0.45, 0.1)) for _ in n)
    prob = I.Problem(2, n, ((0.0, 1.0),) * 2, D, 0.0, T, N, 16, I.uniform_nodes(3), I.uniform_nodes(2), (),
                     (I.Term(1.0, facs, I.T_EXP, (rate, 0.0)),), 3, 1e-12)
    sys_ = osolver.ModalSystem(prob)
    fine = osolver.sequential_fine(sys_)
    with pe.Solver(prob, precision=precision) as s:
        s.solve(tol=0.0)  # all N iterations: the fixed point on every slice
        got = [s.modal(m) for m in range(N + 1)]
    errors = [_rel(got[m], fine[m], sys_.norm_w) for m in range(1, N + 1)]
    assert max(errors) <= (1e-6 if precision else 1e-12), errors
