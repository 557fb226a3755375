"""GPU: what the batch's calls owe their caller beside the numbers: the times they report, the order with the caller's
stream, threads, and what a finished solve keeps.
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


def test_times_are_those_of_the_solve_with_a_callers_stream(pe):
    import torch

    stream = torch.cuda.Stream()
    with pe.BatchSolver(I.config4(count=6), stream=stream) as b:
        for _ in range(3):
            info = b.solve(tol=1e-6)
            assert info["ms_prepare"] > 0.0 and info["ms_iterations"] > 0.0
    torch.cuda.synchronize()
