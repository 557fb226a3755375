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


@pytest.mark.parametrize("own_stream", [False, True], ids=["default", "callers"])
def test_a_buffer_is_written_after_its_last_reader(pe, own_stream):
    """One device buffer for every solution, read by work of the caller's stream that has not run yet when the next call
    is made."""
    import torch

    probs = I.config4(count=4)
    stream = torch.cuda.Stream() if own_stream else None
    with pe.BatchSolver(probs, stream=stream) as b, torch.cuda.stream(stream):
        b.solve(tol=1e-6)
        want = [b.solution(i) for i in range(4)]
        modal = [b.modal(i, 1) for i in range(4)]
        buf = torch.empty(max(p.ndof for p in probs), dtype=torch.float64, device="cuda")
        for fetch, ref in ((lambda i: b.solution(i, out=buf), want), (lambda i: b.modal(i, 1, out=buf), modal)):
            kept = []
            for i, p in enumerate(probs):
                fetch(i)
                torch.cuda._sleep(20000000)  # about 10 ms of another kernel
                kept.append(buf[:p.ndof].clone())
            for i, k in enumerate(kept):
                assert np.array_equal(k.cpu().numpy(), ref[i]), i


@pytest.mark.parametrize("device", [False, True], ids=["host", "device"])
def test_threads_fetch_from_one_batch(pe, device):
    """Several threads fetch solutions of one batch at once (the calls release the interpreter's lock): the transforms
    share the batch's scratch."""
    import threading

    import torch

    probs = I.config4(count=5)
    with pe.BatchSolver(probs) as b:
        b.solve(tol=1e-6)
        want = [b.solution(i) for i in range(5)]
        wrong = []

        def fetch(seed):
            rng = np.random.default_rng(seed)
            for i in rng.integers(0, 5, 40):
                if device:
                    out = torch.empty(probs[i].ndof, dtype=torch.float64, device="cuda")
                    got = b.solution(int(i), out=out).cpu().numpy()
                else:
                    got = b.solution(int(i))
                if not np.array_equal(got, want[i]):
                    wrong.append(int(i))

        ts = [threading.Thread(target=fetch, args=(s,)) for s in range(6)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        assert not wrong


@pytest.mark.parametrize("engine", [0, 1], ids=["simt", "tc"])
def test_autotune_leaves_a_finished_solve_as_it_is(pe, engine):
    probs = I.config4(count=5)
    with pe.BatchSolver(probs, fine_engine=engine) as b:
        b.solve(tol=1e-6)

        def results():
            r, k = b.status()
            return [r, k] + [b.modal(i, m) for i, p in enumerate(probs) for m in (0, 1, p.N)] + \
                [b.solution(i) for i in range(len(probs))]

        before = results()
        b.autotune(None)
        for x, y in zip(before, results()):
            assert np.array_equal(x, y)
        b.solve(tol=1e-6)
        for x, y in zip(before[1:], results()[1:]):  # (the residual sums follow the launch shape's items)
            assert np.array_equal(x, y)
