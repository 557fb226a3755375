"""GPU: shards of a grid whose weights come from the response table although a shard alone has too few modes for one.

A sharded context's per-mode arithmetic is the whole grid's, so its modal iterates are the unsharded solve's bit for
bit; which form the weights take has to follow from the whole grid too.
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


@pytest.mark.parametrize("n,precision", [((160, 131), 1), ((256, 200), 0), ((31, 30, 26), 1)],
                         ids=["plane_mixed", "plane_fp64", "box_mixed"])
@pytest.mark.parametrize("parts", [2, 7])
def test_shards_take_the_whole_grids_weights(pe, n, precision, parts):
    from paper_2412_01138_gb300 import shard

    prob = I.scaled(I.config2() if len(n) == 2 else I.config3(), n, N=4, M=16)
    with pe.Solver(prob, precision=precision) as s:
        s.set_problem()
        s.iterate()
        want = [s.modal(m) for m in range(prob.N + 1)]
    got = []
    for rg in shard.shard_ranges(n[0], parts):
        with pe.Solver(prob, precision=precision, mode_range=rg) as s:
            s.set_problem()
            s.iterate_sums()
            got.append([s.modal(m) for m in range(prob.N + 1)])
    for m in range(prob.N + 1):
        assert np.array_equal(np.concatenate([g[m] for g in got]), want[m]), m
