"""GPU: the folded matrix form of the DST-I (axes whose n + 1 is not a power of two) against dense products.

Sizes where it can go wrong: odd and even n (an odd one has a middle index that is its own mirror), fewer
indices than a chunk of 32, one more than a chunk, tiles of 8, 16 and 32 outputs with a remainder,
pencil counts around 32 and 64 and large enough for the wide tiles, contiguous and strided pencils with short
and long inner extents, short axes with an FFT form that take it in float64, in place.  Bound: a folded sum has n/2 + 1 rounded terms, so each output is within
(n/2 + 3) u sum |S||x| of the product, and the 2-norm of |S||x| is at most sqrt(n) times that of x:
(n/2 + 3) u sqrt(n) relative, u = 2^-53 or 2^-24.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(2,), (4,), (5,), (6,), (33,), (64,), (65,), (66,), (257,), (1000,), (4, 2), (5, 33), (33, 5), (64, 64),
         (100, 37), (37, 100), (200, 117), (129, 300), (20, 700), (1200, 9), (6, 5, 4), (10, 33, 17), (40, 66, 9),
         (12, 250, 130), (63, 34, 100),
         (7, 400), (31, 400), (19, 17, 15), (63, 500)]


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_01138_gb300 import pe

    pe.lib()
    return pe, torch


def _dense(x):
    for a, n in enumerate(x.shape):
        j = np.arange(1, n + 1)
        S = math.sqrt(2.0 / (n + 1)) * np.sin(np.pi * (np.outer(j, j) % (2 * (n + 1))) / (n + 1))
        x = np.moveaxis(np.tensordot(S, x, axes=(1, a)), 0, a)
    return x


@pytest.mark.parametrize("n", SIZES, ids=["x".join(map(str, n)) for n in SIZES])
@pytest.mark.parametrize("f32", [False, True], ids=["float64", "float32"])
def test_folded_matrix_form_matches_dense_products(env, n, f32):
    pe, torch = env
    x = np.random.default_rng(sum(n)).standard_normal(n)
    x = x.astype(np.float32) if f32 else x
    ref = _dense(x.astype(np.float64))
    u = 2.0 ** (-24 if f32 else -53)
    bound = sum((v / 2 + 3) * u * math.sqrt(v) for v in n)
    d = torch.tensor(x.reshape(-1), device="cuda")
    out = torch.empty_like(d)
    pe.dst(len(n), n, d, out, f32=f32)
    pe.dst(len(n), n, d, d, f32=f32)
    for got in (out, d):
        err = np.linalg.norm(got.cpu().numpy().astype(np.float64).reshape(n) - ref) / np.linalg.norm(ref)
        assert err <= bound, (err, bound)


@pytest.mark.parametrize("m", [15, 31, 63, 127, 255, 511, 1023])
@pytest.mark.parametrize("pencils", [1, 2, 5, 70])
@pytest.mark.parametrize("strided", [False, True], ids=["contiguous", "strided"])
def test_few_float64_pencils(env, m, pencils, strided):
    """The block-wide half-length FFT at every length, one pencil and an odd number of them (the last pair is
    half empty).  Its prefix sum adds up to N/2 = (m + 1)/2 values of an FFT of log2 N stages: N log2 N u relative."""
    pe, torch = env
    n = (m,) if pencils == 1 else ((m, pencils) if strided else (pencils, m))
    x = np.random.default_rng(m + pencils).standard_normal(n)
    d = torch.tensor(x.reshape(-1), device="cuda")
    pe.dst(len(n), n, d, d)
    ref = _dense(x)
    err = np.linalg.norm(d.cpu().numpy().reshape(n) - ref) / np.linalg.norm(ref)
    bound = (m + 1) * math.log2(m + 1) * 2.0 ** -53
    if pencils > 1:  # the other axis in the matrix form
        bound += (pencils / 2 + 3) * 2.0 ** -53 * math.sqrt(pencils)
    assert err <= bound, (err, bound)


@pytest.mark.parametrize("n", [(511, 305), (511, 3648), (511, 3649), (2, 511, 3500)],
                         ids=["511x305", "511x3648", "511x3649", "2x511x3500"])
def test_strided_511_float32(env, n):
    """The two-pass kernel of 511 strided float32 values: in its blocks of 8 pencils, at the last and the first count
    of the two block sizes, with ragged tails and several blocks to a CTA, and with blocks that cross a plane.
    Ten butterfly stages: 10 sqrt(10) u relative, and the other axes in the matrix form."""
    pe, torch = env
    x = np.random.default_rng(sum(n)).standard_normal(n).astype(np.float32)
    d = torch.tensor(x.reshape(-1), device="cuda")
    out = torch.empty_like(d)
    pe.dst(len(n), n, d, out, f32=True)
    pe.dst(len(n), n, d, d, f32=True)
    ref = _dense(x.astype(np.float64))
    u = 2.0 ** -24
    bound = 10 * math.sqrt(10) * u + sum((v / 2 + 3) * u * math.sqrt(v) for v in n if v != 511)
    for got in (out, d):
        err = np.linalg.norm(got.cpu().numpy().astype(np.float64).reshape(n) - ref) / np.linalg.norm(ref)
        assert err <= bound, (err, bound)


@pytest.mark.parametrize("m", [2, 5, 36, 301, 1030])
@pytest.mark.parametrize("pencils", [1, 2, 3, 7, 8, 9])
@pytest.mark.parametrize("strided", [False, True], ids=["contiguous", "strided"])
@pytest.mark.parametrize("f32", [False, True], ids=["float64", "float32"])
def test_few_pencils_in_the_matrix_form(env, m, pencils, strided, f32):
    """A warp's share of every sum, at both parities of the length, fewer outputs than a warp makes, every group size,
    a ragged last group and the first count that goes to the tiles at any length.  Sums of n/2 products and a tree, as above."""
    pe, torch = env
    n = (m,) if pencils == 1 else ((m, pencils) if strided else (pencils, m))
    x = np.random.default_rng(m + pencils).standard_normal(n)
    x = x.astype(np.float32) if f32 else x
    d = torch.tensor(x.reshape(-1), device="cuda")
    pe.dst(len(n), n, d, d, f32=f32)
    ref = _dense(x.astype(np.float64))
    u = 2.0 ** (-24 if f32 else -53)
    bound = sum((v / 2 + 3) * u * math.sqrt(v) for v in n)
    err = np.linalg.norm(d.cpu().numpy().astype(np.float64).reshape(n) - ref) / np.linalg.norm(ref)
    assert err <= bound, (err, bound)


@pytest.mark.parametrize("n,periodic", [((517,), (True,)), ((517, 8), (True, False)), ((45, 2), (True, True))],
                         ids=["517", "517x8", "45x2"])
def test_few_periodic_pencils(env, n, periodic):
    """A periodic line and thin grids whose Hartley transforms have few pencils, against the oracle at the
    periodic tests' bounds."""
    from oracle import solver as osolver
    from test_gpu_periodic import _problem, _rel

    pe, _ = env
    prob = _problem(n, periodic, N=3, M=4)
    sys_ = osolver.ModalSystem(prob)
    fine = osolver.sequential_fine(sys_)
    for precision, tol in ((pe.PE_FP64, 1e-12), (pe.PE_MIXED, 1e-6)):
        with pe.Solver(prob, precision=precision) as s:
            s.solve(tol=0.1 * tol)
            assert _rel(s.solution(prob.N).reshape(prob.n), sys_.to_nodal(fine[-1])) <= tol
