"""The register kernels of the FP32 and mixed roundings (Jacobi on the rows of
the centre matrix, or the one that starts the FP64 SVD, whose rotations the
cluster replays; panel QR) at the edges of their variants: vectors of 32 / 64 / 128
entries and one more, blocks of 1 / 2 / 4 columns (up to 32, 64, 128 of them)
and one more, wide and tall centre matrices, and beyond what they take.

Tolerance.  A rounding factorises 2 L matrices of at most n columns; each
factorisation is backward stable to c sqrt(n) u with u = 2^-24 and a modest c
(8 here), and the 2 L errors add like independent ones: 8 sqrt(n) u sqrt(2 L)
relative to the norm, for an untruncated sum.  A truncated one is compared by
its distance from the exact sum, which may exceed the oracle's by that much."""
import numpy as np
import pytest

import synth
from oracle import mps as M

pytestmark = pytest.mark.gpu
U = 2.0 ** -24


@pytest.fixture(scope="module")
def tl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_07615_gb300 import tnlbm as T
    return T


def _float(cores):
    return [c.astype(np.float32).astype(np.float64) for c in cores]


@pytest.fixture(params=[1, 3], ids=["fp32", "mixed"])
def prec(request):
    return request.param


# (sites, bonds of the two terms, chi): the centre matrices are m x n with m up to
# the summed bond (or 2^k, 2^(L-k)) and n = 2 chi or twice the bond to the right
@pytest.mark.parametrize("L,a,b,chi", [
    (3, 1, 1, 2), (6, 3, 5, 8), (9, 9, 7, 16), (12, 15, 17, 32), (12, 16, 17, 33), (12, 30, 34, 64), (12, 32, 33, 65),
    (15, 64, 64, 128), (15, 65, 64, 129), (15, 127, 3, 130),
    (12, 32, 32, 1), (12, 32, 32, 16), (12, 33, 30, 17), (15, 64, 64, 32), (15, 64, 64, 64), (15, 64, 65, 33)])
def test_sum_of_two(tl, prec, L, a, b, chi):
    A = _float(synth.random_mps(L, synth.feasible_ranks(L, a), 1))
    B = _float(synth.random_mps(L, synth.feasible_ranks(L, b), 2))
    dA, dB = tl.DeviceMps.from_cores(A, a, prec), tl.DeviceMps.from_cores(B, b, prec)
    D = tl.DeviceMps(L, max(chi, a, b), prec)
    tl.lincomb_round([[tl.plain(dA), tl.plain(dB, -0.5)]], [D], chi, 0.0)
    exact = M.to_tensor(A) - 0.5 * M.to_tensor(B)
    ref = M.to_tensor(M.lincomb_round([(1.0, A), (-0.5, B)], chi, 0.0))
    tol = 8.0 * np.sqrt(2.0 * (a + b)) * U * np.sqrt(2.0 * L)
    norm = np.linalg.norm(exact)
    err, opt = np.linalg.norm(M.to_tensor(D.cores()) - exact) / norm, np.linalg.norm(ref - exact) / norm
    assert err <= opt + tol


@pytest.mark.parametrize("terms", ["same", "cancel", "ones", "zero"])
def test_rank_deficient_sums(tl, prec, terms):
    """Centre matrices with zero and repeated directions (their rows are not
    orthonormal and must carry nothing)."""
    L = 9
    A = _float(synth.random_mps(L, synth.feasible_ranks(L, 12), 3))
    dA = tl.DeviceMps.from_cores(A, 12, prec)
    spec = {"same": [tl.plain(dA), tl.plain(dA, 2.0)], "cancel": [tl.plain(dA), tl.plain(dA, -1.0)],
            "ones": [tl.ones(3.0), tl.ones(-1.0)], "zero": [tl.plain(dA, 0.0), tl.ones(0.0)]}[terms]
    ref = {"same": 3.0 * M.to_tensor(A), "cancel": 0.0 * M.to_tensor(A),
           "ones": 2.0 * M.to_tensor(M.ones(L)), "zero": 0.0 * M.to_tensor(A)}[terms]
    D = tl.DeviceMps(L, 24, prec)
    tl.lincomb_round([spec], [D], 24, 0.0)
    scale = max(np.linalg.norm(ref), np.linalg.norm(M.to_tensor(A)))
    tol = 8.0 * np.sqrt(48.0) * U * np.sqrt(2.0 * L)
    assert np.linalg.norm(M.to_tensor(D.cores()) - ref) <= tol * scale
