"""Dense contraction of MPS and TT-SVD of dense fields at the edges of their kernels'
tiles: bonds around the 16/32-wide steps of the digit products and the 128 up to
which they are taken, lattices on both sides of the 64^3 from which they are, rows
that are not finite; eigenproblems below, at and beyond 128 columns."""
import numpy as np
import pytest

import synth
from oracle import mps as M, quantics as q

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_07615_gb300 import tnlbm as T
    return T


def device(tl, cores, cap, prec):
    import torch
    X = tl.DeviceMps(len(cores), cap, prec)
    flat = torch.zeros(X.data.numel(), dtype=X.data.dtype)
    for k, c in enumerate(cores):
        o = tl.mps_offset(X.L, cap, k)
        flat[o:o + c.size] = torch.from_numpy(np.ascontiguousarray(c).reshape(-1)).to(flat.dtype)
    X.data.copy_(flat)
    X.ranks.copy_(torch.tensor([1] + [c.shape[2] for c in cores], dtype=torch.int32))
    return X


def field(cores):
    """The dense [x][y][z] field in 64 bits."""
    L = len(cores)
    left = np.ones((1, 1))
    for c in cores[:L // 2]:
        left = np.einsum("la,asb->lsb", left, c).reshape(-1, c.shape[2])
    right = np.ones((1, 1))
    for c in cores[:L // 2 - 1:-1]:
        right = np.einsum("asb,bq->asq", c, right).reshape(c.shape[0], -1)
    return q.decode((left @ right).reshape((2,) * L))


@pytest.mark.parametrize("n,bond,cap", [(1, 2, 2), (2, 5, 8), (4, 33, 64), (5, 64, 64), (6, 1, 1), (6, 15, 16),
                                        (6, 33, 45), (6, 64, 64), (6, 128, 128), (6, 128, 129), (7, 31, 128)])
@pytest.mark.parametrize("prec", [0, 1])
def test_to_dense(tl, n, bond, cap, prec):
    dt = np.float64 if prec == 0 else np.float32
    cores = [c.astype(dt).astype(np.float64) for c in synth.random_mps(3 * n, synth.feasible_ranks(3 * n, bond), 11 * bond + n)]
    ref = field(cores)
    got = tl.to_dense(device(tl, cores, cap, prec)).cpu().numpy().astype(np.float64)
    # FP32 output: its rounding; the sums: 128 roundings of 1.1e-16 of terms a few times the largest value
    tol = (6e-8 * np.abs(ref) if prec else 0.0) + 1e-13 * np.abs(ref).max()
    assert (np.abs(got - ref) <= tol).all()


def test_to_dense_rows_not_finite(tl):
    """An infinity in a core's first half reaches the cells whose prefix holds it, no others."""
    cores = [c.astype(np.float32).astype(np.float64) for c in synth.random_mps(18, synth.feasible_ranks(18, 8), 3)]
    ref = field(cores)
    bad = [c.copy() for c in cores]
    bad[8][0, 1, 2] = np.inf
    got = tl.to_dense(device(tl, bad, 8, 1)).cpu().numpy()
    hit = np.zeros((2,) * 18, dtype=bool)
    hit[(slice(None),) * 8 + (1,)] = True
    hit = q.decode(hit.astype(float)) > 0.5
    assert not np.isfinite(got[hit]).any()
    assert np.abs(got[~hit] - ref[~hit]).max() <= 1e-6 * np.abs(ref).max()


def test_output_fields_sum_the_populations(tl):
    """rho and u of 64^3 FP32 populations, FP64 sums, against the dense populations."""
    from oracle import lattice
    lat = lattice.D3Q19
    sim = tl.Sim(6, tau=0.7, chi_max=16, eps=1e-7, precision=1, force=(1e-5, 0.0, 0.0))
    pops = []
    for i in range(19):
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
        rest = [np.full((1, 2, 1), w[i] if k == 0 else 1.0) for k in range(18)]
        noise = synth.random_mps(18, synth.feasible_ranks(18, 15), 100 + i)
        noise[0] = noise[0] * (1e-3 * w[i] / np.abs(field(noise)).max())
        pops.append([c.astype(np.float32).astype(np.float64) for c in M.add(rest, noise)])
    sim.set_populations(pops)
    rho, u = sim.macroscopic()
    f = np.array([field(p) for p in pops])
    c = np.array(lat.c)
    r = f.sum(0)
    assert np.abs(rho - r).max() <= 1e-13
    for d in range(3):
        j = np.tensordot(c[:, d].astype(float), f, 1) + (0.5e-5 if d == 0 else 0.0)
        assert np.abs(u[d] - j / r).max() <= 1e-13
    sim.close()


@pytest.mark.parametrize("n,bond,chi,prec", [(2, 2, 2, 0), (4, 3, 3, 0), (4, 20, 16, 0), (5, 48, 48, 0), (5, 64, 64, 1),
                                             (6, 90, 80, 0)])
def test_from_dense_bound(tl, n, bond, chi, prec):
    """TT-SVD with a rank cap: cores of orthonormal columns, and an error of at most the
    root of the summed squared tails of the field's unfoldings."""
    import torch
    L = 3 * n
    cores = synth.random_mps(L, synth.feasible_ranks(L, bond), 7 + bond)
    x = field(cores)
    x /= np.linalg.norm(x)
    X = tl.from_dense(torch.tensor(x, dtype=torch.float64 if prec == 0 else torch.float32, device="cuda"), chi, chi, 0.0)
    out = X.cores()
    for c in out[:-1]:
        m = np.asarray(c, dtype=np.float64).reshape(-1, c.shape[2])
        assert np.abs(m.T @ m - np.eye(m.shape[1])).max() <= (1e-12 if prec == 0 else 1e-5)
    err = np.linalg.norm(field([np.asarray(c, dtype=np.float64) for c in out]) - x)
    t = q.encode(x).reshape(-1)
    tails = 0.0
    for k in range(1, L):
        m = t.reshape(2 ** k, -1)
        s2 = np.linalg.eigvalsh(m @ m.T if m.shape[0] <= m.shape[1] else m.T @ m)[::-1]
        tails += max(0.0, s2[chi:].sum())
    # what the Gram matrices cannot resolve: 64 eps m per bond, squared norms
    floor = (L - 1) * 64 * 2.3e-16 * 2 * chi
    assert err ** 2 <= tails * (1 + 1e-6) + floor + (1e-9 if prec else 0.0)
