"""rho and u where the capacities of the populations and of the mask lie on both sides of
the 128 up to which FP32 fields are joined by digits: one scratch serves both, and its
size is no monotonic function of the capacity."""
import numpy as np
import pytest

import synth
from oracle import lattice, mps as M, quantics as q

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


@pytest.mark.parametrize("chi,chi_mask", [(128, 256), (256, 128), (96, 129), (150, 48)])
@pytest.mark.parametrize("prec", [0, 1])
def test_fields_with_two_capacities(tl, chi, chi_mask, prec):
    """64^3 with a solid box and a body force, against the dense populations."""
    lat = lattice.D3Q19
    dt = np.float32 if prec else np.float64
    solid = np.zeros((64, 64, 64), dtype=np.uint8)
    solid[16:32, 8:40, 32:48] = 1
    force = np.array([1e-3, -2e-3, 5e-4])
    sim = tl.Sim(6, tau=0.7, chi_max=chi, eps=1e-7, precision=prec, force=tuple(force), solid=solid, chi_mask=chi_mask)
    w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
    pops = []
    for i in range(19):
        rest = [np.full((1, 2, 1), w[i] if k == 0 else 1.0) for k in range(18)]
        noise = synth.random_mps(18, synth.feasible_ranks(18, 7), 300 + i)
        noise[0] = noise[0] * (1e-3 * w[i] / np.abs(q.decode(M.to_tensor(noise))).max())
        pops.append([c.astype(dt).astype(np.float64) for c in M.add(rest, noise)])
    sim.set_populations(pops)
    rho, u = sim.macroscopic()
    sim.close()
    f = np.array([q.decode(M.to_tensor(p)) for p in pops])
    c = np.array(lat.c, dtype=float)
    r = f.sum(0)
    # 19 populations of order one summed in FP64; the box has few singular values, of one size,
    # kept to FP64 rounding, and a mask stored in FP32 carries 18 roundings of 6e-8
    tol = 1e-13 + 1e-12 * np.abs(force).max() + (18 * 6e-8 * np.abs(force).max() if prec else 0.0)
    assert np.abs(rho - r).max() <= 1e-13
    for d in range(3):
        ref = (np.tensordot(c[:, d], f, 1) + 0.5 * force[d] * (1.0 - solid)) / r
        assert np.abs(u[d] - ref).max() <= tol
