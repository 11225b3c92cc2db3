"""FP64 roundings whose refinement hands over to the FP64 sweeps, at every kind of cluster
size: a wide centre matrix (more columns than rows) with equal singular values, whose
directions are the result and which small tangents cannot separate."""
import numpy as np
import pytest

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


def equal_values(L, k, r, r1, rng):
    """Cores of an MPS that is an isometry on both sides of bond k, r equal singular values
    there, bond k + 1 of r1 <= r."""
    q = lambda m, n: np.linalg.qr(rng.standard_normal((m, n)))[0]
    bonds = [min(2 ** j, r) for j in range(k + 1)] + [min(2 ** (L - j), r1) for j in range(k + 1, L + 1)]
    cores = [q(bonds[j] * 2, bonds[j + 1]).reshape(bonds[j], 2, bonds[j + 1]) for j in range(k)]
    cores += [q(2 * bonds[j + 1], bonds[j]).T.reshape(bonds[j], 2, bonds[j + 1]) for j in range(k, L)]
    return cores


def flat_field(cores):
    left = np.ones((1, 1))
    for c in cores[:len(cores) // 2]:
        left = np.einsum("la,asb->lsb", left, c).reshape(-1, c.shape[2])
    right = np.ones((1, 1))
    for c in cores[:len(cores) // 2 - 1:-1]:
        right = np.einsum("asb,bq->asq", c, right).reshape(c.shape[0], -1)
    return (left @ right).reshape(-1)


# jobs: the clusters get 16, 8 .. 2 CTAs on 152 SMs; (r, r1): centre matrices of r x 2 r1
@pytest.mark.parametrize("jobs", [1, 9, 18, 40, 60])
@pytest.mark.parametrize("r,r1,chi", [(120, 64, 64), (33, 20, 40), (100, 62, 70)])
def test_equal_singular_values(tl, jobs, r, r1, chi):
    L, k = 15, 7
    rng = np.random.default_rng(1000 * jobs + r)
    ops = [equal_values(L, k, r, r1, rng) for _ in range(min(jobs, 3))]
    dev = [tl.DeviceMps.from_cores(o, max(r, r1), tl.nat.FP64) for o in ops]
    dst = [tl.DeviceMps(L, chi, tl.nat.FP64) for _ in range(jobs)]
    tl.lincomb_round([[tl.plain(dev[j % len(dev)])] for j in range(jobs)], dst, chi, 1e-12)
    for j in range(jobs):
        got = [np.asarray(c) for c in dst[j].cores()]
        x, y = flat_field(ops[j % len(dev)]), flat_field(got)
        for c in got[1:]:
            m = c.reshape(c.shape[0], -1)
            # right-orthonormal to FP64 rounding of products of 128 terms
            assert np.abs(m @ m.T - np.eye(m.shape[0])).max() <= 1e-12
        # a projection: |x|^2 = |y|^2 + |x - y|^2, and no more is cut than the tails
        tails = sum((np.linalg.svd(x.reshape(2 ** b, -1), compute_uv=False)[chi:] ** 2).sum() for b in range(1, L))
        n2 = x @ x
        assert abs(n2 - y @ y - (x - y) @ (x - y)) <= 1e-12 * n2
        assert (x - y) @ (x - y) <= tails * (1 + 1e-9) + (1e-12) ** 2 * n2 + 1e-24 * n2
