"""FP64 roundings whose centre SVDs are refined, against 64-bit fields: what the refinement does to
W and V may cost rounding only."""
import numpy as np
import pytest

from oracle import mps as M, quantics as q

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def tl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2512_07615_gb300 import tnlbm as T
    return T


def train(L, r, rng):
    """A random tensor train of bond r with orthonormal rows, entries of order one."""
    b = [min(r, 2 ** k, 2 ** (L - k)) for k in range(L + 1)]
    return [np.sqrt(2.0) * np.linalg.qr(rng.standard_normal((2 * b[k + 1], b[k])))[0].T.reshape(b[k], 2, b[k + 1])
            for k in range(L)]


def population(L, bond, seed):
    """A constant and trains of bond four whose amplitudes fall over eight decades, as a sum
    of blocks (bonds of at most 2^k and 2^(L - k) at the ends)."""
    rng = np.random.default_rng(seed)
    parts = (bond - 1) // 4
    terms = [(1.0 / 18.0, M.ones(L))] + [(1e-3 / 18.0 * 10.0 ** (-8.0 * i / (parts - 1)), train(L, 4, rng)) for i in range(parts)]
    c = M.lincomb(terms)
    for k in range(L):
        if 2 ** (k + 1) <= c[k].shape[2]:
            m = c[k].reshape(2 ** (k + 1), -1)
            c[k], c[k + 1] = np.eye(len(m)).reshape(-1, 2, len(m)), np.einsum("ab,bsc->asc", m, c[k + 1])
    for k in range(L - 1, 0, -1):
        if 2 ** (L - k) <= c[k].shape[0]:
            m = c[k].reshape(c[k].shape[0], -1)
            c[k], c[k - 1] = np.eye(m.shape[1]).reshape(m.shape[1], 2, -1), np.einsum("asb,bc->asc", c[k - 1], m)
    return c


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_untruncated_shift(tl, axis):
    """A shift of a 64^3 population without truncation: centre matrices of 90 x 180 whose
    singular values go down to rounding.  Four products a site (R W, QR, X V, Q U S) of
    sums of at most 180 terms leave sqrt(4 L 180) u of the largest value; the largest of 2^18
    cells is allowed half as much again."""
    L, bond = 18, 45
    x = population(L, bond, 11)
    X = tl.DeviceMps.from_cores(x, bond, tl.nat.FP64)
    dst = tl.DeviceMps(L, 2 * bond, tl.nat.FP64)
    tl.lincomb_round([[tl.shift(X, axis, 1)]], [dst], 2 * bond, 1e-16)
    got = q.decode(M.to_tensor([np.asarray(c) for c in dst.cores()]))
    ref = np.roll(q.decode(M.to_tensor(x)), -1, axis)
    assert np.abs(got - ref).max() <= 1.5 * np.sqrt(4 * L * 4 * bond) * U * np.abs(ref).max()


def isometries(L, k, sig, r1, rng):
    """Cores of an MPS that is an isometry on both sides of bond k, the singular values sig
    there and a bond of r1 to its right; and the 2^(L-k) rows of their right vectors."""
    r = len(sig)
    bonds = [min(2 ** j, r) for j in range(k + 1)] + [min(2 ** (L - j), r1) for j in range(k + 1, L + 1)]
    orth = lambda m, n: np.linalg.qr(rng.standard_normal((m, n)))[0]
    cores = [orth(bonds[j] * 2, bonds[j + 1]).reshape(bonds[j], 2, bonds[j + 1]) for j in range(k)]
    cores += [orth(2 * bonds[j + 1], bonds[j]).T.reshape(bonds[j], 2, bonds[j + 1]) for j in range(k, L)]
    rows = right_rows(cores[k:])
    cores[k] = cores[k] * sig[:, None, None]
    return cores, rows


def right_rows(cores):
    right = np.ones((1, 1))
    for c in reversed(cores):
        right = np.einsum("asb,bq->asq", c, right).reshape(c.shape[0], -1)
    return right


# r columns of 2 r1 entries: as many rows as columns (V is the result) and fewer (W is)
@pytest.mark.parametrize("r,r1,chi", [(120, 60, 60), (100, 62, 62), (64, 32, 32), (100, 50, 50)])
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_small_directions(tl, r, r1, chi, seed):
    """Ten decades of singular values cut at chi: the kept directions against the discarded ones.
    The rows of the centre matrix are graded as the singular values are, so its
    rounding turns a pair by ~u sqrt(n) (1 / q - q)^-1, q the ratio of neighbours, and the
    sweeps' own tolerance, 16 * 2 u sqrt(n) of a pair's cosine, by as much as that."""
    L, k = 15, 7
    rng = np.random.default_rng(100 * r + seed)
    sig = 10.0 ** (-10.0 * np.arange(r) / (r - 1))
    cores, rows = isometries(L, k, sig, r1, rng)
    X = tl.DeviceMps.from_cores(cores, r, tl.nat.FP64)
    dst = tl.DeviceMps(L, chi, tl.nat.FP64)
    tl.lincomb_round([[tl.plain(X)]], [dst], chi, 1e-14)
    got = right_rows([np.asarray(c) for c in dst.cores()][k:])
    assert got.shape[0] == chi
    ratio = sig[1] / sig[0]
    assert np.abs(got @ rows[chi:].T).max() <= 32 * U * np.sqrt(2 * r1) / (1 / ratio - ratio)


def close_values(tl, r, r1, chi, width, gap, seed):
    """The largest part of a kept direction along a discarded one, where the cut at chi lies in the
    middle of `width` singular values of relative distance gap."""
    L, k = 15, 7
    rng = np.random.default_rng(1000 * r + seed)
    sig = 10.0 ** (-np.arange(r) / (r - 1))
    sig[chi - width // 2:chi + width // 2] = sig[chi] * (1.0 - gap * np.arange(width))
    cores, rows = isometries(L, k, sig, r1, rng)
    mix = np.linalg.qr(rng.standard_normal((r, r)))[0]
    cores[k] = np.einsum("ab,bsc->asc", mix, cores[k])
    X = tl.DeviceMps.from_cores(cores, r, tl.nat.FP64)
    dst = tl.DeviceMps(L, chi, tl.nat.FP64)
    tl.lincomb_round([[tl.plain(X)]], [dst], chi, 1e-14)
    got = right_rows([np.asarray(c) for c in dst.cores()][k:])
    return np.abs(got @ rows[chi:].T).max()


# The sweeps' tolerance of a pair's cosine, 16 * 2 u sqrt(n), and the centre matrix's rounding, four
# products of sums of n terms at s_0 / s_chi <= 4, over the difference of the pair's squares:
def close_bound(r1, gap):
    return (32 + 4 * 4) * U * np.sqrt(2 * r1) / (2 * gap)


# fewer rows than columns: the sweeps finish what the refinement leaves of close values
@pytest.mark.parametrize("r,r1,chi", [(100, 62, 62), (60, 40, 40)])
@pytest.mark.parametrize("seed", [0, 1, 2, 3])
def test_sweeps_of_close_values(tl, r, r1, chi, seed):
    assert close_values(tl, r, r1, chi, 8, 1e-9, seed) <= close_bound(r1, 1e-9)


# as many rows as columns: the refinement may leave close values as they are, but not across the cut
@pytest.mark.parametrize("r,r1,chi", [(64, 32, 32), (120, 60, 60)])
@pytest.mark.parametrize("width,gap", [(2, 1e-7), (2, 1e-9), (8, 1e-9), (24, 1e-7)])
@pytest.mark.parametrize("seed", [0, 1, 2, 3])
def test_cut_between_close_values(tl, r, r1, chi, width, gap, seed):
    assert close_values(tl, r, r1, chi, width, gap, seed) <= close_bound(r1, gap)
