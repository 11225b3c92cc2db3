"""FP64-accurate centre SVDs at the edges of their paths, in mixed precision and FP64,
against the dense FP64 sums: few columns (the leader's sweeps up to 16 of them, 5 in
mixed precision), one size within a CTA's registers, and beyond them the FP32
sweeps over the cluster (ncol just above 128, odd counts, up to 256; columns up to 256
and up to 512 entries) and the sizes past those."""
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


def flat_field(cores):
    """The field in site order, in 64 bits."""
    left = np.ones((1, 1))
    for c in cores[:len(cores) // 2]:
        left = np.einsum("la,asb->lsb", left, c).reshape(-1, c.shape[2])
    right = np.ones((1, 1))
    for c in cores[:len(cores) // 2 - 1:-1]:
        right = np.einsum("asb,bq->asq", c, right).reshape(c.shape[0], -1)
    return (left @ right).reshape(-1)


# centre matrices at the widest bond: (sum of the operands' bonds) x 2 chi
@pytest.mark.parametrize("bond,chi,terms", [(2, 2, 2), (3, 3, 2), (8, 8, 2), (9, 9, 2), (45, 90, 2), (65, 65, 2), (67, 67, 2), (100, 100, 2), (128, 128, 2), (70, 140, 2),
                                            (90, 128, 3), (50, 200, 2), (90, 140, 3)])
@pytest.mark.parametrize("prec", [0, 3])
def test_rounded_sum(tl, bond, chi, terms, prec):
    n, L = 6, 18
    dt = np.float64 if prec == 0 else np.float32
    prec = tl.nat.FP64 if prec == 0 else tl.nat.MIXED
    ops = []
    for t in range(terms):
        c = synth.random_mps(L, synth.feasible_ranks(L, bond), 1000 * terms + 10 * bond + t)
        # bonds whose singular values fall over six decades, as those of smooth fields do
        for k in range(L - 1):
            c[k] = c[k] * 10.0 ** (-6.0 * np.arange(c[k].shape[2]) / c[k].shape[2])
        ops.append([x.astype(dt).astype(np.float64) for x in c])
    coef = [1.0, -0.43, 0.7][:terms]
    dst = tl.DeviceMps(L, chi, prec)
    tl.lincomb_round([[tl.plain(device(tl, o, bond, prec), a) for o, a in zip(ops, coef)]], [dst], chi,
                     1e-10 if dt == np.float64 else 1e-7)
    ref = sum(a * flat_field(o) for o, a in zip(ops, coef))
    got = [np.asarray(c, dtype=np.float64) for c in dst.cores()]
    norm = np.linalg.norm(ref)
    # right-orthonormal cores, up to their storage's rounding
    for c in got[1:]:
        m = c.reshape(c.shape[0], -1)
        assert np.abs(m @ m.T - np.eye(m.shape[0])).max() <= (1e-12 if dt == np.float64 else 3e-6)
    tails = 0.0
    for k in range(1, L):
        m = ref.reshape(2 ** k, -1)
        tails += (np.linalg.svd(m, compute_uv=False)[chi:] ** 2).sum()
    eps = 1e-10 if dt == np.float64 else 1e-7
    # the discarded part, the truncation tolerance, and the storage's rounding over L cores
    tol = np.sqrt(tails) * (1 + 1e-6) + eps * norm + (1e-13 if dt == np.float64 else 1e-6 * L) * norm
    assert np.linalg.norm(flat_field(got) - ref) <= tol
