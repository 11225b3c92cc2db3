"""Scratch of a rounding launch that runs one CTA a job: none for the refinement, which clusters
alone do."""
import threading

import pytest

import synth

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


def peak(tl, prec, jobs, bond):
    """Most device memory in use while `jobs` sums of two MPS are rounded, above that before."""
    import torch
    L = 12
    x = tl.DeviceMps.from_cores(synth.random_mps(L, synth.feasible_ranks(L, bond), 3), bond, prec)
    dst = [tl.DeviceMps(L, bond, prec) for _ in range(jobs)]
    run = lambda: tl.lincomb_round([[tl.plain(x), tl.plain(x, -0.5)]] * jobs, dst, bond, 1e-7)
    run()                                            # modules and tables of the first call
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    worker = threading.Thread(target=run)
    worker.start()
    low = before
    while worker.is_alive():
        low = min(low, torch.cuda.mem_get_info()[0])
    worker.join()
    return before - low


def test_scratch_of_single_cta_jobs(tl):
    """160 jobs leave no room for clusters.  Mixed precision then needs the FP64 Jacobi matrices beyond what
    FP32 does, by the bonds' capacities 128 columns of 128 and of 128 entries, two apart from each
    other's banks (a quarter more and 16 MB for alignment and granularity are allowed); the
    rotations' log alone would be four times as much."""
    jobs = 160
    extra = peak(tl, tl.nat.MIXED, jobs, 64) - peak(tl, tl.nat.FP32, jobs, 64)
    assert extra <= 1.25 * jobs * 8 * 2 * 128 * 130 + 16 * 2 ** 20
