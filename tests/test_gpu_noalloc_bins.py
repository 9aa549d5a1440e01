"""The allocation-free cut-offs form a bin's v_ran once or per particle by the
particles a bin: both sides of that line agree with the context's path, and many
bins of few particles cost no more than few bins."""
import numpy as np
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t
    return p3t


@pytest.mark.parametrize("n,bins", [(1, 1), (255, 1), (256, 1), (1023, 4), (1024, 4), (1025, 4),
                                    (1000, 4096), (70_000, 273), (70_000, 274)])
def test_radii_on_both_sides_of_the_line(P, n, bins):
    s = disks.equal_mass_ring(n, seed=n)
    prm = P.Params(vran_bins=bins)
    a, b = P.State.from_numpy(s), P.State.from_numpy(s)
    P.p3t_cutoffs_noalloc(prm, a)
    ctx = P.p3t_create(prm, 0)
    try:
        P.p3t_cutoffs(ctx, b)
        torch.cuda.synchronize()
        assert P.p3t_status(ctx)[0] == 0
    finally:
        P.p3t_destroy(ctx)
    # the bins' sums: exact in one, in index order in FP64 in the other
    for p, q in ((a.r_out, b.r_out), (a.r_search, b.r_search)):
        p, q = p.cpu().numpy(), q.cpu().numpy()
        assert np.all(q > 0.0) and np.abs(p / q - 1.0).max() <= 1e-13


def test_many_bins_of_few_particles_cost_no_more(P):
    def us(bins):
        st = P.State.from_numpy(disks.equal_mass_ring(1000, seed=1))
        prm, best = P.Params(vran_bins=bins), np.inf
        for _ in range(30):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(8):
                P.p3t_cutoffs_noalloc(prm, st)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best
    # 2.2 times when one block formed all bins' v_ran
    assert us(4096) <= 1.6 * us(256)
