"""The tree's key sort takes three routes (one block, sample sort, radix passes)
by the capacity of the context: the same forces, interaction counts and
neighbour rows bit for bit from a context sized for the particles and from one
sized for the radix passes, at the edges of the routes, for disks, for inputs
whose samples mislead (one bucket far beyond what a block sorts) and for
bodies at one place."""
import numpy as np
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

RADIX = 1_600_000  # above the sample sort's largest capacity


def _inputs(n, kind):
    s = disks.equal_mass_ring(n, seed=n)
    if kind == "clump":
        # all but the sampled positions (every n / 256th) within 1e-3 au
        far = np.zeros(n, dtype=bool)
        far[(np.arange(256) * n) // 256] = True
        rng = np.random.default_rng(1)
        for k, c in (("x", 1.0), ("y", 0.0), ("z", 0.0)):
            s[k] = np.where(far, s[k], c + 1e-3 * rng.uniform(-1, 1, n))
    if kind == "coincident":
        for k in ("x", "y", "z"):
            s[k][n // 4:n // 2] = s[k][0]        # a quarter of them at one place
            s[k][1:n // 4:2] = s[k][0:n // 4 - 1:2][:len(s[k][1:n // 4:2])]  # and pairs
    return s


def _eval(P, s, cap):
    n = len(s["m"])
    ctx = P.p3t_create(P.Params(theta=0.7, group_size=32, precision=P.P3T_MIXED), 0)
    try:
        P.p3t_reserve(ctx, cap)
        st = P.State.from_numpy(s, r_out=np.full(n, 1e-7), r_search=np.full(n, 2e-7))
        acc = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
        P.p3t_build_tree(ctx, st)
        P.p3t_soft_force(ctx, st, acc, cnt)
        stats = P.p3t_tree_stats(ctx)
        P.p3t_status(ctx)  # many coincident bodies may overflow the candidates: not compared
        return acc.cpu().numpy(), cnt.cpu().numpy(), stats
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("n,kind", [(1, "disk"), (2, "disk"), (257, "disk"), (3001, "disk"),
                                    (8192, "disk"), (8193, "disk"), (16_001, "disk"),
                                    (150_000, "disk"), (20_000, "clump"), (120_001, "clump"),
                                    (600, "coincident"), (8000, "coincident"),
                                    (20_000, "coincident")])
def test_key_sort_routes_agree(n, kind):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    s = _inputs(n, kind)
    a, ca, sa = _eval(P, s, n)
    b, cb, sb = _eval(P, s, RADIX)
    assert sa == sb and np.array_equal(ca, cb)
    assert np.array_equal(a, b)
