"""Members of neighbour clusters close to percolation: in index order at the
sizes where their sort changes form (a warp's 32 and 256, a block's 8,192, the
slices above), and in a time that does not grow with the clusters' number and
size beyond what the same particles cost in small clusters."""
import numpy as np
import pytest
import torch

from tests.gpu_util import need_gpu
from tests.test_gpu_cluster_members import test_members_in_index_order as members_in_index_order

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(31, 32, 33, 255, 256, 257), (8191, 8192, 8193),
                                   (8193, 9000, 40_000, 5, 600), (33,) * 300 + (300,) * 90,
                                   (8200,) * 12])
@pytest.mark.parametrize("singles", [0, 1030])
def test_members_in_index_order_near_percolation(sizes, singles):
    members_in_index_order(sizes, singles)


def _neighbours_us(P, n, size, count):
    """Shortest time of the neighbour and cluster stage: `count` chains of
    `size` bodies, in random order, the other bodies apart."""
    rs, rng = 1e-6, np.random.default_rng(1)
    k = np.arange(n)
    on = k < size * count
    x = np.where(on, 1.0 + 0.9 * rs * (k % size), rng.uniform(1.0, 2.0, n))
    y = np.where(on, 1e-3 * (k // size), rng.uniform(0.0, 1.0, n))
    p, o = rng.permutation(n), np.zeros(n)
    s = dict(x=x[p], y=y[p], z=np.where(on, 0.0, 1.0)[p], vx=o, vy=o, vz=o, m=np.full(n, 1e-12))
    st = P.State.from_numpy(s, r_out=np.full(n, rs / 2), r_search=np.full(n, rs))
    ctx = P.p3t_create(P.Params(theta=0.7, group_size=64), 0)
    try:
        P.p3t_reserve(ctx, n)
        P.p3t_build_tree(ctx, st)
        P.p3t_soft_force(ctx, st, torch.zeros(3, n, dtype=torch.float64, device="cuda"))
        off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        idx = torch.zeros(4 * n, dtype=torch.int32, device="cuda")
        best = np.inf
        for _ in range(8):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            P.p3t_neighbours(ctx, st, off, idx)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * e[0].elapsed_time(e[1]))
        assert P.p3t_status(ctx)[0] == 0
        return best
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("size,count", [(40, 2000), (300, 300), (1030, 87), (9000, 10)])
def test_no_slower_near_percolation(size, count):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    # the same neighbour pairs in chains of nine; 10 to 40 times that when one
    # block took the large clusters one after another.  Four: the union-find of
    # long chains alone takes up to 1.7 times that of short ones
    assert _neighbours_us(P, 100_000, size, count) <= 4 * _neighbours_us(P, 100_000, 9, 10_000)
