"""Members of neighbour clusters in index order at the sizes where their sort
changes form: a thread's eight, a block's 1,024 and the listing above."""
import numpy as np
import pytest
import torch

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [(2,), (2, 3, 7, 8, 9), (2, 8, 9, 33, 300, 1023, 1024, 1025),
                                   (2048, 2049, 5000), (2,) * 700 + (9,) * 20])
@pytest.mark.parametrize("singles", [0, 513])
def test_members_in_index_order(sizes, singles):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    # clusters are chains with links below the search radius, far apart
    rs = 1e-5
    x, cl = [], []
    for c, m in enumerate(sizes):
        x.append(1.0 + 0.9 * rs * np.arange(m))
        cl.append(np.full(m, c))
    x.append(np.full(singles, 2.0))
    cl.append(len(sizes) + np.arange(singles))
    x, cl = np.concatenate(x), np.concatenate(cl)
    n = len(x)
    perm = np.random.default_rng(n).permutation(n)
    x, cl = x[perm], cl[perm]
    z = np.zeros(n)
    s = dict(x=x, y=1e-3 * cl, z=z, vx=z, vy=z, vz=z, m=np.full(n, 1e-12))
    st = P.State.from_numpy(s, r_out=np.full(n, rs / 2), r_search=np.full(n, rs))
    ctx = P.p3t_create(P.Params(precision=P.P3T_FP64), 0)
    try:
        P.p3t_reserve(ctx, n)
        P.p3t_build_tree(ctx, st)
        acc = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        P.p3t_soft_force(ctx, st, acc)
        off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        idx = torch.zeros(4 * n + 64, dtype=torch.int32, device="cuda")
        t = P.p3t_copy_clusters(ctx, P.p3t_neighbours(ctx, st, off, idx), n)
        torch.cuda.synchronize()
        assert P.p3t_status(ctx)[0] == 0
    finally:
        P.p3t_destroy(ctx)
    counts = t["counts"].cpu().numpy()
    assert list(counts) == [singles, len(sizes), sum(sizes), max(sizes)]
    # clusters by their smallest member, members ascending
    want = sorted((np.flatnonzero(cl == c) for c in range(len(sizes))), key=lambda m: m[0])
    o = t["cl_off"].cpu().numpy()[:len(sizes) + 1]
    assert np.array_equal(o, np.concatenate([[0], np.cumsum([len(m) for m in want])]))
    assert np.array_equal(t["cl_mem"].cpu().numpy()[:sum(sizes)], np.concatenate(want))
    assert np.array_equal(np.sort(t["singles"].cpu().numpy()[:singles]),
                          np.flatnonzero(cl >= len(sizes)))
