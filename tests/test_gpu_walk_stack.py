"""The walk's stack: a tree whose frontier is far wider than any disk's (cubes of
bodies nested at seven scales, walked to the leaves) gives the forces of the
all-pairs kernels, and a context for a few thousand bodies stays small."""
import numpy as np
import pytest
import torch

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t
    return p3t


@pytest.mark.parametrize("precision,tol", [(0, 1.2e-13), (1, 5e-6)])
@pytest.mark.parametrize("scale_bodies", [4300, 4500])  # a small context and a large one
def test_wide_and_deep_tree(P, scale_bodies, precision, tol):
    # cubes of bodies at scales of 8^-k, all with one corner in common: the last
    # one that a walk reaches first, so that every level waits with some 100 nodes
    # (2,490 in all with rounds of 32)
    rng = np.random.default_rng(1)
    x = np.concatenate([-rng.uniform(0.0, 1.0, (scale_bodies, 3)) * 8.0 ** -k for k in range(7)])
    n = len(x)
    z = np.zeros(n)
    s = dict(x=x[:, 0], y=x[:, 1], z=x[:, 2], vx=z, vy=z, vz=z, m=np.full(n, 1e-9))
    # no cut-off, so that the sums are plain: r_out far below every distance
    st = P.State.from_numpy(s, r_out=np.full(n, 1e-12), r_search=np.full(n, 1e-12))
    f64 = dict(dtype=torch.float64, device="cuda")
    acc, ref = torch.zeros(3, n, **f64), torch.zeros(3, n, **f64)
    ctx = P.p3t_create(P.Params(theta=0.0, leaf_size=4, group_size=64, precision=precision), 0)
    try:
        P.p3t_reserve(ctx, n)
        P.p3t_build_tree(ctx, st)
        assert P.p3t_tree_stats(ctx)["depth"] >= 18
        P.p3t_soft_force(ctx, st, acc)
        P.p3t_soft_force_direct(ctx, st, ref)
        assert P.p3t_status(ctx)[0] == 0
    finally:
        P.p3t_destroy(ctx)
    # either kernel: a term's error, a few roundings of its magnitude (see
    # test_gpu_all_pairs), and the sums', n / 32 roundings in FP64 and 32 in FP32
    q, mag = torch.as_tensor(x).cuda(), []
    for i in range(0, n, 500):
        d2 = ((q[i:i + 500, None] - q[None]) ** 2).sum(2)
        d2[d2 == 0.0] = np.inf
        mag.append((1e-9 / d2).sum(1))
    assert bool(((acc - ref).abs() <= 2 * tol * torch.cat(mag)).all())


@pytest.mark.parametrize("n,most", [(1000, 9e6), (5000, 64e6)])
def test_small_contexts_are_small(P, n, most):
    torch.zeros(1, device="cuda")
    ctx, before = [], torch.cuda.mem_get_info()[0]
    try:
        for _ in range(8):
            ctx.append(P.p3t_create(P.Params(group_size=64), 0))
            P.p3t_reserve(ctx[-1], n)
        used = (before - torch.cuda.mem_get_info()[0]) / 8
    finally:
        for c in ctx:
            P.p3t_destroy(c)
    # particle and node buffers of 2.5 and 8 MB, stacks of 4 and 48
    assert used <= most
