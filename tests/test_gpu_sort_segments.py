"""Several systems in one context: a block sorts each system's keys when none is
above its limit, otherwise one sort of all is followed by a pass by system.
Every system's forces, candidates and nodes have the bits it has alone."""
import numpy as np
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _disk(n, coincident):
    s = disks.equal_mass_narrow(n, seed=n, planted=False)
    s = {k: s[k].copy() for k in disks.KEYS}
    if coincident and n > 8:
        for k in ("x", "y", "z"):
            s[k][n // 4:n // 2] = s[k][0]
    return s


def _eval(P, s, seg, precision):
    n = len(s["m"])
    ctx = P.p3t_create(P.Params(theta=0.7, group_size=32, precision=precision), 0)
    try:
        if seg is not None:
            P.p3t_set_segments(ctx, seg)
        P.p3t_reserve(ctx, n)
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


# 8,192 entries a run, 16,384 a block's limit; 16,385 sends all to the one sort
@pytest.mark.parametrize("sizes", [(1, 5, 31, 33), (8192, 1, 8193), (16384, 700, 9001, 16383),
                                   (16385, 700, 8193)])
@pytest.mark.parametrize("coincident", [False, True])
@pytest.mark.parametrize("precision", [0, 1])
def test_systems_keep_their_bits(sizes, coincident, precision):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    ds = [_disk(n, coincident and n < 1000) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)])
    both = _eval(P, {k: np.concatenate([d[k] for d in ds]) for k in disks.KEYS}, off, precision)
    counts, nodes = np.zeros(2, dtype=np.int64), 0
    for d, a, b in zip(ds, off[:-1], off[1:]):
        one = _eval(P, d, None, precision)
        assert np.array_equal(both[0][:, a:b], one[0])
        counts += one[1]
        nodes += one[2]["n_nodes"]
    assert np.array_equal(both[1], counts) and both[2]["n_nodes"] == nodes
