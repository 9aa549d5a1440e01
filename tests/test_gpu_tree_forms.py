"""The tree stages take their form from the size of the whole context: one
block orders the nodes of a small one, a radix pass those of a large one, and
a leaf's moments are formed by eight lanes or by one thread.  A disk's forces,
candidates and counts have the same bits alone and beside a larger system."""
import numpy as np
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _step(P, s, seg, leaf, precision):
    n = len(s["m"])
    ctx = P.p3t_create(P.Params(leaf_size=leaf, precision=precision), 0)
    try:
        if seg is not None:
            P.p3t_set_segments(ctx, seg)
        P.p3t_reserve(ctx, n)
        st = P.State.from_numpy(s)
        P.p3t_cutoffs(ctx, st)
        P.p3t_build_tree(ctx, st)
        acc = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
        P.p3t_soft_force(ctx, st, acc, cnt)
        assert P.p3t_status(ctx)[0] == 0
        return acc.cpu().numpy(), cnt.cpu().numpy(), P.p3t_tree_stats(ctx)
    finally:
        P.p3t_destroy(ctx)


# 250,000 others have more leaves than eight lanes each take (some 19,000), and
# any number of nodes above a block's; n crosses a leaf, a tile of 256, and
# (leaf 1 at 600, leaf 16 at 6,000) a block's node capacity
@pytest.mark.parametrize("precision", ["P3T_FP64", "P3T_MIXED"])
@pytest.mark.parametrize("n,leaf", [(1, 16), (2, 1), (9, 8), (17, 16), (33, 32), (257, 16),
                                    (600, 1), (3001, 16), (6000, 16)])
def test_forms_agree(n, leaf, precision):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    prec = getattr(P, precision)
    a = disks.equal_mass_narrow(n, seed=n, planted=False)
    b = disks.equal_mass_ring(250_000, seed=5)
    alone = _step(P, a, None, leaf, prec)
    other = _step(P, b, None, leaf, prec)
    both = _step(P, {k: np.concatenate([a[k], b[k]]) for k in disks.KEYS},
                 [0, n, n + 250_000], leaf, prec)
    assert np.array_equal(both[0][:, :n], alone[0])
    assert np.array_equal(both[0][:, n:], other[0])
    assert np.array_equal(both[1], alone[1] + other[1])
    assert both[2]["n_nodes"] == alone[2]["n_nodes"] + other[2]["n_nodes"]
    assert both[2]["n_leaves"] == alone[2]["n_leaves"] + other[2]["n_leaves"]
