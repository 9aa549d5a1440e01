"""The mixed walk's units of work: whatever the number of its warps, and so the
groups whose rests follow their first 32 targets at once, every target is
walked once, with the same bits and interaction counts."""
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


# groups of more than 32: fewer than the warps of one block an SM (31,000), some
# (60,000) and many times more than those of any grid (400,000)
@pytest.mark.parametrize("n", [31_000, 60_000, 400_000])
def test_units_cover_every_target(n):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    ctx = P.p3t_create(P.Params(theta=0.7, group_size=64, precision=P.P3T_MIXED), 0)
    try:
        P.p3t_reserve(ctx, n)
        st = P.State.from_numpy(disks.wide_power_law(n, seed=n))
        P.p3t_cutoffs(ctx, st)
        P.p3t_build_tree(ctx, st)
        out = []
        for blocks in (1, 2, 3, 6):
            P.p3t_set_tuning(ctx, 8, blocks)
            acc = torch.full((3, n), float("nan"), dtype=torch.float64, device="cuda")
            cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
            P.p3t_soft_force(ctx, st, acc, cnt)
            out.append((acc, cnt))
        assert P.p3t_status(ctx)[0] == 0
    finally:
        P.p3t_destroy(ctx)
    assert torch.isfinite(out[0][0]).all() and (out[0][1] > 0).all()
    for acc, cnt in out[1:]:
        assert torch.equal(acc, out[0][0]) and torch.equal(cnt, out[0][1])
