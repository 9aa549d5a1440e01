"""The backward pass takes the last segment from the forward pass and recomputes
the others up to their last drift: the gradients have the same bits (the
tree VJP adds atomically: the same to rounding) when every segment is
recomputed, and when one tape is used twice."""
import numpy as np
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("force,hard", [("direct", "kepler"), ("tree", "kepler"), ("tree", "p3t")])
@pytest.mark.parametrize("steps,checkpoint", [(1, 1), (3, 1), (4, 2), (5, 3), (3, 8)])
def test_kept_segment_equals_the_recomputed_one(force, hard, steps, checkpoint):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import adjoint as AD, p3t as P
    n = 600
    s = disks.adjoint_disk(n, 7, m=1e-7)
    x = torch.as_tensor(np.stack([s["x"], s["y"], s["z"]])).cuda()
    v = torch.as_tensor(np.stack([s["vx"], s["vy"], s["vz"]])).cuda()
    m = torch.as_tensor(s["m"]).cuda()
    prm = P.Params(group_size=64, precision=P.P3T_FP64)
    ro, rs = AD.cutoffs(prm, x, v, m, with_search=True)
    run = AD.SoftKDK(prm, n, steps, checkpoint, force=force, hard=hard)
    try:
        xn, vn, tape = run.forward(x, v, m, ro, rs)
        lx = torch.as_tensor(np.random.default_rng(1).normal(size=(3, n))).cuda()
        lv = torch.as_tensor(np.random.default_rng(2).normal(size=(3, n))).cuda()
        first = run.backward(tape, lx, lv)
        again = run.backward(tape, lx, lv)
        whole = run.backward(dict(tape, last=None), lx, lv)
        run.status()
    finally:
        run.close()
    for a, b, c in zip(first, again, whole):
        assert torch.isfinite(a).all() and a.abs().max() > 0.0
        # the tree VJP's atomic sums are not in a fixed order
        tol = 0.0 if force == "direct" else 1e-11 * float(a.abs().max())
        assert float((a - b).abs().max()) <= tol and float((a - c).abs().max()) <= tol
