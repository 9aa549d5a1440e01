"""The FP64 walks take their targets in chunks whose size follows the size of
the whole system: a disk's forces and interaction counts have the same bits
whatever the chunk, and its tree VJP the same values to rounding."""
import numpy as np
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _eval(P, s, seg, group, theta):
    n = len(s["m"])
    ctx = P.p3t_create(P.Params(theta=theta, group_size=group, precision=P.P3T_FP64), 0)
    try:
        if seg is not None:
            P.p3t_set_segments(ctx, seg)
        P.p3t_reserve(ctx, n)
        st = P.State.from_numpy(s)
        P.p3t_cutoffs(ctx, st)
        P.p3t_build_tree(ctx, st)
        f64 = dict(dtype=torch.float64, device="cuda")
        acc, cnt = torch.zeros(3, n, **f64), torch.zeros(2, dtype=torch.int64, device="cuda")
        P.p3t_soft_force(ctx, st, acc, cnt)
        gx, gm = torch.zeros(3, n, **f64), torch.zeros(n, **f64)
        P.p3t_soft_force_vjp_tree(ctx, st, 0.5, acc / acc.abs().max(), gx, gm)
        assert P.p3t_status(ctx)[0] == 0
        return acc.cpu().numpy(), cnt.cpu().numpy(), gx.cpu().numpy(), gm.cpu().numpy()
    finally:
        P.p3t_destroy(ctx)


# alone 1, 31, 33 or 700 particles take single targets; beside 40,000 or
# 90,000 others (a system of its own) chunks of four and eight
@pytest.mark.parametrize("n", [1, 31, 33, 700])
@pytest.mark.parametrize("other,group,theta", [(40_000, 64, 0.5), (90_000, 20, 0.5),
                                               (90_000, 0, 0.0)])
def test_forces_do_not_depend_on_the_chunk(n, other, group, theta):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    if theta == 0.0:
        other = min(other, 20_000)  # the other system's pairs count too
    s = disks.equal_mass_narrow(n, seed=n, planted=False)
    if n == 700:  # an oversized leaf: 70 bodies at one place
        for k in ("x", "y", "z"):
            s[k][100:170] = s[k][100]
    o = disks.equal_mass_ring(other, seed=3)
    both = {k: np.concatenate([s[k], o[k]]) for k in disks.KEYS}
    a, ca, gxa, gma = _eval(P, s, None, group, theta)
    b, cb, gxb, gmb = _eval(P, both, [0, n, n + other], group, theta)
    assert np.array_equal(a, b[:, :n])
    assert np.all(cb >= ca)
    if n > 1:
        # the scale of lam differs between the two calls
        f = np.abs(a).max() / np.abs(b).max()
        assert np.abs(gxa * f - gxb[:, :n]).max() <= 1e-11 * np.abs(gxb[:, :n]).max()
        assert np.abs(gma * f - gmb[:n]).max() <= 1e-11 * np.abs(gmb[:n]).max()
