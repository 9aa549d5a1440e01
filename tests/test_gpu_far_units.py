"""The FP64 walks' far test in units of length far from one: lengths times a
power of two leave every decision of the walk and every mantissa as they are, so
forces and neighbour rows are those of the unscaled disk bit for bit, and the
tree VJP the same to the rounding of its atomic sums."""
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


def _eval(P, power):
    n, f = 3000, 2.0 ** power
    s = disks.equal_mass_ring(n, seed=5)
    s = {k: s[k] * (f if k in "xyz" else 1.0) for k in s}
    ro = np.random.default_rng(n).uniform(2e-3, 2e-2, n) * f
    st = P.State.from_numpy(s, r_out=ro, r_search=1.2 * ro)
    lam = torch.as_tensor(np.random.default_rng(1).normal(size=(3, n))).cuda()
    f64 = dict(dtype=torch.float64, device="cuda")
    ctx = P.p3t_create(P.Params(theta=0.5, group_size=64, precision=P.P3T_FP64), 0)
    try:
        P.p3t_reserve(ctx, n)
        P.p3t_build_tree(ctx, st)
        acc, cnt = torch.zeros(3, n, **f64), torch.zeros(2, dtype=torch.int64, device="cuda")
        P.p3t_soft_force(ctx, st, acc, cnt)
        off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        idx = torch.zeros(64 * n, dtype=torch.int32, device="cuda")
        P.p3t_neighbours(ctx, st, off, idx)
        gx, gm = torch.zeros(3, n, **f64), torch.zeros(n, **f64)
        P.p3t_soft_force_vjp_tree(ctx, st, 1.0, lam, gx, gm)
        assert P.p3t_status(ctx)[0] == 0
        return (acc.cpu().numpy() * f ** 2, cnt.cpu().numpy(), off.cpu().numpy(),
                idx[:int(off[-1])].cpu().numpy(), gx.cpu().numpy() * f ** 3,
                gm.cpu().numpy() * f ** 2)
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("power", [83, 72, 64, 60, -60])  # reaches of 1e23 down to 1e-20
def test_forces_and_rows_in_any_unit_of_length(P, power):
    a, b = _eval(P, 0), _eval(P, power)
    assert a[3].size > 3000
    for q in range(4):
        assert np.array_equal(a[q], b[q])
    for q in (4, 5):
        assert np.abs(a[q] - b[q]).max() <= 1e-11 * np.abs(a[q]).max()
