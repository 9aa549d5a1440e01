"""FP64 pair sums at distances whose square or inverse cube leaves the range of
a double, and bodies without a finite place.  Two bodies inside gamma times
their cut-off radius add nothing to each other's force however near they are;
a pair so far apart that r^2 is infinite, and a body at NaN or infinity, adds
nothing to the others' forces and an infinitely far one none to the energy."""
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


def _sums(P, s, ro, tree):
    n = len(s["m"])
    st = P.State.from_numpy(s, r_out=ro, r_search=ro)
    lam = torch.as_tensor(np.random.default_rng(4).normal(size=(3, n))).cuda()
    f64 = dict(dtype=torch.float64, device="cuda")
    acc, gx, gm, e = (torch.zeros(3, n, **f64), torch.zeros(3, n, **f64), torch.zeros(n, **f64),
                      torch.zeros(4, **f64))
    ctx = P.p3t_create(P.Params(theta=0.0, precision=P.P3T_FP64), 0)
    try:
        if tree:
            P.p3t_reserve(ctx, n)
            P.p3t_build_tree(ctx, st)
            P.p3t_soft_force_vjp_tree(ctx, st, 1.0, lam, gx, gm)
        else:
            P.p3t_soft_force_direct(ctx, st, acc)
            P.p3t_soft_force_vjp(ctx, st, 1.0, lam, gx, gm)
        P.p3t_energy(ctx, st, e)
        assert P.p3t_status(ctx)[0] == 0
        return [t.cpu().numpy() for t in (acc, gx, gm, e)]
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("tree", [False, True])
@pytest.mark.parametrize("n", [65, 300])
@pytest.mark.parametrize("gap", [1e-104, 1e-140, 1e-156])
def test_bodies_at_almost_one_place(P, tree, n, gap):
    s = disks.equal_mass_ring(n, seed=n)
    ro = np.full(n, 1e-2)
    for k in ("x", "y", "z"):
        s[k][0] = s[k][n // 2] = 0.0  # all others at 1 au: beyond every radius
    base = _sums(P, s, ro, tree)
    s["x"][0] = gap
    near = _sums(P, s, ro, tree)
    for a, b in zip(base[:3], near[:3]):
        # the same sums (the gap is far below the others' distances' rounding),
        # the tree VJP's to the rounding of its atomic additions
        tol = 1e-12 * np.abs(a).max() if tree else 0.0
        assert np.isfinite(b).all() and np.abs(a - b).max() <= tol
    want = -s["m"][0] * s["m"][n // 2] / gap
    assert abs(near[3][3] - want) <= 1e-9 * abs(want)


@pytest.mark.parametrize("far", [1e155, 1e200])
@pytest.mark.parametrize("n", [65, 300])
def test_bodies_beyond_the_range_of_squares(P, n, far):
    s = disks.equal_mass_ring(n, seed=n)
    ro = np.full(n, 1e-2)
    keep = np.arange(n) != n // 2
    base = _sums(P, {k: s[k][keep] for k in s}, ro[keep], False)
    s["y"][n // 2] = far
    got = _sums(P, s, ro, False)
    # the body itself feels nothing, the others feel nothing of it (the split of
    # the sources may reorder their sums: n additions' rounding of some 30 times
    # the largest sum's terms)
    assert np.all(got[0][:, n // 2] == 0.0)
    assert np.abs(got[0][:, keep] - base[0]).max() <= 1e-12 * np.abs(base[0]).max()
    assert np.isfinite(got[1]).all() and np.isfinite(got[2]).all()
    assert abs(got[3][3] - base[3][3]) <= 1e-13 * abs(base[3][3])


@pytest.mark.parametrize("where", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n", [65, 300])
def test_bodies_without_a_place_add_no_force(P, n, where):
    s = disks.equal_mass_ring(n, seed=n)
    ro = np.full(n, 1e-2)
    keep = np.arange(n) != n // 2
    base = _sums(P, {k: s[k][keep] for k in s}, ro[keep], False)[0]
    s["z"][n // 2] = where
    acc = _sums(P, s, ro, False)[0]
    assert np.all(acc[:, n // 2] == 0.0)
    assert np.abs(acc[:, keep] - base).max() <= 1e-12 * np.abs(base).max()
