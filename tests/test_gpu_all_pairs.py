"""The all-pairs kernels' far and near forms and the energy's tile pairs.

Direct force: every body's sum against NumPy, with bodies all far apart, all
within each other's cut-off radii, and half and half (chunks that switch from
one form to the other).  A term's error is a few rounding errors of its
Newtonian magnitude m / r^2 (the changeover weight's absolute error included:
|K' y| <= 2.5 times y's), so the bound is on |error| / sum m / r^2: 3e-6 in FP32
(24-bit terms, 8 to 10 roundings of 6e-8 in r^-3 and K), 1e-14 in FP64.

Energy: the pair sum against NumPy at the edges of the 256-body tiles; FP32
terms 1e-6 relative, FP64 1e-13; two bodies at one place give minus infinity
in FP64 and no term in the mixed path."""
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


def _state(kind, n):
    s = disks.equal_mass_ring(n, seed=n)
    if kind != "far":
        c = disks.clump(n, seed=2, size=2e-3)
        k = np.arange(n) >= (n // 2 if kind == "half" else 0)
        for q in ("x", "y", "z"):
            s[q] = np.where(k, c[q], s[q])
    return s


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind,n", [("far", 33), ("far", 700), ("near", 65), ("near", 700),
                                    ("half", 129), ("half", 700)])
def test_direct_far_and_near_forms(P, kind, n, precision):
    s = _state(kind, n)
    ro = np.random.default_rng(n).uniform(0.2e-3, 2e-3, n)
    st = P.State.from_numpy(s, r_out=ro, r_search=2 * ro)
    ctx = P.p3t_create(P.Params(precision=precision))
    try:
        acc = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        P.p3t_soft_force_direct(ctx, st, acc)
        assert P.p3t_status(ctx)[0] == 0
        a = acc.cpu().numpy()
    finally:
        P.p3t_destroy(ctx)
    x = np.stack([s["x"], s["y"], s["z"]])
    d = x[:, :, None] - x[:, None, :]
    r = np.sqrt((d * d).sum(0))
    np.fill_diagonal(r, np.inf)
    u = np.clip((r / np.maximum(ro[:, None], ro[None, :]) - 0.1) / 0.9, 0.0, 1.0)
    K = u ** 4 * (35 - 84 * u + 70 * u ** 2 - 20 * u ** 3)
    ref = -(s["m"][None, :] * K / r ** 3 * d).sum(2)
    mag = (s["m"][None, :] / r ** 2).sum(1)
    assert (np.abs(a - ref).max(0) <= (1e-14 if precision == 0 else 3e-6) * mag).all()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n", [1, 2, 255, 256, 257, 512, 513, 1025])
def test_energy_tile_pairs(P, n, precision):
    s = disks.equal_mass_ring(n, seed=n)
    x = np.stack([s["x"], s["y"], s["z"]])

    def pairs(s, x):
        r = np.sqrt(((x[:, :, None] - x[:, None, :]) ** 2).sum(0))
        r[r == 0.0] = np.inf
        return -0.5 * (s["m"][:, None] * s["m"][None, :] / r).sum()

    def run(s):
        ctx = P.p3t_create(P.Params(precision=precision))
        try:
            e = torch.zeros(4, dtype=torch.float64, device="cuda")
            P.p3t_energy(ctx, P.State.from_numpy(s), e)
            assert P.p3t_status(ctx)[0] == 0
            return e.cpu().numpy()
        finally:
            P.p3t_destroy(ctx)
    e = run(s)
    ek = 0.5 * (s["m"] * (s["vx"] ** 2 + s["vy"] ** 2 + s["vz"] ** 2)).sum()
    es = -(s["m"] / np.sqrt((x * x).sum(0))).sum()
    assert abs(e[1] - ek) <= 1e-13 * ek and abs(e[2] - es) <= 1e-13 * abs(es)
    tol = 1e-13 if precision == 0 else 1e-6
    assert abs(e[3] - pairs(s, x)) <= tol * abs(pairs(s, x))
    assert e[0] == e[1] + e[2] + e[3]
    if n < 2:
        return
    for k in ("x", "y", "z"):  # the first and the last body at one place
        s[k][n - 1] = s[k][0]
    x = np.stack([s["x"], s["y"], s["z"]])
    e = run(s)
    if precision == 0:
        assert e[3] == -np.inf
    else:
        assert abs(e[3] - pairs(s, x)) <= tol * abs(pairs(s, x))
