"""The block-step criterion of small clusters in units far from the paper's.
Lengths stay, times grow by a power of two: every value of a correct
integration is then scaled exactly, also where the criterion's squared norms
and their products leave FP32's range, so the one-warp clusters have the bits
of the plain kernel, and the lanes' gradients those of unscaled units."""
import numpy as np
import pytest
import torch

from tests.gpu_util import need_gpu
from tests.test_gpu_hermite_warp import K, _clusters

pytestmark = pytest.mark.gpu

# accelerations of 2^(-2 k): 1 to 1e-14, and 1e10
POWERS = [0, 12, 14, 15, 16, 17, 18, 20, 23, -17]


@pytest.fixture(scope="module")
def P():
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t
    return p3t


def _scaled(s, power):
    f = {k: 1.0 if k in "xyz" else 2.0 ** (-power if k != "m" else -2 * power) for k in s}
    return {k: s[k] * f[k] for k in s}


def _table(P, sizes):
    n = int(np.sum(sizes))
    t = dict(label=torch.zeros(n, dtype=torch.int32), singles=torch.zeros(n, dtype=torch.int32),
             cl_off=torch.as_tensor(np.concatenate([[0], np.cumsum(sizes)])),
             cl_mem=torch.arange(n, dtype=torch.int32),
             counts=torch.tensor([0, len(sizes), n, max(sizes)]))
    t = {k: a.cuda() for k, a in t.items()}
    return t, P.Clusters(*[t[k].data_ptr() for k in ("label", "singles", "cl_off", "cl_mem",
                                                     "counts")])


def _params(P, power, **kw):
    return P.Params(dt_soft=2.0 ** (power - 6), m_star=2.0 ** (-2 * power), **kw)


def _step(P, s, sizes, power, warp_max):
    n = len(s["m"])
    st = P.State.from_numpy(_scaled(s, power), r_out=np.full(n, 1e-3), r_search=np.full(n, 2e-3))
    prm = _params(P, power)
    ctx = P.p3t_create(prm)
    try:
        P.p3t_reserve(ctx, n)
        P.p3t_set_tuning(ctx, warp_max, 0)
        rec = torch.zeros(n, dtype=torch.int32, device="cuda")
        P.p3t_set_diag(ctx, hermite_steps=rec)
        t, cl = _table(P, sizes)
        P.p3t_hard_step(ctx, st, cl, prm.dt_soft)
        assert P.p3t_status(ctx)[0] == 0
        return {k: getattr(st, k).cpu().numpy() for k in K}, rec.cpu().numpy()
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("power", POWERS)
@pytest.mark.parametrize("nc", [3, 5])
def test_one_warp_steps_in_any_units(P, nc, power):
    s = _clusters(nc, 40, nc)
    a, ra = _step(P, s, [nc] * 40, power, 8)
    b, rb = _step(P, s, [nc] * 40, power, 2)
    assert ra.max() > 50 and np.array_equal(ra, rb)
    for k in K:
        assert np.array_equal(a[k], b[k]), k


def _gradients(P, s, nc, power):
    n = len(s["m"])
    z = _scaled(s, power)
    st = P.State.from_numpy(z, r_out=np.full(n, 1e-3), r_search=np.full(n, 2e-3))
    lam = np.random.default_rng(nc).normal(size=(6, n))
    prm = _params(P, power, precision=P.P3T_FP64)
    ctx = P.p3t_create(prm)
    try:
        P.p3t_reserve(ctx, n)
        t, cl = _table(P, [nc] * (n // nc))
        l = torch.as_tensor(lam).cuda()
        lx, lv = l[:3].contiguous(), 2.0 ** power * l[3:]
        gm = torch.zeros(n, dtype=torch.float64, device="cuda")
        P.p3t_hard_step_vjp(ctx, st, cl, prm.dt_soft, lx, lv, gm)
        assert P.p3t_status(ctx)[0] == 0
        return lx.cpu().numpy(), lv.cpu().numpy() * 2.0 ** -power, gm.cpu().numpy() * 4.0 ** -power
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("power", POWERS[1:])
@pytest.mark.parametrize("nc", [2, 4, 10])
def test_gradients_in_any_units(P, nc, power):
    s = _clusters(nc, 12, nc)
    s["x"][nc:2 * nc] += 1e-3 * np.arange(nc)  # no two at one place
    a, b = _gradients(P, s, nc, 0), _gradients(P, s, nc, power)
    for g, h in zip(a, b):
        assert np.isfinite(g).all() and np.abs(g).max() > 0.0
        assert np.array_equal(g, h)
