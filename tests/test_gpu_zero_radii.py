"""Gradients with bodies of zero cut-off radius (massless bodies under
P3T_CUT_HILL, radii that the caller sets): K = 1 for their pairs with each
other, K by the other's radius otherwise, no NaN."""
import numpy as np
import pytest
import torch

from oracle import adjoint_oracle as A
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t
    return p3t


@pytest.mark.parametrize("zeros", [1, 5, 200])
def test_tree_vjp_with_zero_cutoff_radii(P, zeros):
    # every particle a target of the direct part (theta = 0): the oracle's sum
    n = 200
    rng = np.random.default_rng(zeros)
    x = np.array([[1.0], [0.0], [0.0]]) + rng.normal(0.0, 0.02, (3, n))
    m, lam = rng.uniform(1e-6, 4e-6, n), rng.normal(size=(3, n))
    ro = rng.uniform(0.01, 0.06, n)
    ro[:zeros] = 0.0
    m[0] = 0.0
    q = torch.tensor(x.T.copy(), requires_grad=True)
    mm = torch.tensor(m, requires_grad=True)
    a = A.soft_force(q, mm, torch.tensor(np.maximum(ro, 1e-300)))
    ex, em = torch.autograd.grad((a * torch.tensor(lam.T)).sum(), (q, mm))
    z = np.zeros(n)
    s = dict(x=x[0], y=x[1], z=x[2], vx=z, vy=z, vz=z, m=m)
    st = P.State.from_numpy(s, r_out=ro, r_search=np.full(n, 1e-3))
    f64 = dict(dtype=torch.float64, device="cuda")
    ctx = P.p3t_create(P.Params(theta=0.0, group_size=64, precision=P.P3T_FP64), 0)
    try:
        P.p3t_reserve(ctx, n)
        P.p3t_build_tree(ctx, st)
        gx, gm = torch.zeros(3, n, **f64), torch.zeros(n, **f64)
        P.p3t_soft_force_vjp_tree(ctx, st, 1.0, torch.as_tensor(lam).cuda(), gx, gm)
        assert P.p3t_status(ctx)[0] == 0
        gx, gm = gx.cpu().numpy(), gm.cpu().numpy()
    finally:
        P.p3t_destroy(ctx)
    ex, em = ex.numpy().T, em.numpy()
    assert np.abs(gx - ex).max() <= 1e-12 * np.abs(ex).max()
    assert np.abs(gm - em).max() <= 1e-12 * np.abs(em).max()


@pytest.mark.parametrize("nc", [3, 4, 10])
def test_cluster_gradients_with_zero_cutoff_radii(P, nc):
    # two members of zero radius, beside others in the changeover: the bits of
    # a radius far below every distance
    rng = np.random.default_rng(nc)
    x = np.array([[1.0], [0.0], [0.0]]) + 4e-4 * rng.normal(size=(3, nc))
    v = np.array([[0.0], [1.0], [0.0]]) + 5e-4 * rng.normal(size=(3, nc))
    s = dict(zip(("x", "y", "z", "vx", "vy", "vz"), (*x, *v)), m=rng.uniform(0.5e-9, 2e-9, nc))
    lam = rng.normal(size=(6, nc))

    def run(radius):
        ro = np.full(nc, 1e-3)
        ro[:2] = radius
        st = P.State.from_numpy(s, r_out=ro, r_search=np.full(nc, 2e-3))
        i32 = dict(dtype=torch.int32, device="cuda")
        t = dict(label=torch.zeros(nc, **i32), singles=torch.zeros(nc, **i32),
                 cl_off=torch.tensor([0, nc], device="cuda"), cl_mem=torch.arange(nc, **i32),
                 counts=torch.tensor([0, 1, nc, nc], device="cuda"))
        ctx = P.p3t_create(P.Params(precision=P.P3T_FP64))
        try:
            P.p3t_reserve(ctx, 64)
            cl = P.Clusters(*[t[k].data_ptr() for k in ("label", "singles", "cl_off", "cl_mem",
                                                        "counts")])
            l = torch.as_tensor(lam).cuda()
            lx, lv = l[:3].contiguous(), l[3:].contiguous()
            gm = torch.zeros(nc, dtype=torch.float64, device="cuda")
            P.p3t_hard_step_vjp(ctx, st, cl, 1.0 / 64.0, lx, lv, gm)
            assert P.p3t_status(ctx)[0] == 0
            return [t.cpu().numpy() for t in (lx, lv, gm)]
        finally:
            P.p3t_destroy(ctx)
    for a, b in zip(run(0.0), run(1e-30)):
        assert np.isfinite(b).all() and np.array_equal(a, b)
