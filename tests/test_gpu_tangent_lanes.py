"""The hard part's adjoint by lanes (clusters of 2 to 10 members) and by
threads (11 to 16): gradients of one hard step of single clusters against
central differences of the forward step (1e-4 of the largest component: the
differences' own truncation, and a block step whose level flips), for members
in the changeover, inside it and beyond each other's cut-off radii."""
import numpy as np
import pytest
import torch

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

K = ("x", "y", "z", "vx", "vy", "vz")


@pytest.mark.parametrize("nc,sep", [(2, 3e-4), (2, 6e-5), (2, 3e-3), (3, 3e-4), (4, 4e-4),
                                    (7, 6e-4), (10, 8e-4), (11, 8e-4)])
def test_cluster_gradients_against_differences(nc, sep):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    rng = np.random.default_rng(nc)
    dt = 1.0 / 64.0
    x = np.array([[1.0], [0.0], [0.0]]) + sep * rng.normal(size=(3, nc))
    v = np.array([[0.0], [1.0], [0.0]]) + 5e-4 * rng.normal(size=(3, nc))
    m = rng.uniform(0.5e-9, 2e-9, nc)
    lam = rng.normal(size=(6, nc))
    f64 = dict(dtype=torch.float64, device="cuda")
    ctx = P.p3t_create(P.Params(eta=0.003, eta0=0.0003, precision=P.P3T_FP64))
    try:
        P.p3t_reserve(ctx, 64)
        i32 = dict(dtype=torch.int32, device="cuda")
        t = dict(label=torch.zeros(nc, **i32), singles=torch.zeros(nc, **i32),
                 cl_off=torch.tensor([0, nc], device="cuda"), cl_mem=torch.arange(nc, **i32),
                 counts=torch.tensor([0, 1, nc, nc], device="cuda"))
        cl = P.Clusters(*[t[k].data_ptr() for k in ("label", "singles", "cl_off", "cl_mem",
                                                    "counts")])

        def state(x, v, m):
            s = dict(zip(K, (*x, *v)), m=m)
            return P.State.from_numpy(s, r_out=np.full(nc, 1e-3), r_search=np.full(nc, 2e-3))

        def value(x, v, m):
            st = state(x, v, m)
            P.p3t_hard_step(ctx, st, cl, dt)
            return sum(float((lam[q] * getattr(st, k).cpu().numpy()).sum())
                       for q, k in enumerate(K))
        st = state(x, v, m)
        l = torch.as_tensor(lam).cuda()
        lx, lv, gm = l[:3].contiguous(), l[3:].contiguous(), torch.zeros(nc, **f64)
        P.p3t_hard_step_vjp(ctx, st, cl, dt, lx, lv, gm)
        assert P.p3t_status(ctx)[0] == 0
        g = [lx.cpu().numpy(), lv.cpu().numpy(), gm.cpu().numpy()[None]]
        for what, (a, h) in enumerate(((x, 1e-3 * sep), (v, 1e-7), (m[None], 1e-12))):
            d = np.zeros_like(a)
            for idx in np.ndindex(a.shape):
                b = a.copy()
                b[idx] += h
                c = a.copy()
                c[idx] -= h
                args = [[x, v, m], [x, v, m]]
                args[0][what], args[1][what] = (b, c) if what < 2 else (b[0], c[0])
                d[idx] = (value(*args[0]) - value(*args[1])) / (2 * h)
            assert np.abs(g[what] - d).max() <= 1e-4 * max(np.abs(d).max(), 1e-3)
    finally:
        P.p3t_destroy(ctx)
