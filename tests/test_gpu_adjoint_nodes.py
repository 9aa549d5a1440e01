"""The tree VJP's node part is gathered by leaf: deep trees, leaves of one
member and oversized ones, against the oracle's autograd over the same lists."""
import numpy as np
import pytest
import torch

from oracle import adjoint_oracle as AO
from oracle import oracle as O
from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu, oracle_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("leaf,group", [(1, 0), (16, 64), (32, 20)])
@pytest.mark.parametrize("n,clump,size", [(2, 0, 0.0), (40, 0, 0.0), (700, 90, 1e-9),
                                          (700, 90, 3e-5)])
def test_node_adjoint_matches_oracle(n, clump, size, leaf, group):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    s = disks.equal_mass_narrow(n, seed=n, planted=False)
    rng = np.random.default_rng(n + clump)
    s["m"][:] *= rng.uniform(0.5, 2.0, n)
    for k in ("x", "y", "z") if clump else ():   # in one cell of the deepest level, or nearly
        s[k][100:100 + clump] = s[k][100] + size * rng.uniform(-1.0, 1.0, clump)
    prm = P.Params(theta=0.5, precision=P.P3T_FP64, leaf_size=leaf, group_size=group)
    op = oracle_params(prm)
    ro, rs, _, _ = O.cutoffs(s, op)
    lam = rng.normal(size=(3, n))
    st = P.State.from_numpy(s, r_out=ro, r_search=rs)
    ctx = P.p3t_create(prm, 0)
    try:
        gx = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        gm = torch.zeros(n, dtype=torch.float64, device="cuda")
        P.p3t_build_tree(ctx, st, False)
        P.p3t_soft_force_vjp_tree(ctx, st, 1.0, torch.as_tensor(lam, device="cuda"), gx, gm)
        torch.cuda.synchronize()
        assert P.p3t_status(ctx)[0] == 0
        g_x, g_m = gx.cpu().numpy().T, gm.cpu().numpy()
    finally:
        P.p3t_destroy(ctx)
    L = O.tree_lists(s, ro, rs, op)
    x = torch.tensor(np.stack([s["x"], s["y"], s["z"]], 1), requires_grad=True)
    m = torch.tensor(s["m"], requires_grad=True)
    (AO.tree_force(x, m, torch.tensor(ro), L) * torch.tensor(lam.T)).sum().backward()
    rx, rm = x.grad.numpy(), m.grad.numpy()
    assert np.isfinite(rx).all() and np.isfinite(rm).all()
    assert np.abs(g_x - rx).max() <= 1e-11 * np.abs(rx).max()
    assert np.abs(g_m - rm).max() <= 1e-11 * np.abs(rm).max()
