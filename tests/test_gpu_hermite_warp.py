"""The one-warp Hermite integration of clusters of two to five members against
the four-warp kernel's plain one (a cluster above hermite_warp_max members):
the same state and corrector steps bit for bit, over pairs inside gamma r_out,
across the changeover and beyond it, planar and coincident members, with and
without collisions."""
import numpy as np
import pytest
import torch

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

K = ("x", "y", "z", "vx", "vy", "vz")


def _clusters(nc, count, seed):
    """count clusters of nc members around (1, 0, 0): separations from well
    inside gamma r_out = 1e-4 to beyond r_out = 1e-3, one planar, one with two
    members at the same place."""
    rng = np.random.default_rng(seed)
    sep = np.exp(rng.uniform(np.log(2e-5), np.log(2e-3), count))[:, None, None]
    x = np.array([1.0, 0.0, 0.0]) + sep * rng.normal(size=(count, nc, 3))
    v = np.array([0.0, 1.0, 0.0]) + np.sqrt(1e-9 / sep) * rng.normal(size=(count, nc, 3))
    x[0, :, 2] = v[0, :, 2] = 0.0
    x[1, 1] = x[1, 0]
    s = {k: np.ascontiguousarray(a[..., q].ravel())
         for q, (k, a) in enumerate(zip(K, (x, x, x, v, v, v)))
         for q in (q % 3,)}
    s["m"] = rng.uniform(0.5e-9, 2e-9, count * nc)
    return s


def _run(P, s, sizes, warp_max, coll):
    n = len(s["m"])
    st = P.State.from_numpy(s, r_out=np.full(n, 1e-3), r_search=np.full(n, 2e-3),
                            r_phys=np.full(n, 2e-6) if coll else None)
    ctx = P.p3t_create(P.Params(f_radius=1.0 if coll else 0.0))
    try:
        P.p3t_reserve(ctx, n)
        P.p3t_set_tuning(ctx, warp_max, 0)
        rec = torch.zeros(n, dtype=torch.int32, device="cuda")
        P.p3t_set_diag(ctx, hermite_steps=rec)
        off = np.concatenate([[0], np.cumsum(sizes)])
        t = dict(label=torch.zeros(n, dtype=torch.int32), singles=torch.zeros(n, dtype=torch.int32),
                 cl_off=torch.as_tensor(off), cl_mem=torch.arange(n, dtype=torch.int32),
                 counts=torch.tensor([0, len(sizes), n, max(sizes)]))
        t = {k: a.cuda() for k, a in t.items()}
        cl = P.Clusters(*[t[k].data_ptr() for k in ("label", "singles", "cl_off", "cl_mem",
                                                    "counts")])
        P.p3t_hard_step(ctx, st, cl, 1.0 / 64.0)
        pending = P.p3t_collisions_pending(ctx)
        assert P.p3t_status(ctx)[0] == 0
        return {k: getattr(st, k).cpu().numpy() for k in K}, rec.cpu().numpy(), pending
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("nc", [2, 3, 4, 5])
@pytest.mark.parametrize("coll", [False, True])
def test_one_warp_clusters_have_the_plain_bits(nc, coll):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    count = 40
    s = _clusters(nc, count, 100 * nc + coll)
    a, ra, pa = _run(P, s, [nc] * count, 8, coll)
    # the same clusters in the four-warp kernel; pairs with a third member far
    # beyond every r_out, which adds exact zeros
    t, pick = s, np.arange(count * nc)
    if nc == 2:
        far = {k: np.full(count, 0.0) for k in K}
        far.update(x=np.full(count, -1.0), vy=np.full(count, -1.0), m=np.full(count, 1e-9))
        t = {k: np.concatenate([s[k].reshape(count, 2), far[k][:, None]], 1).ravel() for k in s}
        pick = (np.arange(count)[:, None] * 3 + np.arange(2)).ravel()
    b, rb, pb = _run(P, t, [max(nc, 3)] * count, 2, coll)
    for k in K:
        assert np.array_equal(a[k], b[k][pick]), k
    assert np.array_equal(ra, rb[pick]) and pa == pb
    assert ra.max() > 50 and (pa > 0) == coll
