"""Cut-off radii where the radial bins are hard to decide or the lengths are far
from one: many narrow bins, a range that is one number, zero or 60 decades
wide, particles on the axis and massless ones, against the oracle."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu, oracle_params

pytestmark = pytest.mark.gpu


def _disk(kind, n):
    s = {k: v.copy() for k, v in disks.equal_mass_narrow(n, seed=n, planted=False).items()
         if np.ndim(v)}
    f = {"far": 1e40, "near": 1e-40}.get(kind, 1.0)
    if kind == "axis":
        s["x"][n // 2] = s["y"][n // 2] = 0.0
        s["z"][n // 2] = 0.7
        s["m"][::3] = 0.0
    if kind == "circle":   # one R to the last bit: no range
        s["x"][:], s["y"][:] = 1.5, 0.0
    if kind == "spread":   # 60 decades, the speeds far from escape
        f = 10.0 ** np.random.default_rng(n).integers(-30, 31, n)
    for k in ("x", "y", "z"):
        s[k] *= f
    return s


@pytest.mark.parametrize("kind", ["annulus", "far", "near", "axis", "circle", "spread"])
@pytest.mark.parametrize("n,bins", [(1, 1), (2, 4096), (257, 256), (6000, 257), (6000, 2048),
                                    (50000, 4096), (50000, 0)])
def test_cutoffs_match_oracle(kind, n, bins):
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t as P
    s = _disk(kind, n)
    prm = P.Params(vran_bins=bins)
    with np.errstate(all="ignore"):
        ro, rs, _, _ = O.cutoffs(s, oracle_params(prm))
    st = P.State.from_numpy(s)
    ctx = P.p3t_create(prm, 0)
    try:
        P.p3t_cutoffs(ctx, st)
        torch.cuda.synchronize()
        assert P.p3t_status(ctx)[0] == 0
    finally:
        P.p3t_destroy(ctx)
    pairs = [(st.r_out, ro), (st.r_search, rs)]
    if kind in ("annulus", "axis", "circle"):  # |u|^2 within its fixed-point sums
        na = P.State.from_numpy(s)
        P.p3t_cutoffs_noalloc(prm, na)
        pairs += [(na.r_out, ro), (na.r_search, rs)]
    for got, ref in pairs:
        got = got.cpu().numpy()
        assert np.all(np.isfinite(ref)) and np.max(np.abs(got - ref) / np.abs(ref)) < 1e-13
