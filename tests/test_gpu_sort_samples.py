"""The samples of the tree's key sort: positions that no order of the input in
rows misleads (a lattice stored row by row is built as fast as in random order),
and, with bodies put where the samples are taken, a bucket far beyond what a
block sorts: the same forces bit for bit as from the radix passes, every device
status clean."""
import numpy as np
import pytest
import torch

from paper_2007_15432_gb300 import disks
from tests.gpu_util import need_gpu
from tests.test_gpu_sort_paths import RADIX

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    need_gpu()
    from paper_2007_15432_gb300 import build
    build.build()
    from paper_2007_15432_gb300 import p3t
    return p3t


def _samples(n):
    """The positions that the sort of n keys samples."""
    buckets = 16
    while buckets < 1024 and buckets * 1000 < n:
        buckets *= 2
    ns = min(4096 // buckets, 8) * buckets
    i = np.arange(ns, dtype=np.uint32)
    h = i.copy()
    for mul, shift in ((0x85ebca6b, 16), (0xc2b2ae35, 13)):  # MurmurHash3's finalizer
        h ^= h >> np.uint32(shift)
        h *= np.uint32(mul)
    h ^= h >> np.uint32(16)
    return i.astype(np.int64) * n // ns + ((h.astype(np.int64) >> 16) * (n // ns) >> 16)


def _eval(P, s, cap):
    n = len(s["m"])
    ctx = P.p3t_create(P.Params(theta=0.7, group_size=32, precision=P.P3T_MIXED), 0)
    try:
        P.p3t_reserve(ctx, cap)
        st = P.State.from_numpy(s, r_out=np.full(n, 1e-7), r_search=np.full(n, 2e-7))
        acc = torch.zeros(3, n, dtype=torch.float64, device="cuda")
        cnt = torch.zeros(2, dtype=torch.int64, device="cuda")
        P.p3t_build_tree(ctx, st)
        P.p3t_soft_force(ctx, st, acc, cnt)
        stats = P.p3t_tree_stats(ctx)
        assert P.p3t_status(ctx)[0] == 0
        a = acc.cpu().numpy()
        assert np.isfinite(a).all() and (n == 1 or np.abs(a).max() > 0.0)
        return a, cnt.cpu().numpy(), stats
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("n,clump", [(3001, 0), (8193, 0), (20_000, 1), (120_001, 1),
                                     (20_000, 2)])
def test_sort_routes_agree_and_report_nothing(P, n, clump):
    s = disks.equal_mass_ring(n, seed=n)
    if clump:
        rng, far = np.random.default_rng(1), np.zeros(n, dtype=bool)
        at = _samples(n)
        far[at if clump == 1 else at[:len(at) // 2]] = True
        for k, c in (("x", 1.0), ("y", 0.0), ("z", 0.0)):
            s[k] = np.where(far, s[k], c + 1e-3 * rng.uniform(-1, 1, n))
    a, ca, sa = _eval(P, s, n)
    b, cb, sb = _eval(P, s, RADIX)
    assert sa == sb and np.array_equal(ca, cb) and ca[0] > 0
    assert np.array_equal(a, b)


def _build_us(P, x):
    n = len(x)
    z = np.zeros(n)
    s = dict(x=x[:, 0], y=x[:, 1], z=x[:, 2], vx=z, vy=z, vz=z, m=np.full(n, 1e-9))
    st = P.State.from_numpy(s, r_out=np.full(n, 1e-7), r_search=np.full(n, 2e-7))
    ctx = P.p3t_create(P.Params(precision=P.P3T_MIXED), 0)
    try:
        P.p3t_reserve(ctx, n)
        best = np.inf
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            P.p3t_build_tree(ctx, st)
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, 1e3 * e[0].elapsed_time(e[1]))
        assert P.p3t_status(ctx)[0] == 0
        return best
    finally:
        P.p3t_destroy(ctx)


@pytest.mark.parametrize("row", [64, 128, 256])
def test_a_lattice_in_rows_is_built_as_fast(P, row):
    # 2^17 and 2^20 bodies: samples at even strides of 128 and 256 bodies took
    # them all from one or a few columns
    for n in (1 << 17, 1 << 20):
        k = np.arange(n)
        side = int(np.sqrt(n // row))
        x = np.stack([k % row, k // row % side, k // (row * side)], 1) * 1e-3
        x = x + np.random.default_rng(2).uniform(0, 1e-4, x.shape)
        mixed = x[np.random.default_rng(3).permutation(n)]
        a, b = _build_us(P, x), _build_us(P, mixed)
        print(f"row {row} n {n}: {a:.1f} us in rows, {b:.1f} in random order")
        assert a <= 1.5 * b
