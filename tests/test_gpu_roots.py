"""The roots of the kernels (p3t_internal.cuh, cutoff_math.cuh) by a small test
program built from the same headers: against exact rational values over the
exponent range, with bounds from their series and roundings (u = 2^-53), and
against CUDA's functions outside the seeds' ranges and at the edges.

  seed          |e| = |1 - x y^2| <= 2^-19 in range; y = rsqrt(x), e = 0 outside
  x^(-1/2)      y^2's rounding reaches e (u / 2 of the root), the last fma u, the
                series' rest 5/16 e^3 < 2^-58: 1.6 u
  x^(-3/2)      y^2 u / 2, y^3 u, the last fma u, the rest 2.2 e^3 < 2^-55: 2.8 u
  x^(-1/4)      z^4's three roundings 3/4 u, the last fma u, the rest e^4 / 10: 1.9 u
  x^(1/3)       z^3's rounding u / 3 and the last fma u, twice (w^2), two products
                2 u, the rest 2/9 e^3 < u / 200: 4.8 u"""
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
U = 2.0 ** -53


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    need_gpu()
    d = tmp_path_factory.mktemp("roots")
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "-fmad=false", "-I", os.path.join(ROOT, "include"), "-o", str(d / "roots"),
                    os.path.join(ROOT, "tests", "cuda", "roots_check.cu")], check=True)

    def run(*args):
        return subprocess.run([str(d / "roots"), *args], check=True, capture_output=True,
                              text=True).stdout

    def evaluate(x):
        np.asarray(x, dtype=np.float64).tofile(d / "in")
        run("eval", str(d / "in"), str(d / "out"))
        return np.fromfile(d / "out").reshape(-1, 10)
    return run, evaluate


def test_rsqrt_normal_is_rsqrtf_for_every_normal_float(program):
    assert int(program[0]("rsqrtf")) == 0


def test_seed_residual_over_every_leading_mantissa(program):
    assert 0.0 < float(program[0]("seed")) <= 2.0 ** -19


# (column, power p of x^p, range of exponents, bound in u)
@pytest.mark.parametrize("col,num,den,lo,hi,bound", [(2, -1, 2, -511, 512, 1.6),
                                                     (3, -3, 2, -511, 512, 2.8),
                                                     (4, -1, 2, -511, 512, 1.6),
                                                     (5, -1, 4, -511, 512, 1.9),
                                                     (6, 1, 3, -99, 98, 4.8)])
def test_roots_against_exact_values(program, col, num, den, lo, hi, bound):
    rng = np.random.default_rng(col)
    e = np.concatenate([rng.integers(lo, hi + 1, 4000), [lo, lo, hi, hi]])
    m = np.concatenate([rng.uniform(1.0, 2.0, 4000), [1.0, 2.0 - 2.0 ** -52] * 2])
    x = np.ldexp(m, e)
    r = program[1](x)[:, col]
    worst = 0.0
    for a, b in zip(x, r):
        # b^den x^-num = (1 + d)^den for a relative error d
        q = Fraction(b) ** den / Fraction(a) ** num
        worst = max(worst, abs(float(q - 1)) / den)
    assert worst <= bound * U


def test_ranges_end_in_cudas_functions(program):
    rng = np.random.default_rng(9)
    tiny, huge = np.nextafter(0.0, 1.0), np.finfo(np.float64).max
    edge = np.array([0.0, tiny, 2.0 ** -1022, huge, np.inf, np.nan])
    low = np.ldexp(rng.uniform(1, 2, 500), rng.integers(-1073, -511, 500))
    high = np.ldexp(rng.uniform(1, 2, 500), rng.integers(513, 1024, 500))
    o = program[1](np.concatenate([edge[1:], low, high]))
    for c, ref in ((0, 7), (4, 7), (5, 8)):
        assert np.array_equal(o[:, c], o[:, ref], equal_nan=True)
    assert np.all(o[:, 1] == 0.0)
    o = program[1](edge)
    # the seed, 1 / r and r^-3 of a pair at one place and at infinity, the root of 0
    assert np.all(o[0, [0, 1, 2, 3, 4]] == 0.0) and np.all(o[4, [0, 1, 2, 3, 4, 5]] == 0.0)
    assert o[0, 5] == np.inf
    low = np.ldexp(rng.uniform(1, 2, 500), rng.integers(-1073, -99, 500))
    high = np.ldexp(rng.uniform(1, 2, 500), rng.integers(99, 1024, 500))
    o = program[1](np.concatenate([edge, -edge[:4], low, high]))
    assert np.array_equal(o[:, 6], o[:, 9], equal_nan=True)
