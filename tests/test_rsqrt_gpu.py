"""The FP64 reciprocal square root of the bond lengths against exact arithmetic and CUDA's.

From 2^-60 to 2^60 it is one cubic step from an FP32 seed.  Bound: the seed is within
2^-22.4 (rsqrt.approx.ftz.f32) plus 2^-24 (its argument cut to 24 bits), so e = 1 - x y^2
is below 2^-21 and the step's own error, 5/16 e^3, below 2^-64; rounding x y moves e by
2^-53, so y by 2^-54, and the last operation rounds once more (2^-53).  The other roundings
act on terms below 2^-21 of y.  Together 1.5 * 2^-53 (1 + 2^-10).  Outside that range, and
for zeros, infinities, NaN and negative numbers, the bits are CUDA's."""
import ctypes as ct
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1411_3487_gb300 import build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def both():
    build.build()
    out_dir = os.path.join(HERE, "_build")
    os.makedirs(out_dir, exist_ok=True)
    so = os.path.join(out_dir, "librsqrt_check.so")
    tmp = so + f".tmp{os.getpid()}"
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler",
                    "-fPIC", os.path.join(HERE, "rsqrt_check.cu"), "-o", tmp], check=True)
    os.replace(tmp, so)
    fn = ct.CDLL(so).rsqrt_check
    fn.argtypes = [ct.c_void_p] * 3 + [ct.c_int]

    def call(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        own, cuda = np.empty_like(x), np.empty_like(x)
        assert fn(x.ctypes.data, own.ctypes.data, cuda.ctypes.data, x.size) == 0
        return own, cuda
    return call


def test_error_within_its_range(both):
    rng = np.random.default_rng(0)
    lo, hi = 2.0 ** -60, 2.0 ** 60
    edges = np.concatenate([np.nextafter(lo, [lo, 1.0]), [lo], np.nextafter(hi, [1.0, 0.0]),
                            2.0 ** np.arange(-60.0, 60.0), np.nextafter(2.0 ** np.arange(-59.0, 61.0), 0.0),
                            np.nextafter(2.0 ** np.arange(-60.0, 60.0), np.inf)])
    x = np.concatenate([edges, rng.uniform(1, 4, 6000) * 4.0 ** rng.integers(-30, 30, 6000), rng.uniform(1, 4, 6000)])
    x = x[(x >= lo) & (x < hi)]
    own, _ = both(x)
    worst = Fraction(0)
    for a, y in zip(x.tolist(), own.tolist()):
        # y = (1 + d) / sqrt(x): x y^2 - 1 = 2 d + d^2
        worst = max(worst, abs(Fraction(a) * Fraction(y) ** 2 - 1))
    assert worst < 2 * Fraction(3, 2) / 2 ** 53 * (1 + Fraction(1, 2 ** 10)), float(worst)


def test_the_rest_is_cudas(both):
    tiny, big = np.nextafter(2.0 ** -60, 0.0), 2.0 ** 60
    rng = np.random.default_rng(1)
    x = np.concatenate([[0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, -2.0 ** -70, -2.0 ** 70, tiny, big, 5e-324, 2.0 ** -1022,
                         np.nextafter(2.0 ** -1022, 0.0), np.finfo(np.float64).max, 2.0 ** -100, 2.0 ** 100],
                        2.0 ** rng.uniform(-1074, -60, 500), 2.0 ** rng.uniform(60, 1023.9, 500), -2.0 ** rng.uniform(-60, 60, 200)])
    own, cuda = both(x)
    assert np.array_equal(own.view(np.int64)[~np.isnan(cuda)], cuda.view(np.int64)[~np.isnan(cuda)])
    assert np.array_equal(np.isnan(own), np.isnan(cuda))
    assert own[0] == np.inf and own[1] == -np.inf and own[2] == 0.0 and np.isnan(own[3:6]).all()
