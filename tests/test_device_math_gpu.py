"""Arithmetic helpers of the kernels, compiled from the package's headers into a
small library of their own and compared with exact sums."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

from paper_1410_5584_gb300 import _build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def device_math(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("device_math") / "libdevice_math.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "device_math.cu")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.NVCC_FLAGS, "-shared", src, "-o", out], check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("n", [1, 2, 19, 76, 128])
@pytest.mark.parametrize("kind", ["mean_zero", "one_sign", "cancelling", "mixed_sizes"])
def test_float_sums_are_within_their_bound(device_math, n, kind):
    """|s - exact| <= (2 n 2^-24)^3 sum |v| + 2^-52 |exact| (the bound of the sum with K = 3 and the rounding of its
    value to a double); pairs of floats do not keep it beyond a few terms."""
    rng = np.random.default_rng(n)
    v = rng.standard_normal((4096, n)).astype(np.float32)
    if kind == "one_sign":
        v = np.abs(v)
    elif kind == "cancelling":
        v = np.abs(v)
        v[:, n // 2:] *= -1
    elif kind == "mixed_sizes":
        v *= np.exp2(rng.integers(-40, 20, v.shape)).astype(np.float32)
    got = np.empty(len(v))
    f32p, f64p = (ctypes.POINTER(t) for t in (ctypes.c_float, ctypes.c_double))
    assert device_math.float_sum(v.ctypes.data_as(f32p), n, len(v), got.ctypes.data_as(f64p)) == 0
    exact = np.array([math.fsum(r) for r in v.astype(np.float64)])
    bound = (2 * n * 2.0 ** -24) ** 3 * np.abs(v.astype(np.float64)).sum(axis=1) + 2.0 ** -52 * np.abs(exact)
    assert np.all(np.abs(got - exact) <= bound)


def test_float_sums_of_infinities(device_math):
    inf = np.float32(np.inf)
    v = np.array([[1, inf, 2, 3], [1, -inf, 2, 3], [inf, 1, -inf, 2], [np.nan, 1, 2, 3]], dtype=np.float32)
    got = np.empty(4)
    f32p, f64p = (ctypes.POINTER(t) for t in (ctypes.c_float, ctypes.c_double))
    assert device_math.float_sum(v.ctypes.data_as(f32p), 4, 4, got.ctypes.data_as(f64p)) == 0
    assert got[0] == np.inf and got[1] == -np.inf and np.isnan(got[2:]).all()


@pytest.mark.parametrize("exponent", [-100, -63, -20, -3, -2, -1, 0, 1, 2, 3, 20, 64, 99])
def test_reciprocals_are_correctly_rounded(device_math, exponent):
    """Every mantissa of one exponent of the densities' range: one Newton-Raphson step gives __frcp_rn's values, and
    rsqrt_hw those of rsqrtf."""
    differ = (ctypes.c_uint * 2)()
    assert device_math.compare(exponent, differ) == 0
    assert list(differ) == [0, 0]
