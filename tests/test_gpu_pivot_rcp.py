"""The pivots' reciprocal against 1 / x over all exponents and at the edges of the mantissa.

Error: the FP32 start y is off by less than e = 2^-21 (hardware reciprocal 2^-23, mantissa cut at 2^-23), the series
leaves e^3 < 2^-63 of the value, and the last multiply-add rounds once; the result lies in [1/2, 1] before its exponent
is put back, where a unit in the last place is 2^-53.  So it differs from the correctly rounded 1 / x by one unit at
most, and only where 1 / x is within 2^-9 units of a tie.  Outside the normal range the division itself is used."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from tests.conftest import ROOT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    from paper_1005_0088_gb300 import build as b
    lib = str(tmp_path_factory.mktemp("rcp") / "probe.so")
    subprocess.run([b._nvcc()] + b.ARCH + ["-std=c++17", "-O3", "-I" + b.CSRC, "-shared", "-Xcompiler", "-fPIC",
                                           os.path.join(ROOT, "tests", "pivot_rcp_probe.cu"), "-o", lib], check=True)
    f = ctypes.CDLL(lib).pivot_probe

    def call(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y, bad = np.zeros_like(x), np.zeros(x.size, np.int32)
        ptr = ctypes.c_void_p
        assert f(x.ctypes.data_as(ptr), y.ctypes.data_as(ptr), bad.ctypes.data_as(ptr), x.size) == 0
        return y, bad

    return call


def test_reciprocal(probe):
    rng = np.random.default_rng(1)
    bits = rng.integers(1 << 52, 0x7FE << 52, 2_000_000)                 # normal numbers, every exponent
    edge = np.array([0, 1, 2, (1 << 29) - 1, 1 << 29, (1 << 52) - 1, (1 << 52) - 2, 1 << 51])
    bits = np.concatenate([bits, (edge[None, :] + (np.arange(1, 0x7FF)[:, None] << 52)).ravel()]).astype(np.int64)
    x = bits.view(np.float64)
    y, bad = probe(x)
    want = 1.0 / x
    ulps = np.abs(y.view(np.int64) - want.view(np.int64))
    assert ulps.max() <= 1 and not bad.any()
    normal = want >= 2.0 ** -1022
    off = np.flatnonzero((ulps > 0) & normal)
    assert off.size < 1e-2 * x.size
    for i in off[:300]:                                                  # near a tie of two neighbours
        mid = (Fraction(float(y[i])) + Fraction(float(want[i]))) / 2
        unit = abs(Fraction(float(y[i])) - Fraction(float(want[i])))
        assert abs(Fraction(1) / Fraction(float(x[i])) - mid) < unit / 512
    power = bits % (1 << 52) == 0
    assert np.array_equal(y[power], want[power])


def test_outside_the_normal_range(probe):
    sub = np.array([1, 2, 3, 1 << 51, (1 << 52) - 1], dtype=np.int64).view(np.float64)
    x = np.concatenate([[0.0, -0.0, np.inf, np.nan, 2.0 ** 1022, 2.0 ** 1023, 1.7976931348623157e308], sub])
    y, bad = probe(x)
    with np.errstate(divide="ignore", over="ignore"):
        want = 1.0 / x
    assert np.array_equal(y, want, equal_nan=True)
    assert bad.tolist() == [1, 1, 1, 1] + [0] * (x.size - 4)
