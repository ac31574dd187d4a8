"""The FP64 kernels' own reciprocal, square root and quotients (wcc_d3.cuh) round
as the IEEE operations do: bit for bit against CUDA's division and square root
over random fractions at every exponent, at the edges of the ranges they take
(2^+-1000, 2^+-240), on the values next to powers of two and to exact squares, on
fractions of all ones, and on zeros, subnormals, infinities, NaN and negative numbers."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2104_04347_gb300 import build

pytestmark = pytest.mark.gpu

OPS = ["recip", "sqrt", "sqrt_and_recip", "quotient", "cfl_quotients"]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fp64_ops") / "fp64_ops.so")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "fp64_ops.cu")
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", src, "-o", so], check=True)
    return ctypes.CDLL(so)


def _compare(lib, a, b):
    a, b = np.ascontiguousarray(a), np.ascontiguousarray(b)
    bad = np.zeros(5, dtype=np.uint64)
    ptr = lambda x: ctypes.c_void_p(x.ctypes.data)
    assert lib.fp64_ops_compare(ptr(a), ptr(b), ctypes.c_longlong(a.size), ptr(bad)) == 0
    return dict(zip(OPS, bad.tolist()))


def _bits(sign, exponent, fraction):
    u = (sign.astype(np.uint64) << np.uint64(63)) | (exponent.astype(np.uint64) << np.uint64(52)) | fraction.astype(np.uint64)
    return u.view(np.float64)


def _random(rng, n, lo, hi):
    return _bits(rng.integers(0, 2, n), rng.integers(lo, hi, n), rng.integers(0, 1 << 52, n))


@pytest.mark.parametrize("lo,hi", [(0, 2048), (1020, 1027), (1, 60), (1990, 2047), (780, 790), (1260, 1268)])
def test_random_fractions(lib, lo, hi):
    rng = np.random.default_rng(lo)
    n = 1 << 24
    a = _random(rng, n, lo, hi)
    assert not any(_compare(lib, np.abs(a), _random(rng, n, lo, hi)).values())
    assert not any(_compare(lib, a, _random(rng, n, 1000, 1046)).values())


def test_hard_fractions(lib):
    # next to powers of two, all ones but a few bits, squares and their neighbours
    # (roots next to a representable number or to the middle of two)
    rng = np.random.default_rng(7)
    n = 1 << 22
    near = rng.integers(0, 64, n)
    frac = np.where(rng.integers(0, 2, n) == 1, near, (1 << 52) - 1 - near)
    a = _bits(np.zeros(n, dtype=np.int64), rng.integers(700, 1340, n), frac)
    assert not any(_compare(lib, a, a[::-1]).values())
    m = (1.0 + rng.integers(0, 1 << 26, n) * 2.0 ** -26)
    sq = m * m  # exact: 27-bit factors
    mid = np.sqrt(_random(rng, n, 1023, 1025) ** 2) ** 2
    for x in (sq, mid):
        u = np.ascontiguousarray(x).view(np.uint64)
        for d in range(-3, 4):
            y = (u + np.uint64(d % (1 << 64))).view(np.float64) * 4.0 ** rng.integers(-400, 400, n)
            assert not any(_compare(lib, y, m).values())


def test_special_values(lib):
    tiny, one = 5e-324, 1.0
    v = np.array([0.0, tiny, 2.2250738585072014e-308, 2.0 ** -1001, 2.0 ** -1000, 2.0 ** -999, 2.0 ** -241, 2.0 ** -240,
                  one, np.nextafter(one, 2.0), np.nextafter(one, 0.0), 2.0 ** 240, 2.0 ** 241, 2.0 ** 999, 2.0 ** 1000,
                  2.0 ** 1001, 1.7976931348623157e308, np.inf, np.nan])
    v = np.concatenate([v, -v])
    a, b = np.repeat(v, v.size), np.tile(v, v.size)
    assert not any(_compare(lib, a, b).values())
