"""Arithmetic written out in the kernels: the FP64 reciprocal of the pivots and
the rounding of right-hand sides to FP32, against the division and the
conversion."""
import ctypes as C
import os
import subprocess
import tempfile

import numpy as np
import pytest

from paper_1711_10579_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def dev():
    so = os.path.join(tempfile.mkdtemp(prefix="arith"), "arith_device.so")
    subprocess.check_call([os.path.join(build._cuda_home(), "bin", "nvcc"), *build.ARCH, "-O3",
                           "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-o", so,
                           os.path.join(HERE, "arith_device.cu")])
    return C.CDLL(so)


def _mantissas(rng, n):
    m = 1.0 + rng.random(n)
    m[:64] = 1.0 + np.arange(64) * 2.0 ** -52  # next to one and to two
    m[64:128] = 2.0 - (1 + np.arange(64)) * 2.0 ** -52
    return m


@pytest.mark.gpu
def test_reciprocal_against_the_division(dev):
    """Within the iteration's range (exponents of 2^+-100) at most one unit in the
    last place from the correctly rounded 1 / x: its own error is below 0.51 units
    (the truncated cube of e <= 1.5 x 2^-23 and two roundings).  Outside, zeros,
    denormals, infinities and NaN: the division's bits."""
    rng = np.random.default_rng(5)
    x = []
    for e in (-100, -99, -53, -24, -1, 0, 1, 24, 52, 99, 100):
        x.append(np.ldexp(_mantissas(rng, 4096), e))
    x.append(np.ldexp(_mantissas(rng, 65536), rng.integers(-100, 101, 65536)))
    inside = np.concatenate(x)
    outside = np.concatenate(
        [np.ldexp(_mantissas(rng, 256), e) for e in (-1022, -500, -102, -101, 101, 102, 500, 1023)]
        + [np.array([0.0, 5e-324, 1e-310, np.inf, np.nan, np.finfo(np.float64).max])])
    v = np.concatenate([inside, -inside, outside, -outside])
    out, div = np.empty_like(v), np.empty_like(v)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    assert dev.arith_recip(ptr(v), ptr(out), ptr(div), v.size) == 0
    k = 2 * inside.size
    with np.errstate(divide="ignore", over="ignore"):
        exact = 1.0 / v
    assert np.array_equal(div[:k], exact[:k])
    assert np.max(np.abs(out[:k].view(np.int64) - exact[:k].view(np.int64))) <= 1
    same = (out[k:].view(np.int64) == div[k:].view(np.int64)) | (np.isnan(out[k:]) & np.isnan(div[k:]))
    assert np.all(same)


@pytest.mark.gpu
def test_narrowing_against_the_conversion(dev):
    """Half a unit in the last place over the FP32 range (ties away from zero where
    the conversion rounds to even); what overflows or is not finite does not come
    out finite, except a NaN, whose scenario the stop test has already ended."""
    rng = np.random.default_rng(6)
    v = np.concatenate([np.ldexp(_mantissas(rng, 4096), e) for e in (-126, -100, -30, -1, 0, 1, 30, 126)]
                       + [np.array([0.0, 1.0 + 2.0 ** -24, 1.0 + 3 * 2.0 ** -24])])
    v = np.concatenate([v, -v])
    out = np.empty(v.size, np.float32)
    ptr = lambda a: a.ctypes.data_as(C.c_void_p)
    assert dev.arith_narrow(ptr(v), ptr(out), v.size) == 0
    half = 0.5 * np.spacing(np.abs(v.astype(np.float32))).astype(np.float64)
    assert np.all(np.abs(out.astype(np.float64) - v) <= half)
    assert np.array_equal(np.signbit(out), np.signbit(v))
    big = np.array([np.inf, -np.inf, 1e300, -1e300])
    out = np.empty(big.size, np.float32)
    assert dev.arith_narrow(ptr(big), ptr(out), big.size) == 0
    assert not np.any(np.isfinite(out))
