"""The FP64 cube root (Manning's friction, the critical depth of an inflow) and
the truncation to FP32 that decides whether a stationary wave's exact bound is
looked at (gf_fp64.cuh), on the host: the root within one ulp of the exact one
for FP32 estimates anywhere within 2^-20, checked in integers; the truncation
bit for bit, with its range's ends."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
DP = C.POINTER(C.c_double)


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("cbrt") / "cbrt_shim.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                           "-I", os.path.join(HERE, "..", "paper_2403_15435_gb300", "csrc"),
                           os.path.join(HERE, "cbrt_shim.cpp"), "-o", so])
    return C.CDLL(so)


def cbrt(shim, x, err):
    out = np.empty_like(x)
    shim.cbrt_ops.argtypes = [C.c_int, DP, C.c_double, DP]
    native = shim.cbrt_ops(len(x), x.ctypes.data_as(DP), err, out.ctypes.data_as(DP))
    return out, native


@pytest.mark.parametrize("err", [0.0, 2.0 ** -24, 2.0 ** -21, 2.0 ** -20])
def test_cube_root_within_an_ulp(shim, err):
    rng = np.random.default_rng(5)
    x = np.concatenate([
        np.ldexp(rng.uniform(0.5, 1.0, 4000), rng.integers(-1017, 1020, 4000)),
        np.ldexp(rng.uniform(0.5, 1.0, 4000), rng.integers(-30, 12, 4000)),  # depths, q^2 / g
        np.ldexp(1.0 + rng.integers(0, 8, 200) * 2.0 ** -52, rng.integers(-40, 40, 200)),
        np.ldexp(1.0 - rng.integers(1, 8, 200) * 2.0 ** -53, rng.integers(-40, 40, 200)),
        np.arange(1.0, 41.0) ** 3])
    y, native = cbrt(shim, x, err)
    assert native == 0
    for a, r in zip(x, y):
        lo, hi = Fraction(np.nextafter(r, 0.0)), Fraction(np.nextafter(r, np.inf))
        assert lo ** 3 < Fraction(a) < hi ** 3, (a, r)


def test_cube_root_at_the_ends_of_the_range_is_the_native_one(shim):
    x = np.array([0.0, 5e-324, 2.0 ** -1074, 2.0 ** -1022, 2.0 ** -1020, 1.7e308, 2.0 ** 1023,
                  np.inf, np.nan])
    y, native = cbrt(shim, x, 2.0 ** -20)
    assert native == len(x)
    with np.errstate(all="ignore"):
        assert np.allclose(y, np.cbrt(x), rtol=1e-15, atol=0.0, equal_nan=True)


def test_truncation_to_fp32(shim):
    rng = np.random.default_rng(6)
    n = 100000
    x = np.concatenate([
        np.ldexp(rng.uniform(0.5, 1.0, n), rng.integers(-126, 128, n)) * rng.choice([-1.0, 1.0], n),
        rng.integers(0, 1 << 62, n, dtype=np.uint64).view(np.float64),  # up to 2
        -rng.integers(0, 1 << 62, n, dtype=np.uint64).view(np.float64),
        [0.0, -0.0, 5e-324, -1e-300, 2.0 ** -126, -2.0 ** -126, np.nextafter(2.0 ** -126, 0.0),
         1.0, -1.0, np.nextafter(1.0, 0.0), np.nextafter(2.0 ** 127, 0.0), 2.0 ** 127, -2.0 ** 127,
         2.0 ** 128, 1e300, np.inf, -np.inf, np.nan]])
    got = np.empty(len(x), np.uint32)
    shim.trunc_ops(len(x), x.ctypes.data_as(DP), got.ctypes.data_as(C.POINTER(C.c_uint32)))
    a = np.abs(x)
    ok = (a >= 2.0 ** -126) & (a < 2.0 ** 127)
    f = x[ok].astype(np.float32)  # to nearest: one down where that went up
    want = np.where(np.abs(f.astype(np.float64)) > a[ok], np.nextafter(f, np.float32(0.0)), f)
    assert np.array_equal(got[ok], want.view(np.uint32))
    assert (got[a < 2.0 ** -126] == 0).all()
    big = got[(a >= 2.0 ** 127) | np.isnan(x)].view(np.float32)
    assert len(big) > 0 and np.isnan(big).all()
