"""The integer forms of the FP64 operations (gf_fp64.cuh) against the host's
IEEE arithmetic, bit for bit: quotients, square roots, scalings by two and
comparisons, over random significands and exponents, exact products and
squares, near-ties, zeros, denormals, infinities and NaN, for reciprocal seeds
anywhere within the error the device's approximations may have."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fp64") / "fp64_shim.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-ffp-contract=off",
                           "-I", os.path.join(HERE, "..", "paper_2403_15435_gb300", "csrc"),
                           os.path.join(HERE, "fp64_shim.cpp"), "-o", so])
    f = C.CDLL(so).fp64_ops
    dp = C.POINTER(C.c_double)
    f.argtypes = [C.c_int, dp, dp, C.c_double, dp, dp, dp, dp, C.POINTER(C.c_uint8)]
    f.restype = None

    def run(a, b, err):
        out = [np.empty_like(a) for _ in range(4)]
        fl = np.empty(len(a), np.uint8)
        p = lambda x: x.ctypes.data_as(dp)
        f(len(a), p(a), p(b), err, *[p(x) for x in out], fl.ctypes.data_as(C.POINTER(C.c_uint8)))
        return out, fl
    return run


def operands(rng, n):
    u = lambda lo, hi: rng.integers(lo, hi, n, dtype=np.uint64)
    m = np.uint64(1) << np.uint64(52)
    near1 = (u(1021, 1026) << np.uint64(52))
    kinds = [
        u(0, 1 << 63) * np.uint64(2) + u(0, 2),                  # any bits
        near1 | u(0, 1 << 52),
        near1 | u(0, 16),
        near1 | (m - np.uint64(1) - u(0, 16)),
        (u(0, 2047) << np.uint64(52)) | u(0, 1 << 52),
        np.ldexp(rng.integers(1, 1000, n).astype(float), rng.integers(-20, 20, n)).view(np.uint64),
        np.where(rng.random(n) < 0.5, 0.0, -np.exp(rng.uniform(-12, 5, n))).view(np.uint64),
        rng.choice(np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1e-308, 1.7e308]), n).view(np.uint64),
    ]
    pick = rng.integers(0, len(kinds), n)
    return np.choose(pick, kinds).view(np.float64)


def same(x, y):
    return (x.view(np.uint64) == y.view(np.uint64)) | (np.isnan(x) & np.isnan(y))


@pytest.mark.parametrize("err", [0.0, 2.0 ** -24, 2.0 ** -23, 2.0 ** -22])
def test_integer_forms_equal_ieee(ops, err):
    rng = np.random.default_rng(17)
    n = 400000
    a, b = operands(rng, n), operands(rng, n)
    with np.errstate(all="ignore"):
        a = np.where(rng.random(n) < 0.25, a * b, a)      # exact quotients among them
        a = np.where(rng.random(n) < 0.1, a * a, a)       # exact squares
        (q, r, h, d), fl = ops(a, b, err)
        assert same(q, a / b).all()
        assert same(r, np.sqrt(a)).all()
        assert same(h, 0.5 * a).all() and same(d, 2.0 * a).all()
        ok = ~(np.isnan(a) | np.isnan(b))
        want = ((a < b) * 1 | (a < 0) * 2 | (a > 0) * 4 | (a == 0) * 8 | (a > 1e-3) * 16)
        assert (fl[ok] == want[ok]).all()
    assert ((fl[np.isnan(a)] & 16) == 0).all()  # NaN is never above a threshold
