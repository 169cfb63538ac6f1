"""The integer AVG quotient (csrc/quotient.cuh), built for the host, against IEEE float64 division."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("q") / "libquotient.so")
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-o", so,
                           os.path.join(HERE, "quotient_host.cpp")])
    return ctypes.CDLL(so)


def p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def check(lib, x, c):
    x, c = np.ascontiguousarray(x, np.float64), np.ascontiguousarray(c, np.uint32)
    out, ok = np.zeros(x.size, np.uint64), np.zeros(x.size, np.uint8)
    lib.quotients(p(x), p(c), ctypes.c_int64(x.size), p(out), p(ok))
    with np.errstate(all="ignore"):
        ref = x / c.astype(np.float64)
    ok = ok.astype(bool)
    assert np.array_equal(out[ok], ref.view(np.uint64)[ok])
    return ok, ref


@pytest.mark.parametrize("kind", ["random", "small", "exact", "ties", "powers", "edges"])
def test_quotient_is_the_ieee_one(lib, kind):
    rng = np.random.default_rng(5)
    n = 1_000_000
    c = np.exp2(rng.uniform(0, 32, n)).astype(np.uint64).clip(1, 2 ** 32 - 1)
    if kind == "random":
        x = rng.standard_normal(n) * np.exp2(rng.integers(-900, 900, n).astype(np.float64))
    elif kind == "small":
        x, c = rng.integers(-10 ** 6, 10 ** 6, n).astype(np.float64), rng.integers(1, 1000, n)
    elif kind == "exact":  # quotients that are representable
        q = rng.integers(1, 2 ** 21, n).astype(np.float64)
        x = q * c
    elif kind == "ties":  # (k + 1/2) units of the quotient times a power of two
        c = np.uint64(1) << rng.integers(0, 32, n).astype(np.uint64)
        x = rng.integers(2 ** 52, 2 ** 53, n).astype(np.float64)
    elif kind == "powers":
        x, c = np.exp2(rng.integers(-1000, 1000, n).astype(np.float64)), c | 1
    else:
        x = np.repeat([0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, 2.2250738585072014e-308,
                       1.7976931348623157e308, np.nextafter(2.0, 0), np.nextafter(1.0, 2)], 8)
        c = np.tile([1, 2, 3, 2 ** 31 - 1, 2 ** 31, 2 ** 31 + 1, 2 ** 32 - 2, 2 ** 32 - 1], 12)
    ok, ref = check(lib, x, c)
    normal = np.isfinite(ref) & ((np.abs(ref) >= 2.3e-308) | (ref == 0)) & ((np.abs(x) >= 2.3e-308) | (np.abs(x) == 0))
    assert np.all(ok[normal])  # only subnormal and non-finite cases are left to a float64 division


def test_int64_to_float64(lib):
    rng = np.random.default_rng(6)
    v = np.concatenate([rng.integers(-2 ** 63, 2 ** 63 - 1, 500_000), rng.integers(-2 ** 54, 2 ** 54, 500_000),
                        [0, 1, -1, 2 ** 53, 2 ** 53 + 1, 2 ** 54 + 2, 2 ** 54 + 6, 2 ** 63 - 1, -2 ** 63, -2 ** 63 + 1]])
    v = v.astype(np.int64)
    out = np.zeros(v.size, np.uint64)
    lib.conversions(p(v), ctypes.c_int64(v.size), p(out))
    assert np.array_equal(out, v.astype(np.float64).view(np.uint64))
