"""The integer-pipe FP64 arithmetic of the data preparation (csrc/lisa_soft64.cuh), compiled for the host
with g++: the square root and the product are IEEE's bit for bit wherever the form answers, and the
fixed-point sum of squares keeps its bound for any number of terms."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2507_06300_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("soft64") / "soft64.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-x", "c++", "-I", CSRC,
                    os.path.join(HERE, "_soft64_host.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _spread(rng, n):
    """Doubles of any exponent and sign, significands anywhere and next to both ends."""
    m = 1.0 + rng.random(n)
    m[::5] = 1.0 + rng.integers(0, 64, m[::5].size) * 2.0 ** -52
    m[1::5] = 2.0 - rng.integers(1, 64, m[1::5].size) * 2.0 ** -52
    with np.errstate(over="ignore", under="ignore"):
        v = np.ldexp(m, rng.integers(-1074, 1024, n)) * rng.choice([-1.0, 1.0], n)
    v[:9] = 0.0, -0.0, 5e-324, np.inf, -np.inf, np.nan, 2.2250738585072014e-308, 1.7976931348623157e308, 1.0
    return v


def test_sqrt_half(lib):
    rng = np.random.default_rng(1)
    n = 400000
    v = np.concatenate([np.abs(_spread(rng, n)), np.round(rng.uniform(1, 1 << 26, n)) ** 2 * 2.0, -rng.random(10)])
    out, ok = np.zeros(v.size, np.uint64), np.zeros(v.size, np.uint8)
    lib.host_sqrt_half(_p(v), _p(out), _p(ok), ctypes.c_int64(v.size))
    ok = ok.astype(bool)
    normal = np.isfinite(v) & (v >= 2.0 ** -1021)
    assert not ok[~normal].any() and ok[normal][:n].mean() > 0.9
    assert np.array_equal(out[ok].view(np.float64), np.sqrt(0.5 * v[ok]))


def test_mul(lib):
    rng = np.random.default_rng(2)
    n = 400000
    a, x = np.abs(_spread(rng, n)), _spread(rng, n)[rng.permutation(n)]
    a = np.where(np.isfinite(a) & (a >= 2.0 ** -1022), a, 1.5)
    out, ok = np.zeros(n, np.uint64), np.zeros(n, np.uint8)
    lib.host_mul(_p(a), _p(x), _p(out), _p(ok), ctypes.c_int64(n))
    ok = ok.astype(bool)
    with np.errstate(all="ignore"):
        ref = a * x
    inside = np.isfinite(x) & (np.abs(x) >= 2.0 ** -1022) & (np.abs(ref) < 2.0 ** 1022) & (np.abs(ref) >= 2.0 ** -1021)
    assert np.array_equal(ok[inside], np.ones(inside.sum(), bool))
    assert np.array_equal(out[ok].view(np.float64), ref[ok])


@pytest.mark.parametrize("order", ["large_first", "large_last", "random"])
@pytest.mark.parametrize("n", [1, 2, 7, 300, 200000])
def test_square_sum(lib, n, order):
    """One large term and n - 1 small ones (squares down to 2^-66 of the large one's, where each loses up to
    all of itself): the sum is never above the exact one, and below it by less than three units of 2^-62 of
    the largest square's binade per term (two for the square's truncation, one for the shift of the sum)."""
    rng = np.random.default_rng(n)
    v = np.ldexp(1.0 + rng.random(n), rng.integers(-33, -20, n)) * rng.choice([-1.0, 1.0], n)
    v[0] = 1.25
    if order == "large_last":
        v = v[::-1].copy()
    if order == "random":
        v = np.ldexp(v, rng.integers(-30, 30, n))[rng.permutation(n)]
    top, acc = ctypes.c_uint32(), ctypes.c_uint64()
    E = lib.host_square_sum(_p(v), ctypes.c_int64(n), ctypes.byref(top), ctypes.byref(acc))
    unit = Fraction(2) ** (2 * (E - 1023) - 62)
    got = ((top.value << 64) + acc.value) * unit
    lo = np.frexp(v)[1].min() - 60   # exact sum of squares as integers of a common scale
    exact = sum(int(t) ** 2 for t in np.ldexp(v, -lo).astype(object)) * Fraction(2) ** int(2 * lo)
    assert 0 <= exact - got < 3 * n * unit
