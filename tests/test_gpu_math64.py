"""The FP64 path's own exponential, division and reciprocal (csrc/lisa_math64.cuh) against extended
precision (numpy's longdouble, 64 bits or more), in units of the result's last place.

Bounds, from the arithmetic: the result is rounded once, after a correction that is exact to 2^-60 of it, so
half a unit; the exponential's series may neglect up to (0.85 ln2 / 8192)^4 / 24 = 1.1e-18, 0.01 units, and its
linear term is rounded to 2^-66."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
EXP, DIV, REC = 0, 1, 2


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    import torch
    from paper_2507_06300_gb300 import build
    so = str(tmp_path_factory.mktemp("probe") / "math64.so")
    r = subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-cudart", "static",
                        os.path.join(HERE, "_math64_probe.cu"), "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(so)
    tab = np.zeros(lib.probe_table_doubles())
    lib.probe_table(tab.ctypes.data_as(ctypes.c_void_p))
    tab_d = torch.as_tensor(tab, device="cuda")

    def run(what, a, b=None):
        a = np.ascontiguousarray(a, np.float64)
        a_d = torch.as_tensor(a, device="cuda")
        b_d = torch.as_tensor(np.ascontiguousarray(a if b is None else b, np.float64), device="cuda")
        out = torch.empty_like(a_d)
        torch.cuda.synchronize()
        ptr = lambda t: ctypes.c_void_p(t.data_ptr())
        assert lib.probe_run(what, ptr(a_d), ptr(b_d), ptr(tab_d), ptr(out), ctypes.c_int64(a.size)) == 0
        return out.cpu().numpy()
    return run


def ulps(y, ref):
    """|y - ref| in units of the last place of the double nearest to ref."""
    return np.abs((y.astype(np.longdouble) - ref) / np.spacing(np.abs(ref).astype(np.float64))).astype(np.float64)


@pytest.mark.parametrize("span", [1e-300, 1e-8, 0.3, 3.0, 30.0, 99.999])
def test_exp10(probe, span):
    rng = np.random.default_rng(3)
    v = rng.uniform(-span, span, 100000)
    assert ulps(probe(EXP, v), np.power(np.longdouble(10), v.astype(np.longdouble))).max() <= 0.52


def test_exp10_edges(probe):
    """Zero, the smallest numbers, the table's nodes and the midpoints between them with their neighbours,
    and the ends of the range (|v| < 100)."""
    j = np.concatenate([np.arange(-70, 70), np.arange(-8200, 8200, 41), np.arange(-2_700_000, 2_700_000, 997)])
    node = np.concatenate([j, j + 0.5]) * (np.log10(2.0) / 8192.0)
    v = np.concatenate([[0.0, -0.0, 5e-324, -5e-324, 2.2e-308, 1e-200, -1e-200, 2.0 ** -60, -(2.0 ** -60), 1.0, -1.0, 2.0, 50.0,
                         np.nextafter(100.0, 0.0), np.nextafter(-100.0, 0.0)],
                        node, np.nextafter(node, 200.0), np.nextafter(node, -200.0)])
    v = v[np.abs(v) < 100.0]
    y = probe(EXP, v)
    assert ulps(y, np.power(np.longdouble(10), v.astype(np.longdouble))).max() <= 0.52
    assert np.all(y[v == 0.0] == 1.0)


def mantissas(rng, n):
    """Positive numbers: significands anywhere in [1, 2) and next to both ends, exponents to 2^+-899."""
    m = 1.0 + rng.random(n)
    m[::4] = 1.0 + rng.integers(0, 64, m[::4].size) * 2.0 ** -52
    m[1::4] = 2.0 - rng.integers(1, 64, m[1::4].size) * 2.0 ** -52
    return m


def test_division(probe):
    rng = np.random.default_rng(4)
    n = 200000
    a, b = mantissas(rng, n), mantissas(rng, n)[rng.permutation(n)]
    eb = rng.integers(-899, 900, n)
    ea = np.clip(eb + rng.integers(-100, 100, n), -899, 899)
    a, b = np.ldexp(a, ea), np.ldexp(b, eb)
    ref = a.astype(np.longdouble) / b.astype(np.longdouble)
    assert ulps(probe(DIV, a, b), ref).max() <= 0.501


def test_reciprocal(probe):
    rng = np.random.default_rng(5)
    n = 200000
    b = np.ldexp(mantissas(rng, n), rng.integers(-899, 900, n))
    assert ulps(probe(REC, b), np.longdouble(1) / b.astype(np.longdouble)).max() <= 0.501
