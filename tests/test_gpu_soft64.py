"""The data preparation's integer-pipe arithmetic at its edges, against numpy: the synthesis rounds as
IEEE FP64 does, bit for bit, and the periodogram's fixed-point sums keep the tolerance of the FP64
ones, for values of every exponent, zeros, subnormals, infinities and NaNs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _spread(rng, n, lo=-1074, hi=1024):
    """Doubles of random significands over the binary exponents lo..hi, either sign, with the edges."""
    with np.errstate(over="ignore", under="ignore"):
        v = np.ldexp(rng.uniform(0.5, 1.0, n), rng.integers(lo, hi + 1, n)) * rng.choice([-1.0, 1.0], n)
    edge = np.array([0.0, -0.0, 5e-324, 2.2250738585072014e-308, 2.225073858507201e-308, 1.7976931348623157e308, np.inf,
                     -np.inf, np.nan, 1.0, 2.0, 4.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52])
    v[:edge.size] = edge
    return v


@pytest.mark.parametrize("n", [1, 255, 40001])
def test_synthesis_rounds_like_ieee(n):
    import torch
    from paper_2507_06300_gb300 import binding as B
    rng = np.random.default_rng(n)
    m = max(n, 14)
    S = rng.permutation(np.abs(_spread(rng, m)))[:n]
    S = np.concatenate([S, np.round(rng.uniform(1, 1 << 26, n)) ** 2 * 2.0]) if n > 1 else S   # exact roots
    z = np.stack([_spread(rng, max(S.size, 14))[:S.size], np.ldexp(rng.standard_normal(S.size), rng.integers(-60, 60, S.size))],
                 axis=-1)
    d = B.fd_synthesize(torch.as_tensor(S[None], device="cuda"), torch.as_tensor(z[None], device="cuda")).cpu().numpy()[0]
    with np.errstate(all="ignore"):
        a = np.sqrt(0.5 * S)
        ref = a[:, None] * z
    assert np.array_equal(d, ref, equal_nan=True)


@pytest.mark.parametrize("width", [1, 11, 12, 13, 64, 257])
def test_periodogram_of_wide_ranges(width):
    import torch
    from paper_2507_06300_gb300 import binding as B
    rng = np.random.default_rng(width)
    nb, C = 300, 2
    n = nb * width
    d = np.ldexp(rng.standard_normal((C, n, 2)), rng.integers(-200, 200, (C, n, 1)))
    d[0, : n // 3] *= 2.0 ** -300                  # small squares, some below the normal range
    d[0, 5 * width] = np.inf
    d[1, 7 * width, 1] = np.nan
    d[1, 8 * width:9 * width] = 0.0
    d[1, 9 * width:10 * width] = 5e-324
    d[1, 11 * width] = 1e200                       # the square overflows
    off = torch.arange(nb + 1, dtype=torch.int64, device="cuda") * width
    P = B.averaged_periodogram(torch.as_tensor(d, device="cuda"), 1e-4, 1e-8, off)[0].cpu().numpy()
    with np.errstate(all="ignore"):
        # math.fsum-like reference: extended precision where the platform has it, scaled against underflow
        x = d.astype(np.longdouble)
        ref = ((x * x).sum(axis=-1).reshape(C, nb, width).sum(axis=-1) / width).astype(np.float64)
    ref[1, 11] = np.inf
    assert np.array_equal(np.isnan(P), np.isnan(ref)) and np.array_equal(np.isinf(P), np.isinf(ref))
    ok = np.isfinite(ref)
    # 1e-14 relative, and a few units of the smallest subnormal (squares that underflow in FP64)
    assert np.all(np.abs(P[ok] - ref[ok]) <= 1e-14 * np.abs(ref[ok]) + 2.0 * width * 5e-324)
