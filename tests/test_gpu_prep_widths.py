"""The averaged periodogram's forms (fixed point on the integer pipes, FP64 one channel after the other, FP64 all
channels together): bins of every width beside each other, few bins and many, against extended-precision
sums.  All terms are positive, so a sum of n squares in FP64 is within (2 n + 8) 2^-53 of itself; the fixed
point's bound, 3 n 2^-62, lies below."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _widths(rng, kind, nb):
    if kind == "narrow_and_wide":   # mean about 13: bins on both sides of the fixed point's line, some far wider
        w = rng.choice([1, 2, 3, 11, 12, 13, 14, 30], nb)
        w[rng.permutation(nb)[:nb // 100 + 1]] = 211
        return w
    if kind == "ones_and_wide":     # mean below 12: one lane per bin
        w = np.ones(nb, np.int64)
        w[rng.permutation(nb)[:nb // 200 + 1]] = 1500
        return w
    if kind == "wide":              # mean above 256: eight lanes per bin
        return rng.integers(1, 700, nb)
    return rng.integers(0, 40, nb)  # empty bins among them


@pytest.mark.parametrize("channels", [1, 2, 3])
@pytest.mark.parametrize("kind,nb", [("narrow_and_wide", 300), ("narrow_and_wide", 21000), ("ones_and_wide", 90000),
                                     ("ones_and_wide", 400), ("wide", 200), ("wide", 10000), ("empty", 22000)])
def test_every_width(kind, nb, channels):
    import torch
    from paper_2507_06300_gb300 import binding as B
    rng = np.random.default_rng(nb + channels)
    w = _widths(rng, kind, nb)
    off = np.concatenate([[0], np.cumsum(w)]).astype(np.int64)
    n = int(off[-1])
    d = np.ldexp(rng.standard_normal((channels, n, 2)), rng.integers(-40, 40, (channels, n, 1)))
    d[:, : n // 3] *= 2.0 ** -600                      # squares below the normal range
    big = [int(v) for v in rng.choice(np.flatnonzero(w), 3, replace=False)]
    d[0, off[big[0]]] = np.inf
    d[-1, off[big[1] + 1] - 1, 1] = np.nan
    d[0, off[big[2]]] = 1e200                          # the square overflows
    P, f, nu = B.averaged_periodogram(torch.as_tensor(d, device="cuda"), 1e-4, 1e-8, torch.as_tensor(off, device="cuda"))
    P = P.cpu().numpy()
    np.testing.assert_array_equal(nu.cpu().numpy(), w)
    with np.errstate(all="ignore"):
        x = d.astype(np.longdouble)
        c = np.concatenate([np.zeros((channels, 1), np.longdouble), (x * x).sum(axis=-1)], axis=1)
        live = np.flatnonzero(w)
        ref = np.full((channels, nb), np.nan)
        ref[:, live] = (np.add.reduceat(c[:, 1:], off[:-1][live], axis=1) / w[live]).astype(np.float64)
    if big[2] not in big[:2]:
        ref[0, big[2]] = np.inf if not np.isnan(ref[0, big[2]]) else np.nan
    assert np.array_equal(np.isnan(P), np.isnan(ref)) and np.array_equal(np.isinf(P), np.isinf(ref))
    ok = np.isfinite(ref)
    # (plus a few units of the smallest subnormal: squares that underflow in FP64)
    tol = (2.0 * w + 8.0) * 2.0 ** -53 * np.abs(ref) + 4.0 * np.maximum(w, 1) * 5e-324
    assert np.all(np.abs(P[ok] - ref[ok]) <= tol[ok])
