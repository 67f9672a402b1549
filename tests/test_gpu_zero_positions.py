"""Knot positions and band edges at zero (1 Hz), of either sign: -0.0 and +0.0 are one position, so a
knot at the band's edge is refused and a pair of them is a duplicate, as in the oracle."""
import numpy as np
import pytest

import oracle
from paper_2507_06300_gb300 import synth
from tests._workloads import gpu_eval, oracle_dataset
from tests.test_gpu_grad import gpu_grad

pytestmark = pytest.mark.gpu
FP32, FP64 = 0, 1
EDGE = {-1: (0.05, 0.9), 0: (0.05, 20.0), 1: (1.1, 20.0)}   # bins below, around and above 1 Hz


@pytest.mark.parametrize("precision", [FP64, FP32])
@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("side,edge", [(-1, 0.0), (-1, -0.0), (1, 0.0), (1, -0.0), (0, None)])
def test_zero_positions(side, edge, kind, precision):
    lo, hi = EDGE[side]
    wl = synth.workload("tiny", n_bins=64, n_states=6, kmin=3, kmax_draw=3, kind=kind, f_min=lo, f_max=hi)
    k = wl.knots
    if side < 0:
        wl.x_hi[:] = edge
    elif side > 0:
        wl.x_lo[:] = edge
    P = oracle_dataset(wl)["P"]
    # states 0, 1: no knot at zero; 2, 3: one at -0.0, +0.0; 4: both, next to each other; 5: apart
    k.x[3], k.w[3], wl.theta[3] = k.x[2], k.w[2], wl.theta[2]
    k.x[2, 0, 1], k.x[3, 0, 1] = -0.0, 0.0
    k.x[4, 3, :2] = -0.0, 0.0
    k.x[5, 2, 0], k.x[5, 2, 2] = 0.0, -0.0
    ds = oracle_dataset(wl)
    ds["P"] = P
    L_ref, st_ref = oracle.loglike(ds, wl.theta, k.as_dict())
    assert np.array_equal(st_ref != 0, [False, False, side != 0, side != 0, True, True])
    L, st = gpu_eval(wl, P, precision)
    np.testing.assert_array_equal(st & ~32, st_ref)
    assert np.all(np.isneginf(L[st_ref != 0]))
    Lg, G, st_g, _ = gpu_grad(wl, P, precision)
    np.testing.assert_array_equal(st_g & ~32, st_ref)
    assert np.all(np.isneginf(Lg[st_ref != 0])) and np.all(G[st_ref != 0] == 0.0) and np.all(np.isfinite(G))
    if side == 0:   # a knot at zero is the same knot whatever its sign
        assert L[2] == L[3] and np.array_equal(G[2], G[3])
