"""The FP64 path where exponents leave the range of its short forms (100 decades): states lifted or lowered by
120 decades beside ordinary ones in the same warps, log L and template gradients against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2507_06300_gb300 import synth
from tests._workloads import gpu_eval, oracle_dataset
from tests.test_gpu_grad import gpu_grad

pytestmark = pytest.mark.gpu
FP64 = 1


@pytest.mark.parametrize("sgwb", [0, 1, 2])
@pytest.mark.parametrize("n_bins,n_states", [(3, 1), (65, 5), (700, 33)])
def test_wide_exponents(n_bins, n_states, sgwb):
    """At the tolerances of ordinary states: 1e-12 of log L and of the template gradients' condition scale.  (The
    knots' gradients go through the reverse map, whose error at close knots and at components without any
    bin exceeds that bound whichever form the bins take.)"""
    wl = synth.workload("tiny", n_bins=n_bins, n_states=n_states, kmin=0, kmax_draw=6, sgwb_model=sgwb)
    wl.f_ref[:] = 3e-3
    w = wl.knots.w
    w[0::3, 0, :] += 120.0
    w[1::6, 1, :] -= 120.0
    if sgwb:
        w[2::6, 3, :] += 130.0
    ds = oracle_dataset(wl)
    L_ref, G_ref, sc, St = oracle.loglike_grad_scale(ds, wl.theta, wl.knots.as_dict())
    ok = (St & ~32) == 0
    L, _ = gpu_eval(wl, ds["P"], FP64)
    np.testing.assert_allclose(L[ok], L_ref[ok], rtol=1e-12, atol=0)
    Lg, G, _, _ = gpu_grad(wl, ds["P"], FP64)
    np.testing.assert_allclose(Lg[ok], L_ref[ok], rtol=1e-12, atol=0)
    assert np.all((np.abs(G - G_ref) <= 1e-12 * sc)[ok, :5]) and np.all(np.isfinite(G))
