"""The FP32 gradient's fallback pass (states beyond the FP32 range) at the edges of its choice of ranges: few
flagged states take the adjoint's ranges, many take longer ones that hold several of them."""
import numpy as np
import pytest

from paper_2507_06300_gb300 import synth
from tests._workloads import oracle_dataset
from tests.test_gpu_grad import gpu_grad

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("n_bins,n_states", [(1, 700), (127, 400), (129, 320), (2049, 90), (2050, 300), (4097, 300),
                                             (9001, 200)])
def test_fallback_ranges(n_bins, n_states, kind):
    """Every state's first noise spline lifted by 45 decades (its sums leave the FP32 range), against calls in
    which one state alone is lifted: every per-bin value is the same, only the grouping of the FP64 sums
    differs (2^-53 per sum, through the reverse map), so each component agrees to 1e-9 of the state's
    largest one and log L to 1e-13."""
    wl = synth.workload("tiny", n_bins=n_bins, n_states=n_states, kmin=0, kmax_draw=8)
    wl.knots.kind = kind
    wl.f_ref[:] = 3e-3
    P = oracle_dataset(wl)["P"]
    w0 = wl.knots.w.copy()
    wl.knots.w[:, 0, :] += 45.0
    lifted = wl.knots.w.copy()
    L, G, St, _ = gpu_grad(wl, P, 0)
    ok = (St & ~32) == 0
    assert ok.sum() >= n_states // 2 and np.all(np.isfinite(L[ok])) and np.all(np.isfinite(G))
    for s in np.flatnonzero(ok)[[0, ok.sum() // 2, -1]]:
        wl.knots.w[:] = w0
        wl.knots.w[s] = lifted[s]
        L1, G1, _, _ = gpu_grad(wl, P, 0)
        np.testing.assert_allclose(L1[s], L[s], rtol=1e-13, atol=0)
        assert np.all(np.abs(G1[s] - G[s]) <= 1e-9 * np.abs(G[s]).max()), s
