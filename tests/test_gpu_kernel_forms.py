"""The kernel forms of small problems and of many states against the forms that they stand in for."""
import numpy as np
import pytest

import oracle
from tests import _forms
from tests._workloads import fp32_tolerance, fp32_tolerance_full, gpu_eval, oracle_dataset

pytestmark = pytest.mark.gpu
FP32 = 0


@pytest.mark.parametrize("n_channels,sgwb", [(2, 0), (2, 1), (2, 2), (3, 0), (3, 1), (3, 2)])
@pytest.mark.parametrize("n_bins,n_states", [(1, 65), (63, 100), (66, 128), (577, 129), (2000, 128), (4097, 70)])
def test_chunk_kernel_is_the_fused_kernel(n_bins, n_states, n_channels, sgwb):
    """More than 64 states on few bins take the one-chunk kernel; beside a data set of one state the same
    call takes the fused kernel, on the same 64-bin chunks: the same bits.  And the FP32 bound against the
    oracle."""
    wl, P = _forms.chunk_workload(n_bins, n_states, n_channels, sgwb)
    L, St = gpu_eval(wl, P, FP32)
    L2, St2 = _forms.eval_beside(wl, P)
    np.testing.assert_array_equal(St, St2)
    np.testing.assert_array_equal(L, L2)
    ds = oracle_dataset(wl)
    L_ref, St_ref = oracle.loglike(ds, wl.theta, wl.knots.as_dict())
    np.testing.assert_array_equal(St & ~32, St_ref & ~32)
    ok = St_ref == 0
    if n_bins >= 2000:   # (the bound is one of many bins' sum)
        assert np.all(np.abs(L[ok] - L_ref[ok]) <= fp32_tolerance(L_ref, wl, P)[ok])


@pytest.mark.parametrize("sgwb", [0, 1, 2])
@pytest.mark.parametrize("n_bins,n_states", [(2, 65), (63, 70), (130, 129), (1025, 66), (4097, 200)])
def test_dense_one_warp_form_against_rows(n_bins, n_states, sgwb):
    """More than 64 states, 128 to an item: one warp per CTA.  With 64 to an item the same call takes the form
    whose threads split a state's bins over rows.  Every bin's term is the same; the FP32 sums run over other
    chunks of at most 16 terms, so each side is within 16 x 2^-24 = 1e-6 of the summed magnitudes, which are at
    most twice the scale of the FP32 bound (1e-6 of it): four bounds."""
    wl, P9 = _forms.dense_workload(n_bins, n_states, sgwb)
    L1, S1 = _forms.dense_eval(wl, P9, 128)
    L4, S4 = _forms.dense_eval(wl, P9, 64)
    np.testing.assert_array_equal(S1, S4)
    ok = S1 == 0
    assert np.all(np.abs(L1 - L4)[ok] <= 4.0 * fp32_tolerance_full(L4, wl, P9)[ok])
