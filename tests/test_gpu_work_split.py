"""Small problems, whose work items and adjoint ranges the library splits to fill the GPU: log L and the
gradient against the oracle at the edges of the split (one bin past a chunk, ragged last tiles, state
counts that leave rows and lanes empty), at the tolerances of the unsplit paths."""
import numpy as np
import pytest

from paper_2507_06300_gb300 import synth
from tests._workloads import fp32_tolerance, gpu_eval, oracle_batched, oracle_dataset
from tests.test_gpu_grad import gpu_grad

pytestmark = pytest.mark.gpu
FP32, FP64 = 0, 1


def _wl(n_bins, n_states, **kw):
    return synth.workload("tiny", n_bins=n_bins, n_states=n_states, kmin=0, kmax_draw=8, **kw)


@pytest.mark.parametrize("precision", [FP64, FP32])
@pytest.mark.parametrize("n_bins,n_states", [(1, 1), (63, 3), (65, 17), (129, 33), (513, 40), (577, 65), (1025, 129),
                                             (4097, 130)])
def test_loglike_split(precision, n_bins, n_states):
    wl = _wl(n_bins, n_states)
    P, L_ref, St = oracle_batched(wl)
    L, St_gpu = gpu_eval(wl, P, precision)
    np.testing.assert_array_equal(St_gpu, St)
    ok = St == 0
    if precision == FP64:
        np.testing.assert_allclose(L[ok], L_ref[ok], rtol=1e-12, atol=0)
    else:
        assert np.all(np.abs(L[ok] - L_ref[ok]) <= fp32_tolerance(L_ref, wl, P)[ok])


@pytest.mark.parametrize("precision", [FP64, FP32])
@pytest.mark.parametrize("n_bins,n_states,kind", [(1, 2, 0), (127, 5, 0), (128, 33, 1), (129, 32, 0), (2049, 31, 0),
                                                  (4100, 40, 1)])
def test_gradient_split(precision, n_bins, n_states, kind):
    """A small problem's gradient (128-bin ranges) against the same states and data inside a data
    object with enough other work to keep 2,048-bin ranges.  Every per-bin value and FP32 chunk sum is
    the same; only the grouping of the float-float and FP64 sums differs (2^-46 per sum), so each
    component agrees to 1e-9 of the state's largest one."""
    import torch
    from paper_2507_06300_gb300 import binding as B
    wl = _wl(n_bins, n_states)
    wl.knots.kind = kind
    wl.f_ref[:] = 3e-3
    ds_o = oracle_dataset(wl, 0)
    P = ds_o["P"]
    L1, G1, St, _ = gpu_grad(wl, P, precision)
    # the filler: one more dataset of 2,048-bin ranges x 32 states on every warp the rule asks for
    n_fill, s_fill = 2048 * 64, 1024
    fill = synth.workload("tiny", n_bins=n_fill, n_states=s_fill, kmin=0, kmax_draw=0, kmax=wl.knots.kmax)
    f = np.concatenate([wl.f, fill.f])
    k, kf = wl.knots, fill.knots
    ds = B.Dataset(n_channels=3, freq=f, nu=np.concatenate([wl.nu, fill.nu]),
                   periodogram=np.concatenate([P, np.ones((3, n_fill))], axis=1),
                   response=np.concatenate([wl.R, fill.R], axis=1), bin_offset=np.array([0, n_bins, n_bins + n_fill]),
                   state_offset=np.array([0, n_states, n_states + s_fill]), x_lo=np.full(2, wl.x_lo[0]),
                   x_hi=np.full(2, wl.x_hi[0]), f_ref=np.full(2, wl.f_ref[0]))
    cat = lambda a, b: torch.as_tensor(np.concatenate([a, b]), device="cuda")
    count, x, w, th = cat(k.count, kf.count), cat(k.x, kf.x), cat(k.w, kf.w), cat(wl.theta, fill.theta)
    buf, st = ds.spline_setup(count, x, w, k.kmax, kind, precision)
    L2, G2 = ds.psd_loglike_grad(th, count, x, w, k.kmax, kind, buf, precision)
    L2, G2 = L2.cpu().numpy()[:n_states], G2.cpu().numpy()[:n_states]
    np.testing.assert_array_equal(st.cpu().numpy()[:n_states], St)
    ds.close()
    assert np.all(np.isfinite(G1)) and np.all(np.isfinite(L1[St == 0]))
    np.testing.assert_allclose(L1, L2, rtol=1e-13, atol=0)
    assert np.all(np.abs(G1 - G2) <= 1e-9 * np.abs(G2).max(axis=1, keepdims=True))


@pytest.mark.parametrize("n_bins,n_states", [(2, 65), (63, 70), (130, 129), (1025, 66)])
def test_dense_one_warp_ctas(n_bins, n_states):
    """The dense covariance with more than 64 states (one warp per CTA, staged pieces, items split in segments)
    at ragged sizes against tiles of one piece: the same FP32 sums, so only the order of their FP64 sum and the
    last rounding of log L may differ.  Permuting the states permutes the results."""
    from tests._workloads import fp32_tolerance_full, oracle_dataset_full
    wl = synth.workload("tiny", cov_model=1, n_bins=n_bins, n_states=n_states)
    P9 = oracle_dataset_full(wl)["P9"]
    L, St = gpu_eval(wl, P9, FP32)
    Lr, Sr = gpu_eval(wl, P9, FP32, tiling=dict(tile_bins=64, states_per_cta=128, group=2))
    np.testing.assert_array_equal(St, Sr)
    ok = St == 0
    # 1e-13 of the summed magnitudes (the FP32 bound is 1e-6 of them) and 4 roundings of log L
    tol = 1e-7 * fp32_tolerance_full(Lr, wl, P9) + 4 * 2.3e-16 * np.abs(Lr)
    assert np.all(np.abs(L[ok] - Lr[ok]) <= tol[ok])
    o = np.random.default_rng(n_states).permutation(n_states)
    k = wl.knots
    kn = synth.Knots(count=k.count[o].copy(), x=k.x[o].copy(), w=k.w[o].copy(), kmax=k.kmax, kind=k.kind)
    Lp, Sp = gpu_eval(wl, P9, FP32, theta=wl.theta[o].copy(), knots=kn)
    np.testing.assert_array_equal(Sp, St[o])
    assert np.all(np.abs(Lp - L[o])[Sp == 0] <= tol[o][Sp == 0])


@pytest.mark.parametrize("run", [1, 2, 63, 64, 65, 130])
def test_fp64_runs_of_equal_nu(run):
    """The FP64 kernels take one logarithm per run of bins with equal nu (at most 64): log L of the forward
    call and of the gradient call with nu changing every `run` bins, some of it zero."""
    wl = _wl(700, 40)
    wl.nu = np.array([4.0, 0.0, 7.0, 1.0, 128.0])[(np.arange(700) // run) % 5]
    P, L_ref, St = oracle_batched(wl)
    Lg, _, _, L = gpu_grad(wl, P, FP64)
    ok = St == 0
    np.testing.assert_allclose(L[ok], L_ref[ok], rtol=1e-12, atol=0)
    np.testing.assert_allclose(Lg[ok], L_ref[ok], rtol=1e-12, atol=0)


@pytest.mark.parametrize("n_bins,n_states", [(1, 1), (15, 2), (31, 3), (64, 16), (1001, 5), (4097, 1), (700, 17)])
def test_fp64_rows(n_bins, n_states):
    """The FP64 likelihood of few states: each warp's lanes split the bins in rows, some of them empty, at
    the tolerance of many states."""
    wl = _wl(n_bins, n_states)
    P, L_ref, St = oracle_batched(wl)
    L, St_gpu = gpu_eval(wl, P, FP64)
    np.testing.assert_array_equal(St_gpu, St)
    ok = St == 0
    np.testing.assert_allclose(L[ok], L_ref[ok], rtol=1e-12, atol=0)


@pytest.mark.parametrize("n_bins,n_states", [(700, 1), (701, 6), (1024, 16)])
def test_fp64_rows_dense(n_bins, n_states):
    """The same for the dense covariance."""
    import oracle
    from tests._workloads import oracle_dataset_full
    wl = synth.workload("tiny", cov_model=1, n_bins=n_bins, n_states=n_states)
    ds = oracle_dataset_full(wl)
    L_ref, St_ref = oracle.loglike_full(ds, wl.theta, wl.knots.as_dict())
    L, _ = gpu_eval(wl, ds["P9"], FP64)
    ok = St_ref == 0
    np.testing.assert_allclose(L[ok], L_ref[ok], rtol=1e-12, atol=0)
