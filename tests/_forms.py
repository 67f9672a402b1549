"""Calls that reach the kernel forms of small problems and of many states: the one-chunk likelihood kernel
(more than 64 states on few bins), the one-warp dense kernel (more than 64 states) and the fallback pass's
longer ranges.  Shared by the release and the bounds-checked tests."""
import numpy as np

from paper_2507_06300_gb300 import synth
from tests._workloads import gpu_eval, oracle_dataset, oracle_dataset_full


def chunk_workload(n_bins, n_states, n_channels, sgwb):
    """Cold and hot states; every fifth has a pair of close knots on the first spline (ill-conditioned
    intervals: masked bins), every seventh amplitudes 1e7 times the injected ones (channel products beyond
    2^125: the guarded redo)."""
    wl = synth.workload("tiny", n_bins=n_bins, n_states=n_states, n_channels=n_channels, sgwb_model=sgwb, kmin=2, kmax_draw=6)
    wl.f_ref[:] = 3e-3
    rng = np.random.default_rng(n_bins + n_states)
    k = wl.knots
    for s in range(0, n_states, 5):
        k.x[s, 0, 1] = k.x[s, 0, 0] + rng.uniform(2e-5, 2e-4) * (1 if k.x[s, 0, 0] < -2 else -1)
    wl.theta[::7, :2] *= 1e7
    return wl, oracle_dataset(wl)["P"]


def eval_beside(wl, P, precision=0):
    """The same data set and states in a data object with a second data set (64 bins, one state) in front."""
    import torch
    from paper_2507_06300_gb300 import binding as B
    one = synth.workload("tiny", n_bins=64, n_states=1, n_channels=wl.n_channels, sgwb_model=wl.sgwb_model, kmin=0,
                         kmax_draw=0, kmax=wl.knots.kmax)
    cat = lambda a, b, ax=0: np.concatenate([a, b], axis=ax)
    two = lambda v: np.full(2, float(v[0]))
    n, S = wl.n_bins, wl.n_states
    ds = B.Dataset(n_channels=wl.n_channels, freq=cat(one.f, wl.f), nu=cat(one.nu, wl.nu),
                   periodogram=cat(np.ones((wl.n_channels, 64)), P, 1),
                   response=cat(one.R, wl.R, 1) if wl.sgwb_model else None, bin_offset=np.array([0, 64, 64 + n]),
                   state_offset=np.array([0, 1, 1 + S]), x_lo=two(wl.x_lo), x_hi=two(wl.x_hi), f_ref=two(wl.f_ref),
                   sgwb_model=wl.sgwb_model)
    k, ko = wl.knots, one.knots
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    count, x, w, th = dev(cat(ko.count, k.count)), dev(cat(ko.x, k.x)), dev(cat(ko.w, k.w)), dev(cat(one.theta, wl.theta))
    buf, st = ds.spline_setup(count, x, w, k.kmax, k.kind, precision)
    L = ds.psd_loglike(th, buf, k.kmax, precision).cpu().numpy()[1:]
    st = st.cpu().numpy()[1:]
    ds.close()
    return L, st


def dense_workload(n_bins, n_states, sgwb):
    wl = synth.workload("tiny", cov_model=1, n_bins=n_bins, n_states=n_states, sgwb_model=sgwb)
    wl.f_ref[:] = 3e-3
    return wl, oracle_dataset_full(wl)["P9"]


def dense_eval(wl, P9, states_per_cta):
    return gpu_eval(wl, P9, 0, tiling=dict(tile_bins=512, states_per_cta=states_per_cta, group=4))
