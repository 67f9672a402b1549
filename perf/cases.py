"""The calls this framework is timed on: what a program that uses it has it do, over the real range.

A case is one call (or the short fixed sequence of calls a user makes together) on one set of
sizes and options:

  host     ``Evaluator.loglike_host``: a host-side sampler's step, pinned inputs in, log L out
  step     ``Evaluator.replay``: the same step on device-resident inputs (spline setup + log L)
  grad     ``Dataset.spline_setup`` + ``Dataset.psd_loglike_grad`` with kept buffers: one
           likelihood-and-gradient call of the sampler's MALA move
  psd      ``Dataset.spline_setup`` + ``Dataset.model_psd``: the model PSD of posterior draws
  simulate ``fd_synthesize`` + ``averaged_periodogram``: a simulated realisation and its averaged
           periodogram, the inputs of a dataset

Inputs follow the shapes of ``synth`` (its frequency grid, response stand-in, Table I priors): bins
uniform in 0.1-29 mHz, periodograms Gamma-scattered around the injected PSD, half of an ensemble's
states near the injection (cold chains) and half from the priors (hot chains), knot positions
uniform in log10 f in any order, amplitudes N(0, 0.1).  Knots of one spline stay 1e-3 decades
apart (closer pairs of prior draws give PSD values of hundreds of decades, states that no chain
keeps), which still leaves ill-conditioned intervals in the ensembles.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2507_06300_gb300 import binding as B
from paper_2507_06300_gb300 import synth

F64 = torch.float64
MIN_GAP = 1.0e-3   # smallest distance of two knots of a spline, decades in f

ARM, CLIGHT, H0H = 2.5e9, 299792458.0, 1.0e5 / 3.0856775814913673e22


def _ens(name, call, channels, bins, states, kmin, kmax, **kw):
    """An ensemble case: its defaults are the averaged A, E, T periodogram with a power-law
    background, Akima splines and the FP32 path."""
    c = dict(name=name, call=call, channels=channels, bins=bins, states=states, kmin=kmin, kmax=kmax, datasets=1,
             nu=64, sgwb=1, kind=0, precision=0, dense=False, mixed=True)
    c.update(kw)
    return c


def listed():
    return [
        # a host sampler on a short A, E record: 32 walkers x 4 temperatures; latency and launches
        _ens("host_small", "host", 2, 2000, 128, 2, 4, nu=16),
        # the paper's step: 64 walkers x 16 temperatures on the full averaged record
        _ens("step_paper", "step", 3, 131072, 1024, 0, 20),
        # many records at once, uneven lengths, few cold states on each
        _ens("step_batched", "step", 3, 24000, 16, 0, 30, datasets=128, mixed=False),
        # the largest ensemble: 32 temperatures x 256 walkers, broken power law, 0-40 knots
        _ens("step_full", "step", 3, 524288, 8192, 0, 40, nu=128, sgwb=2),
        # the dense A, E, T covariance with its three correlation splines
        _ens("step_dense", "step", 3, 131072, 1024, 0, 20, dense=True),
        # the double-precision option: checking an ensemble of 20 x 20 states; an odd bin count
        _ens("step_fp64", "step", 3, 65537, 400, 0, 10, precision=1),
        # one MALA call of the small sampler
        _ens("grad_small", "grad", 2, 2000, 128, 2, 4, nu=16),
        # one MALA call of the paper's 20 x 20 ensemble on a coarse record, odd bin count
        _ens("grad_20x20", "grad", 3, 8191, 400, 0, 10),
        # the large gradient: 256 walkers x 8 temperatures
        _ens("grad_large", "grad", 3, 131072, 2048, 6, 10),
        # gradient in double precision, natural cubic splines
        _ens("grad_fp64", "grad", 3, 16384, 400, 0, 10, kind=1, precision=1),
        # posterior PSD bands: the model PSD of 64 cold draws
        _ens("psd_posterior", "psd", 3, 131072, 64, 0, 10, precision=1, mixed=False),
        # a simulated year of data: 64 samples a bin
        dict(name="simulate", call="simulate", channels=3, bins=131072, width=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["host", "step", "step", "step", "grad", "grad", "psd", "simulate"])
    if call == "simulate":
        width = _log_int(rng, 1, 300)
        bins = _log_int(rng, 2000, 131072 * 64 // max(width, 64))
        return dict(call=call, channels=rng.choice([2, 3]), bins=bins, width=width)
    precision = 1 if call == "psd" or rng.random() < 0.25 else 0
    dense = call == "step" and rng.random() < 0.2
    # state-bins of the largest listed case of each kind
    if call == "psd":
        most = 64 * 131072
    elif call == "grad":
        most = 400 * 16384 if precision else 2048 * 131072
    elif dense:
        most = 8 * 10 ** 6 if precision else 1024 * 131072
    else:
        most = 400 * 65537 if precision else 1024 * 262144
    bins = _log_int(rng, 500, 262144)
    states = _log_int(rng, 4, 4096)
    datasets = rng.choice([1, 1, 1, _log_int(rng, 2, 64)])
    if datasets > 1:
        bins, states = min(bins, 65536), min(states, 64)
    while bins * states * datasets > most:
        if states > 8 and (states > 256 or bins <= 4096):
            states = -(-states * 2 // 3)
        elif bins > 500:
            bins = bins * 2 // 3 + 1
        else:
            datasets = max(1, datasets // 2)
    kmax = rng.choice([0, 1, 2, 4, 7, 10, 10, 20, 20, 40])
    return dict(call=call, channels=3 if dense else rng.choice([2, 3, 3]), bins=bins, states=states,
                kmin=rng.choice([0, 0, kmax // 2, kmax]), kmax=kmax, datasets=datasets,
                nu=rng.choice([1, 4, 16, 64, 128]) if not dense else rng.choice([16, 64, 128]),
                sgwb=rng.choice([0, 1, 1, 1, 2]), kind=rng.choice([0, 0, 0, 1]), precision=precision, dense=dense,
                mixed=rng.random() < 0.6 and call != "psd")


# ---- inputs -------------------------------------------------------------------------------------

def _templates(f, R):
    """Per unit amplitude^2 (Table I units) at the frequencies f: noise of A / E and T from the optical
    metrology and the test masses, and the background per unit h^2 Omega and response."""
    u = 2.0 * np.pi * f * ARM / CLIGHT
    su, cu = np.sin(u), np.cos(u)
    pref = su ** 6
    omc = 2.0 * np.sin(0.5 * u) ** 2
    oms = 1.0e-24 * (1.0 + (2.0e-3 / f) ** 4) * (2.0 * np.pi * f / CLIGHT) ** 2
    tm = 1.0e-30 * (1.0 + (0.4e-3 / f) ** 2) * (1.0 + (f / 8.0e-3) ** 4) / (2.0 * np.pi * f * CLIGHT) ** 2
    go = np.stack([32.0 * pref * (2.0 + cu) * oms] * 2 + [64.0 * pref * omc * oms])
    gt = np.stack([128.0 * pref * (1.0 + cu + cu * cu) * tm] * 2 + [128.0 * pref * omc * omc * tm])
    gh = R * (3.0 * H0H ** 2 / (4.0 * np.pi ** 2 * f ** 3)) if R is not None else None
    return go, gt, gh


def _knots(rng, S, nsp, kmin, kmax, x_lo, x_hi):
    """Counts uniform in kmin..kmax, positions uniform at least MIN_GAP apart, in any order."""
    count = rng.integers(kmin, kmax + 1, size=(S, nsp)).astype(np.int32)
    j = np.arange(kmax)
    live = j < count[:, :, None]
    u = np.where(live, rng.random((S, nsp, kmax)), 2.0)
    u = np.sort(u, axis=2)
    room = (x_hi - x_lo) - (count[:, :, None] + 1) * MIN_GAP
    x = np.where(live, x_lo + u * room + (j + 1) * MIN_GAP, 0.0)
    order = np.argsort(np.where(live, rng.random((S, nsp, kmax)), 2.0), axis=2)
    x = np.take_along_axis(x, order, axis=2)
    w = 0.1 * rng.standard_normal((S, nsp, kmax + 2))
    jw = np.arange(kmax + 2)
    w = np.where((jw == 0) | (jw == kmax + 1) | ((jw >= 1) & (jw <= count[:, :, None])), w, 0.0)
    return count, np.ascontiguousarray(x), np.ascontiguousarray(w)


def _inputs(case, seed):
    """The numpy inputs of an ensemble case, from the seed alone."""
    rng = np.random.default_rng([int(seed), 77])
    C, nd, sg = case["channels"], case["datasets"], case["sgwb"]
    dense = case["dense"]
    lens = [case["bins"]] if nd == 1 else [int(v) for v in rng.integers(max(1, case["bins"] // 3), case["bins"] * 5 // 3 + 2,
                                                                        size=nd)]
    true = np.empty((nd, 5))
    fs, Ps, Rs, Xs, thetas = [], [], [], [], []
    x_lo, x_hi = math.log10(synth.F_MIN), math.log10(synth.F_MAX)
    f_ref = 3.0e-3 if sg == 2 else 1.0e-3
    S1 = case["states"]
    for d, n in enumerate(lens):
        lA, n1 = (-12.0, 2.0 / 3.0) if nd == 1 else (rng.uniform(-13.0, -11.0), rng.uniform(-1.0, 3.0))
        true[d] = (15.0, 3.0, lA, n1, -1.0 if sg == 2 else n1)
        f = synth.freq_grid(n)
        R = synth.response_standin(f, C) if sg else None
        go, gt, gh = _templates(f, R)
        noise = 15.0 ** 2 * go[:C] + 3.0 ** 2 * gt[:C]
        back = 0.0
        if sg:
            sl = np.where(f < f_ref, true[d, 3], true[d, 4])
            back = 10.0 ** lA * (f / f_ref) ** sl * gh
        nu = np.full(n, float(case["nu"]))
        if dense:
            W = synth.complex_wishart_unit(rng, nu)
            P9 = _colour(noise, noise + back, W)
            Ps.append(P9[:3])
            Xs.append(P9[3:])
        else:
            Ps.append((noise + back) * synth.gamma_multipliers(rng, C, nu))
        fs.append(f)
        if sg:
            Rs.append(R)
        if case["mixed"]:
            cold = S1 // 2
            thetas += [synth.draw_theta(rng, cold, "posterior", true[d], sg),
                       synth.draw_theta(rng, S1 - cold, "prior", true[d], sg)]
        else:
            thetas.append(synth.draw_theta(rng, S1, "posterior", true[d], sg))
    nsp = C + (1 if sg else 0) + (3 if dense else 0)
    count, x, w = _knots(rng, S1 * nd, nsp, case["kmin"], case["kmax"], x_lo, x_hi)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    return dict(f=np.concatenate(fs), nu=np.full(int(off[-1]), float(case["nu"])), P=np.concatenate(Ps, axis=1),
                R=np.concatenate(Rs, axis=1) if sg else None, X=np.concatenate(Xs, axis=1) if dense else None,
                bin_offset=off, state_offset=np.arange(nd + 1, dtype=np.int64) * S1, x_lo=x_lo, x_hi=x_hi, f_ref=f_ref,
                theta=np.concatenate(thetas), count=count, x=x, w=w, nsp=nsp)


def _colour(noise, total, W):
    """P = L W L^T with L the Cholesky factor of the injected covariance (constant correlations
    z = 0.05, 0.03, -0.04 of the noise, the background on the diagonal), per bin: the auto-powers and the
    real parts of P_AE, P_AT, P_ET, [6, N]."""
    z = np.array(synth.Z_INJ)
    s = 1.0 / np.sqrt(1.0 + z * z)
    r = z * s
    cor = {(1, 0): r[0], (2, 0): r[1], (2, 1): r[0] * r[1] + s[0] * s[1] * r[2]}
    n = noise.shape[1]
    Cm = np.zeros((n, 3, 3))
    for c in range(3):
        Cm[:, c, c] = total[c]
    for (a, b), v in cor.items():
        Cm[:, a, b] = Cm[:, b, a] = v * np.sqrt(noise[a] * noise[b])
    L = np.linalg.cholesky(Cm)
    M = np.zeros((n, 3, 3), dtype=np.complex128)
    for c in range(3):
        M[:, c, c] = W[c]
    for k, (a, b) in enumerate(((0, 1), (0, 2), (1, 2))):
        M[:, a, b] = W[3 + 2 * k] + 1j * W[4 + 2 * k]
        M[:, b, a] = np.conj(M[:, a, b])
    P = L @ M @ np.transpose(L, (0, 2, 1))
    return np.stack([P[:, c, c].real for c in range(3)] + [P[:, a, b].real for a, b in ((0, 1), (0, 2), (1, 2))])


def _simulation(case, seed):
    """PSD, standard normal draws and bin offsets of a simulated record (device tensors)."""
    C, n = case["channels"], case["bins"] * case["width"]
    f = synth.freq_grid(n)
    go, gt, _ = _templates(f, None)
    psd = torch.as_tensor(15.0 ** 2 * go[:C] + 3.0 ** 2 * gt[:C], device="cuda")
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 2 + 1)
    z = torch.randn((C, n, 2), generator=g, dtype=F64, device="cuda")
    off = torch.arange(case["bins"] + 1, dtype=torch.int64, device="cuda") * case["width"]
    return dict(psd=psd, z=z, off=off, f0=float(f[0]), df=float((f[-1] - f[0]) / max(n - 1, 1)))


# ---- prepare / run ----------------------------------------------------------------------------

def prepare(case, seed):
    if case["call"] == "simulate":
        st = _simulation(case, seed)
        st["d"] = torch.empty_like(st["z"])
        st["call"] = "simulate"
        return st
    q = _inputs(case, seed)
    nd = case["datasets"]
    ds = B.Dataset(n_channels=case["channels"], freq=q["f"], nu=q["nu"], periodogram=q["P"], response=q["R"],
                   bin_offset=q["bin_offset"], state_offset=q["state_offset"], x_lo=np.full(nd, q["x_lo"]),
                   x_hi=np.full(nd, q["x_hi"]), f_ref=np.full(nd, q["f_ref"]), sgwb_model=case["sgwb"],
                   cov_model=B.COV_FULL if case["dense"] else B.COV_DIAGONAL, periodogram_cross=q["X"])
    kmax, kind, prec = case["kmax"], case["kind"], case["precision"]
    st = dict(call=case["call"], ds=ds, kmax=kmax, kind=kind, prec=prec)
    if case["call"] in ("host", "step"):
        ev = B.Evaluator(ds, kmax, kind, prec)
        st["ev"] = ev
        if case["call"] == "host":
            h = ev.host_inputs()
            for dst, k in zip(h, ("theta", "count", "x", "w")):
                dst.copy_(torch.as_tensor(q[k]))
            st["args"] = (*h, torch.empty(ds.n_states, dtype=F64).pin_memory())
            ev.capture_host(*st["args"])
        else:
            ev.load(*(torch.as_tensor(q[k]) for k in ("theta", "count", "x", "w")))
            ev.capture()
    else:
        for k in ("theta", "count", "x", "w"):
            st[k] = torch.as_tensor(q[k], device="cuda")
        st["buf"] = torch.empty(ds.spline_buf_bytes(kmax, prec), dtype=torch.uint8, device="cuda")
        if case["call"] == "grad":
            st["ws"] = torch.empty(ds.workspace_bytes(kmax, prec, True), dtype=torch.uint8, device="cuda")
        else:
            st["out"] = torch.empty(ds.n_channels * ds.n_states * case["bins"] if nd == 1 else
                                    int(ds.n_channels * case["states"] * ds.n_bins), dtype=F64, device="cuda")
    return st


def run(state):
    call = state["call"]
    if call == "simulate":
        d = B.fd_synthesize(state["psd"], state["z"], out=state["d"])
        P, f, nu = B.averaged_periodogram(d, state["f0"], state["df"], state["off"])
        return {"d": d, "P": P, "f": f, "nu": nu}
    if call == "host":
        return {"logL": state["ev"].loglike_host(*state["args"]), "status": state["ev"].status}
    if call == "step":
        return {"logL": state["ev"].replay(), "status": state["ev"].status}
    ds = state["ds"]
    _, status = ds.spline_setup(state["count"], state["x"], state["w"], state["kmax"], state["kind"], state["prec"],
                                buf=state["buf"])
    if call == "psd":
        return {"psd": ds.model_psd(state["theta"], state["buf"], state["kmax"], out=state["out"]), "status": status}
    L, g = ds.psd_loglike_grad(state["theta"], state["count"], state["x"], state["w"], state["kmax"], state["kind"],
                               state["buf"], state["prec"], workspace=state["ws"])
    return {"logL": L, "grad": g, "status": status}


# ---- the work a pass cannot do without ---------------------------------------------------------

def work(case):
    C = case["channels"]
    if case["call"] == "simulate":
        n = C * case["bins"] * case["width"]
        # PSD, draws in; data out; data in again; the periodogram out
        return {"bytes": 8.0 * n + 16.0 * n + 16.0 * n + 16.0 * n + 8.0 * case["bins"] * (C + 3), "flops": 8.0 * n}
    nsp = C + (1 if case["sgwb"] else 0) + (3 if case["dense"] else 0)
    S = case["states"] * case["datasets"]
    bins = case["bins"] * case["datasets"]
    sb = float(case["states"]) * bins
    size = 8 if case["precision"] else 4
    knots = S * (8.0 * 5 + nsp * (4.0 + 8.0 * case["kmax"] + 8.0 * (case["kmax"] + 2)))
    fields = 3 + 2 * C + (C if case["sgwb"] else 0) + (3 if case["dense"] else 0)
    data = float(size) * fields * bins
    # per state and bin: each spline's cubic (7) and its exponential (1), the background's exponent (3), the
    # channels' PSD (6), and the term's reciprocal, logarithm, products and sums
    per = 8.0 * nsp + 3.0 + 6.0 * C
    if case["call"] == "psd":
        return {"bytes": data + knots + 8.0 * C * sb, "flops": sb * (per + C)}
    per += 4.0 * C
    if case["dense"]:
        per += 90.0
    out = 8.0 * S
    if case["call"] == "grad":
        per += 12.0 * C + 8.0 * nsp + 10.0
        out += 8.0 * S * (5 + nsp * (2 * case["kmax"] + 2))
    return {"bytes": data + knots + out, "flops": sb * per}


# ---- 64-bit values ------------------------------------------------------------------------------

def _shift(v, d, fill=0.0):
    """v[..., j + d] along the last axis, `fill` outside."""
    if d == 0:
        return v
    pad = torch.full(v.shape[:-1] + (abs(d),), fill, dtype=v.dtype, device=v.device)
    return torch.cat([v[..., d:], pad], -1) if d > 0 else torch.cat([pad, v[..., :d]], -1)


def _spline(count, x, w, x_lo, x_hi, kind):
    """Left knots [S, a, k], coefficients about them and the interior knots (for the search)."""
    S, A, k = x.shape
    j = torch.arange(k, device=x.device)
    n = count.long()[..., None]
    key = torch.where(j < n, x.detach(), torch.full_like(x, math.inf))
    order = torch.argsort(key, dim=-1)
    inner = torch.gather(key, -1, order)
    xs, ws = torch.gather(x, -1, order), torch.gather(w[..., 1:k + 1], -1, order)
    J = torch.arange(k + 2, device=x.device)
    px = torch.cat([torch.full((S, A, 1), x_lo, dtype=F64, device=x.device), xs, xs[..., :1] * 0 if k else
                    torch.zeros((S, A, 1), dtype=F64, device=x.device)], -1)
    py = torch.cat([w[..., :1], ws, torch.zeros((S, A, 1), dtype=F64, device=x.device)], -1)
    X = torch.where(J <= n, px, x_hi + (J - n - 1).to(F64))
    Y = torch.where(J <= n, py, torch.where(J == n + 1, w[..., k + 1:k + 2], torch.zeros_like(py)))
    K = n + 2
    h = X[..., 1:] - X[..., :-1]
    h = torch.cat([h, torch.ones_like(h[..., :1])], -1)
    m = torch.cat([(Y[..., 1:] - Y[..., :-1]), torch.zeros_like(Y[..., :1])], -1) / h
    m = torch.where(J < K - 1, m, torch.zeros_like(m))
    zero = torch.zeros_like(m)
    if kind == 1:
        hm, mm = _shift(h, -1), _shift(m, -1)
        row = (J >= 1) & (J <= K - 2)
        lower, diag = torch.where(row, hm, zero), torch.where(row, 2.0 * (hm + h), torch.ones_like(h))
        upper, rhs = torch.where(row, h, zero), torch.where(row, 6.0 * (m - mm), zero)
        M = torch.diag_embed(diag) + torch.diag_embed(upper[..., :-1], 1) + torch.diag_embed(lower[..., 1:], -1)
        d2 = torch.linalg.solve(M, rhs[..., None])[..., 0]
        dn = _shift(d2, 1)
        cb, cc, cd = m - h * (2.0 * d2 + dn) / 6.0, 0.5 * d2, (dn - d2) / (6.0 * h)
    else:
        a2, a1, b1 = _shift(m, -2), _shift(m, -1), _shift(m, 1)
        second, before = J == 1, J == K - 2
        wl = torch.where(before & ~second, (m - a1).abs(), (b1 - m).abs())
        wr = torch.where(second, (m - a1).abs(), (a1 - a2).abs())
        den = wl + wr
        ok = den > 0
        s = torch.where(ok, (wl * a1 + wr * m) / torch.where(ok, den, torch.ones_like(den)), 0.5 * (a1 + m))
        s = torch.where(J == 0, 1.5 * m - 0.5 * b1, s)
        s = torch.where(J == K - 1, 1.5 * a1 - 0.5 * a2, s)
        s = torch.where(J < K, s, zero)
        sn = _shift(s, 1)
        cb, cc, cd = s, (3.0 * m - 2.0 * s - sn) / h, (s + sn - 2.0 * m) / (h * h)
    lin = K < 4
    return X, (Y, torch.where(lin, m, cb), torch.where(lin, zero, cc), torch.where(lin, zero, cd)), inner


def _values(sp, xb):
    """Spline values [S, a, N] at the bins."""
    X, coef, inner = sp
    S, A, k = inner.shape
    if k:
        jj = torch.searchsorted(inner.reshape(S * A, k).contiguous(), xb.expand(S * A, -1).contiguous(), right=True)
        jj = jj.reshape(S, A, -1)
    else:
        jj = torch.zeros((S, A, xb.numel()), dtype=torch.int64, device=xb.device)
    t = xb - torch.gather(X, -1, jj)
    a, b, c, d = (torch.gather(v, -1, jj) for v in coef)
    return a + t * (b + t * (c + t * d))


def _model(case, th, sp, T, f_ref):
    """Noise, background and total PSD [S, C, N] and the last three splines' values of some states."""
    C, sg = case["channels"], case["sgwb"]
    v = _values(sp, T["x"])
    D = (th[:, 0, None, None] ** 2 * T["go"][:C] + th[:, 1, None, None] ** 2 * T["gt"][:C]) * 10.0 ** v[:, :C]
    back = torch.zeros_like(D)
    if sg:
        n2 = th[:, 4:5] if sg == 2 else th[:, 3:4]
        sl = torch.where(T["ell"] < 0, th[:, 3:4], n2)
        back = (10.0 ** (th[:, 2:3] + v[:, C]) * 2.0 ** (sl * T["ell"]))[:, None] * T["gh"]
    return D, back, D + back, v[:, -3:]


def _tables(q, d):
    b0, b1 = int(q["bin_offset"][d]), int(q["bin_offset"][d + 1])
    f = q["f"][b0:b1]
    R = q["R"][:, b0:b1] if q["R"] is not None else None
    go, gt, gh = _templates(f, R)
    T = dict(x=np.log10(f), ell=np.log2(f / q["f_ref"]), go=go, gt=gt, P=q["P"][:, b0:b1], nu=q["nu"][b0:b1])
    if gh is not None:
        T["gh"] = gh
    if q["X"] is not None:
        T["X"] = q["X"][:, b0:b1]
    return {k: torch.as_tensor(np.ascontiguousarray(v), device="cuda") for k, v in T.items()}


def _loglike(case, th, sp, T, f_ref):
    D, back, tot, z = _model(case, th, sp, T, f_ref)
    if not case["dense"]:
        return -((T["P"] / tot + torch.log(tot)).sum(1) * T["nu"]).sum(-1)
    # C = s_a s_b K_ab with s_c = sqrt(C_cc) and K = G R G + diag(h), g_c^2 = D_c / C_cc, h_c = 1 - g_c^2: the
    # determinant and the adjugate's diagonal as sums of non-negative products
    s0, s1, s2 = (1.0 / torch.sqrt(1.0 + z[:, k] ** 2) for k in range(3))
    r0, r1, r2 = z[:, 0] * s0, z[:, 1] * s1, z[:, 2] * s2
    r12 = r0 * r1 + s0 * s1 * r2
    e = r0 * r2 * s1 - r1 * s0
    m01, m02, m12 = s0 * s0, s1 * s1, (s1 * s2) ** 2 + e * e
    g = D / tot
    h = back / tot
    g0, g1, g2, h0, h1, h2 = g[:, 0], g[:, 1], g[:, 2], h[:, 0], h[:, 1], h[:, 2]
    A0 = g1 * g2 * m12 + h1 * (h2 + g2) + h2 * g1
    A1 = g0 * g2 * m02 + h0 * (h2 + g2) + h2 * g0
    A2 = g0 * g1 * m01 + h0 * (h1 + g1) + h1 * g0
    det = h0 * A0 + g0 * (g1 * g2 * (s0 * s1 * s2) ** 2 + h1 * (g2 * m02 + h2) + h2 * g1 * m01)
    q = torch.sqrt(D) / tot
    X = T["X"]
    B01 = s1 * (r1 * r2 * s0 - r0 * s1) * g2 - h2 * r0
    B02 = s0 * e * g1 - h1 * r1
    B12 = -(s0 * s1 * r2 * g0 + h0 * r12)
    off = q[:, 0] * q[:, 1] * X[0] * B01 + q[:, 0] * q[:, 2] * X[1] * B02 + q[:, 1] * q[:, 2] * X[2] * B12
    tr = A0 * T["P"][0] / tot[:, 0] + A1 * T["P"][1] / tot[:, 1] + A2 * T["P"][2] / tot[:, 2] + 2.0 * off
    return -((tr / det + torch.log(det) + torch.log(tot).sum(1)) * T["nu"]).sum(-1)


def exact(case, seed):
    """The outputs in 64 bits; None for the largest ensembles (too many state-bins for 20 seconds)."""
    if case["call"] == "simulate":
        q = _simulation(case, seed)
        d = torch.sqrt(0.5 * q["psd"])[..., None] * q["z"]
        n = case["width"]
        P = (d * d).sum(-1).reshape(case["channels"], case["bins"], n).mean(-1)
        b0 = q["off"][:-1].to(F64)
        return {"d": d, "P": P, "f": q["f0"] + q["df"] * (b0 + 0.5 * (n - 1)), "nu": torch.full_like(b0, float(n))}
    sb = case["states"] * case["datasets"] * case["bins"]
    if sb > 3.0e8:
        return None
    q = _inputs(case, seed)
    th, count, x, w = (torch.as_tensor(q[k], device="cuda") for k in ("theta", "count", "x", "w"))
    grad = case["call"] == "grad"
    Ls, Gs, Ps = [], [], []
    for d in range(case["datasets"]):
        T = _tables(q, d)
        s0, s1 = int(q["state_offset"][d]), int(q["state_offset"][d + 1])
        step = max(1, int((3.0e6 if grad or case["dense"] else 8.0e6) // max(1, T["x"].numel())))
        for a in range(s0, s1, step):
            b = min(a + step, s1)
            leaves = [v[a:b].clone().requires_grad_(grad) for v in (th, x, w)]
            with torch.set_grad_enabled(grad):
                sp = _spline(count[a:b], leaves[1], leaves[2], q["x_lo"], q["x_hi"], case["kind"])
                if case["call"] == "psd":
                    Ps.append(_model(case, leaves[0], sp, T, q["f_ref"])[2].reshape(-1))
                    continue
                L = _loglike(case, leaves[0], sp, T, q["f_ref"])
                Ls.append(L.detach())
                if grad:
                    gt, gx, gw = torch.autograd.grad(L.sum(), leaves, allow_unused=True)
                    gx = torch.zeros_like(leaves[1]) if gx is None else gx
                    Gs.append(torch.cat([gt, torch.cat([gw, gx], -1).reshape(b - a, -1)], -1))
    if case["call"] == "psd":
        return {"psd": torch.cat(Ps), "status": None}
    out = {"logL": torch.cat(Ls), "status": None}
    if grad:
        out["grad"] = torch.cat(Gs)
    elif case["call"] == "host":
        out["logL"] = out["logL"].cpu()
    return out
