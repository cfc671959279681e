"""What this library is timed on: the work a user has it do, through the public
entry points of the Python binding.

Three kinds of pass:

* ``eval``: one batched likelihood, ``Sampler.eval_lnl`` of unit-cube points on
  the device. The points are draws from the prior: the initial live set of a
  run, an importance or calibration sample.
* ``step``: one nested-sampling iteration through host buffers: the run is
  resumed from its checkpoint (``restore``), advanced by one iteration
  (``step_host``, whose dead points a user's program collects) and its live set
  is read back.
* ``serve``: a few analyses of different durations and live-point counts
  submitted to the continuous-batching server, each for a fixed number of
  iterations (the server's cap), and driven until all are done.

Grids, priors, live-point counts and precisions are those of the workloads in
``gwinputs`` and ``bench.py`` (4 to 256 s segments from 20 Hz, 1 to 3
detectors, compact binaries of 10-40 solar masses or low-mass inspirals of
1.1-1.5, 200-2000 live points with half of them replaced per iteration), on
seeded synthetic data: an injection from the prior at a target SNR plus
stationary Gaussian noise. Both precisions are used in earnest: FP64 as the
reference form, mixed for throughput.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2509_24949_gb300 as g

MC, Q, CHI1, CHI2, DL, COSI, PSI, PHIC, TC, RA, SINDEC = range(11)
FIXED, UNIFORM, VOLUME = 0, 1, 2
TSUN = 4.925490947641267e-6          # G Msun / c^3 [s]
C_SI = 299792458.0
MPC = 3.085677581491367e22
R_EARTH = 6.371e6
F_LO = 20.0
SLICE_EVALS = 3.76                   # likelihood evaluations per slice step (measured over the workloads)
SERVE_ITERATIONS = 20                # per served analysis


def listed():
    heavy, low = "heavy", "low-mass"
    return [
        # the smallest call: a handful of points of the single-detector, 4-parameter
        # analysis (512 bins), where the call's latency is what a user sees
        dict(name="eval 512 bins fp64", kind="eval", duration=511 / 492, f_hi=512.0, n_det=0, mass=heavy,
             precision="fp64", points=64, coarse=0, snr=20.0),
        # the initial live set of a 4 s analysis
        dict(name="eval 4017 bins fp64", kind="eval", duration=4.0, f_hi=1024.0, n_det=3, mass=heavy,
             precision="fp64", points=1000, coarse=0, snr=20.0),
        # batches of prior draws on the 32 s and 256 s grids, in both precisions
        dict(name="eval 64897 bins fp64", kind="eval", duration=32.0, f_hi=2048.0, n_det=3, mass=heavy,
             precision="fp64", points=2048, coarse=0, snr=20.0),
        dict(name="eval 64897 bins mixed", kind="eval", duration=32.0, f_hi=2048.0, n_det=3, mass=heavy,
             precision="mixed", points=8192, coarse=0, snr=20.0),
        dict(name="eval 519169 bins fp64", kind="eval", duration=256.0, f_hi=2048.0, n_det=3, mass=low,
             precision="fp64", points=2048, coarse=0, snr=30.0),
        dict(name="eval 519169 bins mixed", kind="eval", duration=256.0, f_hi=2048.0, n_det=3, mass=low,
             precision="mixed", points=8192, coarse=0, snr=30.0),
        # the heterodyned likelihood (relative binning about the injection) on 1024 coarse bins
        dict(name="eval 1024 coarse bins fp64", kind="eval", duration=256.0, f_hi=2048.0, n_det=3, mass=low,
             precision="fp64", points=8192, coarse=1024, snr=30.0),
        # one iteration: the smallest analysis, the 4 s analysis in FP64, the 32 s and
        # the 256 s analysis in mixed precision (the benchmark's step)
        dict(name="step 512 bins fp64", kind="step", duration=511 / 492, f_hi=512.0, n_det=0, mass=heavy,
             precision="fp64", n_live=200, coarse=0, snr=20.0),
        dict(name="step 4017 bins fp64", kind="step", duration=4.0, f_hi=1024.0, n_det=3, mass=heavy,
             precision="fp64", n_live=1000, coarse=0, snr=20.0),
        dict(name="step 64897 bins mixed", kind="step", duration=32.0, f_hi=2048.0, n_det=3, mass=heavy,
             precision="mixed", n_live=2000, coarse=0, snr=20.0),
        dict(name="step 519169 bins mixed", kind="step", duration=256.0, f_hi=2048.0, n_det=3, mass=low,
             precision="mixed", n_live=2000, coarse=0, snr=30.0),
        # the serving loop over analyses of 4, 8, 16 and 32 s that share the GPU
        dict(name="serve 4 analyses mixed", kind="serve", duration=4.0, f_hi=2048.0, n_det=3, mass=heavy,
             precision="mixed", n_live=500, analyses=4, coarse=0, snr=20.0),
    ]


def _evals(case):
    if case["kind"] == "eval":
        return case["points"]
    dim = 4 if case["n_det"] == 0 else 11
    per_iteration = case["n_live"] // 2 * 5 * dim * SLICE_EVALS
    return per_iteration if case["kind"] == "step" else per_iteration * SERVE_ITERATIONS * case["analyses"]


def _bins_read(case):
    """Mean number of grid bins below the signal's end (f_ISCO) over prior draws."""
    rng = np.random.default_rng(7)
    mc = rng.uniform(*_mass_range(case), 4096)
    q = rng.uniform(0.25, 1.0, 4096)
    eta = q / (1 + q) ** 2
    fisco = 1.0 / (6.0 ** 1.5 * math.pi * mc * TSUN * eta ** -0.6)
    span = np.clip(fisco, F_LO, case["f_hi"]) - F_LO
    return float(np.mean(span * case["duration"])) + 1.0


def _cost(case):
    """Rough work of a pass in point-bins, FP64 ones weighted by their rate."""
    bins = min(_bins_read(case), 4.0 * case["coarse"]) if case["coarse"] else _bins_read(case)
    return _evals(case) * (bins + 400.0) * (60.0 if case["precision"] == "fp64" else 1.0)


def draw(rng):
    """Another case of these ranges: any duration, live-point and batch size."""
    def spread(a, b):
        return math.exp(rng.uniform(math.log(a), math.log(b)))

    kind = rng.choice(["eval", "eval", "eval", "step", "step", "serve"])
    mass = "heavy" if kind == "serve" else rng.choice(["heavy", "heavy", "low-mass"])
    duration = round(spread(64.0, 256.0) if mass == "low-mass" else spread(4.0, 32.0 if kind == "serve" else 64.0), 2)
    case = dict(kind=kind, duration=duration, f_hi=rng.choice([512.0, 1024.0, 2048.0]), n_det=rng.choice([1, 2, 3, 3]),
                mass=mass, precision=rng.choice(["fp64", "mixed"]), coarse=0, snr=round(rng.uniform(10.0, 40.0), 2))
    if kind == "eval":
        case["points"] = int(spread(64, 8193))
        if mass == "low-mass" and rng.random() < 0.3:
            case["coarse"] = int(spread(256, 1025))
    else:
        case["n_live"] = int(spread(200, 2001)) if kind == "step" else int(spread(200, 801))
        if kind == "serve":
            case["precision"] = "mixed"
            case["analyses"] = rng.randint(2, 4)
    limit = max(_cost(c) for c in listed() if (c["kind"] == "serve") == (kind == "serve"))
    if kind == "step" and _bins_read(case) > 20000:
        case["precision"] = "mixed"     # an FP64 iteration on the long grids takes seconds
    size, least = ("points", 64) if kind == "eval" else ("n_live", 200)
    while _cost(case) > limit and case[size] > least:
        case[size] = max(least, int(case[size] * 0.7))
    return case


# ------------------------------------------------------------------ inputs
def _mass_range(case):
    return (10.0, 40.0) if case["mass"] == "heavy" else (1.1, 1.5)


def _prior(case):
    """Kinds and bounds of the 11 parameters; n_det = 0: the idealised single
    detector with chirp mass, mass ratio, time and phase free."""
    kind = np.full(11, UNIFORM, dtype=np.int32)
    lo, hi = np.zeros(11), np.zeros(11)
    box = {MC: _mass_range(case), Q: (0.25, 1.0), CHI1: (-0.5, 0.5), CHI2: (-0.5, 0.5),
           DL: (100.0, 2000.0) if case["mass"] == "heavy" else (10.0, 2000.0), COSI: (-1.0, 1.0),
           PSI: (0.0, math.pi), PHIC: (0.0, 2 * math.pi), TC: (-0.1, 0.1), RA: (0.0, 2 * math.pi), SINDEC: (-1.0, 1.0)}
    for p, (a, b) in box.items():
        lo[p], hi[p] = a, b
    kind[DL] = VOLUME
    if case["n_det"] == 0:
        for p, v in {CHI1: 0.0, CHI2: 0.0, DL: 100.0, COSI: 1.0, PSI: 0.0, RA: 0.0, SINDEC: 0.0}.items():
            kind[p], lo[p], hi[p] = FIXED, v, v
    return kind, lo, hi


def _theta(u, kind, lo, hi):
    """Unit-cube points [m, d] -> physical parameters [m, 11] (torch, FP64)."""
    th = torch.empty(u.shape[0], 11, dtype=torch.float64, device=u.device)
    i = 0
    for p in range(11):
        a, b = float(lo[p]), float(hi[p])
        if kind[p] == FIXED:
            th[:, p] = a
            continue
        x = u[:, i]
        i += 1
        th[:, p] = a + (b - a) * x if kind[p] == UNIFORM else (a ** 3 + x * (b ** 3 - a ** 3)) ** (1.0 / 3.0)
    return th


def _freqs(case, device):
    n = int(round((case["f_hi"] - F_LO) * case["duration"])) + 1
    return F_LO + torch.arange(n, dtype=torch.float64, device=device) * (1.0 / case["duration"])


def _psd(f):
    return 1e-46 * ((f / 30.0) ** -4 + 2.0 + 2.0 * (f / 200.0) ** 2)


def _detectors(n_det, seed):
    """Seeded detectors on the Earth's sphere with orthogonal horizontal arms."""
    rng = np.random.default_rng(seed)
    u = rng.standard_normal((n_det, 3))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    x = rng.standard_normal((n_det, 3))
    x -= np.sum(x * u, axis=1, keepdims=True) * u
    x /= np.linalg.norm(x, axis=1, keepdims=True)
    return R_EARTH * u, x, np.cross(u, x)


# TaylorF2 (3.5PN with aligned-spin terms) in plain torch
def _phase_coefficients(th):
    """Coefficients [m, 8] of f^-5/3, f^-1, f^-2/3, f^-1/3, ln f, f^1/3,
    f^1/3 ln f, f^2/3 and the constant [m] of the phase (without time shifts)."""
    pi = math.pi
    q, c1, c2 = th[:, Q], th[:, CHI1], th[:, CHI2]
    eta, delta = q / (1 + q) ** 2, (1 - q) / (1 + q)
    cs, ca = 0.5 * (c1 + c2), 0.5 * (c1 - c2)
    beta = (113 / 12) * (cs + delta * ca - (76 / 113) * eta * cs)
    sigma = (79 / 8) * eta * c1 * c2
    gamma = (732985 / 2268 - 24260 / 81 * eta - 340 / 9 * eta ** 2) * cs + (732985 / 2268 + 140 / 9 * eta) * delta * ca
    a = (pi * th[:, MC] * TSUN * eta ** -0.6) ** (1.0 / 3.0)     # v = a f^(1/3)
    K = 3.0 / (128.0 * eta)
    p2 = 3715 / 756 + 55 / 9 * eta
    p3 = -16 * pi + 4 * beta
    p4 = 15293365 / 508032 + 27145 / 504 * eta + 3085 / 72 * eta ** 2 - 10 * sigma
    p5 = pi * (38645 / 756 - 65 / 9 * eta) - gamma
    p6 = (11583231236531 / 4694215680 - 640 / 3 * pi ** 2 - 6848 / 21 * 0.5772156649015329
          + (-15737765635 / 3048192 + 2255 / 12 * pi ** 2) * eta + 76055 / 1728 * eta ** 2 - 127825 / 1296 * eta ** 3
          - 6848 / 21 * torch.log(4 * a))
    p7 = pi * (77096675 / 254016 + 378515 / 1512 * eta - 74045 / 756 * eta ** 2)
    coef = torch.stack([K * a ** -5, K * p2 * a ** -3, K * p3 * a ** -2, K * p4 / a, K * p5, K * p6 * a,
                        -6848 / 63 * K * a, K * p7 * a ** 2], dim=1)
    const = -th[:, PHIC] - 0.25 * pi + K * p5 * (1 + 3 * torch.log(math.sqrt(6.0) * a))
    return coef, const


def _basis(f):
    c, lf = f ** (1.0 / 3.0), torch.log(f)
    return torch.stack([c ** -5, 1 / f, c ** -2, 1 / c, lf, c, c * lf, c ** 2])


def _antennas(th, geom):
    """Q_d = F+ (1 + cos^2 i)/2 - i Fx cos i as (re, im) [m, D] and the delays [m, D]."""
    ci = th[:, COSI:COSI + 1]
    if geom is None:
        return 0.5 * (1 + ci ** 2), torch.zeros_like(ci), torch.zeros_like(ci)
    pos, xa, ya = (torch.as_tensor(v, dtype=torch.float64, device=th.device) for v in geom)
    sa, ca = torch.sin(th[:, RA]), torch.cos(th[:, RA])
    sp, cp = torch.sin(th[:, PSI]), torch.cos(th[:, PSI])
    sd = th[:, SINDEC]
    cd = torch.sqrt(1 - sd ** 2)
    X = torch.stack([sa * cp - sp * ca * sd, -ca * cp - sp * sa * sd, sp * cd], dim=1)
    Y = torch.stack([-sa * sp - cp * ca * sd, ca * sp - cp * sa * sd, cp * cd], dim=1)
    n = torch.stack([cd * ca, cd * sa, sd], dim=1)
    xX, xY, yX, yY = X @ xa.T, Y @ xa.T, X @ ya.T, Y @ ya.T
    fp = 0.5 * ((xX ** 2 - yX ** 2) - (xY ** 2 - yY ** 2))
    fc = xX * xY - yX * yY
    return fp * 0.5 * (1 + ci ** 2), -fc * ci, -(n @ pos.T) / C_SI


def _amplitude(th):
    return math.sqrt(5 / 24) * math.pi ** (-2 / 3) * (C_SI / MPC) * (th[:, MC] * TSUN) ** (5 / 6) / th[:, DL]


def _last_bin(th, f):
    """Last grid index at or below f_ISCO (-1: none)."""
    eta = th[:, Q] / (1 + th[:, Q]) ** 2
    fisco = 1.0 / (6.0 ** 1.5 * math.pi * th[:, MC] * TSUN * eta ** -0.6)
    return torch.searchsorted(f, fisco, right=True) - 1


def _snr(th, f, S, df, geom):
    qre, qim, _ = _antennas(th, geom)
    P = torch.cumsum(4 * df * f ** (-7 / 3) / S, 0)
    j = _last_bin(th, f)
    p = torch.where(j >= 0, P[j.clamp(min=0)], torch.zeros_like(th[:, 0]))
    return torch.sqrt(_amplitude(th) ** 2 * (qre ** 2 + qim ** 2).sum(1) * p)


def _problem(case, seed):
    """Detectors, prior, data and the injected parameters of one analysis."""
    dev = torch.device("cuda")
    kind, lo, hi = _prior(case)
    dim = int(np.sum(kind != FIXED))
    nd = max(1, case["n_det"])
    geom = None if case["n_det"] == 0 else _detectors(nd, 1000 + seed)
    f = _freqs(case, dev)
    S, df = _psd(f), 1.0 / case["duration"]
    rng = np.random.default_rng(3000 + seed)
    th = _theta(torch.as_tensor(rng.random((4096, dim)), device=dev), kind, lo, hi)
    if case["n_det"] == 0:
        # distance fixed so that the injection has the target SNR; noise-free data
        th = th[:1]
        dl = th[:, DL] * _snr(th, f, S, df, geom) / case["snr"]
        th[:, DL] = dl
        lo[DL] = hi[DL] = float(dl)
    else:
        # the first prior draw whose distance can be scaled to the target SNR inside the prior
        dl = th[:, DL] * _snr(th, f, S, df, geom) / case["snr"]
        ok = torch.nonzero((dl >= lo[DL]) & (dl <= hi[DL])).flatten()
        i = int(ok[0]) if ok.numel() else int(torch.argmin((torch.log(dl) - math.log(0.5 * hi[DL])).abs()))
        th = th[i:i + 1].clone()
        th[:, DL] = dl[i].clamp(float(lo[DL]), float(hi[DL]))
    coef, const = _phase_coefficients(th)
    qre, qim, dt = _antennas(th, geom)
    phase = (coef @ _basis(f) + const[:, None]) + 2 * math.pi * f * (th[:, TC:TC + 1] + dt.reshape(-1, 1))
    # h_d = conj(G_d) f^(-7/6) exp(-i Psi_d), G_d = A conj(Q_d)
    amp = _amplitude(th) * f ** (-7 / 6) * (torch.arange(f.numel(), device=dev) <= _last_bin(th, f))
    data = amp * torch.complex(qre.reshape(-1, 1), qim.reshape(-1, 1)) * torch.exp(-1j * phase)
    if case["n_det"] != 0:
        noise = np.random.default_rng(2000 + seed).standard_normal((2, nd, f.numel()))
        data = data + torch.sqrt(S / (4 * df)) * torch.complex(*torch.as_tensor(noise, device=dev))
    return dict(kind=kind, lo=lo, hi=hi, dim=dim, geom=geom, f=f, S=S, df=df, nd=nd, data=data, theta=th[0])


def _arguments(case, pb):
    """Keyword arguments of Sampler and Server.submit."""
    pos, xa, ya = pb["geom"] if pb["geom"] is not None else (None, None, None)
    args = dict(kind=pb["kind"], lo=pb["lo"], hi=pb["hi"], data=pb["data"].cpu().numpy(),
                psd=np.tile(pb["S"].cpu().numpy(), (pb["nd"], 1)), f0=F_LO, df=pb["df"], pos=pos, xarm=xa, yarm=ya,
                ideal=pb["geom"] is None)
    if case["coarse"]:
        args.update(coarse_bins=case["coarse"], theta_fid=pb["theta"].cpu().numpy())
    return args


def _points(case, seed, dim):
    return torch.as_tensor(np.random.default_rng(5000 + seed).random((case["points"], dim)), device="cuda")


def prepare(case, seed):
    prec = g.NS_FP64 if case["precision"] == "fp64" else g.NS_MIXED
    if case["kind"] == "serve":
        requests = []
        for i in range(case["analyses"]):
            sub = dict(case, duration=case["duration"] * 2 ** i if case["duration"] * 2 ** i <= 32.0 else case["duration"])
            requests.append(dict(_arguments(sub, _problem(sub, seed + 100003 * i)), n_live=case["n_live"] + 37 * i,
                                 dlogz_stop=-1.0, seed=4000 + seed + i))
        return dict(kind="serve", server=g.Server(precision=prec, max_iter=SERVE_ITERATIONS), requests=requests, dim=11)
    pb = _problem(case, seed)
    args = _arguments(case, pb)
    if case["kind"] == "eval":
        return dict(kind="eval", sampler=g.Sampler(n_live=64, precision=prec, seed=4000 + seed, **args),
                    u=_points(case, seed, pb["dim"]))
    sp = g.Sampler(n_live=case["n_live"], precision=prec, seed=4000 + seed, **args)
    k = sp.k
    return dict(kind="step", sampler=sp, start=sp.checkpoint(), dead_u=np.zeros((k, sp.dim)), dead_logl=np.zeros(k),
                dead_logw=np.zeros(k))


def run(state):
    if state["kind"] == "eval":
        return {"logl": state["sampler"].eval_lnl(state["u"])}
    if state["kind"] == "step":
        sp = state["sampler"]
        sp.restore(state["start"])
        sp.step_host(out_u=state["dead_u"], out_logl=state["dead_logl"], out_logw=state["dead_logw"])
        u, logl = sp.live()
        return {"live_u": u, "live_logl": logl, "dead_u": state["dead_u"], "dead_logl": state["dead_logl"],
                "dead_logw": state["dead_logw"]}
    srv = state["server"]
    ids = [srv.submit(**r) for r in state["requests"]]
    srv.run_until_idle()
    return [srv.result(i, state["dim"]) for i in ids]


def work(case):
    """Bytes: the points, the results and the strain data (two doubles per
    detector and bin below the mean cutoff, or per coarse bin), each once. Flops:
    one complex multiply-add per evaluation, detector and bin read."""
    nd, dim = max(1, case["n_det"]), 4 if case["n_det"] == 0 else 11
    bins = min(_bins_read(case), float(case["coarse"])) if case["coarse"] else _bins_read(case)
    evals = _evals(case)
    rows = case["points"] if case["kind"] == "eval" else 3 * case["n_live"]
    if case["kind"] == "serve":
        rows = case["analyses"] * case["n_live"] * (1 + SERVE_ITERATIONS // 2)
    return {"bytes": rows * 8.0 * (dim + 1) + 16.0 * nd * bins * case.get("analyses", 1), "flops": evals * bins * nd * 8.0}


def exact(case, seed):
    """The log-likelihoods of an ``eval`` case by the per-bin definition in plain
    torch, FP64; the relative-binning likelihood has its own definition (summary
    data between coarse edges), and the sampler's cases have no closed value."""
    if case["kind"] != "eval" or case["coarse"]:
        return None
    pb = _problem(case, seed)
    th = _theta(_points(case, seed, pb["dim"]), pb["kind"], pb["lo"], pb["hi"])
    f, S, df = pb["f"], pb["S"], pb["df"]
    coef, const = _phase_coefficients(th)
    qre, qim, dt = _antennas(th, pb["geom"])
    last, basis = _last_bin(th, f), _basis(f)
    w = 4 * df * f ** (-7 / 6) * pb["data"] / S
    P = torch.cumsum(4 * df * f ** (-7 / 3) / S, 0)
    A = _amplitude(th)
    out = torch.empty_like(A)
    rows = max(1, int(2 ** 26 // f.numel()))
    for i in range(0, th.shape[0], rows):
        s = slice(i, i + rows)
        n = int(last[s].max()) + 1
        live = torch.arange(max(n, 1), device=f.device) <= last[s, None]
        psi = coef[s] @ basis[:, :max(n, 1)] + const[s, None]
        total = torch.zeros_like(A[s])
        for d in range(pb["nd"]):
            ph = psi + 2 * math.pi * f[:live.shape[1]] * (th[s, TC:TC + 1] + dt[s, d:d + 1])
            c, sn = torch.cos(ph) * live, torch.sin(ph) * live
            wr, wi = w[d, :live.shape[1]].real, w[d, :live.shape[1]].imag
            zr, zi = c @ wr - sn @ wi, sn @ wr + c @ wi
            total += A[s] * (qre[s, d] * zr + qim[s, d] * zi)
        pj = torch.where(last[s] >= 0, P[last[s].clamp(min=0)], torch.zeros_like(A[s]))
        out[s] = total - 0.5 * A[s] ** 2 * (qre[s] ** 2 + qim[s] ** 2).sum(1) * pj
    return {"logl": out}
