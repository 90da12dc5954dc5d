"""The calls that a program built on this library spends its time in.

Each case is one pass through the public entry points of
``paper_2009_11742_gb300.rom``: the rank-2 leapfrog in FP32, FP64 and on the
tensor cores, the rank-1 run, the Monte Carlo study with its ensemble
statistics, a batch of uneven models, the adjoint, the statistics alone and
the full-order model.  ``listed()`` names twelve of them, ``draw()`` makes
more over the same ranges.

Operators, periods and receiver rows follow ``inputs.make_problem`` (random
skew-coupled operators, periods of 30 to 60 steps).  The time step is given
instead of computed from a singular value: dt = 0.5 / (1 + sqrt(Ks / Kv)),
the large-matrix limit of 0.5 / ||Asv||_2 for entries of variance 1 / Kv.
States start from seeded noise, as a run that resumes from a checkpoint does.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2009_11742_gb300 import inputs, rom

DEVICE = "cuda"
PROBS = (0.05, 0.5, 0.95)  # the median and the 5-95 % band


def listed():
    return [
        # a quick look at a small ensemble: launch and per-step latency only
        dict(name="rank2-f32-tiny", kind="rank2", prec="fp32", Kv=100, Ks=90, M=5, R=3, r=5, N=50),
        # the benchmark's model: K = 512, 256 realizations, 64 receivers
        dict(name="rank2-f32-k512", kind="rank2", prec="fp32", Kv=512, Ks=512, M=256, R=64, r=10, N=1000),
        # the largest model and ensemble in FP32
        dict(name="rank2-f32-k1024", kind="rank2", prec="fp32", Kv=1024, Ks=1024, M=1024, R=64, r=10, N=100),
        # the same on the tensor cores, in exact BF16 slices
        dict(name="rank2-bf16s-k1024", kind="rank2", prec="bf16s", Kv=1024, Ks=1024, M=1024, R=64, r=10,
             N=200),
        # the FP64 check run of a small model
        dict(name="rank2-f64-k128", kind="rank2", prec="fp64", Kv=128, Ks=128, M=16, R=0, r=0, N=1000),
        # one realization on its own: two matrix-vector products a step
        dict(name="rank1-f32-k512", kind="rank1", prec="fp32", Kv=512, Ks=512, M=1, R=64, r=10, N=1000),
        # the Monte Carlo study: 512 realizations of a ragged model, then the
        # mean and the 5-95 % band of every seismogram
        dict(name="uq-f32-k436", kind="uq", prec="fp32", Kv=436, Ks=417, M=512, R=64, r=10, N=1000),
        # the bands alone, over traces that an earlier run left on the device
        dict(name="stats-m512", kind="stats", nrec=1000, R=64, M=512),
        # many uneven models at once
        dict(name="batched-f32-16", kind="batched", prec="fp32", njobs=16, sizes=0, N=200),
        # waveform inversion: misfit and gradients with checkpoints
        dict(name="adjoint-f32-k512", kind="adjoint", prec="fp32", Kv=512, Ks=512, M=128, R=64, N=256, c=64),
        # the full-order model, many forcings at once: bound by memory
        dict(name="fom-f32-m32", kind="fom", prec="fp32", Nr=512, Nt=2048, M=32, R=64, r=10, N=128),
        # the full-order model, one forcing
        dict(name="fom-f32-m1", kind="fom", prec="fp32", Nr=512, Nt=2048, M=1, R=64, r=10, N=512),
    ]


def _log(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["rank2", "rank2", "rank2", "rank2", "rank1", "uq", "stats", "batched", "adjoint", "fom",
                       "fom"])
    if kind in ("rank2", "rank1", "uq", "adjoint"):
        prec = rng.choice(["fp32", "fp32", "bf16s", "fp64"]) if kind == "rank2" else (
            rng.choice(["fp32", "fp32", "fp64"]) if kind in ("rank1", "adjoint") else "fp32")
        kmax = 512 if prec == "fp64" else 1024  # the FP64 kernels stop at K = 512
        K = _log(rng, 16, kmax)
        Ks = max(1, K - rng.choice([0, 0, 1, 7, K // 16]))
        M = 1 if kind == "rank1" else _log(rng, 2, 1024 if kind == "rank2" else 512)
        # at most a tenth of the largest listed case's work, for the slower types
        share = {"fp32": 6e10, "bf16s": 1.2e11, "fp64": 1.5e9}[prec] / (3 if kind == "adjoint" else 1)
        nmax = max(8, min(1500 if prec != "bf16s" else 400, int(share / (4.0 * K * Ks * M))))
        N = _log(rng, max(8, nmax // 4), nmax)
        R = _log(rng, 1, 100)
        case = dict(kind=kind, prec=prec, Kv=K, Ks=Ks, M=M, R=R, N=N)
        if kind == "adjoint":
            case["c"] = rng.choice([0, 16, 64])
        else:
            case["r"] = min(N, rng.choice([1, 5, 10, 10]))
            if case["r"] == 1:
                case["R"] = min(R, 32)
        return case
    if kind == "stats":
        M = _log(rng, 8, 2000)
        R = _log(rng, 1, 100)
        return dict(kind="stats", nrec=_log(rng, 10, max(10, min(2000, 32_000_000 // (M * R)))), R=R, M=M)
    if kind == "batched":
        return dict(kind="batched", prec=rng.choice(["fp32", "fp32", "auto"]), njobs=rng.randint(3, 16),
                    sizes=rng.randint(1, 10**6), N=_log(rng, 20, 100))
    prec = rng.choice(["fp32", "fp32", "fp64"])
    Nr, Nt, M = _log(rng, 32, 512), _log(rng, 64, 2048), _log(rng, 1, 40)
    cost = Nr * Nt * M * (6 if prec == "fp64" else 1)
    N = max(16, min(512, int(512 * 2048 * 32 * 100 / cost)))
    if cost > 512 * 2048 * 40:
        M, N = max(1, M // 6), 64
    return dict(kind="fom", prec=prec, Nr=Nr, Nt=Nt, M=M, R=_log(rng, 1, 64), r=rng.choice([5, 10]),
                N=_log(rng, max(8, N // 4), N))


# ----------------------------------------------------------------- inputs --
def _dt(Kv, Ks):
    return 0.5 / (1.0 + math.sqrt(Ks / Kv))


def _problem(case, seed):
    return inputs.make_problem(case["Kv"], case["Ks"], case["M"], case["R"], seed=seed,
                               dt=_dt(case["Kv"], case["Ks"]),
                               period_range=(31.0, 69.0) if case["kind"] == "uq" else (30.0, 60.0))


def _np_dtype(case):
    return np.float64 if case.get("prec") == "fp64" else np.float32


def _torch_dtype(case):
    return torch.float64 if case.get("prec") == "fp64" else torch.float32


def _noise(seed, *shapes):
    """Seeded float32 noise of each shape, on the host."""
    rng = np.random.default_rng([seed, 77])
    return [0.2 * rng.standard_normal(s, dtype=np.float32) for s in shapes]


def _device_noise(seed, shape, scale):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(1000 + seed)
    return scale * torch.randn(shape, generator=g, device=DEVICE, dtype=torch.float32)


def _periods(p, case):
    return torch.as_tensor(p.T.astype(_np_dtype(case)), device=DEVICE)


def _trace_buffer(case, M):
    if not case.get("r"):
        return None
    return torch.zeros((case["N"] // case["r"], M, case["R"]), dtype=_torch_dtype(case), device=DEVICE)


def _batch_sizes(case):
    return inputs.batched_sizes(case["njobs"], case["sizes"])


def _batch_problem(K, M, seed, i):
    return inputs.make_problem(K, K, M, 0, seed=100 * seed + i + 1, dt=_dt(K, K))


def _stat_traces(case, seed):
    """Seismograms: quiet (exactly zero) first records, then a decaying
    wave train whose amplitude differs from receiver to receiver."""
    nrec, R, M = case["nrec"], case["R"], case["M"]
    x = _device_noise(seed, (nrec, M, R), 1.0)
    rec = torch.arange(nrec, device=DEVICE, dtype=torch.float32)[:, None, None]
    amp = torch.exp(-3.0 * rec / nrec) * (rec >= nrec // 20)
    return x * amp * (1.0 + torch.arange(R, device=DEVICE, dtype=torch.float32) / R)


def _fom_setup(case, seed):
    """Noise at the scale of the waves (stress = rho vs v), a pulse under
    way (the clock starts at 75 s), periods of 60 to 80 s."""
    Nr, Nt, M = case["Nr"], case["Nt"], case["M"]
    dt = _torch_dtype(case)
    states = [_device_noise(3 * seed + i, (n, M), s).to(dt) for i, (n, s) in enumerate(
        ((Nr * (Nt - 1), 1e-5), ((Nr - 1) * (Nt - 1), 100.0), (Nr * (Nt - 2), 100.0)))]
    rng = np.random.default_rng([seed, 5])
    T = rng.uniform(60.0, 80.0, M).astype(np.float32)
    recv = np.sort(rng.integers(0, Nt - 1, case["R"])) + (Nr - 1) * (Nt - 1)  # at the surface
    return states, torch.as_tensor(T, device=DEVICE).to(dt), torch.as_tensor(recv.astype(np.int32),
                                                                             device=DEVICE)


FOM_N0 = 1500
FOM_DEPTH = 640e3


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "stats":
        st["traces"] = _stat_traces(case, seed)
    elif kind == "fom":
        f = rom.Fom(case["Nr"], case["Nt"])
        st["fom"], st["src"] = f, f.source_index(FOM_DEPTH)
        st["states"], st["T"], st["recv"] = _fom_setup(case, seed)
        st["traces"] = torch.zeros((case["N"] // case["r"], case["R"], case["M"]), dtype=_torch_dtype(case),
                                   device=DEVICE)
    elif kind == "batched":
        st["items"] = []
        for i, (K, M) in enumerate(_batch_sizes(case)):
            p = _batch_problem(K, M, seed, i)
            V, S = _noise(100 * seed + i, (K, M), (K, M))
            st["items"].append((rom.Rom.from_problem(p), rom.Rom.new_state(K, M, "fp32", fill=V),
                                rom.Rom.new_state(K, M, "fp32", fill=S), _periods(p, case), None))
    else:
        p = _problem(case, seed)
        M, prec = case["M"], case["prec"]
        st["rom"] = rom.Rom.from_problem(p)
        V, S = _noise(seed, (case["Kv"], M), (case["Ks"], M))
        st["V"] = rom.Rom.new_state(case["Kv"], M, prec, fill=V)
        st["S"] = rom.Rom.new_state(case["Ks"], M, prec, fill=S)
        st["T"] = _periods(p, case)
        if kind == "rank1":
            st["V"], st["S"], st["T"] = st["V"].t().reshape(-1), st["S"].t().reshape(-1), float(p.T[0])
        if kind == "adjoint":
            st["ystar"] = _device_noise(seed, (case["N"], M, case["R"]), 0.2).to(_torch_dtype(case))
        else:
            st["traces"] = _trace_buffer(case, M)
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "stats":
        return rom.trace_stats(state["traces"], PROBS)
    if kind == "fom":
        V, S1, S2 = state["states"]
        state["fom"].run(V, S1, S2, case["N"], src=state["src"], T=state["T"], recv=state["recv"], r=case["r"],
                         traces=state["traces"], prec=case["prec"], n0=FOM_N0)
        return V, S1, S2, state["traces"]
    if kind == "batched":
        rom.run_batched(state["items"], case["N"], prec=case["prec"])
        return [x for item in state["items"] for x in (item[1], item[2])]
    h = state["rom"]
    if kind == "adjoint":
        return rom.adjoint(h, state["V"], state["S"], state["T"], state["ystar"], case["N"],
                           ckpt_every=case["c"])
    out = [state["V"], state["S"]]
    if kind == "rank1":
        h.run_rank1(state["V"], state["S"], state["T"], case["N"], r=case["r"], trace=state["traces"],
                    prec=case["prec"])
    else:
        h.run_rank2(state["V"], state["S"], state["T"], case["N"], r=case["r"], traces=state["traces"],
                    prec=case["prec"])
    if state["traces"] is not None:
        out.append(state["traces"])
    if kind == "uq":
        out.extend(rom.trace_stats(state["traces"], PROBS))
    return out


# -------------------------------------------------- what a pass comes to --
def _rom_work(Kv, Ks, M, R, N, nrec, es):
    flops = 4.0 * Kv * Ks * M * N + 2.0 * R * Kv * M * nrec
    nbytes = es * (2.0 * Kv * Ks + Kv + R * Kv + 2.0 * (Kv + Ks) * M + M + float(nrec) * R * M)
    return nbytes, flops


def work(case):
    kind = case["kind"]
    es = 8 if case.get("prec") == "fp64" else 4
    if kind == "stats":
        n = case["nrec"] * case["R"]
        return {"bytes": 4.0 * n * case["M"] + 8.0 * n * (1 + len(PROBS)), "flops": 1.0 * n * case["M"]}
    if kind == "fom":
        n = (case["Nr"] * (3.0 * case["Nt"] - 4) - (case["Nt"] - 1)) * case["M"]
        # four products and sums a velocity row, two a stress row (each with
        # the update), once per step; a step cannot start before the last
        # one's field is there, which at these sizes does not stay on chip
        nv = case["Nr"] * (case["Nt"] - 1.0) * case["M"]
        fits = 2 * n * es < 100e6
        return {"bytes": 2.0 * es * n * (1 if fits else case["N"]),
                "flops": (8.0 * nv + 4.0 * (n - nv)) * case["N"]}
    if kind == "batched":
        w = [_rom_work(K, K, M, 0, case["N"], 0, es) for K, M in _batch_sizes(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "adjoint":
        # a forward and a reverse sweep; each trace is formed and carried back
        b, f = _rom_work(case["Kv"], case["Ks"], case["M"], case["R"], case["N"], case["N"], es)
        return {"bytes": b, "flops": 2.0 * f}
    b, f = _rom_work(case["Kv"], case["Ks"], case["M"], case["R"], case["N"],
                     case["N"] // case["r"] if case["r"] else 0, es)
    if kind == "uq":
        b += 8.0 * (case["N"] // case["r"]) * case["R"] * (1 + len(PROBS))
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the distance to `exact` that the listed and a few
    dozen drawn cases showed."""
    kind, prec = case["kind"], case.get("prec")
    if kind == "stats":
        return {"rel": 1e-13}
    if kind == "fom":
        return {"rel": 1e-13} if prec == "fp64" else {"rel": 4e-6}
    if prec == "fp64":
        return {"rel": 2e-14}
    if prec in ("bf16s", "auto"):
        return {"rel": 1e-5}
    return {"rel": 5e-6}


# --------------------------------------------- the same sums, in 64 bits --
def _signal(wavelet, t, T):
    """Source signal of period T at time t, delayed by 1.5 T."""
    a = math.pi * (t - 1.5 * T) / T
    if wavelet == rom.ROM_WAVELET_GAUSS1:
        return -math.sqrt(2.0 * math.e) * a * torch.exp(-a * a)
    return (1.0 - 2.0 * a * a) * torch.exp(-a * a)


def _ricker_dT(t, T):
    """d/dT of the Ricker signal: u = pi^2 (t / T - 1.5)^2."""
    u = (math.pi * (t / T - 1.5)) ** 2
    du = -2.0 * math.pi**2 * (t / T - 1.5) * t / T**2
    return (2.0 * u - 3.0) * torch.exp(-u) * du


def _f64(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), device=DEVICE)


def _leapfrog(p, V, S, T, N, r):
    """V, S after N steps, and the traces (records x M x R) of every r-th."""
    Avs, Asv, g, C = (_f64(x) for x in (p.Avs, p.Asv, p.g, p.C))
    traces = []
    for n in range(N):
        V = V + p.dt * (Avs @ S + torch.outer(g, _signal(rom.ROM_WAVELET_RICKER, n * p.dt, T)))
        S = S + p.dt * (Asv @ V)
        if r and (n + 1) % r == 0:
            traces.append((C @ V).t())
    return V, S, torch.stack(traces) if traces else None


def _exact_stats(traces):
    x, _ = torch.sort(traces.double(), dim=1)
    M = x.shape[1]
    q = []
    for pr in PROBS:
        h = (M - 1) * pr
        i = min(int(math.floor(h)), M - 1)
        lo, hi = x[:, i], x[:, min(i + 1, M - 1)]
        q.append(lo + (hi - lo) * (h - i))
    return traces.double().mean(dim=1), torch.stack(q)


def _exact_adjoint(case, p, V, S, T, ystar):
    Avs, Asv, g, C = (_f64(x) for x in (p.Avs, p.Asv, p.g, p.C))
    _, _, traces = _leapfrog(p, V, S, T, case["N"], 1)
    res = traces - ystar
    lv, ls, gT = torch.zeros_like(V), torch.zeros_like(S), torch.zeros_like(T)
    for n in reversed(range(case["N"])):
        lv = lv + 2.0 * (C.t() @ res[n].t()) + p.dt * (Asv.t() @ ls)
        gT = gT + p.dt * (g @ lv) * _ricker_dT(n * p.dt, T)
        ls = ls + p.dt * (Avs.t() @ lv)
    return float((res * res).sum()), lv, ls, gT


def _exact_fom(case, seed):
    Nr, Nt, M, N, r = (case[k] for k in ("Nr", "Nt", "M", "N", "r"))
    states, T, recv = _fom_setup(case, seed)
    v, s1, s2 = (x.double().view(n, -1, M) for x, n in zip(states, (Nr, Nr - 1, Nr)))
    T = T.double()
    rc, re, rho, vs, dt = 3480e3, 6371e3, 2500.0, 5000.0, 0.05
    mu, dr, dth = rho * vs * vs, (re - rc) / Nr, math.pi / Nt
    rf = rc + dr * torch.arange(Nr + 1, device=DEVICE, dtype=torch.float64)[:, None, None]
    rh = rc + dr * (torch.arange(Nr, device=DEVICE, dtype=torch.float64)[:, None, None] + 0.5)
    sj = torch.sin(dth * torch.arange(1, Nt, device=DEVICE, dtype=torch.float64))[None, :, None]
    sh = torch.sin(dth * (torch.arange(1, Nt - 1, device=DEVICE, dtype=torch.float64) + 0.5))[None, :, None]
    depth_row = min(max(int((re - FOM_DEPTH - rc) / dr), 0), Nr - 1)
    zr, zt = torch.zeros_like(s1[:1]), torch.zeros_like(s2[:, :1])
    traces = []
    for n in range(N):
        flux = torch.cat((zr, rf[1:-1] ** 3 * s1, zr))
        v = v + (dt / rho) * (flux[1:] - flux[:-1]) / (rh**3 * dr)
        flux = torch.cat((zt, sh**2 * s2, zt), dim=1)
        v = v + (dt / rho) * (flux[:, 1:] - flux[:, :-1]) / (rh * sj**2 * dth)
        v[depth_row, 0] += (dt / rho) * _signal(rom.ROM_WAVELET_GAUSS1, (FOM_N0 + n) * dt, T)
        w = v / rh
        s1 = s1 + (dt * mu / dr) * rf[1:-1] * (w[1:] - w[:-1])
        w = v / sj
        s2 = s2 + (dt * mu / dth) * (sh / rh) * (w[:, 1:] - w[:, :-1])
        if (n + 1) % r == 0:
            traces.append(v.view(-1, M)[recv.long()])
    return v.view(-1, M), s1.view(-1, M), s2.view(-1, M), torch.stack(traces)


def exact(case, seed):
    kind = case["kind"]
    if kind == "stats":
        return _exact_stats(_stat_traces(case, seed))
    if kind == "fom":
        return _exact_fom(case, seed)
    if kind == "batched":
        out = []
        for i, (K, M) in enumerate(_batch_sizes(case)):
            p = _batch_problem(K, M, seed, i)
            V, S = _noise(100 * seed + i, (K, M), (K, M))
            out.extend(_leapfrog(p, _f64(V), _f64(S), _f64(p.T), case["N"], 0)[:2])
        return out
    p = _problem(case, seed)
    V, S = (_f64(x) for x in _noise(seed, (case["Kv"], case["M"]), (case["Ks"], case["M"])))
    if kind == "adjoint":
        ystar = _device_noise(seed, (case["N"], case["M"], case["R"]), 0.2).double()
        return _exact_adjoint(case, p, V, S, _f64(p.T), ystar)
    V, S, traces = _leapfrog(p, V, S, _f64(p.T), case["N"], case["r"])
    if kind == "rank1":
        V, S = V.reshape(-1), S.reshape(-1)
    out = [V, S]
    if traces is not None:
        out.append(traces)
    if kind == "uq":
        out.extend(_exact_stats(traces))
    return out
