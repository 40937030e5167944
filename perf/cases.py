"""The calls whose speed matters to a user of the library, with their inputs.

A case names one kind of call, the sizes and the options; ``prepare`` draws the
light curves (``synth``: irregular, seasonal and nightly sampling, individual
errors, periodic signals and pure noise) and makes what a program keeps between
calls (device copies, plans, output buffers), ``run`` is one pass of the call.

Kinds:
  oneshot   periodogram() of one curve from and to host arrays
  session   one curve start to end: Plan, execute, significance, gradients and
            refinement at its peaks, host arrays throughout
  plan      execute() of a kept Plan into a device buffer
  batch     execute_batched(), host arrays or device tensors
  adjoint   execute_batched() and backward_batched() at the peaks it found

Batched calls ask for the fixed launch configuration: float rounding depends on
the configuration, and a program that compares results between processes fixes
it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0901_1913_gb300 import _fc2, synth

TOP_K = 8


def listed():
    return [
        # the quick-start call: a thousand samples over 100 d, three harmonics;
        # allocation, launches and copies count as much as the arithmetic
        dict(name="one short curve", kind="oneshot", prec="mixed", n=1000, N=16384, H=3,
             oversample=2),
        # interactive analysis of one small curve in double, up to the refined peaks
        dict(name="short session in double", kind="session", prec="fp64", n=400, N=2048, H=3,
             oversample=2),
        # a handful of ragged curves from a reduction script, host arrays, grids
        # whose first frequency is not a multiple of the spacing
        dict(name="few ragged curves", kind="batch", prec="mixed", place="host", C=12, n=300,
             N=6001, H=4, T=100.0, f_lo=0.0213, f_hi=11.0, shared=False),
        # one long ground-based curve, 4x oversampled grids, float transforms
        dict(name="long curve", kind="plan", prec="mixed", cadence="nights", n=100_000,
             N=1 << 22, H=6, oversample=4, T=3000.0, f_hi=20.0, gridding="kernel", detrend=0),
        # the same kind of curve for a user who asks for double throughout
        dict(name="long curve in double", kind="plan", prec="fp64", cadence="nights", n=30_011,
             N=1 << 20, H=4, oversample=2, T=3000.0, f_hi=20.0, gridding="kernel", detrend=0),
        # four years of 2-minute space photometry: the largest single problem
        dict(name="large curve", kind="plan", prec="mixed", cadence="regular", n=999_999,
             N=1 << 25, H=8, oversample=2, T=1461.0, f_hi=24.0, gridding="kernel", detrend=0),
        # a slow trend fitted together with the harmonics
        dict(name="trend and harmonics", kind="plan", prec="mixed", cadence="nights", n=20_000,
             N=1 << 18, H=4, oversample=2, T=1000.0, f_hi=12.0, gridding="kernel", detrend=2),
        # the published gridding (nearest lower cell), for comparison with older catalogues
        dict(name="published gridding", kind="plan", prec="mixed", cadence="nights", n=100_000,
             N=1 << 20, H=6, oversample=2, T=3000.0, f_hi=20.0, gridding="paper", detrend=0),
        # the survey: a thousand curves of very uneven length, data kept on the device
        dict(name="survey", kind="batch", prec="mixed", place="device", C=1024, n=2000,
             N=1 << 18, H=6, T=1000.0, f_lo=0.0, f_hi=12.0, shared=False),
        # the candidates of a survey once more in double
        dict(name="survey in double", kind="batch", prec="fp64", place="device", C=32, n=2000,
             N=1 << 18, H=6, T=1000.0, f_lo=0.0, f_hi=12.0, shared=False),
        # all sources of one field, sampled together
        dict(name="shared field", kind="batch", prec="mixed", place="device", C=512, n=2000,
             N=1 << 18, H=4, T=1000.0, f_lo=0.0, f_hi=12.0, shared=True),
        # forward and backward: periodograms and gradients at the peaks found
        dict(name="gradients at peaks", kind="adjoint", prec="mixed", C=128, n=2000, N=1 << 16,
             H=4, T=500.0, f_hi=12.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _span(case, T):
    """A time span no longer than the trial grid resolves (one bin or more per
    peak of the highest harmonic)."""
    return min(T, float(case["N"] // int(case["f_hi"] * case["H"])))


def draw(rng):
    """A case of the listed ranges."""
    kind = rng.choice(["oneshot", "session", "plan", "plan", "batch", "batch", "adjoint"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    if kind in ("oneshot", "session"):
        H = rng.randint(1, 6)
        return dict(kind=kind, prec=prec, n=_log_int(rng, 60, 5000),
                    N=_log_int(rng, 700 * H, 60000), H=H, oversample=rng.choice([2, 4]))
    if kind == "plan":
        case = dict(kind=kind, prec=prec, cadence=rng.choice(["nights", "regular"]),
                    n=_log_int(rng, 1000, 300_000), N=_log_int(rng, 1 << 15, 1 << 21),
                    H=rng.randint(1, 8), oversample=rng.choice([2, 4]),
                    f_hi=rng.choice([12.0, 20.0, 24.0]), detrend=0,
                    gridding=rng.choice(["kernel", "kernel", "kernel", "paper"]))
        case["T"] = _span(case, rng.choice([500.0, 1000.0, 3000.0]))
        if case["cadence"] == "regular":  # searched up to the Nyquist frequency
            case["n"] = max(case["n"], int(2.1 * case["f_hi"] * case["T"]))
        if case["gridding"] == "kernel" and case["H"] <= 6:
            case["detrend"] = rng.choice([0, 0, 1, 2])
        return case
    if kind == "batch":
        place = rng.choice(["host", "device", "device"])
        N = _log_int(rng, 4000, 1 << (15 if place == "host" else 18))
        cells = (1 << 21) if prec == "fp64" else (1 << 26)
        case = dict(kind=kind, prec=prec, place=place, N=N,
                    C=max(2, min(_log_int(rng, 4, 512), cells // N)), n=_log_int(rng, 100, 3000),
                    H=rng.randint(2, 6), f_lo=rng.choice([0.0, 0.0213]),
                    f_hi=rng.choice([11.0, 12.0]), shared=rng.random() < 0.25)
        case["T"] = _span(case, rng.choice([100.0, 500.0, 1000.0]))
        return case
    case = dict(kind=kind, prec="mixed", C=_log_int(rng, 4, 160), n=_log_int(rng, 200, 4000),
                N=_log_int(rng, 8000, 1 << 16), H=rng.randint(1, 6), f_hi=12.0)
    case["T"] = _span(case, 500.0)
    return case


# ---------------------------------------------------------------- inputs

def _curve(case, seed):
    """One curve (t, x, sigma) and its trial grid (f_min, df)."""
    if case["kind"] in ("oneshot", "session"):
        c = synth.short_curve(seed=seed, n=case["n"], N=case["N"])
        return c.t, c.x, c.sigma, c.f_min, c.df
    T, f_hi, n = case["T"], case["f_hi"], case["n"]
    if case["cadence"] == "regular":
        # a regular cadence with 5% of the slots lost
        minutes = 0.95 * T * 24 * 60 / n
        c = synth.large_curve(seed=seed, cadence_min=minutes, years=T / synth.DAY_YEAR,
                              N=case["N"], f_max=f_hi, H=case["H"])
    else:
        c = synth.long_curve(seed=seed, n=n, N=case["N"], T=T, f_max=f_hi, H=case["H"])
    x = c.x
    if case["detrend"]:
        u = c.t / T
        x = x + 0.3 * np.std(x) * (u - 0.7 * u * u)
    return c.t, x, c.sigma, c.f_min, c.df


def _harmonics(case):
    """Harmonic counts of a survey's curves: 2 .. H in turn."""
    return (2 + np.arange(case["C"]) % (case["H"] - 1)).astype(np.int32)


def _batch(case, seed):
    """Concatenated curves and their trial grids."""
    N, T, f_hi = case["N"], case["T"], case["f_hi"]
    if case["kind"] == "adjoint":
        b = synth.adjoint_batch(seed=seed, C=case["C"], n=case["n"], N=N, T=T, f_max=f_hi,
                                H=case["H"])
        return b, b.f_min, b.df
    if case["shared"]:
        b = synth.shared_field(seed=seed, C=case["C"], n=case["n"], N=N, T=T, f_max=f_hi,
                               H=case["H"])
    else:
        b = synth.survey_batch(seed=seed, C=case["C"], N=N, T=T, f_max=f_hi,
                               n_median=float(case["n"]))
        b.H = _harmonics(case)
    if case["f_lo"] > 0.0:
        df = (f_hi - case["f_lo"]) / (N - 1)
        return b, np.full(b.C, case["f_lo"]), np.full(b.C, df)
    return b, b.f_min, b.df


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("oneshot", "session", "plan"):
        t, x, sigma, f_min, df = _curve(case, seed)
        s.update(t=t, x=x, sigma=sigma, f_min=f_min, df=df)
        if kind == "plan":
            s["plan"] = _fc2.Plan(t, x, sigma, case["H"], f_min, df, case["N"],
                                  case["oversample"], case["prec"], top_k=TOP_K,
                                  gridding=case["gridding"], detrend=case["detrend"],
                                  trend_fit=case["detrend"] > 0)
            s["dchi2"] = torch.empty((case["H"], case["N"]), dtype=torch.float64, device="cuda")
        return s
    b, f_min, df = _batch(case, seed)
    s.update(offsets=b.offsets, t=b.t, x=b.x, sigma=b.sigma, H=b.H, f_min=f_min, df=df, N=b.N)
    total = int(np.sum(b.H.astype(np.int64) * b.N))
    if kind == "adjoint" or case["place"] == "device":
        for k in ("t", "x", "sigma"):
            s[k] = torch.from_numpy(s[k]).cuda()
        s["dchi2"] = torch.empty(total, dtype=torch.float32, device="cuda")
    else:
        s["dchi2"] = np.empty(total, dtype=np.float32)
    if kind == "adjoint":
        per_sample = TOP_K * int(b.offsets[-1])
        s["d_dx"] = torch.empty(per_sample, dtype=torch.float64, device="cuda")
        s["d_dsigma"] = torch.empty(per_sample, dtype=torch.float64, device="cuda")
    return s


# ---------------------------------------------------------------- one pass

def _records(recs):
    """Peak records as arrays."""
    return dict(j=np.array([r["j"] for r in recs], dtype=np.int64),
                f=np.array([r["f"] for r in recs]), dchi2=np.array([r["dchi2"] for r in recs]),
                A=np.concatenate([r["A"] for r in recs]))


def _batched(s, shared):
    return _fc2.execute_batched(s["offsets"], s["t"], s["x"], s["sigma"], s["H"], s["f_min"],
                                s["df"], s["N"], 2, s["case"]["prec"], top_k=TOP_K,
                                dchi2=s["dchi2"], autotune="fixed", shared_sampling=shared)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "oneshot":
        d, best, peaks, chi0 = _fc2.periodogram(s["t"], s["x"], s["sigma"], case["H"], s["f_min"],
                                                s["df"], case["N"], case["oversample"],
                                                case["prec"], top_k=TOP_K)
        return dict(dchi2=d, best=_records(best), peaks=_records(peaks), chi0=chi0)
    if kind == "session":
        with _fc2.Plan(s["t"], s["x"], s["sigma"], case["H"], s["f_min"], s["df"], case["N"],
                       case["oversample"], case["prec"], top_k=TOP_K) as p:
            d, best, peaks, chi0 = p.execute()
            log_p, j_min, log_p_min, adj = p.significance(log_p=True)
            g = p.backward([r["j"] for r in peaks if r["j"] >= 0])
        return dict(dchi2=d, best=_records(best), peaks=_records(peaks), chi0=chi0, log_p=log_p,
                    j_min=j_min, log_p_min=log_p_min, adj=adj, **g)
    if kind == "plan":
        d, best, peaks, chi0 = s["plan"].execute(s["dchi2"])
        return dict(dchi2=d, best=_records(best), peaks=_records(peaks), chi0=chi0)
    if kind == "batch":
        d, peaks, _ = _batched(s, case["shared"])
        r = peaks.records
        return dict(dchi2=d, j=r["j"], f=r["f"], peak=r["dchi2"], A=r["A"])
    d, peaks, _ = _batched(s, False)
    r = peaks.records
    g = _fc2.backward_batched(s["offsets"], s["t"], s["x"], s["sigma"], s["H"], s["f_min"],
                              s["df"], s["N"], np.maximum(r["j"], 0), d_dx=s["d_dx"],
                              d_dsigma=s["d_dsigma"])
    return dict(dchi2=d, j=r["j"], peak=r["dchi2"], **g)


# ---------------------------------------------------------------- its work

def work(case):
    """Each sample read once, each periodogram value written once; per trial
    frequency 3 H transforms' share of butterflies and one Cholesky."""
    kind, N, H, n = case["kind"], case["N"], case["H"], case["n"]
    C = case.get("C", 1)
    if kind == "batch" and not case["shared"]:
        n, H = 1.65 * n, float(_harmonics(case).mean())  # n: the mean of the lengths drawn
    out = 4 if kind in ("batch", "adjoint") else 8
    nbytes = C * (24.0 * n + out * H * N)
    transforms = 3.0 * H
    if kind == "batch" and case["shared"]:
        transforms = H + 2.0 * H / C
    flops = C * (N * (transforms * 5.0 * math.log2(N) + (2 * H + 1) ** 3 / 3.0) + 100.0 * n * H)
    if kind in ("adjoint", "session"):
        nbytes += C * TOP_K * 16.0 * n
        flops += C * TOP_K * n * 40.0 * H
    if kind == "session":
        nbytes += 8.0 * H * N
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- 64-bit values

def _dchi2_exact(t, x, sigma, H, f_min, df, N, device):
    """Delta chi^2 [H, N]: per trial frequency the weighted columns
    1, cos, sin, .. orthogonalised one after another (twice), and the data's
    squared projections summed."""
    t, x, sigma = (torch.as_tensor(np.asarray(v), dtype=torch.float64, device=device)
                   for v in (t, x, sigma))
    w = 1.0 / sigma
    tau = t - t.min()
    q0 = (w / torch.linalg.vector_norm(w))
    xbar = torch.sum(w * w * x) / torch.sum(w * w)
    y = w * (x - xbar)
    out = torch.empty((H, N), dtype=torch.float64, device=device)
    n = int(t.shape[0])
    step = max(1, int(2.5e8 / (n * (2 * H + 2))))
    for a in range(0, N, step):
        j = torch.arange(a, min(a + step, N), dtype=torch.float64, device=device)
        ph = torch.remainder((f_min + j * df)[:, None] * tau[None, :], 1.0)
        basis = [q0.expand_as(ph)]
        total = torch.zeros(j.shape[0], dtype=torch.float64, device=device)
        for h in range(1, H + 1):
            arg = torch.remainder(h * ph, 1.0).mul_(2.0 * math.pi)
            for col in (torch.cos(arg).mul_(w), torch.sin(arg).mul_(w)):
                size = torch.linalg.vector_norm(col, dim=1)
                for _ in range(2):
                    for q in basis:
                        col -= torch.sum(q * col, dim=1, keepdim=True) * q
                left = torch.linalg.vector_norm(col, dim=1)
                keep = left > 1e-10 * size
                col *= torch.where(keep, 1.0 / left.clamp_min(1e-300), 0.0)[:, None]
                basis.append(col)
                total = total + (col @ y) ** 2
            out[h - 1, a:a + j.shape[0]] = total
    return out


def exact(case, seed):
    """The periodogram in 64 bits where direct sums over every (trial frequency,
    sample) take seconds; the other outputs hang on which bins are the peaks."""
    kind, H, N = case["kind"], case["H"], case["N"]
    if kind == "plan" and (case["detrend"] or case["gridding"] != "kernel"):
        return None
    cost = case.get("C", 1) * case["n"] * N * (2.0 * H + 1) ** 2
    if kind == "batch" and not case["shared"]:
        cost *= 1.65
    if cost > 1.5e12:
        return None
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if kind in ("oneshot", "session", "plan"):
        t, x, sigma, f_min, df = _curve(case, seed)
        return dict(dchi2=_dchi2_exact(t, x, sigma, H, f_min, df, N, device))
    b, f_min, df = _batch(case, seed)
    rows = []
    for c in range(b.C):
        i = slice(int(b.offsets[c]), int(b.offsets[c + 1]))
        rows.append(_dchi2_exact(b.t[i], b.x[i], b.sigma[i], int(b.H[c]), float(f_min[c]),
                                 float(df[c]), N, device).reshape(-1))
    return dict(dchi2=torch.cat(rows))
