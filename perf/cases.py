"""Measured cases: what a user of the FPW library has it do, through its public
Python entry points, from one short curve to whole batches.

Inputs follow the library's ZTF-like recipe (three 240-day seasons, nights
about 3 days apart, visit pairs 30 minutes apart, sinusoid / eclipse / sawtooth
/ noise curves, flux shifted by its weighted mean) and are made from the seed
alone. A case is a dict of plain values; ``kind`` selects the entry point.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2502_00243_gb300 as G

SEASONS, NIGHTS = 3, 80
EXACT_LIMIT = 6.0e9  # evaluations that the 64-bit reference does in well under 20 s


def listed():
    return [
        # One short curve on a small grid, dense S: the interactive call, where latency counts.
        dict(name="curve_small", kind="curve", n=200, M=10, F=10_000, df=5e-3),
        # One well-sampled survey curve over a deep grid, top peaks only: the usual single-object search.
        dict(name="curve_deep", kind="batch", C=1, n_lo=1000, n_hi=1000, M=20, F=1_000_000, df=1e-4, k=5),
        # A ragged survey batch at the default bin count: the bulk of a catalogue run.
        dict(name="batch_ragged", kind="batch", C=1000, n_lo=50, n_hi=2000, M=20, F=50_000, df=2.5e-4, k=5),
        # Sparse curves (few visits per object) with few bins: many short curves, reduction and peaks count.
        dict(name="batch_sparse", kind="batch", C=4000, n_lo=20, n_hi=150, M=10, F=20_001, df=5e-4, k=5),
        # Fine binning for narrow eclipses.
        dict(name="batch_fine", kind="batch", C=200, n_lo=100, n_hi=3000, M=50, F=50_000, df=1e-4, k=5),
        # A grid uniform in log frequency instead of linear: long-period and multi-decade searches.
        dict(name="batch_loggrid", kind="batch", C=24, n_lo=100, n_hi=2000, M=20, F=100_003, grid="log", f_lo=0.02,
             f_hi=10.0, k=5),
        # Compensated sums, dense S: when the periodogram itself is analysed further.
        dict(name="dense_compensated", kind="dense", C=16, n_lo=100, n_hi=2000, M=20, F=100_000, df=1e-4, accum=2),
        # Several bin counts with every bin offset from one pass (M = 20, 10, 4 from 60 bins).
        dict(name="several_m", kind="multi", C=64, n_lo=100, n_hi=3000, M=60, g0=3, g1=6, g2=15, F=50_000, df=1e-4,
             k=5),
        # One field's curves, all observed in the same exposures.
        dict(name="shared_field", kind="shared", C=512, n=1000, M=20, F=50_000, df=1e-4, k=5),
        # Baseline drift marginalised with three Chebyshev terms, ragged curves.
        dict(name="drift_ragged", kind="drift", C=64, n_lo=50, n_hi=2000, M=20, K=3, F=20_000, df=2.5e-4, k=5),
        # Phase entropy of one field's times over a deep grid.
        dict(name="entropy_deep", kind="entropy", n=1000, M=20, F=1_000_000, df=1e-4),
        # The whole call on host buffers, copies included (pinned inputs), on a coarse first-look grid.
        dict(name="host_batch", kind="host", C=1000, n_lo=100, n_hi=3000, M=20, F=20_000, df=5e-4, k=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["curve", "batch", "batch", "batch", "batch", "dense", "multi", "shared", "drift", "entropy",
                       "host"])
    F = _log_int(rng, 2_000, 100_000)
    df = 10.0 ** rng.uniform(-4.0, -2.5)
    if kind == "curve":
        return dict(kind="curve", n=_log_int(rng, 30, 3000), M=rng.randint(4, 64), F=F, df=df)
    if kind == "entropy":
        return dict(kind="entropy", n=_log_int(rng, 50, 1000), M=rng.randint(5, 50),
                    F=_log_int(rng, 10_000, 1_000_000), df=1e-4)
    n_lo = _log_int(rng, 20, 300)
    n_hi = min(3000, n_lo * rng.randint(2, 20))
    mean = 0.5 * (n_lo + n_hi)
    if kind == "shared":
        n = _log_int(rng, 100, 1000)
        C = rng.randint(40, 512)
        return dict(kind="shared", C=C, n=n, M=rng.randint(8, 50), F=min(F, 50_000), df=df, k=rng.randint(1, 10))
    M = rng.choice([rng.randint(5, 16), rng.randint(17, 33), rng.randint(34, 64)])
    budget = {"batch": 4e10, "host": 3e10, "dense": 1.5e9, "multi": 3e9, "drift": 1.2e9}[kind]
    C = max(1, min(_log_int(rng, 1, 4000), int(budget / (mean * F))))
    c = dict(kind=kind, C=C, n_lo=n_lo, n_hi=n_hi, M=M, F=F, df=df, k=rng.randint(1, 20))
    if kind == "batch" and rng.random() < 0.3:
        c.update(grid="log", f_lo=0.02, f_hi=10.0, C=max(1, C // 10))
        del c["df"]
    if kind == "dense":
        c.update(accum=rng.choice([0, 2]), C=min(C, 64))
        del c["k"]
    if kind == "multi":
        c["M"], c["g0"], c["g1"], c["g2"] = rng.choice([(60, 3, 6, 15), (40, 2, 4, 10), (20, 1, 2, 4), (36, 2, 3, 6)])
    if kind == "drift":
        c.update(K=rng.randint(0, 4), C=min(C, 500))
    return c


# ---------------------------------------------------------------- inputs
def _times(C, ns, gen):
    """Sorted cadence times per curve, as [C, n_max] with valid entries first."""
    n_max = int(ns.max())
    pairs = max(1, -(-n_max // (SEASONS * NIGHTS * 2)))
    need = torch.ceil(ns.double() / (SEASONS * NIGHTS * 2)).clamp_(min=1)
    night = torch.arange(NIGHTS, device="cuda", dtype=torch.float64)[None, None, :] * 3.0
    day = (365.0 * torch.arange(SEASONS, device="cuda", dtype=torch.float64)[None, :, None] + night)
    first = day + 0.1 + 0.3 * torch.rand(C, SEASONS, NIGHTS, generator=gen, device="cuda", dtype=torch.float64)
    p = torch.arange(pairs, device="cuda", dtype=torch.float64) / 24.0
    visit = torch.tensor([0.0, 30.0 / 1440.0], device="cuda", dtype=torch.float64)
    t = (first[:, :, :, None, None] + p[:, None] + visit).reshape(C, -1)
    late = torch.arange(pairs, device="cuda")[None, :] >= need[:, None]  # pair slots this curve does not use
    late = late[:, None, None, :, None].expand(C, SEASONS, NIGHTS, pairs, 2).reshape(C, -1)
    key = torch.rand(t.shape, generator=gen, device="cuda") + 2.0 * late
    t = torch.gather(t, 1, key.argsort(dim=1)[:, :n_max])
    keep = torch.arange(n_max, device="cuda")[None, :] < ns[:, None]
    t = torch.where(keep, t, torch.inf).sort(dim=1).values
    return torch.where(keep, t - t[:, :1], torch.inf), keep


def _fluxes(t, keep, gen):
    """Fluxes and errors of curves with random waveforms at times t [C, n]."""
    C, n = keep.shape

    def logu(lo, hi, *shape):
        u = torch.rand(*shape, generator=gen, device="cuda", dtype=torch.float64)
        return torch.exp(math.log(lo) + u * math.log(hi / lo))

    sigma = logu(0.01, 0.3, C, n)
    period, amp = logu(0.05, 50.0, C, 1), logu(0.2, 5.0, C, 1) * 0.055
    ph = torch.remainder(torch.where(keep, t, 0.0) / period + logu(1.0, 2.0, C, 1), 1.0)
    shape = torch.randint(0, 4, (C, 1), generator=gen, device="cuda")
    s = torch.where(shape == 0, torch.sin(2 * math.pi * ph),
                    torch.where(shape == 1, (ph < 0.08).double(), torch.where(shape == 2, ph - 0.5, 0.0 * ph)))
    x = amp * s + sigma * torch.randn(C, n, generator=gen, device="cuda", dtype=torch.float64)
    w = torch.where(keep, 1.0 / (sigma * sigma), 0.0)
    return x - (w * x).sum(1, keepdim=True) / w.sum(1, keepdim=True), sigma


def _grid(case):
    if case.get("grid") == "log":
        return np.geomspace(case["f_lo"], case["f_hi"], case["F"])
    return 0.01 + case["df"] * np.arange(case["F"], dtype=np.float64)


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if "n" in case:  # one set of times
        C = case.get("C", 1)
        ns = torch.full((1,), case["n"], device="cuda", dtype=torch.int64)
        t, keep = _times(1, ns, gen)
        x, sigma = _fluxes(t.expand(C, -1), keep.expand(C, -1), gen)
        d = dict(t=t[0].contiguous(), x=x.contiguous(), sigma=sigma.contiguous())
    else:
        C, lo, hi = case["C"], case["n_lo"], case["n_hi"]
        ns = torch.randint(lo, hi + 1, (C,), generator=gen, device="cuda")
        parts = []
        for c0 in range(0, C, 500):
            t, keep = _times(ns[c0:c0 + 500].numel(), ns[c0:c0 + 500], gen)
            x, sigma = _fluxes(t, keep, gen)
            parts.append((t[keep], x[keep], sigma[keep]))
        t, x, sigma = (torch.cat([p[j] for p in parts]) for j in range(3))
        off = np.zeros(C + 1, dtype=np.int64)
        np.cumsum(ns.cpu().numpy(), out=off[1:])
        d = dict(t=t, x=x, sigma=sigma, offsets=torch.from_numpy(off).cuda(), offsets_host=off)
    d["freqs"] = torch.from_numpy(_grid(case)).cuda()
    return d


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"], s["ctx"], s["params"] = case, G.Context(0), None
    C, F, k = case.get("C", 1), case["F"], case.get("k", 0)
    rows = C * (3 if case["kind"] == "multi" else 1)
    if case["kind"] in ("curve", "dense"):
        s["S"] = torch.empty(rows * F, dtype=torch.float64, device="cuda")
    if case["kind"] == "entropy":
        s["H"] = torch.empty(F, dtype=torch.float32, device="cuda")
    if case.get("accum"):
        s["params"] = G.fpw_params_default(accum=case["accum"])
    if k:
        s["idx"] = torch.empty(rows * k, dtype=torch.int32, device="cuda")
        s["off"] = torch.empty(rows * k, dtype=torch.int32, device="cuda")
        s["Sk"] = torch.empty(rows * k, dtype=torch.float32, device="cuda")
    if case["kind"] == "host":
        s["host"] = {q: s[q].cpu().pin_memory().numpy() for q in ("offsets", "t", "x", "sigma", "freqs")}
        s["host_idx"] = torch.empty(rows * k, dtype=torch.int32).pin_memory().numpy()
        s["host_S"] = torch.empty(rows * k, dtype=torch.float32).pin_memory().numpy()
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    ctx, p, M, k = s["ctx"], s["params"], case["M"] if "M" in case else 0, case.get("k", 0)
    if kind == "curve":
        G.fpw_periodogram_ex(ctx, None, p, s["t"], s["x"][0], s["sigma"][0], s["freqs"], M, s["S"])
        return [s["S"]]
    if kind == "batch":
        G.fpw_periodogram_batch_ex(ctx, None, p, s["offsets"], s["offsets_host"], s["t"], s["x"], s["sigma"],
                                   s["freqs"], M, k, s["idx"], s["Sk"])
        return [s["idx"], s["Sk"]]
    if kind == "dense":
        G.fpw_periodogram_batch_ex(ctx, None, p, s["offsets"], s["offsets_host"], s["t"], s["x"], s["sigma"],
                                   s["freqs"], M, 0, None, None, s["S"])
        return [s["S"]]
    if kind == "multi":
        G.fpw_periodogram_batch_multi(ctx, None, p, s["offsets"], s["offsets_host"], s["t"], s["x"], s["sigma"],
                                      s["freqs"], M, [case["g0"], case["g1"], case["g2"]], k, s["idx"], s["off"],
                                      s["Sk"])
        return [s["idx"], s["off"], s["Sk"]]
    if kind == "shared":
        G.fpw_periodogram_shared(ctx, None, p, s["t"], s["x"], s["sigma"], s["freqs"], M, k, s["idx"], s["Sk"])
        return [s["idx"], s["Sk"]]
    if kind == "drift":
        G.fpw_periodogram_drift(ctx, None, p, s["offsets"], s["t"], s["x"], s["sigma"], s["freqs"], M, case["K"], 1.0,
                                k, s["idx"], s["Sk"])
        return [s["idx"], s["Sk"]]
    if kind == "entropy":
        G.fpw_phase_entropy(ctx, None, s["t"], s["freqs"], M, s["H"])
        return [s["H"]]
    h = s["host"]
    G.fpw_periodogram_batch_host(ctx, p, h["offsets"], h["t"], h["x"], h["sigma"], h["freqs"], M, k, s["host_idx"],
                                 s["host_S"])
    return [s["host_idx"], s["host_S"]]


def _mean_n(case):
    return case["n"] if "n" in case else 0.5 * (case["n_lo"] + case["n_hi"])


def work(case):
    """Inputs read once, outputs written once; per (observation, frequency) the
    phase (multiply, fraction), the bin (multiply, floor) and the bin's sums,
    per (bin, frequency) the term of the statistic."""
    kind, C, F, k = case["kind"], case.get("C", 1), case["F"], case.get("k", 0)
    n, M = _mean_n(case), case["M"]
    out = {"curve": 8 * F, "dense": 8 * F * C, "entropy": 4 * F, "multi": 36 * C * k}.get(kind, 8 * C * k)
    pairs, cells = n * F, M * F
    if kind == "shared":
        return dict(bytes=8 * n + 16 * n * C + 8 * F + out, flops=4 * pairs + 2 * pairs * C + 4 * cells * C)
    if kind == "entropy":
        return dict(bytes=8 * n + 8 * F + out, flops=5 * pairs + 3 * cells)
    sums = 1 + case["K"] if kind == "drift" else 2
    return dict(bytes=24 * n * C + 8 * F + out, flops=(4 + sums) * pairs * C + 4 * cells * C)


# ---------------------------------------------------------------- 64-bit reference
def _bins(t, f, M):
    """Bins [len(f), n] of times t at frequencies f (binary64 phase, floor, clamp)."""
    p = f[:, None] * t[None, :]
    return torch.floor(M * (p - torch.floor(p))).long().clamp_(0, M - 1)


def _sums(t, f, M, values):
    b = _bins(t, f, M)
    z = torch.zeros(f.numel(), M, dtype=torch.float64, device=f.device)
    return [z.clone().scatter_add_(1, b, v.expand(f.numel(), -1)) for v in values]


def _eq1(A, B):
    return torch.where(B > 0, A * A / torch.where(B > 0, B, 1.0), 0.0).sum(-1)


def _chunks(f, n, M):
    step = max(1, int(3e7 // max(n, M)))
    return [f[i:i + step] for i in range(0, f.numel(), step)]


def _curve_S(t, x, sigma, f, M):
    w = 1.0 / (sigma * sigma)
    return torch.cat([_eq1(*_sums(t, fc, M, (x * w, w))) for fc in _chunks(f, t.numel(), M)])


def _multi_S(t, x, sigma, f, M, groups):
    w = 1.0 / (sigma * sigma)
    rows = [[] for _ in groups]
    for fc in _chunks(f, t.numel(), M):
        A, B = _sums(t, fc, M, (x * w, w))
        for q, g in enumerate(groups):
            best = None
            for o in range(g):
                Ao = torch.roll(A, -o, 1).reshape(-1, M // g, g).sum(-1)
                Bo = torch.roll(B, -o, 1).reshape(-1, M // g, g).sum(-1)
                S = _eq1(Ao, Bo)
                best = S if best is None else torch.maximum(best, S)
            rows[q].append(best)
    return [torch.cat(r) for r in rows]


def _drift_S(t, x, sigma, f, M, K):
    w = 1.0 / (sigma * sigma)
    tau = 2.0 * (t - t.min()) / (t.max() - t.min()) - 1.0
    B = [torch.ones_like(tau), tau]
    while len(B) < K:
        B.append(2.0 * tau * B[-1] - B[-2])
    B = B[:K]
    if K:
        Bm = torch.stack(B, 1)
        H0 = torch.eye(K, dtype=torch.float64, device=t.device) + Bm.T @ (w[:, None] * Bm)
        x = x - Bm @ torch.linalg.solve(H0, Bm.T @ (w * x))
    out = []
    for fc in _chunks(f, t.numel(), M):
        s = _sums(t, fc, M, [w * x, w] + [w * b for b in B])
        z, L = s[0], s[1]
        r = torch.where(L > 0, 1.0 / torch.where(L > 0, L, 1.0), 0.0)
        S = (z * z * r).sum(1)
        if K:
            Q = torch.stack(s[2:], 2)
            v = (Q * (z * r)[:, :, None]).sum(1)
            H = H0 - torch.einsum("fmk,fml,fm->fkl", Q, Q, r)
            H[:, 0, :] = 0.0  # without a prior on the bins the constant term drops out: H_00 = 1, H_0k = 0, v_0 = 0
            H[:, :, 0] = 0.0
            H[:, 0, 0] = 1.0
            v = v.clone()
            v[:, 0] = (s[1] * z * r).sum(1)
            S = S + (v * torch.linalg.solve(H, v[:, :, None])[:, :, 0]).sum(1)
        out.append(S)
    return torch.cat(out)


def _peaks(S, k):
    """The k largest local maxima of S (NaN where there are fewer)."""
    left = torch.cat([S.new_full((1,), -torch.inf), S[:-1]])
    right = torch.cat([S[1:], S.new_full((1,), -torch.inf)])
    p = S[(S > left) & (S >= right)].sort(descending=True).values[:k]
    return torch.cat([p, S.new_full((k - p.numel(),), torch.nan)])


def exact(case, seed):
    kind, M, k = case["kind"], case["M"], case.get("k", 0)
    # drift and several-M references cost about three plain ones; sharing curves cost one matrix product
    cost = _mean_n(case) * case["F"] * case.get("C", 1) * {"drift": 4, "multi": 4, "shared": 0.15}.get(kind, 1)
    if cost > EXACT_LIMIT:
        return None
    d = _inputs(case, seed)
    f = d["freqs"]
    if kind == "curve":
        return [_curve_S(d["t"], d["x"][0], d["sigma"][0], f, M)]
    if kind == "entropy":
        H = []
        for fc in _chunks(f, case["n"], M):
            q = _sums(d["t"], fc, M, (torch.ones_like(d["t"]),))[0] / case["n"]
            H.append(-torch.where(q > 0, q * torch.log(torch.where(q > 0, q, 1.0)), 0.0).sum(1))
        return [torch.cat(H)]
    if kind == "shared":
        w = 1.0 / (d["sigma"] * d["sigma"])
        V = torch.cat([d["x"] * w, w])
        rows = []
        for i in range(0, f.numel(), 256):
            fc = f[i:i + 256]
            b = _bins(d["t"], fc, M)
            H = torch.zeros(case["n"], fc.numel(), M, dtype=torch.float64, device=f.device)
            H.scatter_(2, b.T[:, :, None], 1.0)
            D = (V @ H.reshape(case["n"], -1)).reshape(2, case["C"], fc.numel(), M)
            rows.append(_eq1(D[0], D[1]))
        S = torch.cat(rows, 1)
        return [None, torch.cat([_peaks(r, k) for r in S])]
    out = []
    for c in range(case["C"]):
        a, b = int(d["offsets_host"][c]), int(d["offsets_host"][c + 1])
        t, x, sigma = d["t"][a:b], d["x"][a:b], d["sigma"][a:b]
        if kind == "multi":
            out += [_peaks(S, k) for S in _multi_S(t, x, sigma, f, M, [case["g0"], case["g1"], case["g2"]])]
        elif kind == "drift":
            out.append(_peaks(_drift_S(t, x, sigma, f, M, case["K"]), k))
        elif kind == "dense":
            out.append(_curve_S(t, x, sigma, f, M))
        else:
            out.append(_peaks(_curve_S(t, x, sigma, f, M), k))
    v = torch.cat(out)
    return {"dense": [v], "multi": [None, None, v]}.get(kind, [None, v])
