"""The work a user has this library do, as timed cases.

Every kind of call of the public Python binding that computes something is
here once or more:

  estimate  mm_estimate on device tensors (coefficients, Sigma and R)
  nyquist   mm_coeffs at the data's own Nyquist cutoff, then mm_corr
  host      mm_estimate_host from page-locked host buffers
  corr      mm_corr on coefficients that are already there
  pairwise  mm_corr_pairwise with the positive semi-definite repair
  batch     mm_batch_epps: many small problems, a sweep of cutoffs
  serve     mm_server_submit / mm_server_poll: a burst of requests

A case is a dict of plain values; events and coefficients are made from the
seed on the GPU. Event times follow one of four patterns: "even" (every
second, assets of odd index every `step` seconds), "poisson" (continuous
arrivals, rates spread 30-fold), "grid" (one-second grid, log-normal event
counts) and "day" (one-second grid, busy open and close). Log-prices are
correlated Brownian motions (a market factor, a sector factor per ten assets
and one of each asset's own).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2003_02842_gb300 as mm

DAY_SECONDS = 28800  # one trading day of eight hours
TWO_PI = 2.0 * math.pi


def listed():
    return [
        # the smallest ordinary call: two stocks over a day, about 1400 events each, the cutoff of
        # half the event count; launches and latency are all there is
        dict(name="async_D2_N700", kind="estimate", D=2, N=700, times="grid", events=1600, sd=0.2, kernel="es",
             basis="dirichlet", prec="bf16x3"),
        # a portfolio of ten stocks as a user without a cutoff in mind runs it: the data's Nyquist
        # cutoff, Fejer weights, the Kaiser-Bessel kernel
        dict(name="nyquist_D10", kind="nyquist", D=10, N=14399, times="grid", events=4000, sd=0.7, kernel="kb",
             basis="fejer", prec="bf16x3"),
        # the benchmark's block workload, the ordinary large estimate
        dict(name="block_D100_N10000", kind="estimate", D=100, N=10000, times="poisson", events=7500, kernel="es",
             basis="dirichlet", prec="bf16x3"),
        # the same in double precision throughout, for users who want ten more digits
        dict(name="block_D100_N10000_fp64", kind="estimate", D=100, N=10000, times="poisson", events=7500,
             kernel="es", basis="dirichlet", prec="fp64"),
        # the same from host memory to host memory
        dict(name="block_D100_N10000_host", kind="host", D=100, N=10000, times="poisson", events=7500, kernel="es",
             basis="dirichlet", prec="bf16x3"),
        # the paper's timing table: two synchronous assets of 1e5 points, Gaussian gridding at 1e-12
        dict(name="timing_D2_n100000_fp64", kind="estimate", D=2, N=50000, times="even", events=100000, step=1,
             kernel="gauss", basis="dirichlet", prec="fp64"),
        # the largest single estimate: a whole market day of 500 stocks at the one-second Nyquist cutoff
        dict(name="day_D500_tf32", kind="estimate", D=500, N=14399, times="day", events=20000, kernel="es",
             basis="fejer", prec="3xtf32"),
        # the contraction alone, from coefficients kept from an earlier call
        dict(name="corr_D500", kind="corr", D=500, N=14399, basis="dirichlet", prec="bf16x3"),
        # a cutoff of its own for every asset, and the repair of the indefinite matrix that gives
        dict(name="pairwise_D100_psd", kind="pairwise", D=100, N=10000, basis="fejer", prec="bf16x3"),
        # Monte Carlo replications of a ten-asset day with an Epps sweep over 64 cutoffs
        dict(name="batch_R512_D10", kind="batch", R=512, D=10, N=14399, cutoffs=64, times="grid", events=2000,
             sd=1.0, kernel="es", basis="dirichlet", prec="bf16x3"),
        # the accuracy experiment: thousands of tiny two-asset problems, every cutoff up to 50
        dict(name="batch_R8192_n100", kind="batch", R=8192, D=2, N=50, cutoffs=50, times="even", events=100, step=2,
             kernel="es", basis="fejer", prec="bf16x3"),
        # a burst at the serving form: windows, subsets and cutoff rules of the serving workload
        dict(name="serve_D500", kind="serve", D=500, requests=32, times="day", events=20000, kernel="es",
             basis="fejer", prec="bf16x3"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["estimate", "estimate", "estimate", "nyquist", "host", "corr", "pairwise", "batch", "batch",
                       "serve"])
    basis = rng.choice(["dirichlet", "fejer"])
    prec = rng.choice(["bf16x3", "bf16x3", "3xtf32", "fp64"])
    kernel = rng.choice(["es", "es", "kb", "gauss"])
    c = dict(kind=kind, basis=basis, prec=prec)
    if kind in ("corr", "pairwise"):
        # as many assets as the listed cases, half of them in double precision (64-bit units are narrow)
        top = 500 if kind == "corr" else 130
        D = _log_int(rng, 2, top if prec != "fp64" else top // 2)
        return dict(c, D=D, N=_log_int(rng, 100, 14399 if kind == "corr" else 10000))
    if kind == "serve":
        return dict(c, D=_log_int(rng, 50, 500), requests=rng.randint(8, 32), times="day",
                    events=20000, kernel=kernel, prec=rng.choice(["bf16x3", "3xtf32"]))
    if kind == "batch":
        prec = rng.choice(["bf16x3", "bf16x3", "bf16x3", "fp64"])
        if rng.random() < 0.5:
            N = _log_int(rng, 20, 400)
            return dict(c, R=_log_int(rng, 256, 8192 if prec != "fp64" else 1024), D=rng.randint(2, 3), N=N,
                        cutoffs=min(N, rng.randint(10, 64)), times="even", events=2 * N, step=rng.randint(1, 3),
                        kernel=kernel, prec=prec)
        N = _log_int(rng, 1000, 14399)
        return dict(c, R=_log_int(rng, 8, 256 if prec != "fp64" else 16), D=rng.randint(2, 10), N=N,
                    cutoffs=rng.randint(16, 64), times="grid", events=_log_int(rng, 500, 4000), sd=1.0,
                    kernel=kernel, prec=prec)
    if kind == "nyquist":
        return dict(c, D=_log_int(rng, 2, 60 if prec != "fp64" else 20), N=14399, times="grid",
                    events=_log_int(rng, 500, 10000), sd=0.7, kernel=kernel)
    times = rng.choice(["poisson", "poisson", "grid"])
    D = _log_int(rng, 1 if kind == "estimate" else 2, 300 if prec != "fp64" else 80)
    events = _log_int(rng, 200, 15000)
    return dict(c, D=D, N=_log_int(rng, 50, min(40000, 4000000 // D) if prec != "fp64" else min(20000, 800000 // D)),
                times=times, events=events, sd=0.5, kernel=kernel)


# ------------------------------------------------------------------ inputs
def _generator(case, seed):
    # the same seed gives other inputs to another kind of case
    salt = sum(ord(ch) for ch in case["kind"])
    return torch.Generator(device="cuda").manual_seed(1000003 * (int(seed) + 1) + salt)


def _times(case, gen):
    """Event times of every asset, sorted by (asset, time): (asset index, seconds)."""
    R, D = case.get("R", 1), case["D"]
    n_assets, n = R * D, case["events"]
    if case["times"] == "even":
        stride = torch.where(torch.arange(n_assets, device="cuda") % D % 2 == 1, case["step"], 1)
        sec = torch.arange(n, device="cuda").repeat(n_assets, 1)
        keep = sec % stride[:, None] == 0
        asset, t = keep.nonzero(as_tuple=True)
        return asset, t.double()
    if case["times"] == "poisson":
        # rates uniform on [1/60, 1/2] of the benchmark workload, scaled to `events` on average
        rate = n * (1.0 / 60 + (1.0 / 2 - 1.0 / 60) * torch.rand(n_assets, device="cuda", generator=gen)) * 60.0 / 15.5
        count = torch.poisson(rate.float(), generator=gen).long().clamp(min=3)
        asset = torch.repeat_interleave(torch.arange(n_assets, device="cuda"), count)
        t = DAY_SECONDS * torch.rand(asset.numel(), device="cuda", generator=gen, dtype=torch.float64)
        t, order = t.sort()
        asset, order2 = asset[order].sort(stable=True)
        t = t[order2]
        keep = torch.ones_like(asset, dtype=torch.bool)
        keep[1:] = (asset[1:] != asset[:-1]) | (t[1:] > t[:-1])
        return asset[keep], t[keep]
    # one-second grid; every asset trades in the first two seconds and at the close, so the
    # Nyquist cutoff is that of the grid
    if case["times"] == "grid":
        z = torch.randn(n_assets, device="cuda", generator=gen)
        count = (n * torch.exp(case["sd"] * z)).clamp(100, DAY_SECONDS)
        prob = (count / DAY_SECONDS)[:, None]
    else:
        x = torch.linspace(-1.0, 1.0, DAY_SECONDS, device="cuda").abs()
        prob = (1.0 - torch.exp(-(0.01 + 0.99 * x**0.45) * n / 20000.0))[None, :]
    keep = torch.rand((n_assets, DAY_SECONDS), device="cuda", generator=gen) < prob
    keep[:, :2] = True
    keep[:, -1] = True
    asset, sec = keep.nonzero(as_tuple=True)
    return asset, sec.double()


def _brownian(group, t, gen):
    """A standard Brownian motion per group (days) at the times t, from 0 at the
    group's start. Steps are rounded to 2^-40 so that their sums are exact and the
    same seed gives the same prices everywhere."""
    t, order = t.sort()
    g, order2 = group[order].sort(stable=True)
    t, order = t[order2], order[order2]
    first = torch.ones_like(g, dtype=torch.bool)
    first[1:] = g[1:] != g[:-1]
    dt = torch.diff(t, prepend=t[:1])
    dt[first] = 0.0
    z = torch.randn(t.numel(), device="cuda", generator=gen, dtype=torch.float64)
    w = torch.cumsum(torch.round(z * torch.sqrt(dt / 86400.0) * 2.0**40).long(), 0)
    start = torch.cummax(torch.where(first, torch.arange(t.numel(), device="cuda"), 0), 0).values
    out = torch.empty_like(t)
    out[order] = (w - w[start]).double() * 2.0**-40
    return out


def _events(case, seed):
    """CSR events on the GPU: offsets (int64), times and log-prices (float64)."""
    gen = _generator(case, seed)
    R, D = case.get("R", 1), case["D"]
    asset, t = _times(case, gen)
    problem = asset // D
    sector = problem * (D // 10 + 1) + asset % D // 10
    vol = torch.sqrt(0.05 + 0.25 * torch.rand(R * D, device="cuda", generator=gen, dtype=torch.float64))
    w = (math.sqrt(0.1) * _brownian(problem, t, gen) + math.sqrt(0.3) * _brownian(sector, t, gen) +
         math.sqrt(0.6) * _brownian(asset, t, gen))
    logp = math.log(100.0) + vol[asset] * w
    off = torch.zeros(R * D + 1, device="cuda", dtype=torch.int64)
    off[1:] = torch.bincount(asset, minlength=R * D).cumsum(0)
    return off, t.contiguous(), logp


def _coefficients(case, seed):
    """Coefficients as an earlier call leaves them: complex Gaussian modes of one
    day of returns, correlated across assets."""
    gen = _generator(case, seed)
    dt = torch.complex128 if case["prec"] == "fp64" else torch.complex64
    shape = (case["D"], case["N"] + 1)
    own = torch.randn(shape, device="cuda", generator=gen, dtype=dt)
    market = torch.randn(shape[1:], device="cuda", generator=gen, dtype=dt)
    F = (math.sqrt(0.7) * own + math.sqrt(0.3) * market) * (math.sqrt(0.1 / 3.0) / TWO_PI)
    F[:, 0] = F[:, 0].real.to(dt)
    return F


def _pair_cutoffs(case, seed):
    r = np.random.default_rng([int(seed), 31])
    lo, hi = max(1, case["N"] // 100), case["N"]
    Ns = np.exp(r.uniform(math.log(lo), math.log(hi), case["D"])).round().astype(int).clip(lo, hi)
    Ns[0] = hi
    return [int(x) for x in Ns]


def _sweep(N, count):
    """`count` rising cutoffs, log-spaced from 1 to N."""
    out = []
    for x in np.exp(np.linspace(0.0, math.log(N), count)):
        out.append(max(int(round(x)), out[-1] + 1 if out else 1))
    return [min(x, N - count + 1 + i) for i, x in enumerate(out)]


def _requests(case, seed):
    """Windows of 5 minutes to the whole day, subsets of 10 assets to all, cutoffs by the
    window's Nyquist rule or for sampling every 60 or 600 seconds. Lengths, subset sizes and
    rules belong to the case; the seed chooses where the windows start and which assets are asked for."""
    shape = np.random.default_rng([case["requests"], case["D"]])
    r = np.random.default_rng([int(seed), 47])
    out = []
    for i in range(case["requests"]):
        length = float(shape.uniform(300, DAY_SECONDS))
        k = int(shape.integers(min(10, case["D"]), case["D"] + 1))
        rule = (0.0, 60.0, 600.0)[i % 3]
        t0 = float(r.uniform(0.0, DAY_SECONDS - length))
        assets = np.sort(r.choice(case["D"], size=k, replace=False)).astype(np.int32)
        out.append((t0, t0 + length, assets, rule))
    return out


# ------------------------------------------------------------------ the calls
def prepare(case, seed):
    kind, prec = case["kind"], case["prec"]
    tol = 1e-12 if prec == "fp64" else 1e-6
    real = torch.float64 if prec == "fp64" else torch.float32
    cplx = torch.complex128 if prec == "fp64" else torch.complex64
    st = dict(kind=kind, case=case)
    D, N = case["D"], case.get("N")
    if kind in ("corr", "pairwise"):
        st["plan"] = mm.mm_plan_create(D=D, N_max=N, tol=tol, basis=case["basis"], prec=prec)
        st["F"] = _coefficients(case, seed)
        if kind == "pairwise":
            st["Ns"] = _pair_cutoffs(case, seed)
        st["S"] = torch.empty((D, D), dtype=real, device="cuda")
        st["R"] = torch.empty((D, D), dtype=real, device="cuda")
        return st
    off, t, p = _events(case, seed)
    n_events = t.numel()
    if kind == "serve":
        st["server"] = mm.mm_server_create(D=D, N_max=DAY_SECONDS // 2, max_events=n_events, hbm_budget=16 << 30,
                                           max_slots=8, tol=tol, kernel=case["kernel"], basis=case["basis"],
                                           prec=prec)
        mm.mm_server_load(st["server"], off.cpu().numpy(), t.cpu().numpy(), p.cpu().numpy())
        st["requests"] = _requests(case, seed)
        return st
    if kind == "batch":
        R, J = case["R"], case["cutoffs"]
        st["batch"] = mm.mm_batch_create(reps=R, D=D, N_max=N, max_events=n_events, tol=tol, kernel=case["kernel"],
                                         basis=case["basis"], prec=prec)
        st["cutoffs"] = _sweep(N, J)
        st["S"] = torch.empty((R, J, D, D), dtype=real, device="cuda")
        st["R"] = torch.empty((R, J, D, D), dtype=real, device="cuda")
        st["events"] = (off, t, p)
        return st
    st["plan"] = mm.mm_plan_create(D=D, N_max=N, max_events=n_events, tol=tol, kernel=case["kernel"],
                                   basis=case["basis"], prec=prec)
    if kind == "host":
        st["events"] = tuple(x.cpu().pin_memory() for x in (off, t, p))
        st["S"] = torch.empty((D, D), dtype=real).pin_memory()
        st["R"] = torch.empty((D, D), dtype=real).pin_memory()
        return st
    st["events"] = (off, t, p)
    st["F"] = torch.empty((D, N + 1), dtype=cplx, device="cuda")
    st["S"] = torch.empty((D, D), dtype=real, device="cuda")
    st["R"] = torch.empty((D, D), dtype=real, device="cuda")
    return st


def run(st):
    kind, N = st["kind"], st["case"].get("N")
    if kind == "estimate":
        mm.mm_estimate(st["plan"], *st["events"], N, coeffs=st["F"], sigma=st["S"], R=st["R"])
        return [st["F"], st["S"], st["R"]]
    if kind == "nyquist":
        F, N = mm.mm_coeffs(st["plan"], *st["events"], N=0)
        S, R = mm.mm_corr(st["plan"], F, N, sigma=st["S"], R=st["R"])
        return [F, S, R, N]
    if kind == "host":
        mm.mm_estimate_host(st["plan"], *st["events"], N, sigma=st["S"], R=st["R"])
        return [st["S"], st["R"]]
    if kind == "corr":
        S, R = mm.mm_corr(st["plan"], st["F"], N, sigma=st["S"], R=st["R"])
        return [S, R]
    if kind == "pairwise":
        S, R, clipped = mm.mm_corr_pairwise(st["plan"], st["F"], N, st["Ns"], psd_repair=True, sigma=st["S"],
                                            R=st["R"])
        return [S, R, clipped]
    if kind == "batch":
        S, R = mm.mm_batch_epps(st["batch"], *st["events"], st["cutoffs"], sigma=st["S"], R=st["R"])
        return [S, R]
    tickets = [mm.mm_server_submit(st["server"], t0, t1, assets, dt=dt) for t0, t1, assets, dt in st["requests"]]
    done = {}
    while len(done) < len(tickets):
        for c in mm.mm_server_poll(st["server"], max_items=64, wait=0.01):
            done[c["ticket"]] = c
    return [done[k]["R"] for k in tickets] + [np.array([done[k]["N"] for k in tickets])]


# ------------------------------------------------------------------ the work
def _mean_events(case):
    n = case["events"]
    if case["times"] == "even":
        D = case["D"]
        per = sum(math.ceil(n / (case["step"] if i % 2 else 1)) for i in range(D)) / D
    elif case["times"] == "day":
        x = np.abs(np.linspace(-1.0, 1.0, DAY_SECONDS))
        per = float(np.sum(1.0 - np.exp(-(0.01 + 0.99 * x**0.45) * n / 20000.0)))
    elif case["times"] == "grid":
        per = min(DAY_SECONDS, n * math.exp(0.5 * case["sd"] ** 2))
    else:
        per = n
    return per * case["D"] * case.get("R", 1)


def _work(events, D, N, real, sums=1):
    """One problem: 16 bytes an event, a coefficient written once a mode, Sigma and R; a
    13-point stencil an event, the real transform of the twofold grid, the products of the
    upper triangle."""
    M = 2 * (2 * N + 1)
    return dict(bytes=16.0 * events + 8.0 * (D + 1) + 2.0 * real * D * (N + 1) + 2.0 * real * D * D * sums,
                flops=26.0 * events + 2.5 * D * M * math.log2(M) + D * (D + 1.0) * (2 * N + 1))


def work(case):
    kind, D, N = case["kind"], case["D"], case.get("N")
    real = 8 if case["prec"] == "fp64" else 4
    if kind == "corr":
        return dict(bytes=2.0 * real * D * (N + 1) + 2.0 * real * D * D, flops=D * (D + 1.0) * (2 * N + 1))
    if kind == "pairwise":
        # a pair's cutoff is the smaller of two log-uniform ones: about N / 15 on average; the
        # repair is one symmetric eigendecomposition and the product back, about 10 D^3
        return dict(bytes=2.0 * real * D * (N / 4.6 + 1) + 2.0 * real * D * D,
                    flops=D * (D + 1.0) * 2 * N / 15.0 + 10.0 * D**3)
    if kind == "serve":
        # a request: half the day and about half the assets on average, one of three cutoff rules
        n, k = case["requests"], (D + 10) / 2
        w = [_work(0.5 * _mean_events(case) * k / D, k, m, real) for m in (7200, 120, 12)]
        return dict(bytes=n * sum(x["bytes"] for x in w) / 3, flops=n * sum(x["flops"] for x in w) / 3)
    if kind == "batch":
        R, J = case["R"], case["cutoffs"]
        w = _work(_mean_events(case) / R, D, N, real, sums=J)
        # the coefficients stay inside the call: only Sigma and R at every cutoff come out
        return dict(bytes=R * (w["bytes"] - 2.0 * real * D * (N + 1)), flops=R * w["flops"])
    w = _work(_mean_events(case), D, N, real)
    if kind == "host":
        w["bytes"] -= 2.0 * real * D * (N + 1)
    return w


# ------------------------------------------------------------------ the answer in 64 bits
def _weights(N, basis):
    """Weights of k = 0..N with the conjugate modes folded in, for coefficients of 1/(2 pi)."""
    k = torch.arange(N + 1, device="cuda", dtype=torch.float64)
    w = torch.full_like(k, 1.0 / (2 * N + 1)) if basis == "dirichlet" else (1.0 - k / N) / (N + 1)
    w = w * 2.0
    w[0] *= 0.5
    return w * TWO_PI**2


def _corr(S):
    d = torch.diagonal(S, dim1=-2, dim2=-1)
    inv = torch.where(d > 0, torch.rsqrt(d), torch.full_like(d, math.nan))
    R = S * inv[..., :, None] * inv[..., None, :]
    return torch.where(torch.eye(S.shape[-1], device=S.device, dtype=torch.bool) & (d > 0)[..., None], 1.0, R)


def _sigma(F, basis):
    w = _weights(F.shape[1] - 1, basis)
    S = torch.zeros((F.shape[0],) * 2, device="cuda", dtype=torch.float64)
    for a in range(0, F.shape[1], 4096):
        f = torch.view_as_real(F[:, a:a + 4096].contiguous())
        x = (f * torch.sqrt(w[a:a + 4096])[None, :, None]).reshape(F.shape[0], -1)
        S += x @ x.T
    return S


def _direct(t, logp, N, t0, t1):
    """(1 / 2 pi) sum_h exp(-i k u_h) dp_h, k = 0..N, with k split as B a + b."""
    B = 256
    A = N // B + 1
    u, d = (t[:-1] - t0) / (t1 - t0), logp[1:] - logp[:-1]
    F = torch.zeros((A, B), device="cuda", dtype=torch.complex128)
    for h in range(0, u.numel(), 16384):
        x = u[h:h + 16384, None]
        one = torch.ones_like(x)
        lo = torch.polar(one.expand(-1, B), -TWO_PI * torch.frac(x * torch.arange(B, device="cuda")))
        hi = torch.polar(one.expand(-1, A), -TWO_PI * torch.frac(x * (B * torch.arange(A, device="cuda"))))
        F += hi.T @ (lo * d[h:h + 16384, None])
    return F.reshape(-1)[:N + 1] / TWO_PI


def _exact_estimate(case, seed):
    off, t, p = _events(case, seed)
    N, D = case["N"], case["D"]
    edges = off.tolist()
    t0, t1 = t.min(), t.max()
    if case["kind"] == "nyquist":
        same = torch.repeat_interleave(torch.arange(D, device="cuda"), torch.diff(off))
        gap = torch.where(same[1:] == same[:-1], torch.diff(t), math.inf)
        least = torch.full((D,), math.inf, device="cuda", dtype=torch.float64).scatter_reduce(0, same[1:], gap, "amin")
        N = int(torch.floor((t1 - t0) / (2.0 * least.max())))
    F = torch.stack([_direct(t[a:b], p[a:b], N, t0, t1) for a, b in zip(edges[:-1], edges[1:])])
    S = _sigma(F, case["basis"])
    return F, S, _corr(S), N


def _exact_batch(case, seed):
    off, t, p = _events(case, seed)
    R, D, N, J = case["R"], case["D"], case["N"], case["cutoffs"]
    asset = torch.repeat_interleave(torch.arange(R * D, device="cuda"), torch.diff(off))
    L = int(t.max())  # every problem starts at second 0 and has an event at the last one
    last = torch.ones_like(asset, dtype=torch.bool)
    last[:-1] = asset[1:] != asset[:-1]
    d = torch.zeros_like(p)
    d[:-1] = p[1:] - p[:-1]
    flat = (asset * L + t.long())[~last]
    d, kept = d[~last], asset[~last]
    cut = torch.tensor(_sweep(N, J), device="cuda")
    k = torch.arange(N + 1, device="cuda", dtype=torch.float64)
    two = torch.where(k > 0, 2.0, 1.0)
    S = torch.empty((R, J, D, D), device="cuda", dtype=torch.float64)
    group = max(1, min(R, 2**26 // (D * max(L, (N + 1) * D))))
    for r in range(0, R, group):
        m = min(group, R - r)
        at = (kept >= r * D) & (kept < (r + m) * D)
        x = torch.zeros(m * D * L, device="cuda", dtype=torch.float64)
        x[flat[at] - r * D * L] = d[at]
        F = torch.fft.fft(x.reshape(m, D, L))[..., torch.arange(N + 1, device="cuda") % L] / TWO_PI
        q = (F[:, :, None, :] * F[:, None, :, :].conj()).real * two
        P = q.cumsum(-1)[..., cut].movedim(-1, 1)
        c = cut.double()[None, :, None, None]
        if case["basis"] == "fejer":
            Q = (q * k).cumsum(-1)[..., cut].movedim(-1, 1)
            S[r:r + m] = (P - Q / c) / (c + 1.0)
        else:
            S[r:r + m] = P / (2.0 * c + 1.0)
    S *= TWO_PI**2
    return [S, _corr(S)]


def _exact_serve(case, seed):
    off, t, p = _events(case, seed)
    D = case["D"]
    asset = torch.repeat_interleave(torch.arange(D, device="cuda"), torch.diff(off))
    out, Ns = [], []
    for t0, t1, assets, dt in _requests(case, seed):
        of = torch.full((D,), -1, device="cuda", dtype=torch.int64)
        of[torch.from_numpy(assets).cuda().long()] = torch.arange(len(assets), device="cuda")
        sel = (t >= t0) & (t <= t1) & (of[asset] >= 0)
        a, s, v = of[asset[sel]], t[sel], p[sel]
        same = a[1:] == a[:-1]
        if dt > 0:
            N = max(1, int(math.floor(0.5 * ((t1 - t0) / dt - 1.0))))
        else:
            least = torch.full((len(assets),), math.inf, device="cuda", dtype=torch.float64)
            least = least.scatter_reduce(0, a[1:][same], torch.diff(s)[same], "amin")
            N = int(math.floor((t1 - t0) / (2.0 * float(least[torch.isfinite(least)].max()))))
        N = min(N, DAY_SECONDS // 2)
        first = math.ceil(t0)
        x = torch.zeros((len(assets), int(t1) - first + 1), device="cuda", dtype=torch.float64)
        x[a[:-1][same], s[:-1][same].long() - first] = torch.diff(v)[same]
        u = (torch.arange(x.shape[1], device="cuda") + (first - t0)) / (t1 - t0)
        F = []
        for k in range(0, N + 1, 2048):
            ang = TWO_PI * torch.frac(u[:, None] * torch.arange(k, min(k + 2048, N + 1), device="cuda").double())
            F.append(torch.complex(x @ torch.cos(ang), -(x @ torch.sin(ang))) / TWO_PI)
        out.append(_corr(_sigma(torch.cat(F, 1), case["basis"])))
        Ns.append(N)
    return out + [np.array(Ns)]


def _exact_pairwise(case, seed):
    F = _coefficients(case, seed).to(torch.complex128)
    D = case["D"]
    Ns = _pair_cutoffs(case, seed)
    S = torch.zeros((D, D), device="cuda", dtype=torch.float64)
    for i in range(D):
        n = Ns[i]
        js = [j for j in range(D) if Ns[j] >= n]
        v = ((F[js, :n + 1].conj() * F[i, :n + 1]).real * _weights(n, case["basis"])).sum(1)
        S[i, js] = v
        S[js, i] = v
    lam, V = torch.linalg.eigh(S)
    if (lam < 0).any():
        S = (V * lam.clamp(min=0.0)) @ V.T
    return [S, _corr(S), None]


def exact(case, seed):
    kind = case["kind"]
    if kind == "corr":
        S = _sigma(_coefficients(case, seed).to(torch.complex128), case["basis"])
        return [S, _corr(S)]
    if kind == "pairwise":
        return _exact_pairwise(case, seed)
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "serve":
        return _exact_serve(case, seed)
    F, S, R, N = _exact_estimate(case, seed)
    return [S, R] if kind == "host" else [F, S, R, N] if kind == "nyquist" else [F, S, R]
