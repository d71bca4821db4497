"""The work a user of this library has it do, as cases that can be timed and compared.

``listed()`` are the standing cases, ``draw(rng)`` gives more of the same ranges;
``prepare(case, seed)`` makes what a program has in hand before the call, ``run(state)`` is one
pass through the public entry points, ``work(case)`` the bytes and operations one pass cannot
do without, and ``exact(case, seed)`` the same results in plain 64-bit torch, without this
library.

Kinds of case:

  run           a catalog resident on the device, subtracted to convergence; S_gal and the
                resolved mask in device buffers
  host          the catalog in page-locked host memory, read in place; results to the host
  simulate      a catalog drawn on the device inside the catalog pass, subtracted, and its 100
                coarse-grained bins on the host (the paper's simulator)
  batch         many catalogs in one launch
  serve         a burst of jobs through the request loop
  estimate      the running estimator applied to a given device spectrum
  running_mean  the running mean of a device spectrum without device allocation
"""
from __future__ import annotations

import math

import torch

from paper_2602_18560_gb300 import gbsub, synth

F_MIN, F_MAX = 1e-4, 1e-2
RHO_TH = 7.0
BIAS = 729.0 / 512.0
ESTIMATORS = {"mean": gbsub.MEAN, "median": gbsub.MEDIAN, "median_mean": gbsub.MEDIAN_MEAN}
PRECISIONS = {"fp64": gbsub.FP64, "mixed": gbsub.MIXED}

# Populations.  "synthetic": power law f^-gamma, Gamma(shape) amplitudes, GW-driven chirps.
# "paper": the parameters of the paper's Table I.
BENCH_POP = {"model": "synthetic", "gamma": 3.293, "shape": 2.255}
PLAIN_POP = {"model": "synthetic", "gamma": 11.0 / 3.0, "shape": 2.0}


def listed():
    mm = {"window": 1000, "estimator": "median_mean", "precision": "fp64"}
    return [
        # the smallest catalog of the test and bench sizes: latency and launches
        {"name": "run_1yr_1e4", "kind": "run", "n": 10_000, "years": 1.0, **mm, **PLAIN_POP},
        # an ordinary catalog
        {"name": "run_4yr_1e6", "kind": "run", "n": 1_000_000, "years": 4.0, **mm, **PLAIN_POP},
        # the bench workload: a full galaxy
        {"name": "run_4yr_3e7", "kind": "run", "n": 30_000_000, "years": 4.0, **mm, **BENCH_POP},
        # the paper's own settings: running mean over 2000 bins
        {"name": "run_4yr_1e7_mean", "kind": "run", "n": 10_000_000, "years": 4.0,
         "window": 2000, "estimator": "mean", "precision": "fp64", **PLAIN_POP},
        # odd sizes throughout: catalog, observation time and window, the plain median, and the
        # paper's population, whose Gamma prior puts some sources on long sweeps
        {"name": "run_odd_median", "kind": "run", "n": 3_000_017, "years": 1.87654321,
         "window": 501, "estimator": "median", "precision": "fp64", "model": "paper",
         "alpha_pl": -2.8, "alpha_g": 2.2, "beta_g": 1.3, "mu_g": -21.0, "mu": -22.0,
         "sigma": 0.2, "rho": 0.0},
        # a catalog that lives in host memory, results wanted there
        {"name": "host_4yr_1e7", "kind": "host", "n": 10_000_000, "years": 4.0, **mm,
         **BENCH_POP},
        # parameters in, coarse-grained foreground out
        {"name": "simulate_4yr_3e7", "kind": "simulate", "n": 30_000_000, "years": 4.0, **mm,
         **BENCH_POP},
        # the paper's simulator at a draw of the Table I priors with long sweeps (about half of
        # the draws have them)
        {"name": "simulate_prior_1e7", "kind": "simulate", "n": 10_000_000, "years": 4.0, **mm,
         "model": "paper", "alpha_pl": -3.0, "alpha_g": 2.6, "beta_g": 1.2, "mu_g": -20.5,
         "mu": -22.0, "sigma": 0.2, "rho": 0.5},
        # many catalogs at once, mixed precision
        {"name": "batch_64", "kind": "batch", "catalogs": 64, "n_lo": 100_000,
         "n_hi": 10_000_000, "years": 4.0, "window": 1000, "estimator": "median_mean",
         "precision": "mixed", "grid_div": 4},
        # a burst of served jobs of mixed sizes and observation times
        {"name": "serve_24", "kind": "serve", "jobs": 24, "n_lo": 100_000, "n_hi": 10_000_000,
         **mm},
        # the estimator on a measured spectrum: every bin holds power
        {"name": "estimate_4yr", "kind": "estimate", "years": 4.0, "occupied": 1.0, **mm},
        # the allocation-free running mean of a one-year spectrum
        {"name": "running_mean_1yr", "kind": "running_mean", "n": 312_422, "window": 1000},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["run", "host", "simulate", "batch", "serve", "estimate", "running_mean"],
                       [8, 2, 4, 1, 1, 3, 2])[0]
    if kind == "running_mean":
        return {"kind": kind, "n": _log_uniform(rng, 20_000, 1_300_000),
                "window": _log_uniform(rng, 16, 8192)}
    case = {"kind": kind,
            "window": rng.choice([1000, 2000, _log_uniform(rng, 100, 4096)]),
            "estimator": rng.choice(sorted(ESTIMATORS)),
            "precision": rng.choice(sorted(PRECISIONS))}
    years = rng.choice([1.0, 2.0, 4.0, round(rng.uniform(0.5, 4.0), 8)])
    if kind == "estimate":
        return {**case, "years": years, "occupied": rng.choice([1.0, round(rng.random(), 3)])}
    if kind in ("batch", "serve"):
        many = {"n_lo": _log_uniform(rng, 10_000, 100_000), "n_hi": _log_uniform(rng, 300_000, 3_000_000)}
        if kind == "batch":
            return {**case, "catalogs": rng.randint(4, 32), "years": years,
                    "grid_div": rng.choice([1, 4, 8]), **many}
        return {**case, "jobs": rng.randint(6, 20), **many}
    case["years"] = years
    if kind == "simulate" and rng.random() < 0.5:
        # the paper's priors, the catalog size and the fdot tail as far as the listed case goes
        prior = {**synth.PAPER_PRIOR, "alpha_g": (1.0, 2.6), "beta_g": (1.2, 3.0),
                 "mu_g": (-22.0, -20.5)}
        pop = {k: round(rng.uniform(*prior[k]), 4)
               for k in ("alpha_pl", "alpha_g", "beta_g", "mu_g", "mu", "sigma", "rho")}
        return {**case, "model": "paper", "n": rng.randint(5_000_000, 10_000_000), **pop}
    n_hi = 30_000_000 if kind == "run" else 10_000_000
    return {**case, "n": _log_uniform(rng, 10_000, n_hi), "model": "synthetic",
            "gamma": round(rng.uniform(3.0, 4.5), 3), "shape": round(rng.uniform(1.5, 3.0), 3)}


# ------------------------------------------------------------------ inputs

def _grid(years):
    """(T_obs, first DFT index, bins) of the default band."""
    T = years * synth.YEAR
    k_lo = math.ceil(F_MIN * T)
    return T, k_lo, math.floor(F_MAX * T) - k_lo + 1


def _catalog(case, seed):
    """(A, f, fdot) of the case's population, FP64 on the device."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n = case["n"]

    def uniform():
        return torch.rand(n, generator=g, dtype=torch.float64, device="cuda")

    def gamma(shape):
        a = torch.full((n,), float(shape), dtype=torch.float64, device="cuda")
        return torch._standard_gamma(a, generator=g)

    paper = case["model"] == "paper"
    e = 1.0 + (case["alpha_pl"] if paper else -case["gamma"])  # p(f) ~ f^(e - 1)
    a, b = F_MIN ** e, F_MAX ** e
    f = (a + uniform() * (b - a)).pow_(1.0 / e).clamp_(F_MIN, F_MAX)
    if paper:
        fdot = torch.pow(10.0, case["mu_g"] + gamma(case["alpha_g"]) / case["beta_g"])
        z = torch.randn(n, generator=g, dtype=torch.float64, device="cuda")
        A = f ** (2.0 / 3.0) * torch.pow(10.0, case["mu"] + torch.exp(case["sigma"] * z))
    else:
        A = 1e-23 * gamma(case["shape"]) * (f / 1e-3) ** (2.0 / 3.0)
        mc = (0.2 + 0.6 * uniform()) * 4.925490947e-6  # chirp mass in seconds
        fdot = (96.0 / 5.0) * math.pi ** (8.0 / 3.0) * mc ** (5.0 / 3.0) * f ** (11.0 / 3.0)
    return A, f, fdot


def _spectrum(n, seed, occupied=1.0):
    """A periodogram: a steep smooth level times chi^2_2 scatter, zero outside the occupied bins."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.linspace(0.0, 1.0, n, dtype=torch.float64, device="cuda")
    u = torch.rand(n, generator=g, dtype=torch.float64, device="cuda")
    P = 1e-40 * torch.exp(-9.0 * x) * -torch.log1p(-u)
    if occupied < 1.0:
        P *= torch.rand(n, generator=g, dtype=torch.float64, device="cuda") < occupied
    return P


def _population(case):
    if case["model"] == "paper":
        return synth.PaperPopulation(**{k: case[k] for k in ("alpha_pl", "alpha_g", "beta_g",
                                                             "mu_g", "mu", "sigma", "rho")})
    return synth.Population(gamma=case["gamma"], shape=case["shape"])


def _several(case, seed, count, years):
    """(n, T_obs, seed, population) of a batch's catalogs or a burst's jobs.  The sizes are a
    fixed spread over the case's range, so that every seed is the same amount of work."""
    g = torch.Generator().manual_seed(seed)
    lo, hi = math.log(case["n_lo"]), math.log(case["n_hi"])
    out = []
    for i in range(count):
        u = (i * 0.6180339887498949) % 1.0
        r = torch.rand(2, generator=g, dtype=torch.float64).tolist()
        out.append((int(round(math.exp(lo + u * (hi - lo)))), years[i % len(years)] * synth.YEAR,
                    seed * 4096 + i,
                    synth.Population(gamma=3.0 + 1.5 * r[0], shape=1.5 + 1.5 * r[1])))
    return out


def _context(case, T):
    return gbsub.Subtraction(T_obs=T, window=case["window"],
                             estimator=ESTIMATORS[case["estimator"]],
                             precision=PRECISIONS[case["precision"]])


def _device(n, dtype):
    return torch.empty(n, dtype=dtype, device="cuda")


def _pinned(n, dtype):
    return torch.empty(n, dtype=dtype, pin_memory=True)


def prepare(case, seed):
    return {"kind": case["kind"], **_PREPARE[case["kind"]](case, seed)}


def _prepare_run(case, seed):
    T, _, nb = _grid(case["years"])
    A, f, fdot = _catalog(case, seed)
    s = _context(case, T)
    s.load(A, f, fdot)
    # the arrays stay alive until the context's copies of them have passed
    return {"s": s, "catalog": (A, f, fdot), "S_gal": _device(nb, torch.float64),
            "resolved": _device(case["n"], torch.uint8)}


def _prepare_host(case, seed):
    T, _, nb = _grid(case["years"])
    catalog = []
    for x in _catalog(case, seed):
        catalog.append(_pinned(case["n"], torch.float64))
        catalog[-1].copy_(x)
    return {"s": _context(case, T), "catalog": catalog, "S_gal": _pinned(nb, torch.float64),
            "resolved": _pinned(case["n"], torch.uint8)}


def _prepare_simulate(case, seed):
    T, _, _ = _grid(case["years"])
    return {"s": _context(case, T), "n": case["n"], "seed": seed, "pop": _population(case),
            "paper": case["model"] == "paper"}


def _prepare_batch(case, seed):
    T, _, nb = _grid(case["years"])
    specs = _several(case, seed, case["catalogs"], (case["years"],))
    subs = []
    for n, _, sd, pop in specs:
        s = _context(case, T)
        s.load_generated(n, sd, pop, fused=False)
        gbsub.sub_set_grid_div(s.ctx, case["grid_div"])
        subs.append(s)
    return {"batch": gbsub.Batch(subs), "subs": subs, "n": [n for n, _, _, _ in specs],
            "S_gal": _device(len(subs) * nb, torch.float64).view(len(subs), nb),
            "resolved": _device(sum(n for n, _, _, _ in specs), torch.uint8)}


def _prepare_serve(case, seed):
    years = (1.0, 2.0, 4.0)
    jobs = _several(case, seed, case["jobs"], years)
    srv = gbsub.Server(hbm_budget=40 * 10**9, max_inflight=32, max_contexts=12,
                       window=case["window"], estimator=ESTIMATORS[case["estimator"]],
                       precision=PRECISIONS[case["precision"]])
    for y in years:
        srv.prewarm(y * synth.YEAR, case["n_hi"], 4)
    bins = [_grid(T / synth.YEAR)[2] for _, T, _, _ in jobs]
    return {"server": srv, "jobs": jobs, "bins": bins,
            "S_gal": _pinned(sum(bins), torch.float64),
            "resolved": _pinned(sum(n for n, _, _, _ in jobs), torch.uint8)}


def _prepare_estimate(case, seed):
    T, _, nb = _grid(case["years"])
    return {"s": _context(case, T), "P": _spectrum(nb, seed, case["occupied"]),
            "out": _device(nb, torch.float64)}


def _prepare_running_mean(case, seed):
    return {"n": case["n"], "window": case["window"], "x": _spectrum(case["n"], seed),
            "out": _device(case["n"], torch.float64)}


_PREPARE = {"run": _prepare_run, "host": _prepare_host, "simulate": _prepare_simulate,
            "batch": _prepare_batch, "serve": _prepare_serve, "estimate": _prepare_estimate,
            "running_mean": _prepare_running_mean}


# ------------------------------------------------------------------ one pass

def run(state):
    return _RUN[state["kind"]](state)


def _counts(st):
    return {"iterations": st.iterations, "n_resolved": st.n_resolved,
            "n_candidates": st.n_candidates}


def _run_run(state):
    s = state["s"]
    st = s.run()
    return {"S_gal": s.spectrum(out=state["S_gal"]), "resolved": s.resolved(out=state["resolved"]),
            **_counts(st)}


def _run_host(state):
    state["s"].load(*state["catalog"], mapped=True)
    return _run_run(state)


def _run_simulate(state):
    s = state["s"]
    load = s.load_population if state["paper"] else s.load_generated
    load(state["n"], state["seed"], state["pop"], fused=True)
    st = s.run()
    S, f, count = s.coarse_grain()
    return {"S": S, "f": f, "count": count, **_counts(st)}


def _run_batch(state):
    sts = state["batch"].run()
    at = 0
    for i, (s, n) in enumerate(zip(state["subs"], state["n"])):
        s.spectrum(out=state["S_gal"][i])
        s.resolved(out=state["resolved"][at:at + n])
        at += n
    return {"S_gal": state["S_gal"], "resolved": state["resolved"],
            "n_resolved": sum(st.n_resolved for st in sts),
            "iterations": sum(st.iterations for st in sts)}


def _run_serve(state):
    srv, bin0, src0 = state["server"], 0, 0
    for i, ((n, T, sd, pop), nb) in enumerate(zip(state["jobs"], state["bins"])):
        srv.submit_generated(i, T, n, sd, pop, state["S_gal"][bin0:bin0 + nb],
                             state["resolved"][src0:src0 + n])
        bin0 += nb
        src0 += n
    done = []
    while len(done) < len(state["jobs"]):
        done += srv.poll(timeout_ms=1000)
    for r in done:
        if r["status"] not in (gbsub.OK, gbsub.ENOTCONVERGED):
            raise RuntimeError("job %d ended with %d" % (r["job_id"], r["status"]))
    return {"S_gal": state["S_gal"], "resolved": state["resolved"],
            "n_resolved": sum(r["stats"]["n_resolved"] for r in done)}


def _run_estimate(state):
    return {"out": state["s"].estimate(state["P"], out=state["out"])}


def _run_running_mean(state):
    rc = gbsub.lib().sub_running_mean_noalloc(
        state["x"].data_ptr(), state["out"].data_ptr(), state["n"], state["window"],
        torch.cuda.current_stream().cuda_stream)
    if rc != gbsub.OK:
        raise RuntimeError("sub_running_mean_noalloc: %d" % rc)
    return {"out": state["out"]}


_RUN = {"run": _run_run, "host": _run_host, "simulate": _run_simulate, "batch": _run_batch,
        "serve": _run_serve, "estimate": _run_estimate, "running_mean": _run_running_mean}


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """Bytes: each input read once, each output written once.  Operations: about a hundred per
    source to draw it, twenty to place and test it, and ten per bin to estimate."""
    kind = case["kind"]
    if kind == "running_mean":
        return {"bytes": 16 * case["n"], "flops": 10 * case["n"]}
    if kind in ("batch", "serve"):
        years = (case["years"],) if kind == "batch" else (1.0, 2.0, 4.0)
        jobs = _several(case, 0, case["catalogs" if kind == "batch" else "jobs"], years)
        nb = sum(_grid(T / synth.YEAR)[2] for _, T, _, _ in jobs)
        n = sum(n for n, _, _, _ in jobs)
        # a batch's catalogs are read, a burst's are drawn
        return {"bytes": 8 * nb + n + (24 * n if kind == "batch" else 0),
                "flops": (20 if kind == "batch" else 120) * n + 10 * nb}
    nb = _grid(case["years"])[2]
    if kind == "estimate":
        return {"bytes": 16 * nb, "flops": 10 * nb}
    n = case["n"]
    if kind == "simulate":
        return {"bytes": 100 * 24, "flops": 120 * n + 10 * nb}
    return {"bytes": 25 * n + 8 * nb, "flops": 20 * n + 10 * nb}


# ------------------------------------------------------------------ 64-bit results in plain torch

def exact(case, seed):
    kind = case["kind"]
    if kind == "running_mean":
        x = _spectrum(case["n"], seed)
        return {"out": _window_mean(x, case["window"])}
    if kind == "estimate":
        P = _spectrum(_grid(case["years"])[2], seed, case["occupied"])
        every = torch.arange(P.numel(), device=P.device)
        return {"out": _Estimator(case["estimator"], case["window"]).update(P, every)}
    if kind in ("run", "host"):
        S_gal = _subtract(case, *_catalog(case, seed))
        return None if S_gal is None else {"S_gal": S_gal, "resolved": None, "iterations": None,
                                           "n_resolved": None, "n_candidates": None}
    # the catalogs of the other kinds are this library's own draws
    return None


def _tables(T, k_lo, nb):
    """S_instr (App. C, A channel with the TDI-2 factor) and the response R (App. B)."""
    f = torch.arange(k_lo, k_lo + nb, dtype=torch.float64, device="cuda") / T
    c, arm = 299792458.0, 2.5e9
    x = f * (2.0 * math.pi * arm / c)
    w2 = (2.0 * math.pi * f / c) ** 2
    p_oms = 15e-12 ** 2 * (1.0 + (2e-3 / f) ** 4) * w2
    p_tm = (3e-15 ** 2 * (1.0 + (0.4e-3 / f) ** 2) * (1.0 + (f / 8e-3) ** 4)
            / (2.0 * math.pi * f) ** 4 * w2)
    sin2, cos = torch.sin(x) ** 2, torch.cos(x)
    tdi2 = 4.0 * torch.sin(2.0 * x) ** 2
    S = 8.0 * sin2 * (4.0 * (1.0 + cos + cos * cos) * p_tm + (2.0 + cos) * p_oms) * tdi2
    R = 16.0 * sin2 * x * x * (9.0 / 20.0) / (1.0 + 0.7 * x * x) * tdi2
    return S, R


def _pieces(A, f, fdot, T, k_lo, nb, R):
    """(source, bin, power) of every bin each source's sweep touches; None when the sweeps are
    too long to list."""
    u0 = f * T
    u1 = u0 + fdot * (T * T)
    lo, hi = torch.minimum(u0, u1), torch.maximum(u0, u1)
    ka, kb = torch.floor(lo + 0.5).long(), torch.floor(hi + 0.5).long()
    first, last = ka.clamp(min=k_lo), kb.clamp(max=k_lo + nb - 1)
    count = (last - first + 1).clamp_(min=0)
    if int(count.sum()) > 150_000_000:
        return None
    src = torch.repeat_interleave(torch.arange(A.numel(), device=A.device), count)
    start = torch.cumsum(count, 0) - count
    k = first[src] + torch.arange(src.numel(), device=A.device) - start[src]
    a = torch.maximum(lo[src], k - 0.5)
    b = torch.minimum(hi[src], k + 0.5)
    w = torch.where((ka == kb)[src], torch.ones_like(a), (b - a) / (hi - lo)[src])
    return src, k - k_lo, (T / 5.0) * R[k - k_lo] * A[src] ** 2 * w


def _bounds(rows, n, W):
    """First and last bin of the window of each output in rows."""
    s = rows - W // 2
    return s.clamp(min=0), (s + W - 1).clamp(max=n - 1)


def _windows(x, W, fill):
    """Row j: the W values of output j's window, fill outside the band."""
    left = torch.full((W // 2,), fill, dtype=x.dtype, device=x.device)
    right = torch.full((W,), fill, dtype=x.dtype, device=x.device)
    return torch.cat([left, x, right]).unfold(0, W, 1)


def _blocks(rows, W):
    return rows.split(max(1, 100_000_000 // W))


def _window_mean(x, W, rows=None):
    rows = torch.arange(x.numel(), device=x.device) if rows is None else rows
    win, out = _windows(x, W, 0.0), []
    for r in _blocks(rows, W):
        s, e = _bounds(r, x.numel(), W)
        out.append(win[r].sum(1) / (e - s + 1))
    return torch.cat(out) if out else x[:0]


def _window_median(x, W, rows):
    win, out = _windows(x, W, math.inf), []
    for r in _blocks(rows, W):
        s, e = _bounds(r, x.numel(), W)
        c = e - s + 1
        v = win[r].sort(1).values
        lo, hi = v.gather(1, ((c - 1) // 2)[:, None]), v.gather(1, (c // 2)[:, None])
        out.append((lo + hi)[:, 0] * 0.5)
    return torch.cat(out) if out else x[:0]


class _Estimator:
    """The running estimator, recomputed where its input has changed."""

    def __init__(self, kind, W):
        self.kind, self.W, self.med, self.out = kind, W, None, None

    def _reach(self, rows, n):
        """Outputs whose windows hold one of the bins in rows."""
        flag = torch.zeros(n + 1, dtype=torch.int64, device=rows.device)
        flag[rows + 1] = 1
        before = torch.cumsum(flag, 0)
        s, e = _bounds(torch.arange(n, device=rows.device), n, self.W)
        return torch.nonzero(before[e + 1] > before[s])[:, 0]

    def update(self, P, changed):
        n = P.numel()
        if self.out is None:
            self.out, self.med = torch.zeros_like(P), torch.zeros_like(P)
        rows = self._reach(changed, n)
        if self.kind == "mean":
            self.out[rows] = _window_mean(P, self.W, rows)
        else:
            self.med[rows] = BIAS * _window_median(P, self.W, rows)
            if self.kind == "median":
                self.out = self.med.clone()
            else:
                rows = self._reach(rows, n)
                self.out[rows] = _window_mean(self.med, self.W, rows)
        return self.out


def _subtract(case, A, f, fdot):
    """S_gal after the iterative subtraction (App. D)."""
    T, k_lo, nb = _grid(case["years"])
    S, R = _tables(T, k_lo, nb)
    pieces = _pieces(A, f, fdot, T, k_lo, nb, R)
    if pieces is None:
        return None
    src, j, p = pieces

    def sums(at, values, size):
        return torch.zeros(size, dtype=torch.float64, device=A.device).index_add_(0, at, values)

    rho0 = 4.0 * sums(src, p / S[j], A.numel())
    keep = (rho0 > RHO_TH ** 2 * (1.0 - 1e-12))[src]  # rho never exceeds rho_0
    csrc, cj, cp = src[keep], j[keep], p[keep]
    resolved = torch.zeros(A.numel(), dtype=torch.bool, device=A.device)
    est = _Estimator(case["estimator"], case["window"])
    P, changed = sums(j, p, nb), torch.arange(nb, device=A.device)
    for it in range(101):
        S_gal = est.update(P, changed)
        if it == 100:
            break
        rho2 = 4.0 * sums(csrc, cp / (S + S_gal)[cj], A.numel())
        new = (rho2 > RHO_TH ** 2) & ~resolved
        if not bool(new.any()):
            break
        resolved |= new
        changed = torch.unique(cj[new[csrc]])
        left = ~resolved[src]
        P = sums(j[left], p[left], nb)
    return S_gal
