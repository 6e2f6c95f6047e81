"""Workloads of the CCM library at the sizes its users run, each through the public calls.

A case is one call (or one burst of served jobs) with the series, plan and
buffers that a program keeps between calls already made.  Kinds:

  plan         ccm_plan once, then ccm_run per pass (device or host buffers,
               optionally followed by ccm_convergence on the rho it wrote, or
               ccm_run_ex with the libraries, neighbours and predictions)
  cell         ccm_run_noalloc, one (pair, E, tau, L) cell on the caller's stream
  serve        ccm_submit of a burst of jobs, ccm_poll until all are back
  convergence  ccm_convergence on a rho grid that lies on the device

Series are the coupled logistic maps of ``paper_1905_00565_gb300.inputs``, the
couplings, starting values and noise drawn from the seed.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1905_00565_gb300 import ccm as C
from paper_1905_00565_gb300 import inputs as I

_CTX = None
_STREAM = None


def _context():
    """One context and one stream per program, as a user keeps them."""
    global _CTX, _STREAM
    if _CTX is None:
        torch.cuda.init()
        _CTX = C.ccm_context_create(0)
        _STREAM = torch.cuda.Stream()
    return _CTX, _STREAM


def _plan_case(name, n, E, tau, L, r, variables=2, noise=0.0, theiler=0, weight_floor=0.0,
               host=False, converge=False, details=False):
    c = {"kind": "plan", "n": n, "E": E, "tau": tau, "L": L, "r": r, "variables": variables,
         "noise": noise, "theiler": theiler, "weight_floor": weight_floor, "host": host,
         "converge": converge, "details": details}
    return dict(c, name=name) if name else c


def _log_L(lo, hi, count):
    """count distinct library sizes, log-spaced."""
    return " ".join(str(v) for v in sorted({int(v) for v in I.log_grid(lo, hi, count)}))


def listed():
    return [
        # A latency-critical loop's smallest call: a handful of realizations of one short
        # cell, nothing but launches.
        {"name": "cell-n500", "kind": "cell", "n": 500, "E": 3, "tau": 1, "L": 120, "r": 10},
        # The same call on a longer series with a library of several shared-memory tiles.
        {"name": "cell-n10000", "kind": "cell", "n": 10000, "E": 5, "tau": 2, "L": 1500, "r": 50},
        # The plain single job (both directions, one E and tau), device buffers.
        _plan_case("job-n1000", 1000, "2", "1", "50 100 200 400 800", 100),
        # The paper's baseline scenario with host buffers, and the decision at its end.
        _plan_case("paper-n4000-host", 4000, "1 2 4", "1 2 4", "500 1000 2000", 500, host=True,
                   converge=True),
        # An odd-sized noisy job with the exclusion window and the weight floor.
        _plan_case("options-n2347", 2347, "4 7", "3", "60 217 801 2099", 150, noise=0.01,
                   theiler=10, weight_floor=0.01),
        # A job whose user looks at the neighbours and predictions themselves.
        _plan_case("details-n3001", 3001, "3 6", "2", "97 512 2500", 8, details=True),
        # Short libraries on a long series (how little data still shows the coupling).
        _plan_case("short-libraries-n10000", 10000, "1 2 3 4 5 6 7 8 9 10", "1",
                   "20 35 60 100 150 225", 30),
        # The benchmark's parameter sweep: every E and tau, libraries from 1 % to 90 %.
        _plan_case("sweep-n10000", 10000, "1 2 3 4 5 6 7 8 9 10", "1 2 3 4",
                   _log_L(100, 9000, 20), 250),
        # The long weakly coupled series.
        _plan_case("long-n100000", 100000, "3 4 5 6", "1", "1000 5000 10000 25000 50000", 250,
                   noise=0.01),
        # All ordered pairs of a 64-variable network (63 targets of every library).
        _plan_case("network-v64-n5000", 5000, "2 3 4", "1", _log_L(100, 4500, 8), 25,
                   variables=64),
        # A burst of served jobs of mixed sizes.
        {"name": "serve-burst", "kind": "serve", "jobs": 24, "min_n": 500, "max_n": 8000,
         "r": 100},
        # The convergence decisions of a network sweep's rho grid.
        {"name": "convergence-v64", "kind": "convergence", "rows": 12096, "n_L": 8, "r": 250},
    ]


def _log_int(rng, lo, hi):
    return int(math.floor(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    u = rng.random()
    if u < 0.12:
        n = _log_int(rng, 300, 20000)
        E, tau = rng.randint(1, 10), rng.randint(1, 5)
        n_m = n - (E - 1) * tau
        L = min(n_m, _log_int(rng, E + 10, min(n_m, 4000)))
        return {"kind": "cell", "n": n, "E": E, "tau": tau, "L": L, "r": _log_int(rng, 1, 60)}
    if u < 0.22:
        return {"kind": "serve", "jobs": rng.randint(3, 32), "min_n": rng.randint(400, 900),
                "max_n": _log_int(rng, 1500, 9000), "r": rng.choice([20, 100, 130])}
    if u < 0.32:
        n_L = rng.randint(2, 24)
        return {"kind": "convergence", "rows": _log_int(rng, 20, 12000), "n_L": n_L,
                "r": _log_int(rng, 5, 280)}
    n = _log_int(rng, 400, 100000)
    few = n > 20000
    Es = sorted(rng.sample(range(3 if few else 1, 7 if few else 11), rng.randint(1, 3)))
    taus = sorted(rng.sample(range(1, 6), 1 if few else rng.randint(1, 3)))
    theiler = rng.choice([0, 0, 0, rng.randint(1, 15)])
    n_m = n - (Es[-1] - 1) * taus[-1]
    lo = max(Es[-1] + 2 + 2 * theiler, _log_int(rng, 20, 400))
    if few:
        lo = max(lo, n // 100)
    hi = max(lo + 1, int(n_m * rng.uniform(0.3, 1.0)))
    L = _log_L(lo, hi, rng.randint(2, 9))
    variables = rng.choice([2, 2, 2, rng.randint(3, 24)])
    case = _plan_case("", n, " ".join(map(str, Es)), " ".join(map(str, taus)), L,
                      _log_int(rng, 20, 300), variables=variables,
                      noise=rng.choice([0.0, 0.0, 0.01]), theiler=theiler,
                      weight_floor=rng.choice([0.0, 0.0, 0.0, 0.01]),
                      host=rng.random() < 0.3, converge=rng.random() < 0.3)
    # as many realizations as stay well below the cost of the largest listed case
    most = 0.25 * max(_cost(c) for c in listed() if c["kind"] == "plan")
    while case["r"] > 4 and _cost(case) > most:
        case["r"] = max(4, case["r"] // 2)
    return case


# ------------------------------------------------------------------- sizes --
def _ints(text):
    return [int(v) for v in str(text).split()]


def _pairs(case):
    v = case.get("variables", 2)
    if v == 2:
        return [(1, 0), (0, 1)]
    return [(j, i) for j in range(v) for i in range(v) if i != j]


def _serve_jobs(case):
    """(n, E, tau) of every job of a burst: lengths log-spaced, E and tau cycling."""
    k, a, b = case["jobs"], math.log(case["min_n"]), math.log(case["max_n"])
    return [(int(math.exp(a + (b - a) * ((7 * q) % k) / max(1, k - 1))), 1 + (3 * q) % 10,
             1 + q % 5) for q in range(k)]


def _grids(case):
    """(n, variables, pairs, E list, tau list, L list, r) of every problem in the case."""
    if case["kind"] == "plan":
        return [(case["n"], case["variables"], _pairs(case), _ints(case["E"]),
                 _ints(case["tau"]), _ints(case["L"]), case["r"])]
    if case["kind"] == "cell":
        return [(case["n"], 2, [(1, 0)], [case["E"]], [case["tau"]], [case["L"]], case["r"])]
    return [(n, 2, [(1, 0), (0, 1)], [E], [tau],
             [int(v) for v in I.job_L_grid(n - (E - 1) * tau, E)], case["r"])
            for n, E, tau in _serve_jobs(case)]


def _cost(case):
    """A rough cost for bounding drawn cases: search and epilogue per query, tables per series."""
    n, v, pairs, Es, taus, Ls, r = _grids(case)[0]
    libs = len({j for j, _ in pairs})
    t = len(pairs) / libs
    total = 0.0
    for E in Es:
        for tau in taus:
            n_m = n - (E - 1) * tau
            total += libs * 0.3 * n_m * n_m * E
            for L in Ls:
                total += libs * r * n_m * (min(2.0 * L, 40 + 3.0 * (E + 2) * n_m / L) + 20 * t)
    return total


def work(case):
    """Series (or rho) read once and results written once; the arithmetic the method cannot do
    without: every (query, library point) squared distance once per (variable, E, tau) however
    many realizations share it (3E flops), and per query and realization the E+1 weights (4
    flops each), per target the prediction (2(E+1)) and its share of the skill (6)."""
    if case["kind"] == "convergence":
        v = case["rows"] * case["n_L"] * case["r"]
        return {"bytes": 8 * v + 40 * case["rows"],
                "flops": v * (math.log2(max(2, case["r"])) + case["n_L"] / 2)}
    moved, flops = 0.0, 0.0
    for n, v, pairs, Es, taus, Ls, r in _grids(case):
        libs = len({j for j, _ in pairs})
        moved += 4 * v * n + 8 * len(pairs) * len(Es) * len(taus) * len(Ls) * r
        for E in Es:
            for tau in taus:
                n_m = n - (E - 1) * tau
                flops += libs * 3.0 * E * n_m * min(n_m, sum(Ls) * r)
                flops += len(Ls) * r * n_m * (libs * 4.0 * (E + 1) + len(pairs) * (2.0 * E + 8))
                if case.get("details"):
                    moved += len(pairs) * r * (len(Ls) * 4 * n_m * (E + 2) + 4 * sum(Ls))
    return {"bytes": moved, "flops": flops}


# ------------------------------------------------------------------ inputs --
def _series(n, variables, noise, seed):
    """float32 [variables][n], from the seed alone."""
    rng = np.random.Generator(np.random.Philox(seed))
    if variables == 2:
        bxy, byx = rng.uniform(0.0, 0.1, size=2)
        x0, y0 = rng.uniform(0.2, 0.6, size=2)
        s = I.logistic_pair(n, bxy=float(bxy), byx=float(byx), x0=float(x0), y0=float(y0))
    else:
        s, _ = I.logistic_network(variables, n, 0.05, 1000 * seed)
    return I.add_noise(s, noise, seed + 1) if noise else s


def _rho_grid(case, seed):
    """A rho grid [rows][n_L][r] as sweeps leave it: skill that rises with L in some rows, flat in
    others, its spread shrinking with L, and a few realizations without a value."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rows, n_L, r = case["rows"], case["n_L"], case["r"]
    t = torch.linspace(0.0, 1.0, n_L, dtype=torch.float64, device="cuda")
    top = torch.rand(rows, 1, 1, generator=g, dtype=torch.float64, device="cuda") * 0.9
    slope = torch.rand(rows, 1, 1, generator=g, dtype=torch.float64, device="cuda").round()
    z = torch.randn(rows, n_L, r, generator=g, dtype=torch.float64, device="cuda")
    rho = top * (1.0 - 0.5 * slope * (1.0 - t)[None, :, None])
    rho = (rho + z * (0.08 * (1.2 - t))[None, :, None]).clamp(-1.0, 1.0)
    lost = torch.rand(rows, n_L, r, generator=g, device="cuda") < 1e-4
    return rho.masked_fill(lost, math.nan).contiguous()


class _State:
    """What a program keeps between passes; a plan is given back with its state."""

    plan = None

    def __del__(self):
        if self.plan is not None:
            C.ccm_plan_destroy(self.plan)


def prepare(case, seed):
    ctx, stream = _context()
    st = _State()
    st.case, st.ctx, st.stream, st.seed = case, ctx, stream, seed
    if case["kind"] == "convergence":
        st.rho = _rho_grid(case, seed)
        st.L = 100 * np.arange(1, case["n_L"] + 1, dtype=np.int64)
        st.out = torch.zeros(case["rows"], 40, dtype=torch.uint8, device="cuda")
        return st
    if case["kind"] == "serve":
        st.jobs = []
        for q, (n, v, pairs, E, tau, L, r) in enumerate(_grids(case)):
            rho = np.zeros((len(pairs), 1, 1, len(L), r))
            st.jobs.append((_series(n, v, 0.0, 100 * seed + q), pairs, E, tau, L, r,
                            100 * seed + q, rho))
        return st
    n, v, pairs, E, tau, L, r = _grids(case)[0]
    series = torch.from_numpy(_series(n, v, case.get("noise", 0.0), seed))
    if case["kind"] == "cell":
        st.series = series.cuda()
        st.rho = torch.zeros(r, dtype=torch.float64, device="cuda")
        return st
    shape = (len(pairs), len(E), len(tau), len(L), r)
    # the kernels' own defaults: the choice does not depend on what ran before
    flags = C.CCM_NO_AUTOTUNE
    if case["host"]:
        st.series, st.rho = series.pin_memory(), torch.zeros(shape, dtype=torch.float64).pin_memory()
    else:
        flags |= C.CCM_INPUT_ON_DEVICE | C.CCM_OUTPUT_ON_DEVICE
        st.series, st.rho = series.cuda(), torch.zeros(shape, dtype=torch.float64, device="cuda")
    st.L = np.array(L, np.int64)
    st.plan = C.ccm_plan(ctx, (v, n), pairs, E, tau, L, r, seed, flags,
                         theiler=case["theiler"], weight_floor=case["weight_floor"])
    if case["details"]:
        info = C.ccm_plan_get_info(st.plan)
        st.libraries = torch.zeros(info["library_entries"], dtype=torch.int32, device="cuda")
        st.neighbours = torch.zeros(info["neighbour_entries"], dtype=torch.int32, device="cuda")
        st.predictions = torch.zeros(info["n_queries"], dtype=torch.float32, device="cuda")
    if case["converge"] and not case["host"]:
        rows = len(pairs) * len(E) * len(tau)
        st.out = torch.zeros(rows, 40, dtype=torch.uint8, device="cuda")
    return st


# -------------------------------------------------------------------- pass --
def _decisions(out):
    """The decisions' fields from their 40-byte rows (ccm_convergence_t)."""
    if isinstance(out, np.ndarray):
        out = out.reshape(-1)
        return {"means_jt_z": np.stack([out[f] for f in C.CONVERGENCE_FIELDS[:4]], 1),
                "n_valid": out["n_valid"], "converged": out["converged"]}
    whole = out.view(torch.int32)
    return {"means_jt_z": out.view(torch.float64)[:, :4], "n_valid": whole[:, 8],
            "converged": whole[:, 9]}


def run(st):
    case = st.case
    if case["kind"] == "convergence":
        C.ccm_convergence(st.ctx, st.rho, st.L, out=st.out, stream=st.stream)
        return _decisions(st.out)
    if case["kind"] == "cell":
        C.ccm_run_noalloc(st.series, 1, 0, case["E"], case["tau"], case["L"], case["r"], st.seed,
                          st.rho, st.stream)
        return st.rho
    if case["kind"] == "serve":
        tickets = [C.ccm_submit(st.ctx, *job[:7]) for job in st.jobs]
        for ticket, job in zip(tickets, st.jobs):
            while C.ccm_poll(st.ctx, ticket, job[7], 1000) == C.CCM_PENDING:
                pass
        return [job[7] for job in st.jobs]
    if case["details"]:
        C.ccm_run_ex(st.plan, st.series, st.rho, st.libraries, st.neighbours, st.predictions,
                     st.stream)
        return {"rho": st.rho, "libraries": st.libraries, "neighbours": st.neighbours,
                "predictions": st.predictions}
    if case["host"]:
        C.ccm_run(st.plan, st.series, st.rho)
        if not case["converge"]:
            return st.rho
        return {"rho": st.rho, **_decisions(C.ccm_convergence(st.ctx, st.rho.numpy(), st.L))}
    C.ccm_run(st.plan, st.series, st.rho, st.stream)
    if not case["converge"]:
        return st.rho
    C.ccm_convergence(st.ctx, st.rho, st.L, out=st.out, stream=st.stream)
    return {"rho": st.rho, **_decisions(st.out)}


# ------------------------------------------------------- the same in 64 bits --
def _library(seed, j, E, tau, L, k, n_m):
    """The library of one realization, ascending: the L points with the smallest keys."""
    blocks = (n_m + 7) // 8
    c3 = (j << 16) | (E << 8) | tau
    counter = ((k << 64) | (L << 128) | (c3 << 192)) - 1  # numpy steps the counter first
    w = np.random.Philox(counter=counter % (1 << 256), key=seed).random_raw(4 * blocks)
    v = np.stack([w >> np.uint64(32), w & np.uint64(0xffffffff)], 1).reshape(-1)[:n_m]
    key = (v << np.uint64(32)) | np.arange(n_m, dtype=np.uint64)
    return np.sort(np.argpartition(key, L - 1)[:L]) if L < n_m else np.arange(n_m)


def _pearson(x, y):
    """Pearson of x [n] with every row of y [..., n]; NaN without variance."""
    a, b = x - x.mean(), y - y.mean(-1, keepdim=True)
    return (b @ a) / ((a @ a) * (b * b).sum(-1)).sqrt()


def _exact_grid(series, pairs, Es, taus, Ls, r, seed, theiler, floor, details):
    """rho [pairs][E][tau][L][r] and, when asked, every prediction, in 64 bits."""
    s = torch.from_numpy(series).cuda().double()
    n = s.shape[1]
    rho = torch.zeros(len(pairs), len(Es), len(taus), len(Ls), r, dtype=torch.float64,
                      device="cuda")
    xhat = {}
    for e, E in enumerate(Es):
        for t, tau in enumerate(taus):
            off = (E - 1) * tau
            n_m = n - off
            for j in sorted({p[0] for p in pairs}):
                M = torch.stack([s[j, off - q * tau:off - q * tau + n_m] for q in range(E)])
                d2 = torch.zeros(n_m, n_m, dtype=torch.float64, device="cuda")
                for q in range(E):
                    d2 += (M[q][:, None] - M[q][None, :]) ** 2
                at = torch.arange(n_m, device="cuda")
                near = (at[:, None] - at[None, :]).abs() <= theiler
                d2[near] = math.inf  # the query and its window are no neighbours
                ranked = None
                targets = [p for p, (pj, _) in enumerate(pairs) if pj == j]
                for l, L in enumerate(Ls):
                    ranks = min(n_m, int(math.ceil((E + 1 + 8 * math.sqrt(E + 1) + 12) * n_m / L))
                                + 2 * theiler)
                    by_rank = 2 * ranks < L  # read off every query's whole ranking
                    if by_rank and (ranked is None or ranked.shape[1] < ranks):
                        ranked = d2.sort(dim=1, stable=True).indices[:, :ranks].contiguous()
                    step = max(1, 40_000_000 // (n_m * ranks)) if by_rank else 1
                    for k0 in range(0, r, step):
                        ks = range(k0, min(r, k0 + step))
                        libs = [torch.from_numpy(_library(seed, j, E, tau, L, k, n_m)) for k in ks]
                        libs = torch.stack(libs).cuda()
                        nb = None
                        if by_rank:
                            member = torch.zeros(len(ks), n_m, dtype=torch.bool, device="cuda")
                            member.scatter_(1, libs, True)
                            hit = member[:, ranked[:, :ranks]]
                            place = hit.cumsum(2, dtype=torch.int32)
                            if bool((place[:, :, -1] > E).all()):
                                first = hit & (place <= E + 1)
                                nb = ranked[:, :ranks].expand_as(first)[first]
                                nb = nb.reshape(len(ks), n_m, E + 1)
                        if nb is None:
                            nb = torch.stack([lib[d2[:, lib].sort(dim=1, stable=True)
                                                  .indices[:, :E + 1]] for lib in libs])
                        d = d2[at[None, :, None], nb].sqrt()
                        d1 = d[:, :, :1]
                        u = torch.where(d1 > 0, torch.exp(-d / d1), (d == 0).double())
                        u = u.clamp_min(floor)
                        w = u / u.sum(2, keepdim=True)
                        for p in targets:
                            si = s[pairs[p][1], off:]
                            pred = (w * si[nb]).sum(2)
                            rho[p, e, t, l, k0:k0 + len(ks)] = _pearson(si, pred)
                            if details:
                                for q, k in enumerate(ks):
                                    xhat[p, e, t, l, k] = pred[q]
    flat = torch.cat([xhat[key] for key in sorted(xhat)]) if details else None
    return rho, flat


def _exact_decisions(rho, z_crit=1.6448536269514722):
    """The trend test of every row of rho [rows][n_L][r], L ascending."""
    rows, n_L, r = rho.shape
    fine = torch.isfinite(rho)
    cnt = fine.sum(2)
    zero = torch.where(fine, rho, torch.zeros_like(rho))
    mean = zero.sum(2) / cnt
    J = torch.zeros(rows, dtype=torch.float64, device=rho.device)
    for g in range(n_L):
        for h in range(g):
            step = max(1, (1 << 27) // (r * r))
            for a in range(0, rows, step):
                y, x = rho[a:a + step, g, :, None], rho[a:a + step, h, None, :]
                J[a:a + step] += (y > x).sum((1, 2)) + 0.5 * (y == x).sum((1, 2))
    m = cnt.double()
    N = m.sum(1)
    var = (N * N * (2 * N + 3) - (m * m * (2 * m + 3)).sum(1)) / 72
    z = (J - (N * N - (m * m).sum(1)) / 4) / var.sqrt()
    first, last = mean[:, 0], mean[:, -1]
    return {"means_jt_z": torch.stack([first, last, J, z], 1), "n_valid": N.int(),
            "converged": ((z > z_crit) & (last > first) & (last > 0)).int()}


def exact(case, seed):
    if case["kind"] == "convergence":
        if case["rows"] * (case["n_L"] * case["r"]) ** 2 > 6e10:
            return None
        return _exact_decisions(_rho_grid(case, seed))
    grids = _grids(case)
    # (realization, query) pairs and libraries: more takes over 20 seconds
    units = sum(len(p) * len(E) * len(t) * len(L) * r for _, _, p, E, t, L, r in grids)
    pairs = sum(len({j for j, _ in p}) * len(E) * len(t) * n * sum(L) * r
                for n, _, p, E, t, L, r in grids)
    if units > 60000 or pairs > 3e11 or max(g[0] for g in grids) > 12000:
        return None
    if case["kind"] == "serve":
        return [_exact_grid(_series(n, v, 0.0, 100 * seed + q), p, E, t, L, r, 100 * seed + q, 0,
                            0.0, False)[0] for q, (n, v, p, E, t, L, r) in enumerate(grids)]
    n, v, p, E, t, L, r = grids[0]
    rho, xhat = _exact_grid(_series(n, v, case.get("noise", 0.0), seed), p, E, t, L, r, seed,
                            case.get("theiler", 0), case.get("weight_floor", 0.0),
                            case.get("details", False))
    if case["kind"] == "cell":
        return rho.reshape(-1)
    if case["details"]:
        return {"rho": rho, "libraries": None, "neighbours": None, "predictions": xhat}
    if not case["converge"]:
        return rho
    rows = rho.reshape(-1, len(L), r)
    return {"rho": rho, **(_exact_decisions(rows) if len(L) * r <= 3000 else
                           {"means_jt_z": None, "n_valid": None, "converged": None})}
