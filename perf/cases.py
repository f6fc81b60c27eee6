"""What users of the library have it do, as timed cases.

Each case goes through a public entry point: the persistent engine (submit, wait, read the
result, release), the allocation-free run, the one-trajectory-per-thread kernels in both
precisions with their reduction, and the reduction alone.  Parameter sets are those of the
library's workloads (overdamped sweep, ramp sweep, constant tilt, uneven batch, serving stream);
sizes run from one small request to the largest that finishes in about a second.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1802_05065_gb300 as fpt
from paper_1802_05065_gb300 import api

NAN = float("nan")
# floating-point operations of one step: half a Box-Muller pair (log, sqrt, sin or cos, 4
# multiplies / additions) and the drift update (sin, bias, noise); Heun evaluates the drift twice
FLOPS_EM, FLOPS_HEUN = 12, 20


# ---------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------

def listed() -> list:
    return [
        # the smallest request a user submits: one point of the overdamped sweep, a thousand
        # realisations, for a first look at the distribution (latency of a serial chain of steps)
        dict(name="request_small", path="engine", problem="over", gamma0=0.9, D=0.2, dt=1e-3,
             integrator="em", n=1024, keep=True, bins=100, chunk=16384, service=0, young=0),
        # the headline workload: points of the overdamped sweep together in one engine
        dict(name="sweep", path="sweep", n=2**19, bins=100, chunk=65536, service=0, young=0),
        # coarse steps, ~950 steps per trajectory, millions of realisations: results and refills
        # as frequent as they get
        dict(name="short_many", path="engine", problem="over", gamma0=0.9, D=0.2, dt=0.02,
             integrator="em", n=2**22, keep=False, bins=100, chunk=4096, service=0, young=0),
        # the underdamped junction with Heun at the step it converges at, an odd count
        dict(name="heun_underdamped", path="engine", problem="under", alpha=0.1, gamma0=0.8, D=0.05,
             dt=0.05, integrator="heun", n=250007, keep=False, bins=100, chunk=16384, service=0,
             young=0),
        # switching-current distribution: underdamped, ramped bias, every switching bias kept,
        # fewer realisations than the GPU has lanes (the published histograms have 10^4 .. 10^5)
        dict(name="ramp_switching", path="engine", problem="ramp", alpha=0.05, D=0.01, nu=1e-4,
             dt=0.01, integrator="em", n=30000, keep=True, bins=1000, chunk=16384, service=0,
             young=0),
        # a parameter scan submitted at once: constant and ramped sets of very different lengths
        dict(name="uneven_batch", path="mix", mix_seed=0, sets=24, log2_lo=12, log2_hi=16,
             stop_rse=0.0, bins=200, chunk=16384, service=0, young=0),
        # a server: the engine's own thread, requests with a 1 % standard-error stop rule
        dict(name="serving", path="mix", mix_seed=7, sets=12, log2_lo=12, log2_hi=18,
             stop_rse=0.01, bins=100, chunk=4096, service=1, young=1024),
        # one request inside a program that may not allocate
        dict(name="noalloc", path="noalloc", problem="over", gamma0=0.9, D=0.2, dt=1e-3,
             integrator="em", n=200003, bins=100),
        # the plain single-precision kernel with its reduction
        dict(name="plain_fp32", path="plain", precision="fp32", problem="over", gamma0=0.7, D=0.2,
             dt=1e-3, integrator="em", n=2**18, max_steps=2**40, bins=100),
        # the reference run of the constant tilt in double precision, a bounded step budget
        dict(name="plain_fp64", path="plain", precision="fp64", problem="under", alpha=0.1,
             gamma0=0.8, D=0.05, dt=0.005, integrator="em", n=4096, max_steps=20000, bins=100),
        # double precision to a useful standard error: more trajectories than threads
        dict(name="plain_fp64_large", path="plain", precision="fp64", problem="over", gamma0=0.9,
             D=0.2, dt=1e-3, integrator="em", n=2**16, max_steps=2**40, bins=100),
        # moments and histogram of escape steps a program already has
        dict(name="reduce", path="reduce", mean_steps=19000.0, n=2**24, bins=100, output="time"),
    ]


def _log(rng, lo, hi) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _count(rng, lo, hi) -> int:
    """A trajectory count, log-uniform; ragged in most draws."""
    n = int(_log(rng, lo, hi + 1))
    return n if rng.random() < 0.8 else 1 << (n.bit_length() - 1)


def _problem(rng) -> dict:
    kind = rng.choice(("over", "over", "over", "under", "ramp"))
    integ = rng.choice(("em", "em", "heun"))
    if kind == "over":
        g, D = rng.choice(((0.7, 0.2), (0.9, 0.05), (0.9, 0.1), (0.9, 0.2)))
        return dict(problem="over", gamma0=g, D=D, dt=round(_log(rng, 1e-3, 0.02), 6), integrator=integ)
    if kind == "under":
        return dict(problem="under", alpha=round(_log(rng, 0.05, 0.5), 4), gamma0=0.8, D=0.05,
                    dt=round(_log(rng, 0.02, 0.1) if integ == "heun" else _log(rng, 0.005, 0.02), 6),
                    integrator=integ)
    return dict(problem="ramp", alpha=0.05, D=0.01, nu=round(_log(rng, 1e-4, 1e-3), 7), dt=0.01,
                integrator=integ)


# most trajectory steps of a drawn case, below the sweep's; FP64 runs below the large FP64 case's
MOST_STEPS, MOST_STEPS_64 = 3e10, 1.2e9


def draw(rng) -> dict:
    path = rng.choice(("engine", "engine", "engine", "engine", "mix", "noalloc", "noalloc", "plain32",
                       "plain64", "reduce"))
    bins = rng.choice((50, 64, 100, 200, 333, 1000))
    if path == "reduce":
        return dict(path="reduce", mean_steps=round(_log(rng, 1e3, 1e6), 1), n=_count(rng, 1000, 2**24),
                    bins=bins, output=rng.choice(("time", "bias")))
    if path == "mix":
        stop = rng.choice((0.0, 0.01, 0.02))
        service = rng.choice((0, 1))
        lo = rng.choice((10, 11, 12))
        return dict(path="mix", mix_seed=rng.randrange(1, 1000), sets=rng.randrange(3, 17), log2_lo=lo,
                    log2_hi=rng.randrange(lo + 1, 16), stop_rse=stop, bins=bins,
                    chunk=rng.choice((4096, 16384)), service=service, young=rng.choice((0, 1024)))
    c = _problem(rng)
    mean = _mean_steps(c)
    if path == "engine":
        c.update(path="engine", keep=rng.random() < 0.5, bins=bins, chunk=rng.choice((4096, 16384, 65536)),
                 service=rng.choice((0, 1)), young=0)
        c["n"] = _count(rng, 1000, max(2000, min(2**22, MOST_STEPS / mean)))
    elif path == "noalloc":
        c.update(path="noalloc", bins=bins, n=_count(rng, 1000, max(2000, min(2**19, MOST_STEPS / 3 / mean))))
    elif path == "plain32":
        c.update(path="plain", precision="fp32", max_steps=2**40, bins=bins,
                 n=_count(rng, 1000, max(2000, min(2**18, MOST_STEPS / 5 / mean))))
    else:
        cap = int(_log(rng, 2000, 60000))
        c.update(path="plain", precision="fp64", max_steps=cap, bins=bins,
                 n=_count(rng, 256, min(2**16, MOST_STEPS_64 / min(mean, cap))))
    return c


# ---------------------------------------------------------------------------------------------
# parameter sets
# ---------------------------------------------------------------------------------------------

def _params(c: dict) -> dict:
    """The library's parameter dict of a single-problem case."""
    d = dict(alpha=c.get("alpha", 0.0), D=c["D"], gamma0=c.get("gamma0", 0.0), nu=c.get("nu", 0.0),
             dt=c["dt"], phi0=NAN, v0=0.0, sin_amp=1.0, integrator=c["integrator"], stop_rse=0.0,
             stop_block=4096, precision=c.get("precision", "fp32"), hist_bins=c["bins"],
             max_steps=c.get("max_steps", 2**40), keep_per_traj=int(c.get("keep", False)))
    if c["problem"] == "over":
        d.update(model="overdamped", threshold=2 * math.pi, threshold_mode="from_start",
                 output="time", hist_lo=0.0, hist_hi=round(8 * _mean_steps(c) * c["dt"], 3))
    elif c["problem"] == "under":
        d.update(model="underdamped", threshold=math.pi, threshold_mode="absolute",
                 output="time", hist_lo=0.0, hist_hi=2000.0)
    else:
        steps = math.ceil(1.1 / (c["nu"] * c["dt"]))
        d.update(model="underdamped", threshold=2 * math.pi, threshold_mode="absolute",
                 output="bias", hist_lo=0.5, hist_hi=1.0, max_steps=min(steps, d["max_steps"]))
    return d


SWEEP_POINTS = ((0.7, 0.2), (0.9, 0.05), (0.9, 0.1), (0.9, 0.2))


def _requests(c: dict) -> list:
    """(parameter dict, trajectories) of every request of an engine case."""
    if c["path"] == "sweep":
        return [(_params(dict(c, problem="over", gamma0=g, D=D, dt=1e-3, integrator="em")), c["n"])
                for g, D in SWEEP_POINTS]
    if c["path"] == "mix":
        return _mix(c)
    return [(_params(c), c["n"])]


def _mix(c: dict) -> list:
    """Sets of the uneven batch: alpha, D log-uniform, gamma uniform, half constant, half ramped;
    mean lengths of about 10^3 .. 10^5 steps."""
    r = np.random.Generator(np.random.PCG64(c["mix_seed"]))
    out = []
    while len(out) < c["sets"]:
        alpha, D = float(10 ** r.uniform(-1.3, 0)), float(10 ** r.uniform(-2, -1))
        g, nu = float(r.uniform(0.6, 0.95)), float(10 ** r.uniform(-6, -4))
        n = 2 ** int(r.integers(c["log2_lo"], c["log2_hi"] + 1))
        ramped = len(out) % 2 == 1
        p = dict(alpha=alpha, D=D, gamma0=g, nu=nu if ramped else 0.0, dt=0.01)
        L = _kramers_steps(p)
        if not 1e3 <= L <= 1e5:
            continue
        d = dict(p, model="underdamped", phi0=NAN, v0=0.0, sin_amp=1.0, integrator="em",
                 stop_rse=c["stop_rse"], stop_block=4096, precision="fp32", hist_bins=c["bins"],
                 threshold_mode="absolute", keep_per_traj=0)
        if ramped:
            d.update(threshold=2 * math.pi, output="bias", hist_lo=0.5, hist_hi=1.0,
                     max_steps=int(math.ceil((1.1 - g) / (nu * 0.01))))
        else:
            d.update(threshold=math.pi, output="time", hist_lo=0.0, hist_hi=10 * L * 0.01,
                     max_steps=int(20 * L))
        out.append((d, n))
    return out


# Rough mean lengths, for the work of a case and to bound a drawn one.

def _kramers_steps(p: dict) -> float:
    g, D = p["gamma0"], p["D"]
    w0 = (1.0 - g * g) ** 0.25
    dU = 2.0 * (math.sqrt(1.0 - g * g) - g * math.acos(g))
    t = 2.0 * math.pi / w0 * math.exp(min(dU / D, 700.0))
    t *= max(1.0, D / (p["alpha"] * dU)) if p.get("alpha") else 1.0   # weak damping
    if p.get("nu", 0.0) > 0:
        t = min(t, (1.0 - g) / p["nu"])
    return t / p["dt"]


def _overdamped_mean(g: float, D: float) -> float:
    """Mean first passage over one period of the overdamped tilted washboard."""
    n = 1500
    z = np.linspace(-2 * math.pi, 0.0, n)
    y = math.asin(g) + np.linspace(0.0, 2 * math.pi, n)
    U = lambda x: -np.cos(x) - g * x   # noqa: E731
    f = np.exp((U(y)[:, None] - U(y[:, None] + z[None, :])) / D)
    inner = np.sum((f[:, 1:] + f[:, :-1]) * 0.5, axis=1) * (z[1] - z[0]) / (1 - math.exp(-2 * math.pi * g / D))
    return float(np.sum((inner[1:] + inner[:-1]) * 0.5) * (y[1] - y[0]) / D)


_OVER = {}


def _mean_steps(c: dict) -> float:
    if c["problem"] == "over":
        key = (c["gamma0"], c["D"])
        if key not in _OVER:
            _OVER[key] = _overdamped_mean(*key)
        return _OVER[key] / c["dt"]
    if c["problem"] == "under":
        return _kramers_steps(c)
    return 0.75 / (c["nu"] * c["dt"])


def work(case: dict) -> dict:
    c = case
    if c["path"] == "reduce":
        return {"bytes": 8 * c["n"] + 8 * c["bins"] + 64, "flops": 6 * c["n"]}
    steps, out = 0.0, 0
    if c["path"] in ("engine", "sweep", "mix"):
        for d, n in _requests(c):
            if c["path"] == "mix":
                steps += min(n, 12288 if c["stop_rse"] else n) * min(_kramers_steps(d), d["max_steps"])
            elif c["path"] == "sweep":
                steps += n * _mean_steps(dict(problem="over", gamma0=d["gamma0"], D=d["D"], dt=d["dt"]))
            else:
                steps += n * min(_mean_steps(c), d["max_steps"])
            out += 8 * d["hist_bins"] + 64 + (8 * n if d["keep_per_traj"] else 0)
    else:
        steps = c["n"] * min(_mean_steps(c), c.get("max_steps", 2**48))
        out = 8 * c["n"] + 8 * c["bins"] + 64
    per = FLOPS_HEUN if c.get("integrator") == "heun" else FLOPS_EM
    return {"bytes": out, "flops": per * steps}


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------

def prepare(case: dict, seed: int) -> dict:
    c = dict(case)
    st = {"case": c, "seed": 1000003 * int(seed) + 17}
    if c["path"] in ("engine", "sweep", "mix"):
        st["engine"] = fpt.Engine(0, chunk_steps=c["chunk"], service_thread=c["service"],
                                  young_chunk_steps=c["young"])
        st["requests"] = [(fpt.params_from(d), n, st["seed"] + i, bool(d["keep_per_traj"]))
                          for i, (d, n) in enumerate(_requests(c))]
    elif c["path"] == "noalloc":
        st["params"] = fpt.params_from(_params(c))
        st["steps"] = torch.empty(c["n"], dtype=torch.int64, device="cuda")
        st["sums"] = torch.zeros(8, dtype=torch.int64, device="cuda")
        st["hist"] = torch.zeros(c["bins"], dtype=torch.int64, device="cuda")
    elif c["path"] == "plain":
        st["d"] = _params(c)
    else:
        st["d"], st["steps"] = _reduce_inputs(c, st["seed"])
    return st


def _reduce_inputs(c: dict, seed: int):
    """Escape steps as a run leaves them: exponential above a shortest time, a few per thousand
    censored."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand(c["n"], generator=gen, device="cuda", dtype=torch.float64)
    k = (c["mean_steps"] * (0.05 - 0.95 * torch.log1p(-u))).to(torch.int64) + 1
    cut = int(c["mean_steps"] * 6)
    k = torch.where(k > cut, torch.full_like(k, -1), k)
    d = dict(model="overdamped", alpha=0.0, D=0.2, gamma0=0.1, nu=0.0, dt=1e-3, phi0=NAN, threshold=2 * math.pi,
             threshold_mode="from_start", max_steps=cut, hist_bins=c["bins"], output=c["output"],
             precision="fp64", hist_lo=0.0, hist_hi=5.0 * c["mean_steps"] * 1e-3)
    if c["output"] == "bias":
        d.update(nu=0.8 / (cut * 1e-3), hist_lo=0.1, hist_hi=0.9)
    return d, k


def _reduced(res, hist, sums) -> dict:
    s = np.array([sums.n_done, sums.n_escaped, sums.s1_lo, sums.s1_hi, sums.s2_lo, sums.s2_hi,
                  sums.under, sums.over], dtype=np.uint64).view(np.int64)
    return {"moments": np.array([res.mean, res.var, res.sem]), "sums": s, "hist": hist}


def run(state: dict):
    c = state["case"]
    if "engine" in state:
        eng = state["engine"]
        ids = [eng.submit(p, n, s) for p, n, s, _ in state["requests"]]
        counts, moments, hists, kept = [], [], [], []
        for rid, (p, n, _, keep) in zip(ids, state["requests"]):
            r = eng.wait(rid)
            h, under, over = eng.histogram(rid, p.hist_bins)
            if keep:
                kept.append(eng.per_traj_steps(rid, n))
            eng.release(rid)
            counts.append((r.n_used, r.n_escaped, r.n_censored, r.steps_total, under, over))
            moments.append((r.mean, r.var, r.sem))
            hists.append(h)
        out = {"counts": np.array(counts, dtype=np.int64), "moments": np.array(moments),
               "hist": np.array(hists, dtype=np.int64)}
        if kept:
            out["per_traj"] = kept[0]
        return out
    if c["path"] == "noalloc":
        state["sums"].zero_()
        state["hist"].zero_()
        fpt.run_noalloc(state["params"], c["n"], state["seed"], state["steps"].data_ptr(),
                        state["sums"].data_ptr(), state["hist"].data_ptr(), api.current_stream())
        return {"steps": state["steps"], "sums": state["sums"], "hist": state["hist"]}
    if c["path"] == "plain":
        steps = api.run_plain(state["d"], c["n"], state["seed"])
        return {"steps": steps, "reduced": _reduced(*api.reduce(state["d"], steps))}
    return _reduced(*api.reduce(state["d"], state["steps"]))


# ---------------------------------------------------------------------------------------------
# the same in 64 bits with plain numpy
# ---------------------------------------------------------------------------------------------

def _philox(block, traj, seed: int):
    """Philox4x32-10 words of (block, trajectory) pairs, four uint32 arrays."""
    u64, m32 = np.uint64, np.uint64(0xFFFFFFFF)
    c = [block & m32, block >> u64(32), traj & m32, traj >> u64(32)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = u64(0xD2511F53) * c[0], u64(0xCD9E8D57) * c[2]
        c = [(p1 >> u64(32)) ^ c[1] ^ u64(k0), p1 & m32, (p0 >> u64(32)) ^ c[3] ^ u64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _normals(block0: int, nblocks: int, traj, seed: int):
    """Normals of steps 4 block0 + 1 .. 4 (block0 + nblocks): (steps, trajectories)."""
    b = np.arange(block0, block0 + nblocks, dtype=np.uint64)[:, None]
    x = [w.astype(np.float64) for w in _philox(*np.broadcast_arrays(b, traj[None, :]), seed)]
    u = [(w + 0.5) * 2.0**-32 for w in x]
    ra, rb = np.sqrt(-2 * np.log(u[0])), np.sqrt(-2 * np.log(u[2]))
    ta, tb = 2 * math.pi * u[1], 2 * math.pi * u[3]
    z = np.stack([ra * np.cos(ta), ra * np.sin(ta), rb * np.cos(tb), rb * np.sin(tb)], axis=1)
    return z.reshape(4 * nblocks, traj.size)


def _escape_steps(d: dict, n: int, seed: int):
    """Escape step of trajectories 0 .. n-1 (-1: censored), Euler-Maruyama or Heun in 64 bits."""
    under, heun = d["model"] == "underdamped", d["integrator"] == "heun"
    dt, g0, nudt, a = d["dt"], d["gamma0"], d["nu"] * d["dt"], d["alpha"]
    sigma = math.sqrt(2 * a * d["D"] * dt) if under else math.sqrt(2 * d["D"] * dt)
    phi0 = math.asin(g0)
    th = phi0 + d["threshold"] if d["threshold_mode"] == "from_start" else d["threshold"]
    out = np.full(n, -1, dtype=np.int64)
    ids, phi, v, k = np.arange(n), np.full(n, phi0), np.zeros(n), 0
    while ids.size and k < d["max_steps"]:
        nb = max(4, min(64, 200000 // ids.size))
        z = sigma * _normals(k // 4, nb, ids.astype(np.uint64), seed)
        live = np.ones(ids.size, dtype=bool)
        for row in z:
            if k >= d["max_steps"]:
                break
            k += 1
            g, gp = g0 + nudt * k, g0 + nudt * (k - 1)
            if under and heun:
                a0 = -a * v - np.sin(phi) + gp
                p, q = phi + v * dt, v + a0 * dt + row
                a1 = -a * q - np.sin(p) + g
                phi, v = phi + 0.5 * (v + q) * dt, v + 0.5 * (a0 + a1) * dt + row
            elif under:
                phi, v = phi + v * dt, v + (-a * v - np.sin(phi) + g) * dt + row
            elif heun:
                f0 = gp - np.sin(phi)
                f1 = g - np.sin(phi + f0 * dt + row)
                phi = phi + 0.5 * (f0 + f1) * dt + row
            else:
                phi = phi + (g - np.sin(phi)) * dt + row
            hit = (phi >= th) & live
            if hit.any():
                out[ids[hit]] = k
                live &= ~hit
        if not live.all():
            ids, phi, v = ids[live], phi[live], v[live]
    return out


def _moments(k, d: dict):
    """Mean, unbiased variance and standard error of x over the escaped, from exact integer sums."""
    k = [int(x) for x in k if x >= 0] if len(k) < 2**17 else k[k >= 0]
    n = len(k)
    if n < 2:
        return np.full(3, NAN)
    if isinstance(k, list):
        s1, s2 = sum(k), sum(x * x for x in k)
    else:
        s1 = int(k.sum())
        s2 = int(np.square(k >> 16).sum()) * 2**32 + 2 * int(((k >> 16) * (k & 0xFFFF)).sum()) * 2**16 \
            + int(np.square(k & 0xFFFF).sum())
    a, b = (0.0, d["dt"]) if d["output"] == "time" else (d["gamma0"], d["nu"] * d["dt"])
    var = b * b * ((n * s2 - s1 * s1) / (n * (n - 1)))
    return np.array([a + b * (s1 / n), var, math.sqrt(var / n)])


def exact(case: dict, seed: int):
    c = dict(case)
    s = 1000003 * int(seed) + 17
    if c["path"] == "reduce":
        d, k = _reduce_inputs(c, s)
        return {"moments": _moments(k.cpu().numpy(), d), "sums": None, "hist": None}
    if c["path"] not in ("engine", "plain"):   # no floating outputs, or too many steps
        return None
    d = _params(c)
    mean = min(_mean_steps(c), d["max_steps"])
    if c["n"] * mean > 1e8 or mean * (math.log(c["n"]) + 2) > 4e5 and mean < d["max_steps"]:
        return None
    m = _moments(_escape_steps(d, c["n"], s), d)
    if c["path"] == "plain":
        return {"steps": None, "reduced": {"moments": m, "sums": None, "hist": None}}
    out = {"counts": None, "moments": m[None, :], "hist": None}
    if c["keep"]:
        out["per_traj"] = None
    return out
