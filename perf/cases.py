"""The workloads this engine is timed on: relaxations of every disorder kind in both precisions, from
a single 1024-site chain to 4 chains of 2^25 sites, the trials of the two threshold searches, and the
structure factor.  Sizes, drives and launch shapes are those of the workload presets, of the L = 4096
threshold fixtures and of the threshold searches' defaults.

A case is one of five families:
  relax     a kept handle relaxes its chains from the flat start and records v, ubar and w2 at
            log-spaced steps (reset + observe), reading the line back where it is small
  uneven    the same for a batch of chains of uneven lengths, random field and random bond mixed,
            each at its own drive of a five-point sweep
  trial     one trial of the f_c^L bisection: create a batch, relax and observe, free it
  critical  one trial of the periodic-sample critical-force search: set the line, advance a chunk,
            read the line back (plain FP64, disorder periodic in u)
  sq        the structure factor of the current line
"""
import math

import numpy as np
import torch

import paper_1211_7275_gb300 as qew

RF, RB, RBG_LINEAR, RBG_CUBIC = qew.RF_GAUSS_LINEAR, qew.RB_UNIFORM_CATMULLROM, qew.RB_GAUSS_LINEAR, qew.RB_GAUSS_CATMULLROM
DT = 0.1

# depinning thresholds of the four disorder kinds (the presets' drives; the cubic Gaussian random
# bond's is the L = 4096 fixture's)
F_C = {RF: 0.72057, RB: 0.90749, RBG_LINEAR: 1.5652, RBG_CUBIC: 1.9475}

# launch shapes that the autotuner picks for the large presets of each kind (tile_w, K, tiles_per_cta)
TUNED = {RF: "992,32,2", RB: "480,16,1", RBG_LINEAR: "736,16,1", RBG_CUBIC: "480,16,1"}

# counted lane operations per site-update (elastic force 6, Euler 3, cell test 3, pinning 2 or 8) and
# per disorder draw (one Philox4x32-10 block and its transform), with the share of site-updates that
# draw near the threshold
BASE_OPS = {RF: 14, RB: 20, RBG_LINEAR: 14, RBG_CUBIC: 20}
DRAW_OPS = {RF: 103, RB: 92, RBG_LINEAR: 103, RBG_CUBIC: 103}
DRAWS = {RF: 0.026, RB: 0.03, RBG_LINEAR: 0.18, RBG_CUBIC: 0.05}


def _relax(name, kind, L, batch, steps, n_obs, f=None, fp64=False, tuning="", state=False):
    c = dict(family="relax", kind=kind, L=L, batch=batch, f=F_C[kind] if f is None else f, steps=steps, n_obs=n_obs,
             fp64=fp64, tuning=tuning, state=state)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the plain method at its smallest: one 1024-site chain in the moving regime, 10^4 plain FP64
        # steps, 40 observations
        _relax("tiny_rf_fp64", RF, 1024, 1, 10_000, 40, f=1.0, fp64=True, state=True),
        # the L = 4096 threshold run of 8 samples (t <= 500), Case 3, in the default launch shape
        _relax("rbg_linear_8x4096", RBG_LINEAR, 4096, 8, 5000, 30, state=True),
        # Case 1 on chains of odd length, in the default launch shape
        _relax("rbg_cubic_24x100003", RBG_CUBIC, 100_003, 24, 1000, 30, state=True),
        # the bisection of f_c^L at its defaults (batch 4, 2^14 steps, 30 observations): one trial,
        # handle and all
        dict(name="trial_rf_4x2^18", family="trial", kind=RF, L=1 << 18, batch=4, f=0.725, steps=1 << 14, n_obs=30),
        # the critical force of periodic 512 x 512 samples: one trial's chunk of 2000 plain FP64 steps
        dict(name="critical_rf_16x512", family="critical", kind=RF, L=512, batch=16, period=512, f=0.6, steps=2000),
        # FP64 against FP32-split at 16 x 2^20: the plain FP64 path
        _relax("rf_16x2^20_fp64", RF, 1 << 20, 16, 64, 10, fp64=True),
        # the same chains in FP32-split, long enough for the cell moves to become rare
        _relax("rf_16x2^20", RF, 1 << 20, 16, 8192, 40, tuning=TUNED[RF]),
        # the benchmark: the paper's largest chains
        _relax("rf_4x2^25", RF, 1 << 25, 4, 1024, 40, f=0.7209, tuning=TUNED[RF]),
        # many medium chains, uniform random bond (Case 2)
        _relax("rb_1024x2^16", RB, 1 << 16, 1024, 1024, 40, tuning=TUNED[RB]),
        # the paper's Case 3 at its largest size
        _relax("rbg_linear_4x2^25", RBG_LINEAR, 1 << 25, 4, 512, 30, tuning=TUNED[RBG_LINEAR]),
        # 256 chains of 2^12 .. 2^22 sites, random field and random bond mixed
        dict(name="uneven_256", family="uneven", chains=256, lo=12.0, hi=22.0, length_seed=7275, steps=512, n_obs=30,
             tuning="736,32,1"),
        # S_q of 16 rough lines of 2^20 sites, all modes
        dict(name="sq_16x2^20", family="sq", L=1 << 20, batch=16),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    family = rng.choice(["relax", "relax", "relax", "relax", "fp64", "uneven", "trial", "critical", "sq"])
    off = rng.choice([-0.02, -0.01, 0.0, 0.01, 0.02])
    if family in ("relax", "fp64"):
        fp64 = family == "fp64"
        kind = rng.choice([RF, RB, RBG_LINEAR, RBG_CUBIC])
        L = int(_log_uniform(rng, 1 << 10, 1 << (22 if fp64 else 25)))
        batch = int(_log_uniform(rng, 1, min(1024, (1 << (24 if fp64 else 27)) // L)))
        most = (1e9 if fp64 else 2.5e10) / (L * batch)
        steps = int(min(_log_uniform(rng, 64, 8192), max(16, most)))
        big = batch * L > 1 << 22
        return _relax(None, kind, L, batch, steps, rng.randint(5, 40), f=round(F_C[kind] * (1 + off), 6), fp64=fp64,
                      tuning="" if fp64 or not (big or rng.random() < 0.3) else TUNED[kind],
                      state=batch * L <= 1 << 20 and steps >= 256)
    if family == "uneven":
        chains = int(_log_uniform(rng, 8, 256))
        hi = rng.uniform(16.0, 22.0)
        return dict(family="uneven", chains=chains, lo=rng.uniform(10.0, 13.0), hi=hi, length_seed=rng.randrange(1 << 20),
                    steps=int(_log_uniform(rng, 64, 512)), n_obs=rng.randint(5, 30),
                    tuning=rng.choice(["", "736,32,1", "992,32,2"]))
    if family == "trial":
        return dict(family="trial", kind=rng.choice([RF, RF, RB, RBG_LINEAR]), L=int(_log_uniform(rng, 1 << 12, 1 << 18)), batch=4,
                    f=round(rng.uniform(0.6, 1.6), 5), steps=int(_log_uniform(rng, 1 << 10, 1 << 14)), n_obs=30)
    if family == "critical":
        return dict(family="critical", kind=rng.choice([RF, RBG_CUBIC]), L=int(_log_uniform(rng, 64, 2048)),
                    batch=rng.randint(1, 32), period=int(_log_uniform(rng, 64, 2048)), f=round(rng.uniform(0.2, 0.9), 5),
                    steps=2000)
    L = int(_log_uniform(rng, 1 << 10, 1 << 20))
    return dict(family="sq", L=L, batch=int(_log_uniform(rng, 1, 1 << 4)))


def _steps(n_steps, k):
    """Observation steps: 0 and k log-spaced ones up to n_steps."""
    s = {int(round(n_steps ** (j / (k - 1)))) for j in range(k)} | {0, n_steps}
    return np.asarray(sorted(s), dtype=np.int64)


def _uneven(case):
    rng = np.random.default_rng(case["length_seed"])
    L = np.floor(np.exp2(rng.uniform(case["lo"], case["hi"], size=case["chains"]))).astype(np.int64)
    kind = np.array([RF, RB], dtype=np.int32)[np.arange(case["chains"]) % 2]
    rng.shuffle(kind)
    off = np.array([-0.02, -0.01, 0.0, 0.01, 0.02])[np.arange(case["chains"]) % 5]
    f = np.where(kind == RF, F_C[RF], F_C[RB]) * (1.0 + off)
    return L, f, kind


def _line(L, batch, seed, scale):
    """Rough periodic lines: random walks pinned at both ends, of a few cells' width."""
    rng = np.random.default_rng(seed)
    w = np.cumsum(rng.standard_normal((batch, L)) * scale, axis=1)
    return np.ascontiguousarray(w - w[:, -1:] * (np.arange(1, L + 1) / L)).ravel()


def _critical_start(case, seed):
    return np.abs(_line(case["L"], case["batch"], seed, 0.1))


def _sq_line(case, seed):
    return _line(case["L"], case["batch"], seed, 0.05)


def _tune(r, case):
    if case["tuning"]:
        r.set_tuning(*(int(x) for x in case["tuning"].split(",")))


def prepare(case, seed):
    """What a program holds before the call: the handle (chains, disorder seed, launch shape) and the
    observation steps; for the trials also the start line."""
    fam = case["family"]
    if fam == "relax":
        r = qew.Relaxation(case["L"], case["f"], case["kind"], dt=DT, seed=seed, batch=case["batch"],
                           precision=qew.FP64 if case["fp64"] else qew.FP32_SPLIT)
        _tune(r, case)
        return case, r, _steps(case["steps"], case["n_obs"])
    if fam == "uneven":
        L, f, kind = _uneven(case)
        r = qew.Relaxation(L, f, kind, dt=DT, seed=seed)
        _tune(r, case)
        return case, r, _steps(case["steps"], case["n_obs"])
    if fam == "trial":
        return case, seed, _steps(case["steps"], case["n_obs"])[1:]
    if fam == "critical":
        r = qew.Relaxation(case["L"], case["f"], case["kind"], dt=DT, seed=seed, batch=case["batch"], precision=qew.FP64)
        r.set_disorder_period(case["period"])
        return case, r, _critical_start(case, seed)
    r = qew.Relaxation(case["L"], F_C[RF], RF, dt=DT, seed=seed, batch=case["batch"])
    r.set_state(_sq_line(case, seed))
    return case, r, None


def run(state):
    case, r, what = state
    fam = case["family"]
    if fam == "trial":
        with qew.Relaxation(case["L"], case["f"], case["kind"], dt=DT, seed=r, batch=case["batch"]) as trial:
            obs = trial.observe(what)
        return {"v": obs["v"], "ubar": obs["ubar"], "w2": obs["w2"]}
    if fam == "sq":
        return r.structure_factor()
    if fam == "critical":
        r.set_state(what)
        obs = r.observe([case["steps"]])
        u, _ = r.state()
        return {"v": obs["v"], "ubar": obs["ubar"], "w2": obs["w2"], "u": u}
    r.reset()
    obs = r.observe(what)
    out = {"v": obs["v"], "ubar": obs["ubar"], "w2": obs["w2"]}
    if case.get("state"):
        out["u"], _ = r.state()
    return out


def work(case):
    """Bytes: start line in (where one is given), observables and line out; the line itself can stay on
    chip or in memory between the steps.  Operations: BASE_OPS per site-update and DRAW_OPS per draw."""
    fam = case["family"]
    if fam == "sq":
        n = case["L"] * case["batch"]
        return {"bytes": 8.0 * n + 8.0 * (case["L"] // 2), "flops": 2.5 * n * math.log2(case["L"])}
    if fam == "uneven":
        L, _, kind = _uneven(case)
        ops = sum(float(l) * (BASE_OPS[k] + DRAW_OPS[k] * DRAWS[k]) for l, k in zip(L, kind.tolist()))
        return {"bytes": 24.0 * case["chains"] * len(_steps(case["steps"], case["n_obs"])), "flops": ops * case["steps"]}
    n, k = case["L"] * case["batch"], case["kind"]
    flops = float(n) * case["steps"] * (BASE_OPS[k] + DRAW_OPS[k] * DRAWS[k])
    if fam == "critical":
        return {"bytes": 16.0 * n + 24.0 * case["batch"], "flops": flops}
    seen = 24.0 * case["batch"] * len(_steps(case["steps"], case["n_obs"]))
    return {"bytes": seen + (8.0 * n if case.get("state") else 0.0), "flops": flops}


# ---- the same quantities in plain FP64 torch, from the definitions ----
_MASK = 0xFFFFFFFF


def _philox(i, n, s, tag, seed):
    """Words 0 and 1 of Philox4x32-10 at counter (i, n, s, tag), as int64 tensors in [0, 2^32)."""
    x = [i & _MASK, n & _MASK, s & _MASK, torch.full_like(i, tag)]
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    for _ in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57   # low 64 bits: wraps in two's complement
        x = [((p1 >> 32) & _MASK) ^ x[1] ^ k0, p1 & _MASK, ((p0 >> 32) & _MASK) ^ x[3] ^ k1, p0 & _MASK]
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return x[0], x[1]


def _node(kind, i, n, s, seed, period):
    if period:
        n = torch.remainder(n, period)
    a, b = _philox(i, n, s, {RF: 0, RB: 1, RBG_LINEAR: 2, RBG_CUBIC: 2}[kind], seed)
    if kind == RB:
        return (a.double() + 0.5) * 2.0 ** -31 - 1.0
    return torch.sqrt(-2.0 * torch.log((a.double() + 0.5) * 2.0 ** -32)) * torch.cos(2.0 * math.pi * (b.double() + 0.5) * 2.0 ** -32)


def _simulate(kind, L, batch, f, seed, steps, period=0, u0=None):
    """v, ubar, w2 at the given steps and the last line, of `batch` chains from u0 (default: flat)."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    u = torch.zeros(batch, L, dtype=torch.float64, device=dev) if u0 is None else torch.as_tensor(u0, device=dev).reshape(batch, L).clone()
    first, count = (0, 2) if kind in (RF, RBG_LINEAR) else (-1, 4)
    nodes = [torch.empty(batch * L, dtype=torch.float64, device=dev) for _ in range(count)]
    cell = torch.full((batch * L,), -(1 << 40), dtype=torch.int64, device=dev)
    out = {"v": [], "ubar": [], "w2": []}

    def force():
        fl = torch.floor(u)
        n = fl.reshape(-1).to(torch.int64)
        at = torch.nonzero(n != cell).reshape(-1)
        if at.numel():
            na, site, sample = n[at], at % L, at // L
            for j in range(count):
                nodes[j][at] = _node(kind, site, na + first + j, sample, seed, period)
            cell[at] = na
        d = (u - fl).reshape(-1)
        if kind == RF:
            F = (1.0 - d) * nodes[0] + d * nodes[1]
        elif kind == RBG_LINEAR:
            F = nodes[0] - nodes[1]
        else:
            p0, p1, p2, p3 = nodes
            b = 2.0 * p0 - 5.0 * p1 + 4.0 * p2 - p3
            c = -p0 + 3.0 * p1 - 3.0 * p2 + p3
            F = -0.5 * ((p2 - p0) + 2.0 * b * d + 3.0 * c * d * d)
        return F.reshape(batch, L)

    t = 0
    for target in [int(x) for x in steps]:
        while t < target:
            lap = torch.roll(u, -1, 1) + torch.roll(u, 1, 1) - 2.0 * u
            u = u + DT * (lap + f + force())
            t += 1
        m = u.mean(1)
        out["v"].append(f + force().mean(1))
        out["ubar"].append(m)
        out["w2"].append(((u - m[:, None]) ** 2).mean(1))
    res = {k: torch.stack(v).cpu().numpy() for k, v in out.items()}
    res["u"] = u.reshape(-1).cpu().numpy()
    return res


def exact(case, seed):
    fam = case["family"]
    if fam == "uneven":
        return None   # 256 lengths one by one in FP64: over the time allowed
    if fam == "sq":
        z = np.fft.rfft(_sq_line(case, seed).reshape(case["batch"], case["L"]), axis=1)
        return np.mean(np.abs(z[:, 1:case["L"] // 2 + 1] / case["L"]) ** 2, axis=0)
    n = case["L"] * case["batch"]
    if case["steps"] * (0.6e-3 + 2e-9 * n) > 15.0:
        return None   # the large cases: over the time allowed
    if fam == "critical":
        return _simulate(case["kind"], case["L"], case["batch"], case["f"], seed, [case["steps"]], case["period"],
                         _critical_start(case, seed))
    res = _simulate(case["kind"], case["L"], case["batch"], case["f"], seed,
                    _steps(case["steps"], case["n_obs"])[1 if fam == "trial" else 0:])
    if not case.get("state"):
        del res["u"]
    return res
