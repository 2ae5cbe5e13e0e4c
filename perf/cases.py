"""The work that users of this framework have it do, as cases that can be timed and checked.

Each case is one call pattern of the public Python binding at a size of the repository's
configurations (``workloads``), of its tests or of its benchmark, or of the same ranges:

  single   one run advanced by a window of steps, then read: moment sums, cell data and the
           particle state (a checkpoint)
  restart  a run restored from a host checkpoint, advanced, sampled and saved again
  window   training windows of the surrogate stage taken from a small run, then its fit
  batch    many independent runs advanced together, then the moment sums of all
  serve    micro-solve requests through a pool's request loop
  mms      the whole Micro-Macro-Surrogate hybrid
  bands    the surrogate stage alone: windows, fit, Monte Carlo bands of the profile
  gp       the Gaussian-process variant: fit, prediction and the corrected CFD

A run's random numbers are keyed on its seed, so a case is a pure function of its inputs.
"""
import math

import numpy as np
import torch

from paper_2311_14140_gb300 import (Dsmc, DsmcBatch, DsmcPool, GaussianProcess, Surrogate,
                                    cfd_faces, mms_hybrid)
from paper_2311_14140_gb300 import gp_variant, workloads

SQRT_PI = math.sqrt(math.pi)


# ---------------------------------------------------------------------------------------
# The cases.

def listed():
    f0 = workloads.f0_force
    return [
        # The smallest run in real use: argon hard spheres at Kn = 1, 100 cells x 200, its
        # state in L2, replayed as a CUDA graph: launch latency counts.
        dict(name="hs_kn1_20k", kind="single", omega=0.5, Kn=1.0, n_cells=100, ppc=200,
             F=f0(1.0), steps=64, graph=True, accum=0, collisions=True, group_size=256),
        # The paper's training run (Sec. 3: 200 cells x 50 particles), default options:
        # windows of 100 steps handed to the surrogate, then a fit.
        dict(name="window_200x50", kind="window", omega=0.5, Kn=0.1, n_cells=200, ppc=50,
             F=0.012, window=100, windows=2),
        # The paper's benchmark run (500 particles per cell, 1e5 in all), default options.
        dict(name="channel_200x500", kind="single", omega=0.5, Kn=0.5, n_cells=200, ppc=500,
             F=f0(0.5), steps=50, graph=False, accum=0, collisions=True, group_size=256),
        # A production slice of a mid-sized VHS run with odd sizes: restore a checkpoint
        # from pinned host memory, advance, read, save.
        dict(name="restart_vhs_1m", kind="restart", omega=0.81, Kn=0.3, n_cells=397, ppc=2531,
             F=f0(0.3), steps=24),
        # The large single run: argon VHS at Kn = 0.1, 2,000 cells x 25,000 particles.
        dict(name="vhs_kn0.1_50m", kind="single", omega=0.81, Kn=0.1, n_cells=2000, ppc=25000,
             F=f0(0.1), steps=16, graph=False, accum=0, collisions=True, group_size=256),
        # The same physics with binary64 moment sums, the option for long averages.
        dict(name="vhs_fp64_sums_5m", kind="single", omega=0.81, Kn=0.1, n_cells=1000, ppc=5003,
             F=f0(0.1), steps=16, graph=False, accum=1, collisions=True, group_size=256),
        # 256 uneven runs in one handle (Kn 0.05-10, 50-1,000 cells, 50-400 particles per
        # cell), with the partition the tuner keeps for it.
        dict(name="batch_256", kind="batch", n=256, layout=12345, cells=0, ppc=0, steps=16,
             cta_warps=4, span_particles=8192, graph=True),
        # The design runs of the GP variant: 64 runs of 100 cells x 200, default options.
        dict(name="batch_design_64", kind="batch", n=64, layout=3, cells=100, ppc=200, steps=50,
             cta_warps=0, span_particles=0, graph=False),
        # Continuous batching: 48 requests that share a pool with room for about half.
        dict(name="serve_48", kind="serve", n=48, layout=77, max_steps=384, target_se=0.02,
             sample_start=64, epoch_steps=32, batches=8, pool_particles=3_000_000),
        # The MMS hybrid with the paper's sub-domain (two mean free paths and five buffer
        # cells of width 0.005, 50 particles per cell) and 1,000 Monte Carlo trials.
        dict(name="mms_kn0.1", kind="mms", omega=0.5, Kn=0.1, F=0.012, dy=0.005, ppc=50,
             buffer=5, iterations=3, steps=500, window=100, warmup=200, n_cfd=200, trials=1000),
        # The surrogate stage by itself: 100 windows of 200 cells, fit, 1,000 trials.
        dict(name="bands_1000", kind="bands", Kn=0.1, F=0.012, n_cells=200, ppc=50, steps=100,
             windows=100, n_cfd=200, trials=1000),
        # The GP over 64 design points and the CFD of 8 new cases.
        dict(name="gp_64", kind="gp", n=64, n_cfd=200, tests=8),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["single", "single", "single", "single", "restart", "window", "batch",
                       "batch", "serve", "mms", "bands", "gp"])
    Kn = round(_log(rng, 0.05, 10.0), 4)
    omega = rng.choice([0.5, 0.5, 0.81, 0.81, 0.74, 1.0])
    F = round(workloads.f0_force(Kn) * rng.uniform(0.5, 20.0), 8)
    if kind == "single":
        cells = int(_log(rng, 20, 4000))
        ppc = int(_log(rng, 20, 25000))
        ppc = max(8, min(ppc, 20_000_000 // cells))
        accum = rng.choice([0, 0, 0, 1])
        steps = int(min(96, max(2, (1e8 if accum else 3e8) / (cells * ppc)))) + rng.randint(0, 7)
        return dict(kind=kind, omega=omega, Kn=Kn, n_cells=cells, ppc=ppc, F=F, steps=steps,
                    graph=rng.random() < 0.5, accum=accum, collisions=rng.random() < 0.9,
                    group_size=rng.choice([256, 256, 256, 128, 64]))
    if kind == "restart":
        cells = int(_log(rng, 50, 2000))
        ppc = max(20, int(_log(rng, 2e4, 4e6)) // cells)
        return dict(kind=kind, omega=omega, Kn=Kn, n_cells=cells, ppc=ppc, F=F,
                    steps=rng.randint(4, 40))
    if kind == "window":
        return dict(kind=kind, omega=omega, Kn=round(_log(rng, 0.05, 5.0), 4),
                    n_cells=rng.randint(40, 400), ppc=int(_log(rng, 20, 500)),
                    F=round(rng.uniform(0.004, 0.02), 5), window=rng.choice([50, 100]),
                    windows=rng.randint(1, 3))
    if kind == "batch":
        n = int(_log(rng, 4, 200))
        same = rng.random() < 0.5
        return dict(kind=kind, n=n, layout=rng.randint(1, 1 << 20),
                    cells=rng.randint(50, 300) if same else 0,
                    ppc=rng.randint(50, 400) if same else 0, steps=rng.randint(8, 40),
                    cta_warps=rng.choice([0, 4]), span_particles=rng.choice([0, 8192, 16384]),
                    graph=rng.random() < 0.5)
    if kind == "serve":
        return dict(kind=kind, n=rng.randint(4, 64), layout=rng.randint(1, 1 << 20),
                    max_steps=rng.choice([256, 384, 512]), target_se=rng.choice([0.01, 0.02, 0.05]),
                    sample_start=rng.choice([0, 64]), epoch_steps=rng.choice([16, 32]),
                    batches=8, pool_particles=rng.choice([2_000_000, 4_000_000, 16_000_000]))
    if kind == "mms":
        return dict(kind=kind, omega=rng.choice([0.5, 0.81]), Kn=round(_log(rng, 0.04, 0.2), 4),
                    F=round(rng.uniform(0.006, 0.02), 5), dy=0.005, ppc=rng.randint(40, 200),
                    buffer=5, iterations=rng.randint(1, 4), steps=rng.choice([200, 400, 600]),
                    window=100, warmup=rng.choice([0, 100, 300]), n_cfd=rng.choice([100, 200, 400]),
                    trials=rng.randint(100, 2000))
    if kind == "bands":
        return dict(kind=kind, Kn=round(_log(rng, 0.05, 5.0), 4), F=round(rng.uniform(0.004, 0.02), 5),
                    n_cells=rng.randint(50, 600), ppc=rng.randint(50, 500), steps=100,
                    windows=rng.randint(20, 160), n_cfd=int(_log(rng, 50, 1000)),
                    trials=int(_log(rng, 100, 4000)))
    return dict(kind="gp", n=rng.randint(8, 128), n_cfd=rng.choice([100, 200, 333]),
                tests=rng.randint(1, 16))


# ---------------------------------------------------------------------------------------
# Inputs.

def _seed(seed, k=0):
    return (int(seed) * 1_000_003 + 7919 * k + 17) & 0x7FFFFFFFFFFFFFFF


def _gen(seed, k=0):
    return torch.Generator(device="cuda").manual_seed(_seed(seed, k) % (1 << 62))


def _batch_defs(case, seed):
    """The runs of a batch: their sizes and flow from the case's layout, their random
    numbers from the seed."""
    defs = []
    if case["cells"]:
        Kn, F, _ = workloads.gp_design(case["n"], seed=case["layout"])
        for i in range(case["n"]):
            defs.append(dict(Kn=float(Kn[i]), n_cells=case["cells"], ppc=case["ppc"], omega=0.5,
                             body_force=float(F[i]), seed=_seed(seed, i)))
    else:
        for i, w in enumerate(workloads.batch_instances(case["n"], seed=case["layout"])):
            defs.append(dict(Kn=w.Kn, n_cells=w.n_cells, ppc=w.ppc, omega=w.omega,
                             body_force=w.body_force, seed=_seed(seed, i)))
    return defs


def _windows(case, seed):
    """Raw moment sums of synthetic windows: about steps x ppc samples per cell of a gas with
    velocity and shear profiles like the channel's, every sum with its sampling noise."""
    g = _gen(seed, 5)
    W, n = case["windows"], case["n_cells"]
    cnt = float(case["steps"] * case["ppc"])
    y = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / n
    Kn, F = case["Kn"], case["F"]
    u = (SQRT_PI * F / (2.0 * Kn)) * (y - y * y) + 1.1 * F + 0.3 * F * torch.exp(-y / Kn)
    pxy = F * (2.0 * y - 1.0)

    def noise():
        return torch.randn(W, n, generator=g, device="cuda", dtype=torch.float64)

    out = torch.empty(W, n, 13, device="cuda", dtype=torch.float64)
    N = torch.round(cnt + math.sqrt(cnt) * 0.3 * noise())
    sd = torch.sqrt(0.5 * N)
    out[..., 0] = N
    out[..., 1] = N * u + sd * noise()
    out[..., 2] = sd * noise()
    out[..., 3] = sd * noise()
    for k in (4, 5, 6):
        out[..., k] = 0.5 * N + sd * noise()
    out[..., 7] = N * (0.5 * pxy) + 0.7 * sd * noise()
    for k in (8, 9):
        out[..., k] = 0.7 * sd * noise()
    for k in (10, 11, 12):
        out[..., k] = 2.0 * sd * noise()
    return out


def _gp_inputs(case, seed):
    """Design points, outputs (slip coefficient and stress correction / F at the faces, as
    smooth functions of the inputs with the scatter that fits of short runs have) and new
    cases; host arrays, as the binding takes them."""
    r = np.random.default_rng(_seed(seed, 9))
    n, m = case["n"], case["n_cfd"] + 2
    X = workloads.latin_hypercube(n, 2, seed=int(r.integers(1 << 31)))
    f = np.arange(case["n_cfd"] + 1) / case["n_cfd"]
    Y = np.empty((n, m))
    Y[:, 0] = 1.1 + 0.3 * X[:, 0] - 0.1 * X[:, 0] * X[:, 1] + 0.05 * r.standard_normal(n)
    a = 0.4 + 0.5 * np.sin(2.0 * X[:, 0]) + 0.1 * r.standard_normal(n)
    b = 6.0 + 10.0 * X[:, 0]
    Y[:, 1:] = a[:, None] * (np.exp(-b[:, None] * f) - np.exp(-b[:, None] * (1.0 - f)))
    Y[:, 1:] += 0.01 * r.standard_normal((n, m - 1))
    Xs = r.uniform(size=(case["tests"], 2))
    Kn = np.exp(math.log(workloads.GP_KN[0])
                + Xs[:, 0] * (math.log(workloads.GP_KN[1]) - math.log(workloads.GP_KN[0])))
    fac = workloads.GP_FORCE[0] + Xs[:, 1] * (workloads.GP_FORCE[1] - workloads.GP_FORCE[0])
    F = np.array([workloads.gp_force(k, x) for k, x in zip(Kn, fac)])
    return X, Y, Xs, Kn, F


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "single":
        stream = torch.cuda.Stream() if case["graph"] else None
        st["stream"] = stream
        st["run"] = Dsmc(case["Kn"], case["n_cells"], case["ppc"], omega=case["omega"],
                         body_force=case["F"], seed=_seed(seed), graph=case["graph"],
                         accum=case["accum"], collisions=case["collisions"],
                         group_size=case["group_size"],
                         stream=stream.cuda_stream if stream else None)
        st["state"] = [torch.empty(case["n_cells"] * case["ppc"], device="cuda")
                       for _ in range(4)]
    elif kind == "restart":
        N = case["n_cells"] * case["ppc"]
        st["run"] = Dsmc(case["Kn"], case["n_cells"], case["ppc"], omega=case["omega"],
                         body_force=case["F"], seed=_seed(seed))
        g = _gen(seed, 1)
        cell = torch.arange(N, device="cuda") // case["ppc"]
        y = (cell + torch.rand(N, generator=g, device="cuda")) / case["n_cells"]
        v = [math.sqrt(0.5) * torch.randn(N, generator=g, device="cuda") for _ in range(3)]
        v[0] += case["F"] * (1.0 + (y - y * y) / case["Kn"])
        st["checkpoint"] = [t.float().clamp_(-100, 100).cpu().pin_memory() for t in (y, *v)]
        st["saved"] = [torch.empty(N).pin_memory() for _ in range(4)]
    elif kind == "window":
        st["run"] = Dsmc(case["Kn"], case["n_cells"], case["ppc"], omega=case["omega"],
                         body_force=case["F"], seed=_seed(seed))
        st["surrogate"] = Surrogate(case["Kn"], case["F"], case["n_cells"], case["ppc"])
    elif kind == "batch":
        stream = torch.cuda.Stream() if case["graph"] else None
        st["stream"] = stream
        st["run"] = DsmcBatch(_batch_defs(case, seed), graph=case["graph"],
                              cta_warps=case["cta_warps"], span_particles=case["span_particles"],
                              stream=stream.cuda_stream if stream else None)
    elif kind == "serve":
        st["stream"] = torch.cuda.Stream()
        st["pool"] = DsmcPool(case["pool_particles"], max(2000, case["pool_particles"] // 50),
                              256, 1000, sample_start=case["sample_start"], graph=True,
                              stream=st["stream"].cuda_stream)
        reqs = workloads.serving_requests(case["n"], target_se=case["target_se"],
                                          max_steps=case["max_steps"], seed=case["layout"])
        for i, r in enumerate(reqs):
            r["arrival"] = 0.0
            r["seed"] = _seed(seed, i)
            r["body_force"] *= 20.0
        st["requests"] = reqs
    elif kind == "mms":
        st["seed"] = _seed(seed)
        st["z"] = np.random.default_rng(_seed(seed, 2)).standard_normal((case["trials"], 4))
    elif kind == "bands":
        st["surrogate"] = Surrogate(case["Kn"], case["F"], case["n_cells"], case["ppc"])
        st["windows"] = _windows(case, seed)
        st["z"] = np.random.default_rng(_seed(seed, 2)).standard_normal((case["trials"], 4))
    else:
        st["X"], st["Y"], st["Xs"], st["Kn"], st["F"] = _gp_inputs(case, seed)
    return st


# ---------------------------------------------------------------------------------------
# One pass.

def _fit_out(f):
    return {k: v for k, v in f.items() if k in (
        "n_samples", "n_v", "n_c", "log_evidence_v", "prob_v", "sigma_p", "sigma_p_var",
        "log_evidence_c", "prob_c", "m_c", "S_c", "sel_v", "sel_c")}


def _cells_out(cells):
    off, smax, ncand, nacc = cells
    return dict(offset=off, smax=smax, ncand=ncand.astype(np.int64), nacc=nacc.astype(np.int64))


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "single":
        r = state["run"]
        r.step(case["steps"])
        sums, n = r.moments()
        r.state_into(*state["state"])
        return dict(sums=sums, samples=n, cells=_cells_out(r.cells()), state=state["state"])
    if kind == "restart":
        r = state["run"]
        r.load_state(*state["checkpoint"], step=1000)
        r.reset_samples()
        r.step(case["steps"])
        fields = r.fields()
        sums, n = r.moments()
        r.state_into(*state["saved"])
        return dict(fields=fields, sums=sums, samples=n, state=state["saved"])
    if kind == "window":
        r, s = state["run"], state["surrogate"]
        for _ in range(case["windows"]):
            r.step(case["window"])
            s.add_run(r)
        fit = s.train()
        return dict(fit=_fit_out(fit), cells=_cells_out(r.cells()))
    if kind == "batch":
        b = state["run"]
        b.step(case["steps"])
        sums, n = b.moments_all()
        last = case["n"] - 1
        return dict(sums=sums, samples=n, first=_cells_out(b.cells(0)),
                    last=_cells_out(b.cells(last)), state=list(b.state(last)))
    if kind == "serve":
        res = state["pool"].serve(state["requests"], epoch_steps=case["epoch_steps"],
                                  batches=case["batches"])
        return {k: np.array([r[k] for r in res])
                for k in ("steps", "converged", "u_mean", "u_se", "count", "sum_vx")}
    if kind == "mms":
        h = mms_hybrid(case["Kn"], case["F"], omega=case["omega"], dy=case["dy"], ppc=case["ppc"],
                       buffer=case["buffer"], iterations=case["iterations"], steps=case["steps"],
                       window=case["window"], warmup=case["warmup"], n_cfd=case["n_cfd"],
                       seed=state["seed"], z=state["z"])
        return dict(profile=h["profile"], band_sd=h["band_sd"], samples=h["samples"],
                    interface=np.array(h["interface"]), fit=_fit_out(h["fit"]))
    if kind == "bands":
        s = state["surrogate"]
        s.reset()
        for w in state["windows"]:
            s.add_window(w, case["steps"])
        fit = s.train()
        mean, sd = s.profile(case["n_cfd"], state["z"])
        return dict(fit=_fit_out(fit), mean=mean, sd=sd)
    gp = GaussianProcess(state["X"], state["Y"], gp_variant.GRID)
    pred = gp.predict(state["Xs"])
    prof = np.array([cfd_faces(k, f, case["n_cfd"], p[0], f * p[1:])
                     for k, f, p in zip(state["Kn"], state["F"], pred)])
    out = dict(lml=gp.lml, best=gp.best, pred=pred, profiles=prof)
    gp.close()
    return out


# ---------------------------------------------------------------------------------------
# What a pass cannot do without.

# Operations of one particle and step: its moment products before and after the collisions
# (2 x 33), its share of the candidates (about 0.2 candidates of 90 operations), flight, wall
# test and cell (10).
_STEP_FLOPS = 94


def _dsmc_work(particles, cells, steps):
    # the 16-byte record read and written once per step; the moment sums updated per step
    return dict(bytes=steps * (32 * particles + 208 * cells), flops=steps * _STEP_FLOPS * particles)


def _bands_work(windows, cells, n_cfd, trials):
    return dict(bytes=8 * (13 * windows * cells + 4 * trials + 2 * n_cfd),
                flops=windows * cells * 90 + n_cfd * 150 + trials * n_cfd * 16)


def work(case):
    kind = case["kind"]
    if kind == "single":
        N = case["n_cells"] * case["ppc"]
        w = _dsmc_work(N, case["n_cells"], case["steps"])
        w["bytes"] += 32 * N  # the state read out
        return w
    if kind == "restart":
        N = case["n_cells"] * case["ppc"]
        w = _dsmc_work(N, case["n_cells"], case["steps"])
        w["bytes"] += 64 * N  # the state in, sorted, and out
        return w
    if kind == "window":
        return _dsmc_work(case["n_cells"] * case["ppc"], case["n_cells"],
                          case["window"] * case["windows"])
    if kind == "batch":
        defs = _batch_defs(case, 0)
        return _dsmc_work(sum(d["n_cells"] * d["ppc"] for d in defs),
                          sum(d["n_cells"] for d in defs), case["steps"])
    if kind == "serve":
        reqs = workloads.serving_requests(case["n"], seed=case["layout"])
        least = case["batches"] * case["epoch_steps"]  # steps before a request can end
        return _dsmc_work(sum(r["n_cells"] * r["ppc"] for r in reqs),
                          sum(r["n_cells"] for r in reqs), least)
    if kind == "mms":
        n_sub = math.ceil(2.0 * case["Kn"] / case["dy"] - 1e-9) + case["buffer"]
        steps = case["warmup"] + case["iterations"] * case["steps"]
        w = _dsmc_work(n_sub * case["ppc"], n_sub, steps)
        b = _bands_work(case["iterations"] * case["steps"] // case["window"], n_sub,
                        case["n_cfd"], case["trials"])
        return {k: w[k] + b[k] for k in w}
    if kind == "bands":
        return _bands_work(case["windows"], case["n_cells"], case["n_cfd"], case["trials"])
    n, m, t = case["n"], case["n_cfd"] + 2, case["tests"]
    g = len(gp_variant.GRID)
    # per grid point: the covariance, its factor and a triangular solve per output
    flops = g * (n * n * 10 + n ** 3 / 3 + n * n * m) + 2 * n * n * m + 2 * t * n * m
    return dict(bytes=8 * (2 * n + n * m + 3 * g + g + t * (2 * m + case["n_cfd"])), flops=flops)


# ---------------------------------------------------------------------------------------
# 64-bit values, where a case's outputs are functions of its inputs alone (the runs' outputs
# are those of a seeded particle simulation: they have none).

def _evidence(G, pt, tt, N, st):
    """Bayesian ridge regression by evidence maximisation (no intercept, flat hyperpriors)."""
    k = len(pt)
    ev = np.linalg.eigvalsh(G)
    var = tt / N - (st / N) ** 2
    alpha, beta = 1.0, 1.0 / max(var, 1e-300)
    for _ in range(1000):
        S = np.linalg.inv(beta * G + alpha * np.eye(k))
        m = beta * S @ pt
        gamma = float(np.sum(beta * ev / (alpha + beta * ev)))
        mm = float(m @ m)
        an = 1e30 if mm <= gamma / 1e30 else gamma / mm
        bn = (N - gamma) / float(tt - 2.0 * m @ pt + m @ G @ m)
        done = abs(an - alpha) <= 1e-12 * alpha and abs(bn - beta) <= 1e-12 * beta
        alpha, beta = an, bn
        if done:
            break
    A = beta * G + alpha * np.eye(k)
    S = np.linalg.inv(A)
    m = beta * S @ pt
    E = 0.5 * beta * float(tt - 2.0 * m @ pt + m @ G @ m) + 0.5 * alpha * float(m @ m)
    le = (0.5 * k * math.log(alpha) + 0.5 * N * math.log(beta) - E
          - 0.5 * np.linalg.slogdet(A)[1] - 0.5 * N * math.log(2.0 * math.pi))
    return m, S, le


def _probabilities(le):
    p = np.exp(le - le.max())
    return p / p.sum()


def _tridiagonal(n, rhs, uw):
    """-u'' on n cells with wall values through ghost cells: u for each right side."""
    h = 1.0 / n
    A = (np.diag(np.full(n, -2.0 / h)) + np.diag(np.full(n - 1, 1.0 / h), 1)
         + np.diag(np.full(n - 1, 1.0 / h), -1))
    A[0, 0] = A[-1, -1] = -3.0 / h
    r = np.array(rhs)
    r[..., 0] -= 2.0 * uw / h
    r[..., -1] -= 2.0 * uw / h
    return np.linalg.solve(A, r.T).T


def _exact_bands(case, seed):
    acc = _windows(case, seed).cpu().numpy()
    n, Kn, F = case["n_cells"], case["Kn"], case["F"]
    h, c = 1.0 / n, 2.0 * Kn / SQRT_PI
    table = {0.01: (130, 150, 200), 0.05: (30, 40, 70), 0.1: (20, 40, 10), 0.2: (20, 12, 8),
             0.5: (10, 7, 6), 1.0: (8, 6, 20), 5.0: (7, 6, 5)}  # Table 1 of the paper
    b = table[min(table, key=lambda k: abs(math.log(Kn) - math.log(k)))]
    N = acc[..., 0]
    u, uy = acc[..., 1] / N, acc[..., 2] / N
    P = 2.0 * (N / (case["steps"] * case["ppc"])) * (acc[..., 7] / N - u * uy)
    E = (P[:, 1:-1] + c * (u[:, 2:] - u[:, :-2]) / (2.0 * h)).ravel()
    y = (np.arange(1, n - 1) + 0.5) * h
    phi = np.stack([c * (np.exp(-q * y) - np.exp(-q * (1.0 - y))) for q in b], axis=1)
    Phi = np.tile(phi, (len(acc), 1))
    walls = np.concatenate([1.5 * u[:, 0] - 0.5 * u[:, 1], 1.5 * u[:, -1] - 0.5 * u[:, -2]])
    nv, nc = float(len(walls)), float(len(E))
    le_v, le_c, m_c, S_c = np.empty(2), np.empty(4), np.zeros((4, 3)), np.zeros((4, 3, 3))

    def zero(t):
        be = len(t) / float(t @ t)
        return 0.5 * len(t) * (math.log(be) - math.log(2.0 * math.pi)) - 0.5 * be * float(t @ t)

    le_v[0], le_c[0] = zero(walls), zero(E)
    m, S, le_v[1] = _evidence(np.array([[nv * F * F]]), np.array([F * walls.sum()]),
                              float(walls @ walls), nv, float(walls.sum()))
    sp, sv = float(m[0]), float(S[0, 0])
    for k in (1, 2, 3):
        A = Phi[:, :k]
        m, S, le_c[k] = _evidence(A.T @ A, A.T @ E, float(E @ E), nc, float(E.sum()))
        m_c[k, :k], S_c[k, :k, :k] = m, S

    def pick(le):
        tol = 1e-9 * max(1.0, abs(le.max()))
        return int(np.nonzero(le >= le.max() - tol)[0][0])

    sel_v, sel_c = pick(le_v), pick(le_c)
    z = np.random.default_rng(_seed(seed, 2)).standard_normal((case["trials"], 4))
    uw = (sp + math.sqrt(sv) * z[:, 0]) * F if sel_v else np.zeros(len(z))
    nf = case["n_cfd"]
    S_face = np.zeros((len(z), nf + 1))
    if sel_c:
        L = np.linalg.cholesky(S_c[sel_c][:sel_c, :sel_c])
        w = m_c[sel_c][:sel_c] + z[:, 1:1 + sel_c] @ L.T
        yf = np.arange(nf + 1) / nf
        S_face = w @ np.stack([np.exp(-q * yf) - np.exp(-q * (1.0 - yf)) for q in b[:sel_c]])
    prof = _tridiagonal(nf, -SQRT_PI * F / Kn / nf + np.diff(S_face, axis=1), uw)
    fit = dict(n_samples=None, n_v=nv, n_c=nc, log_evidence_v=le_v, prob_v=_probabilities(le_v),
               sigma_p=sp, sigma_p_var=sv, log_evidence_c=le_c, prob_c=_probabilities(le_c),
               m_c=m_c, S_c=S_c.reshape(4, 9), sel_v=None, sel_c=None)
    return dict(fit=fit, mean=prof.mean(axis=0), sd=prof.std(axis=0, ddof=1))


def _exact_gp(case, seed):
    X, Y, Xs, Kn, F = _gp_inputs(case, seed)
    n, m = Y.shape
    mu, sd = Y.mean(axis=0), Y.std(axis=0)
    Z = (Y - mu) / np.where(sd > 0.0, sd, 1.0)

    def cov(A, B, l1, l2):
        d1, d2 = (A[:, None, 0] - B[None, :, 0]) / l1, (A[:, None, 1] - B[None, :, 1]) / l2
        return np.exp(-0.5 * (d1 * d1 + d2 * d2))

    lml = []
    for l1, l2, s2 in gp_variant.GRID:
        L = np.linalg.cholesky(cov(X, X, l1, l2) + s2 * np.eye(n))
        W = np.linalg.solve(L, Z)
        lml.append(-0.5 * float((W * W).sum()) - m * float(np.log(np.diag(L)).sum())
                   - 0.5 * n * m * math.log(2.0 * math.pi))
    best = int(np.argmax(lml))
    l1, l2, s2 = gp_variant.GRID[best]
    alpha = np.linalg.solve(cov(X, X, l1, l2) + s2 * np.eye(n), Z)
    pred = mu + sd * (cov(Xs, X, l1, l2) @ alpha)
    nf = case["n_cfd"]
    prof = np.stack([_tridiagonal(nf, -SQRT_PI * f / k / nf + np.diff(f * p[1:]), p[0] * f)
                     for k, f, p in zip(Kn, F, pred)])
    return dict(lml=np.array(lml), best=None, pred=pred, profiles=prof)


def exact(case, seed):
    if case["kind"] == "bands":
        return _exact_bands(case, seed)
    if case["kind"] == "gp":
        return _exact_gp(case, seed)
    return None
