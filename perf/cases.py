"""The work that users of this package have it do, as measurable cases.

Every case is a call or a short program through the package's Python entry points:
whole annealing runs (single, batched, learned schedule, partial resampling) from
construction to the results a user reads, the overlap distribution of annealed
populations, the allocation-free weights call and one training iteration of the
schedule controller.

listed()  the fixed cases          draw(rng)  one more of the same ranges
prepare() inputs and handles       run()      one pass, with its outputs
work()    bytes and operations     exact()    64-bit values where they are computed directly
"""
import math

import numpy as np
import torch

from paper_2401_07965_gb300 import controller, pa

RULES = ("multinomial", "systematic", "residual", "poisson", "nearest")

# integer operations per spin update of the Metropolis arithmetic (bit-plane uniforms by
# Philox4x32-10, 32 replicas per site word: 108 operations per site word in 2D, 126 in 3D)
OPS_PER_UPDATE = {2: 108 / 32, 3: 126 / 32}


def listed():
    return [
        # the smallest run in use: a quick look at a small lattice; latency and launches
        {"name": "ising2d_L16_R1000", "kind": "run", "dim": 2, "L": 16, "R": 1000, "steps": 100,
         "theta": 10, "beta_f": 1.0, "rule": "multinomial", "ea": False, "spins": True},
        # the paper's population and schedule (R = 20000, theta = 5, beta_i = i/300), with
        # the final population kept (a checkpoint)
        {"name": "ising2d_L64_R20k", "kind": "run", "dim": 2, "L": 64, "R": 20000, "steps": 300,
         "theta": 5, "beta_f": 1.0, "rule": "nearest", "ea": False, "spins": True},
        # the headline benchmark's run
        {"name": "ising2d_L64_R100k", "kind": "run", "dim": 2, "L": 64, "R": 100000,
         "steps": 200, "theta": 10, "beta_f": 1.0, "rule": "systematic", "ea": False,
         "spins": False},
        # the largest population in use (the single run that weighted averages are held
        # against), where the resampling passes have a million replicas to move
        {"name": "ising2d_L32_R1M", "kind": "run", "dim": 2, "L": 32, "R": 1024000, "steps": 150,
         "theta": 10, "beta_f": 1.0, "rule": "residual", "ea": False, "spins": False},
        # a side that is no power of two, as finite-size scaling studies need, with a
        # glass and a fluctuating population size
        {"name": "ea2d_L48_R20k", "kind": "run", "dim": 2, "L": 48, "R": 20001, "steps": 150,
         "theta": 10, "beta_f": 2.0, "rule": "poisson", "ea": True, "spins": False},
        # spin-glass sampling: many disorder realizations of small 3D lattices in one batch
        {"name": "ea3d_batch_L4_6_8", "kind": "batch", "dim": 3, "sides": "4,6,8", "each": 8,
         "R": 50000, "steps": 100, "theta": 10, "beta_f": 3.0, "rule": "systematic", "ea": True},
        # many small populations of one system, combined by weighted averages
        {"name": "weighted_L32_80runs", "kind": "weighted", "dim": 2, "L": 32, "small": 64,
         "R_small": 2000, "large": 16, "R_large": 8000, "steps": 150, "theta": 10,
         "beta_f": 1.0, "rule": "systematic"},
        # the learned schedule at the small population that its accuracy record uses
        {"name": "learned_L64_R3000", "kind": "learned", "dim": 2, "L": 64, "R": 3000,
         "grid": 800, "budget": 2000, "beta_f": 1.0, "rule": "systematic"},
        # partial resampling (resample only when the effective size falls below half)
        {"name": "partial_L64_R10k", "kind": "partial", "dim": 2, "L": 64, "R": 10000,
         "steps": 200, "theta": 10, "beta_f": 1.0, "rule": "systematic", "alpha": 0.5},
        # the overlap distribution P(q) of two populations per glass sample
        {"name": "overlap_ea2d_L32", "kind": "overlap", "dim": 2, "L": 32, "pairs": 16,
         "R": 100000, "steps": 20, "theta": 5, "beta_f": 3.0},
        # the weights of a population held by another framework, with no allocation
        {"name": "weights_static_L64_R100k", "kind": "weights", "dim": 2, "L": 64, "R": 100000,
         "beta": 0.44, "dbeta": 0.005},
        # one full-batch training iteration of the schedule controller (its trace rows)
        {"name": "mlp_train_12040", "kind": "mlp", "rows": 12040},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(rng, lo, hi):
    return max(2, 2 * round(_log(rng, lo, hi) / 2))


def _fit(updates, limit, c, key, least):
    """Shrink c[key] so that the case stays below `limit` spin updates."""
    u = updates(c)
    if u > limit:
        c[key] = max(least, int(c[key] * limit / u))
    return c


def draw(rng):
    kind = rng.choice(["run2d", "run2d", "run2d", "run3d", "run3d", "batch", "weighted",
                       "learned", "partial", "overlap", "weights", "mlp"])
    rule = rng.choice(RULES)
    theta = int(round(_log(rng, 2, 20)))
    steps = int(round(_log(rng, 60, 300)))
    if kind in ("run2d", "run3d"):
        dim = 2 if kind == "run2d" else 3
        L = (rng.choice([16, 32, 64, _even(rng, 6, 120), _even(rng, 6, 120)]) if dim == 2
             else rng.choice([4, 6, 8, 10, _even(rng, 4, 24)]))
        ea = rng.random() < (0.3 if dim == 2 else 0.7)
        c = {"kind": "run", "dim": dim, "L": L, "R": int(_log(rng, 300, 300000)), "steps": steps,
             "theta": theta, "beta_f": round(rng.uniform(0.6, 1.2) * (2.0 if ea else 1.0), 2),
             "rule": rule, "ea": ea, "spins": rng.random() < 0.25}
        c = _fit(lambda q: q["R"] * q["L"] ** q["dim"] * q["steps"] * q["theta"], 4e11, c, "R",
                 100)
        if c["R"] * c["L"] ** dim > 2e8:
            c["spins"] = False
        return c
    if kind == "batch":
        dim = rng.choice([2, 3])
        sides = sorted({_even(rng, 4, 12) if dim == 3 else _even(rng, 8, 40)
                        for _ in range(rng.choice([1, 2, 3]))})
        c = {"kind": "batch", "dim": dim, "sides": ",".join(map(str, sides)),
             "each": rng.randint(2, 12), "R": int(_log(rng, 500, 60000)), "steps": steps // 2 + 20,
             "theta": theta, "beta_f": round(rng.uniform(1.0, 3.0), 2), "rule": rule,
             "ea": rng.random() < 0.8}
        return _fit(lambda q: q["R"] * q["each"] * sum(s ** dim for s in sides) * q["steps"] *
                    q["theta"], 3e11, c, "R", 100)
    if kind == "weighted":
        c = {"kind": "weighted", "dim": 2, "L": rng.choice([16, 32, 64, _even(rng, 8, 48)]),
             "small": rng.randint(8, 96), "R_small": int(_log(rng, 500, 4000)),
             "large": rng.randint(1, 24), "R_large": int(_log(rng, 4000, 16000)),
             "steps": steps // 2 + 50, "theta": theta, "beta_f": 1.0, "rule": rule}
        return _fit(lambda q: (q["small"] * q["R_small"] + q["large"] * q["R_large"]) *
                    q["L"] ** 2 * q["steps"] * q["theta"], 3e11, c, "theta", 2)
    if kind == "learned":
        return {"kind": "learned", "dim": 2, "L": rng.choice([16, 32, 64]),
                "R": int(_log(rng, 1000, 20000)), "grid": rng.choice([400, 600, 800]),
                "budget": int(rng.uniform(500, 2500)), "beta_f": 1.0, "rule": "systematic"}
    if kind == "partial":
        return {"kind": "partial", "dim": 2, "L": rng.choice([16, 32, 64, _even(rng, 8, 64)]),
                "R": int(_log(rng, 1000, 30000)), "steps": steps // 2 + 50, "theta": theta,
                "beta_f": 1.0, "rule": rule, "alpha": rng.choice([0.2, 0.5, 0.9])}
    if kind == "overlap":
        return {"kind": "overlap", "dim": 2, "L": _even(rng, 8, 64), "pairs": rng.randint(1, 16),
                "R": int(_log(rng, 2000, 100000)), "steps": 10, "theta": 3,
                "beta_f": round(rng.uniform(1.0, 3.0), 2)}
    if kind == "weights":
        return {"kind": "weights", "dim": 2, "L": _even(rng, 16, 128),
                "R": int(_log(rng, 1000, 1000000)), "beta": round(rng.uniform(0.1, 0.8), 3),
                "dbeta": round(_log(rng, 0.001, 0.02), 4)}
    return {"kind": "mlp", "rows": int(_log(rng, 1000, 50000))}


# ---- inputs and handles ----------------------------------------------------------------------

def _runs(case, seed):
    """The run specifications of a batch case."""
    if case["kind"] == "weighted":
        R = [case["R_small"]] * case["small"] + [case["R_large"]] * case["large"]
        return [{"dim": case["dim"], "L": case["L"], "R": r, "ensemble": 0} for r in R]
    runs = []
    for k, L in enumerate(int(s) for s in case["sides"].split(",")):
        for m in range(case["each"]):
            cpl = ("ea", seed & 0xFFFF, 64 * k + m) if case["ea"] else ("ferro",)
            runs.append({"dim": case["dim"], "L": L, "R": case["R"], "couplings": cpl,
                         "ensemble": k})
    return runs


def _energies(case, seed):
    """Energies of a 2D ferromagnet population: a normal distribution about a mean between
    0 and the ground state, on the valid grid of 4."""
    N = case["L"] ** 2
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    b = case["beta"]
    mean, sd = -2.0 * N * math.tanh(1.6 * b), math.sqrt(N * (0.5 + b))
    z = torch.randn(case["R"], generator=g, device="cuda", dtype=torch.float64)
    return (4 * torch.round((mean + sd * z) / 4)).clamp_(-2 * N, 2 * N).to(torch.int32)


def _mlp_inputs(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    B = case["rows"]
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    uni = lambda *s: torch.rand(*s, generator=g, device="cuda")  # noqa: E731
    # features over the ranges of the traces: beta, <E>/N, var(E)/(10 N), 10 ln Q / N,
    # rho_t / R, family entropy, acceptance, L/64
    X = torch.stack([3 * uni(B), -2 * uni(B), 0.2 * uni(B), uni(B), 0.1 * uni(B), uni(B),
                     uni(B), torch.randint(1, 5, (B,), generator=g, device="cuda") / 4.0], 1)
    Yt = torch.stack([0.2 + 2 * uni(B), 0.5 + uni(B)], 1)
    mask = torch.ones(B, 2, device="cuda")
    w = torch.from_numpy(controller.init_params(seed % 1000)).cuda()
    m, v = 1e-3 * rnd(w.numel()), 1e-6 + 1e-4 * uni(w.numel())  # a run some way into training
    return X.contiguous(), Yt.contiguous(), mask, w, m, v


MLP_STEP, MLP_LR = 100, 3e-3


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed, "stream": torch.cuda.Stream()}
    if kind in ("run", "batch", "weighted", "partial", "overlap"):
        n = case["steps"]
        s["betas"] = np.linspace(0.0, case["beta_f"], n + 1)
        s["thetas"] = np.full(n, case["theta"], np.uint32)
    if kind in ("run", "partial"):
        s["couplings"] = ("ea", seed & 0xFFFF, 1) if case.get("ea") else ("ferro",)
    elif kind in ("batch", "weighted"):
        s["runs"] = _runs(case, seed)
    elif kind == "learned":
        s["betas"] = np.linspace(0.0, case["beta_f"], case["grid"] + 1)
        s["params"] = controller.load()
    elif kind == "overlap":
        runs = [{"dim": 2, "L": case["L"], "R": case["R"], "couplings": ("ea", seed & 0xFFFF, m)}
                for m in range(case["pairs"]) for _ in range(2)]
        s["batch"] = pa.Batch(runs, s["betas"], s["thetas"], "systematic", seed,
                              stream=s["stream"])
        s["batch"].step(case["steps"])
        pa.pa_sync(s["batch"].ctx)
        s["pairs"] = [(2 * m, 2 * m + 1) for m in range(case["pairs"])]
    elif kind == "weights":
        s["E"] = _energies(case, seed)
        s["lnQ"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        s["f"] = torch.zeros(case["R"], dtype=torch.int64, device="cuda")
    elif kind == "mlp":
        s["X"], s["Yt"], s["mask"], s["w"], s["m"], s["v"] = _mlp_inputs(case, seed)
        s["g"] = torch.zeros_like(s["w"])
        s["wbf"] = torch.zeros(s["w"].numel(), dtype=torch.int16, device="cuda")
        s["loss"] = torch.zeros(1, device="cuda")
        s["scratch"] = torch.empty(pa.pa_mlp_scratch_bytes(case["rows"]), dtype=torch.uint8,
                                   device="cuda")
    return s


# ---- one pass ----------------------------------------------------------------------------------

def _columns(rows):
    """A trace as one array per quantity."""
    return {k: np.array([r[k] for r in rows]) for k in rows[0] if k != "features"}


def _pad(a, rows):
    """Zero rows up to a fixed number: the population size of some rules and the number of
    steps of a learned schedule are themselves results."""
    out = np.zeros((rows,) + a.shape[1:], a.dtype)
    out[:len(a)] = a
    return out


def _population(p, spins):
    out = {"energies": _pad(p.energies(), p.R_cap), "families": _pad(p.families(), p.R_cap),
           "magnetisations": _pad(p.magnetisations(), p.R_cap)}
    if spins:
        out["spins"] = _pad(p.spins_words(), p.R_cap)
    return out


def run(s):
    return _RUN[s["case"]["kind"]](s["case"], s)


def _run_single(c, s):
    p = pa.Population(c["dim"], c["L"], c["R"], s["betas"], s["thetas"], c["rule"], s["seed"],
                      couplings=s["couplings"], stream=s["stream"])
    if c["kind"] == "partial":
        p.set_partial_resampling(c["alpha"])
    p.step(c["steps"])
    out = {"trace": _columns(p.trace()), "F": p.free_energy()}
    out.update(_population(p, c.get("spins", False)))
    if c["kind"] == "partial":
        out["weights"] = _pad(p.weights(), p.R_cap)
    p.close()
    return out


def _run_learned(c, s):
    p = controller.controlled_run(c["dim"], c["L"], ("ferro",), c["R"], s["betas"], 4, 10,
                                  s["params"], seed=s["seed"], budget=c["budget"],
                                  resampler=c["rule"], stream=s["stream"])
    controller.run_to_end(p)
    rows = p.trace()
    beta, theta = pa.pa_schedule_taken(p.ctx, p.n_steps + 1)
    n = p.n_steps + 1
    out = {"trace": {k: _pad(v, n) for k, v in _columns(rows).items()}, "F": p.free_energy(),
           "beta": _pad(beta, n), "theta": _pad(theta, n),
           "features": _pad(np.array([r["features"] for r in rows], np.float32), n)}
    out.update(_population(p, False))
    p.close()
    return out


def _run_batch(c, s):
    b = pa.Batch(s["runs"], s["betas"], s["thetas"], c["rule"], s["seed"], stream=s["stream"])
    b.step(c["steps"])
    if c["kind"] == "weighted":
        out = {"weighted": _columns(b.weighted(0))}
    else:  # every sample's averages and energies (ground-state search, histograms)
        M = len(s["runs"])
        out = {"last": _columns([b.observables(m) for m in range(M)]),
               "energies": np.concatenate([b.array(m, pa.PA_ARRAY_ENERGY) for m in range(M)])}
    b.close()
    return out


def _run_overlap(c, s):
    hist, P = s["batch"].overlap(s["pairs"])
    return {"hist": hist.view(np.int32), "P": P}


def _run_weights(c, s):
    pa.pa_weights_static(s["E"].data_ptr(), c["R"], c["R"], c["dim"], c["L"], 0, c["dbeta"],
                         s["lnQ"].data_ptr(), s["f"].data_ptr(),
                         torch.cuda.current_stream().cuda_stream)
    return {"lnQ": s["lnQ"], "f": s["f"]}


def _run_mlp(c, s):
    st = torch.cuda.current_stream().cuda_stream
    pa.pa_mlp_gradients(s["w"].data_ptr(), s["X"].data_ptr(), s["Yt"].data_ptr(),
                        s["mask"].data_ptr(), c["rows"], s["g"].data_ptr(), s["loss"].data_ptr(),
                        s["scratch"].data_ptr(), s["scratch"].numel(), st)
    pa.pa_mlp_adam(s["w"].data_ptr(), s["g"].data_ptr(), s["m"].data_ptr(), s["v"].data_ptr(),
                   s["wbf"].data_ptr(), MLP_STEP, MLP_LR, st)
    return {"loss": s["loss"], "grads": s["g"], "params": s["w"], "m": s["m"], "v": s["v"],
            "params_bf16": s["wbf"].view(torch.bfloat16)}


_RUN = {"run": _run_single, "partial": _run_single, "learned": _run_learned, "batch": _run_batch,
        "weighted": _run_batch, "overlap": _run_overlap, "weights": _run_weights,
        "mlp": _run_mlp}


# ---- what a pass cannot do without ---------------------------------------------------------------

def _anneal(dim, L, R, steps, sweeps):
    """Bytes and operations of annealing one population: every replica row is read and
    written once per temperature step, every spin update takes the Metropolis arithmetic."""
    N = L ** dim
    return 2.0 * N / 8 * R * steps, OPS_PER_UPDATE[dim] * N * R * sweeps


def work(case):
    kind = case["kind"]
    if kind in ("run", "partial"):
        b, f = _anneal(case["dim"], case["L"], case["R"], case["steps"],
                       case["steps"] * case["theta"])
    elif kind == "learned":
        b, f = _anneal(case["dim"], case["L"], case["R"], case["grid"] / 4, case["budget"])
    elif kind in ("batch", "weighted"):
        parts = [_anneal(r["dim"], r["L"], r["R"], case["steps"], case["steps"] * case["theta"])
                 for r in _runs(case, 0)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    elif kind == "overlap":
        rows = 2.0 * case["pairs"] * case["R"]
        b = rows * case["L"] ** 2 / 8 + 4.0 * case["pairs"] * (case["L"] ** 2 + 1)
        f = rows * case["L"] ** 2 / 32
    elif kind == "weights":
        b, f = 12.0 * case["R"], 2.0 * case["R"]
    else:
        B, P = case["rows"], pa.PA_MLP_NPARAM
        b, f = 4.0 * B * 12 + 4.0 * 8 * P, 6.0 * B * P
    return {"bytes": b, "flops": f}


# ---- values in 64 bits -----------------------------------------------------------------------------

def exact(case, seed):
    """lnQ of the weights call and the training iteration, in 64 bits.  A run's outputs are
    chains of random decisions (whole numbers, and sums of them) with no such values."""
    if case["kind"] == "weights":
        E = _energies(case, seed).to(torch.float64)
        x = -case["dbeta"] * E
        return {"lnQ": (torch.logsumexp(x, 0) - math.log(case["R"])).reshape(1), "f": None}
    if case["kind"] != "mlp":
        return None
    X, Yt, mask, w, m, v = (t.double() for t in _mlp_inputs(case, seed))
    wr = w.float().bfloat16().double().requires_grad_(True)  # the network runs on BF16 parameters
    parts, o = [], 0
    for shp in ((64, 8), (64,), (64, 64), (64,), (2, 64), (2,)):
        n = math.prod(shp)
        parts.append(wr[o:o + n].reshape(shp))
        o += n
    W1, b1, W2, b2, W3, b3 = parts
    Y = torch.relu(torch.relu(X @ W1.T + b1) @ W2.T + b2) @ W3.T + b3
    loss = (mask * (Y - Yt) ** 2).sum() / (2 * case["rows"])
    loss.backward()
    g = wr.grad
    m1, v1 = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    c1, c2 = 1 - 0.9 ** MLP_STEP, 1 - 0.999 ** MLP_STEP
    w1 = w - MLP_LR * (m1 / c1) / ((v1 / c2).sqrt() + 1e-8)
    return {"loss": loss.detach().reshape(1), "grads": g, "params": w1, "m": m1, "v": v1,
            "params_bf16": w1}
