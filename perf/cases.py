"""Performance cases: the work a user of this package has it do, through its
public entry points, from calls where launches and latency count to
populations that fill the GPU.

  run       one whole population-annealing run: a new population, its schedule
            (cooling from random spins, or heating from ground states), the
            estimators of every step, histograms, energies and spins
  step      two temperature steps of a live population (one up, one down, so
            that the same population serves any number of passes): resample,
            sweep, estimators with the histogram, then every replica's energy
            and occupation
  adaptive  a run with the overlap-controlled temperature steps
  batch     several independent runs advanced together
  lnq       ln Q(dbeta; E) with its first and second derivative by autograd
  mean      a reweighted observable with its gradients
  noalloc   resampling on the caller's device arrays
  spins     reading a population's configurations
"""
import math

import numpy as np
import torch

import paper_1704_01888_gb300 as pa
from paper_1704_01888_gb300 import autograd as ag
from paper_1704_01888_gb300.workloads import beta_t

_PREP_STEPS = 48  # steps that bring the population of a step or spins case to its temperature


def listed():
    return [
        # the smallest plain run: 1000 replicas of 16 x 16, 100 steps, where launches and latency count
        {"name": "run-small", "kind": "run", "q": 10, "L": 16, "R": 1000, "K": 100, "beta": 1.6, "theta": 10,
         "mode": 0, "heat": False, "families": False, "graph": False, "spins": True},
        # the heating branch of a hysteresis loop: ground states at beta = 3, steps of 0.01, one graph
        {"name": "run-heating", "kind": "run", "q": 6, "L": 32, "R": 10000, "K": 300, "beta": 3.0, "theta": 10,
         "mode": 0, "heat": True, "families": False, "graph": True, "spins": False},
        # a temperature step of the plain run at scale (the benchmark's workload), next to beta_t
        {"name": "step-scale", "kind": "step", "q": 10, "L": 64, "R": 100000, "beta": 1.424, "dbeta": 0.008,
         "theta": 10, "mode": 0, "families": False},
        # strong first order: the largest lattices, five planes, families tracked
        {"name": "step-strong", "kind": "step", "q": 20, "L": 256, "R": 20000, "beta": 1.697, "dbeta": 0.006,
         "theta": 20, "mode": 0, "families": True},
        # the paper's width tables: few replicas, many sweeps, a fine grid around beta_t
        {"name": "step-widths", "kind": "step", "q": 8, "L": 64, "R": 1000, "beta": 1.335, "dbeta": 0.001,
         "theta": 100, "mode": 0, "families": False},
        # rows that do not fill whole words, an odd population, the paper's Poisson copy numbers, families
        {"name": "step-ragged", "kind": "step", "q": 3, "L": 100, "R": 5003, "beta": 0.995, "dbeta": 0.01,
         "theta": 10, "mode": 2, "families": True},
        # adaptive steps from infinite temperature
        {"name": "adaptive", "kind": "adaptive", "q": 8, "L": 128, "R": 10000, "beta": 0.3, "theta": 10},
        # different q, L and sizes together
        {"name": "batch", "kind": "batch", "runs": 16, "R": 2000, "K": 40, "theta": 10},
        # the differentiable free energy of a large population
        {"name": "lnq-grad", "kind": "lnq", "L": 128, "R": 200000, "dbeta": 0.004},
        # a reweighted observable with gradients for every replica's value
        {"name": "mean-grad", "kind": "mean", "L": 64, "R": 100000, "dbeta": 0.008},
        # resampling for a host framework that owns the device memory
        {"name": "noalloc", "kind": "noalloc", "L": 64, "R": 100000, "dbeta": 0.008, "mode": 0},
        # configurations of a whole population (of fixed size: resampling off) for the user's own analysis
        {"name": "spins", "kind": "spins", "q": 10, "L": 64, "R": 4000, "beta": 1.424, "theta": 10, "mode": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _lattice(rng, lo=8, hi=256):
    if rng.random() < 0.6:
        return rng.choice([L for L in (8, 16, 32, 48, 64, 96, 128, 192, 256) if lo <= L <= hi])
    return 2 * _log_int(rng, lo // 2, hi // 2)


def _q(rng):
    return rng.choice((2, 3, 4, 5, 6, 8, 10, 10, 12, 20, 20, rng.randint(2, 40)))


def draw(rng):
    kind = rng.choice(("run", "run", "step", "step", "step", "step", "adaptive", "batch", "lnq", "mean", "noalloc",
                       "spins"))
    if kind in ("lnq", "mean"):
        return {"kind": kind, "L": _lattice(rng), "R": _log_int(rng, 1000, 200000),
                "dbeta": round(rng.choice((-1, 1, 1)) * rng.uniform(0.001, 0.01), 4)}
    if kind == "noalloc":
        return {"kind": kind, "L": _lattice(rng), "R": _log_int(rng, 1000, 200000),
                "dbeta": round(rng.uniform(0.001, 0.01), 4), "mode": rng.choice((0, 0, 1, 2))}
    if kind == "batch":
        return {"kind": kind, "runs": rng.randint(2, 24), "R": _log_int(rng, 500, 3000), "K": rng.randint(10, 40),
                "theta": rng.choice((5, 10, 20))}
    q, L, theta = _q(rng), _lattice(rng), rng.choice((5, 10, 10, 20, 50, 100))
    N = L * L
    if kind == "step":
        R = _log_int(rng, 500, max(501, min(100000, int(1e10 / (N * theta)))))
        return {"kind": kind, "q": q, "L": L, "R": R, "beta": round(beta_t(q) * rng.uniform(0.5, 1.1), 3),
                "dbeta": rng.choice((0.001, 0.004, 0.008)), "theta": theta, "mode": rng.choice((0, 0, 0, 2)),
                "families": rng.random() < 0.3}
    if kind == "spins":
        return {"kind": kind, "q": q, "L": L, "R": _log_int(rng, 10, max(11, min(4000, int(2e7 / N)))),
                "beta": round(beta_t(q) * rng.uniform(0.5, 1.1), 3), "theta": 5, "mode": 3}
    L = min(L, 128)
    N = L * L
    theta = min(theta, 20)
    if kind == "adaptive":
        return {"kind": kind, "q": q, "L": L, "R": _log_int(rng, 500, max(501, min(20000, int(1.6e8 / N)))),
                "beta": round(0.3 * beta_t(q) * rng.uniform(0.5, 1.0), 3), "theta": min(theta, 10)}
    K = rng.randint(20, 200)
    R = _log_int(rng, 500, max(501, min(20000, int(1e10 / (N * theta * K)))))
    heat = rng.random() < 0.3
    return {"kind": "run", "q": q, "L": L, "R": R, "K": K, "beta": 3.0 if heat else round(1.1 * beta_t(q), 3),
            "theta": theta, "mode": rng.choice((0, 0, 0, 2)), "heat": heat, "families": rng.random() < 0.3,
            "graph": rng.random() < 0.5, "spins": N * R <= 1000000}


def _params(case, seed, **more):
    return pa.PAParams(q=case["q"], L=case["L"], R=case["R"], seed=int(seed), resample_mode=case.get("mode", 0),
                       track_families=case.get("families", False), **more)


def _betas(case):
    b = np.array([case["beta"] * i / case["K"] for i in range(case["K"] + 1)])
    return b[::-1].copy() if case["heat"] else b


def _energies(case, seed):
    """Energies of a population in one phase near the transition: about -1.2
    per site, a spread of 0.8 sqrt(N), whole numbers in [-2N, 0]."""
    N = case["L"] ** 2
    g = torch.Generator().manual_seed(int(seed))
    e = torch.randn(case["R"], generator=g, dtype=torch.float64) * (0.8 * math.sqrt(N)) - 1.2 * N
    return e.round().clamp(-2 * N, 0).to(torch.int32)


def _observable(case, seed):
    g = torch.Generator().manual_seed(int(seed) + 1)
    return 0.5 + 0.1 * torch.randn(case["R"], generator=g, dtype=torch.float64)


def _batch_runs(case, seed):
    """Runs over q in {5, 6, 8, 10} and L in {16, 32, 48, 64}, each with its own size and schedule."""
    runs = []
    for m in range(case["runs"]):
        q, L = (5, 6, 8, 10)[m % 4], (16, 32, 48, 64)[(m // 4) % 4]
        R = case["R"] + (m * 389) % case["R"]
        betas = np.array([1.1 * beta_t(q) * i / case["K"] for i in range(case["K"] + 1)])
        runs.append((pa.PAParams(q=q, L=L, R=R, seed=int(seed), stream=m), betas, case["theta"]))
    return runs


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "run":
        s["params"] = _params(case, seed, init_mode=pa.INIT_GROUND if case["heat"] else pa.INIT_RANDOM,
                              beta0=case["beta"] if case["heat"] else 0.0)
        s["betas"] = _betas(case)
    elif kind in ("step", "spins"):
        s["pop"] = pa.Population(_params(case, seed))
        s["pop"].run(np.array([case["beta"] * i / _PREP_STEPS for i in range(_PREP_STEPS + 1)]),
                     min(case["theta"], 10))
    elif kind == "adaptive":
        s["params"] = _params(case, seed)
    elif kind == "batch":
        s["runs"] = _batch_runs(case, seed)
    elif kind in ("lnq", "mean"):
        s["E"] = _energies(case, seed).cuda()
        s["dbeta"] = torch.tensor(case["dbeta"], dtype=torch.float64, device="cuda")
        if kind == "mean":
            s["O"] = _observable(case, seed).cuda()
    else:
        s["E"] = _energies(case, seed).cuda()
        s["parent"] = torch.zeros(case["R"] + case["R"] // 4 + 1024, dtype=torch.int32, device="cuda")
        s["lnQ"] = torch.zeros(1, dtype=torch.float64, device="cuda")
        s["R"] = torch.zeros(1, dtype=torch.int32, device="cuda")
        s["seed"] = int(seed)
    return s


_WHOLE = ("R", "n_families", "sumE", "sumE2", "sumMt", "n_near_ties")
_FLOAT = ("beta", "lnQ", "lnZ", "meanE", "meanE2", "C", "meanM", "S_f")


def _columns(obs):
    """Estimators of several steps: one array of the whole numbers, one of the others."""
    return (np.array([[o[k] for k in _WHOLE] for o in obs], dtype=np.int64),
            np.array([[o[k] for k in _FLOAT] for o in obs], dtype=np.float64))


def _padded(a, rows):
    """a in an array of `rows` rows, zeros after its own: a population's size
    and the number of adaptive steps differ from seed to seed."""
    out = np.zeros((rows,) + a.shape[1:], dtype=a.dtype)
    out[: len(a)] = a
    return out


def run(state):
    case, kind = state["case"], state["kind"]
    cap = case["R"] + case["R"] // 4 + 1024
    if kind == "run":
        K = case["K"]
        with pa.Population(state["params"]) as pop:
            obs, hists = pop.run(state["betas"], case["theta"], hist_steps=(K // 2, K), use_graph=case["graph"])
            out = {"obs": _columns(obs), "hists": hists, "E": _padded(pop.energies(), cap)}
            if case["spins"]:
                out["spins"] = _padded(pop.spins(), cap)
        return out
    if kind == "step":
        pop, obs, hists = state["pop"], [], []
        for beta, dbeta in ((case["beta"] + case["dbeta"], case["dbeta"]), (case["beta"], -case["dbeta"])):
            pop.resample(dbeta)
            pop.sweep(beta, case["theta"])
            o, h = pop.observables(with_hist=True)
            obs.append(o)
            hists.append(h)
        out = {"obs": _columns(obs), "hists": hists, "E": _padded(pop.energies(), cap),
               "Mt": _padded(pop.occupations(), cap)}
        if case["families"]:
            out["families"] = _padded(pop.ancestors(), cap)
        return out
    if kind == "adaptive":
        with pa.Population(state["params"]) as pop:
            obs, betas = pop.run_adaptive(case["beta"], case["theta"], max_steps=400)
            return {"obs": [_padded(c, 400) for c in _columns(obs)], "betas": _padded(betas, 400),
                    "E": _padded(pop.energies(), cap)}
    if kind == "batch":
        with pa.Batch(state["runs"]) as b:
            b.run()
            M = len(state["runs"])
            obs = [_columns(b.observables(m)) for m in range(M)]
            return {"whole": np.concatenate([o[0] for o in obs]), "obs": np.concatenate([o[1] for o in obs]),
                    "E": _padded(np.concatenate([np.stack(b.measurements(m), axis=1) for m in range(M)]),
                                 sum(p.R + p.R // 4 + 1024 for p, _, _ in state["runs"]))}
    if kind == "lnq":
        d = state["dbeta"].detach().requires_grad_()
        y = ag.lnQ(d, state["E"])
        (g1,) = torch.autograd.grad(y, d, create_graph=True)
        (g2,) = torch.autograd.grad(g1, d)
        return [y, g1, g2]
    if kind == "mean":
        d = state["dbeta"].detach().requires_grad_()
        O = state["O"].detach().requires_grad_()
        y = ag.reweighted_mean(O, d, state["E"])
        y.backward()
        return [y, O.grad, d.grad]
    if kind == "noalloc":
        E, parent = state["E"], state["parent"]
        pa.resample_noalloc(E.data_ptr(), E.numel(), case["L"], case["dbeta"], case["R"], case["mode"], 7,
                            state["seed"], parent.data_ptr(), parent.numel(), state["lnQ"].data_ptr(),
                            state["R"].data_ptr(), torch.cuda.current_stream().cuda_stream)
        return [parent, state["lnQ"], state["R"]]
    return state["pop"].spins()


def _replica_bytes(q, L):
    """One replica's states at ceil(log2 q) bits per site."""
    return L * L * max(1, math.ceil(math.log2(q))) / 8


def _sweeps(q, L, R, theta, steps):
    """Bytes and integer operations of `steps` temperature steps: each replica
    read and written once per step, its energy and occupation written; about
    5 lane operations per attempt (32 sites per word operation) -- the random
    bits, the proposal, the energy change and the acceptance -- and 3 per site
    measured."""
    return (steps * R * (2 * _replica_bytes(q, L) + 8), steps * R * L * L * (5 * theta + 3))


def work(case):
    kind = case["kind"]
    R = case["R"]
    if kind == "run":
        b, f = _sweeps(case["q"], case["L"], R, case["theta"], case["K"])
        b += R * _replica_bytes(case["q"], case["L"])  # the initial population
        f += R * case["L"] ** 2 * 12  # one Philox word per initial spin
        b += R * case["L"] ** 2 if case["spins"] else 0
    elif kind == "step":
        b, f = _sweeps(case["q"], case["L"], R, case["theta"], 2)
    elif kind == "adaptive":
        # the overlap 0.85 fixes dbeta sigma_E: about 0.4, sigma_E^2 = 2N (1/q)(1 - 1/q) at beta = 0
        sigma = math.sqrt(2 * case["L"] ** 2 * (1 - 1 / case["q"]) / case["q"])
        steps = max(1, math.ceil(case["beta"] * sigma / 0.4), math.ceil(case["beta"] / 0.05))
        b, f = _sweeps(case["q"], case["L"], R, case["theta"], steps)
    elif kind == "batch":
        b = f = 0.0
        for p, betas, theta in _batch_runs(case, 0):
            x, y = _sweeps(p.q, p.L, p.R, theta, betas.size - 1)
            b, f = b + x, f + y
    elif kind == "lnq":
        b, f = 4 * R, 30 * R
    elif kind == "mean":
        b, f = 4 * R + 8 * R + 8 * R, 40 * R
    elif kind == "noalloc":
        b, f = 4 * R + 4 * R, 60 * R
    else:
        b, f = R * (_replica_bytes(case["q"], case["L"]) + case["L"] ** 2), R * case["L"] ** 2
    return {"bytes": float(b), "flops": float(f)}


def exact(case, seed):
    """Reweighting in 64 bits about the lowest (dbeta >= 0) or highest energy;
    the trajectories of the other cases have no closed value."""
    if case["kind"] not in ("lnq", "mean", "noalloc"):
        return None
    E = _energies(case, seed).numpy().astype(np.float64)
    d = case["dbeta"]
    ref = E.min() if d >= 0 else E.max()
    w = np.exp(-d * (E - ref))
    S = math.fsum(w)
    lnq = -d * ref + math.log(S / E.size)
    if case["kind"] == "noalloc":
        return [None, np.array([lnq]), None]
    m1 = math.fsum(w * (E - ref)) / S
    if case["kind"] == "lnq":
        var = math.fsum(w * (E - ref - m1) ** 2) / S
        return [np.float64(lnq), np.float64(-(ref + m1)), np.float64(var)]
    O = _observable(case, seed).numpy()
    mO = math.fsum(w * O) / S
    cov = math.fsum(w * (O - mO) * (E - ref - m1)) / S
    return [np.float64(mO), w / S, np.float64(-cov)]
