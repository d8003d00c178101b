"""Timed cases of the library: what a user's program has it do, through the public binding.

Every case names a ``kind`` (the entry points it goes through) and its sizes:

* ``series``   Metropolis sweeps of small lattices with E and M after every sweep;
* ``sweeps``   one large lattice: a block of sweeps, then E and M (int8 or bit-packed
  layout; ``series`` true: E and M after every sweep of the block);
* ``pa``       a whole population annealing run with a fixed schedule, one lattice
  or a batch of up to three sizes, with each resampling law;
* ``bisect``   a whole annealing run whose temperature steps the library chooses;
* ``pt``       a block of parallel-tempering rounds;
* ``sw``       a block of Swendsen-Wang updates with E and M after each;
* ``mlp``      a minibatch gradient of the schedule network and a batch of proposals.

Outputs are the configurations, energies, magnetisations, statistics and gradients
themselves. All random numbers come from the seed, so a pass is reproducible.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1709_04394_gb300 import gbmc as g

BETA_C = 0.5 * math.log(1.0 + math.sqrt(2.0))
MLP_IN, MLP_HIDDEN = 6, 64


def listed():
    return [
        # validation run of the 2D critical point: one small lattice, E and M after every
        # sweep (the shortest chain of dependent work a user waits for)
        {"name": "series-2d-L16", "kind": "series", "dim": 2, "L": 16, "copies": 1, "sweeps": 2000, "model": "fm"},
        # the headline workload: population annealing of the 2D Ising model
        {"name": "pa-2d-L64", "kind": "pa", "dim": 2, "model": "fm", "L": 64, "R": 100000, "L2": 0, "R2": 0,
         "L3": 0, "R3": 0, "instances": 1, "theta": 10, "steps": 100, "beta_f": 1.0, "law": "multinomial"},
        # spin-glass study: a disorder average at one of the sizes 4, 6, 8, 10, 12 such work uses
        {"name": "pa-3d-ea-L10", "kind": "pa", "dim": 3, "model": "ea", "L": 10, "R": 5000, "L2": 0, "R2": 0,
         "L3": 0, "R3": 0, "instances": 8, "theta": 10, "steps": 30, "beta_f": 3.0, "law": "multinomial"},
        # finite-size scaling: sizes between the powers of two annealed together
        {"name": "pa-2d-mixed", "kind": "pa", "dim": 2, "model": "fm", "L": 24, "R": 20000, "L2": 40, "R2": 10000,
         "L3": 96, "R3": 4000, "instances": 1, "theta": 10, "steps": 20, "beta_f": 0.6, "law": "multinomial"},
        # a small variable population (a pilot run): many short steps, bound by latency and launches
        {"name": "pa-2d-pilot", "kind": "pa", "dim": 2, "model": "fm", "L": 32, "R": 1100, "L2": 0, "R2": 0,
         "L3": 0, "R3": 0, "instances": 1, "theta": 10, "steps": 50, "beta_f": 0.8, "law": "nearest"},
        # adaptive temperature steps by histogram overlap
        {"name": "bisect-2d-L64", "kind": "bisect", "L": 64, "R": 4000, "theta": 10, "beta_f": 0.5},
        # parallel tempering of the 3D spin glass, 32 temperatures per disorder instance
        {"name": "pt-3d-ea-L8", "kind": "pt", "dim": 3, "model": "ea", "L": 8, "instances": 128, "temps": 32,
         "theta": 10, "rounds": 20},
        # one large lattice in the int8 layout, measured every 100 sweeps
        {"name": "sweeps-2d-L4096", "kind": "sweeps", "dim": 2, "model": "fm", "L": 4096, "copies": 1, "sweeps": 100,
         "layout": "int8", "series": False},
        # a large lattice whose size is no power of two
        {"name": "sweeps-2d-L1000", "kind": "sweeps", "dim": 2, "model": "fm", "L": 1000, "copies": 1, "sweeps": 100,
         "layout": "int8", "series": False},
        # the bit-packed layout with time series (autocorrelation measurements)
        {"name": "bitpack-2d-L2048", "kind": "sweeps", "dim": 2, "model": "fm", "L": 2048, "copies": 1, "sweeps": 50,
         "layout": "bitpack", "series": True},
        # cluster updates at the critical point
        {"name": "sw-2d-L1024", "kind": "sw", "dim": 2, "L": 1024, "copies": 1, "updates": 10},
        # the schedule network: one training minibatch, one batch of proposals
        {"name": "mlp-batch", "kind": "mlp", "batch": 128, "points": 1517},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(rng, lo, hi):
    return 2 * max(1, _log_int(rng, lo // 2, hi // 2))


def draw(rng):
    kind = rng.choice(["series", "pa", "pa", "pa", "pa-mixed", "bisect", "pt", "sweeps", "sweeps", "bitpack", "sw", "mlp"])
    if kind == "series":
        dim = rng.choice([2, 2, 3])
        L = _even(rng, 8, 64) if dim == 2 else _even(rng, 4, 16)
        return {"kind": "series", "dim": dim, "L": L, "copies": _log_int(rng, 1, 64), "sweeps": _log_int(rng, 200, 2000),
                "model": rng.choice(["fm", "ea"]) if dim == 3 else "fm"}
    if kind in ("pa", "pa-mixed"):
        dim = 2 if kind == "pa-mixed" else rng.choice([2, 3])
        theta, steps = rng.randint(3, 10), rng.randint(10, 50)
        case = {"kind": "pa", "dim": dim, "model": "fm", "L2": 0, "R2": 0, "L3": 0, "R3": 0, "instances": 1,
                "theta": theta, "steps": steps, "beta_f": round(rng.uniform(0.4, 1.0), 3),
                "law": rng.choice(["multinomial", "nearest", "poisson"])}
        if dim == 3:
            case.update(model=rng.choice(["ea", "ea", "fm"]), L=_even(rng, 4, 16), instances=_log_int(rng, 1, 32),
                        beta_f=round(rng.uniform(0.5, 3.0), 3))
        else:
            case["L"] = _even(rng, 8, 128)
        # up to about 4e9 site updates in all, a tenth of the largest listed run
        most = 4e9 / (theta * steps * case["instances"] * case["L"] ** dim)
        case["R"] = max(200, min(100000, _log_int(rng, 200, max(201, most))))
        if kind == "pa-mixed":
            case.update(law="multinomial", L2=_even(rng, 8, 128), L3=_even(rng, 8, 128), R2=_log_int(rng, 200, 4000),
                        R3=_log_int(rng, 200, 4000))
        return case
    if kind == "bisect":
        return {"kind": "bisect", "L": _even(rng, 16, 96), "R": _log_int(rng, 1000, 10000), "theta": rng.randint(3, 10),
                "beta_f": round(rng.uniform(0.3, 0.5), 3)}
    if kind == "pt":
        return {"kind": "pt", "dim": 3, "model": rng.choice(["ea", "ea", "fm"]), "L": _even(rng, 4, 12),
                "instances": _log_int(rng, 1, 256), "temps": rng.randint(8, 40), "theta": rng.randint(1, 10),
                "rounds": rng.randint(5, 40)}
    if kind == "sweeps":
        dim = rng.choice([2, 2, 3])
        # 2D sizes above the shared-memory ones, multiples of 8 and others; 3D from 18
        L = rng.choice([8 * _log_int(rng, 33, 512), _even(rng, 258, 2048)]) if dim == 2 else _even(rng, 18, 96)
        return {"kind": "sweeps", "dim": dim, "model": rng.choice(["fm", "ea"]) if dim == 3 else "fm", "L": L,
                "copies": rng.choice([1, 1, 1, rng.randint(2, 8)]), "sweeps": _log_int(rng, 10, 100), "layout": "int8",
                "series": rng.random() < 0.3}
    if kind == "bitpack":
        return {"kind": "sweeps", "dim": 2, "model": "fm", "L": 64 * _log_int(rng, 4, 64), "copies": rng.choice([1, 1, rng.randint(2, 4)]),
                "sweeps": _log_int(rng, 10, 100), "layout": "bitpack", "series": rng.random() < 0.5}
    if kind == "sw":
        dim = rng.choice([2, 2, 3])
        L = _even(rng, 16, 1024) if dim == 2 else _even(rng, 8, 64)
        return {"kind": "sw", "dim": dim, "L": L, "copies": max(1, min(256, _log_int(rng, 1, max(2, 2e6 / L**dim)))),
                "updates": rng.randint(2, 20)}
    return {"kind": "mlp", "batch": _log_int(rng, 8, 128), "points": _log_int(rng, 1, 4096)}


class _State:
    """The handles and buffers a user's program keeps; released with the object."""

    def __init__(self, case):
        self.case = case
        self.ctx = g.gbmc_create(0, torch.cuda.current_stream().cuda_stream)
        self.lattices, self.spins = [], []
        self.pa = self.pt = None

    def lattice(self, dim, L, copies, seed, instances=1, model="fm", layout="int8"):
        per_byte = 8 if layout == "bitpack" else 1
        buf = torch.empty(instances * copies * L**dim // per_byte, dtype=torch.int8, device="cuda")
        self.lattices.append(g.lattice_init(
            self.ctx, dim, L, model=g.GBMC_EA_PMJ if model == "ea" else g.GBMC_ISING_FM, start=g.GBMC_START_RANDOM,
            n_instances=instances, n_replicas=copies, seed=seed + 1,
            layout=g.GBMC_BITPACK if layout == "bitpack" else g.GBMC_INT8, spins=buf))
        self.spins.append(buf)
        return self.lattices[-1]

    def __del__(self):
        if self.pa is not None:
            g.pa_free(self.pa)
        if self.pt is not None:
            g.pt_free(self.pt)
        torch.cuda.synchronize()
        for lat in self.lattices:
            g.lattice_free(lat)
        g.gbmc_destroy(self.ctx)


def _ints(*shape):
    return torch.zeros(*shape, dtype=torch.int32, device="cuda")


def prepare(case, seed):
    s = _State(case)
    kind = case["kind"]
    if kind == "series":
        s.lattice(case["dim"], case["L"], case["copies"], seed, model=case["model"])
        s.E, s.M = _ints(case["sweeps"], case["copies"]), _ints(case["sweeps"], case["copies"])
    elif kind == "sweeps":
        s.lattice(case["dim"], case["L"], case["copies"], seed, model=case["model"], layout=case["layout"])
        rows = case["sweeps"] if case["series"] else 1
        s.E, s.M = _ints(rows, case["copies"]), _ints(rows, case["copies"])
    elif kind == "pa":
        nearest = case["law"] != "multinomial"
        for k in ("", "2", "3"):
            if case["L" + k]:
                s.lattice(case["dim"], case["L" + k], case["R" + k], seed + 101 * len(s.lattices), model=case["model"],
                          instances=case["instances"])
        s.seed = seed + 1
        laws = {"multinomial": g.GBMC_RESAMPLE_MULTINOMIAL, "nearest": g.GBMC_RESAMPLE_NEAREST,
                "poisson": g.GBMC_RESAMPLE_POISSON}
        # variable populations: R slots, an expected population a good five sigma below
        start = max(1, int(case["R"] - 8 * math.sqrt(case["R"]))) if nearest else 0
        s.pa = g.pa_create(s.ctx, s.lattices, case["theta"], case["steps"], beta_f=case["beta_f"],
                           resample=laws[case["law"]], initial_replicas=start)
    elif kind == "bisect":
        s.lattice(2, case["L"], case["R"], seed)
        s.seed = seed + 1
        s.pa = g.pa_create(s.ctx, s.lattices, case["theta"], 4096, schedule=g.GBMC_SCHED_BISECTION, beta_f=case["beta_f"])
    elif kind == "pt":
        s.lattice(case["dim"], case["L"], case["temps"], seed, instances=case["instances"], model=case["model"])
        betas = np.geomspace(0.2, 3.0 if case["model"] == "ea" else 0.5, case["temps"])
        s.pt = g.pt_create(s.ctx, s.lattices[0], betas, case["theta"])
        s.E, s.rep = _ints(case["instances"], case["temps"]), _ints(case["instances"], case["temps"])
    elif kind == "sw":
        s.lattice(case["dim"], case["L"], case["copies"], seed)
        # towards equilibrium first: a random start has no clusters worth the name
        g.metropolis_sweeps(s.ctx, s.lattices[0], _sw_beta(case), 20)
        s.E, s.M = _ints(case["updates"], case["copies"]), _ints(case["updates"], case["copies"])
    elif kind == "mlp":
        p, X, T = _mlp_inputs(case, seed)
        s.params, s.X, s.T = p.float().cuda(), X.float().cuda(), T.float().cuda()
        s.grad = torch.zeros(p.numel(), device="cuda")
        s.loss = torch.zeros(1, device="cuda")
        s.Y = torch.zeros(case["points"], device="cuda")
    else:
        raise ValueError("unknown kind %r" % kind)
    return s


def _sw_beta(case):
    return BETA_C if case["dim"] == 2 else 0.2216546


def _beta(case):
    """Temperatures of the plain sweeps: the ferromagnets' critical points, the spin glass below its own."""
    return 1.0 if case["model"] == "ea" else _sw_beta(case)


def run(s):
    case = s.case
    kind = case["kind"]
    if kind == "series":
        g.metropolis_sweeps(s.ctx, s.lattices[0], _beta(case), case["sweeps"], s.E, s.M)
        return {"spins": s.spins[0], "E": s.E, "M": s.M}
    if kind == "sweeps":
        if case["series"]:
            g.metropolis_sweeps(s.ctx, s.lattices[0], _beta(case), case["sweeps"], s.E, s.M)
        else:
            g.metropolis_sweeps(s.ctx, s.lattices[0], _beta(case), case["sweeps"])
            g.observables(s.ctx, s.lattices[0], s.E, s.M)
        return {"spins": s.spins[0], "E": s.E, "M": s.M}
    if kind in ("pa", "bisect"):
        g.pa_reset(s.ctx, s.pa, init=True, seed=s.seed)
        stats, steps = g.pa_run(s.ctx, s.pa, capacity=(case["steps"] if kind == "pa" else 4096) + 1)
        out = {"steps": steps, "betas": g.pa_betas(s.pa)}
        for name in g.PA_STATS_DTYPE.names:
            if name != "pad":
                out[name] = np.ascontiguousarray(stats[name])
        copies = case["R"] * case.get("instances", 1)
        out["E"], out["M"] = _ints(copies), _ints(copies)
        g.pa_energies_out(s.ctx, s.pa, 0, out["E"], out["M"])
        for i, lat in enumerate(s.lattices):
            out["spins%d" % i] = torch.empty_like(s.spins[i])
            g.lattice_copy_out(s.ctx, lat, out["spins%d" % i])
        if case.get("law", "multinomial") != "multinomial":  # slots beyond the population hold nothing
            for k in ("E", "M", "spins0"):
                for population, live in zip(out[k].view(case["instances"], case["R"], -1), stats["n_replicas"][-1]):
                    population[int(live):] = 0
        return out
    if kind == "pt":
        g.pt_step(s.ctx, s.pt, case["rounds"])
        g.pt_state_out(s.ctx, s.pt, rep_of=s.rep, E=s.E)
        return {"spins": s.spins[0], "rep": s.rep, "E": s.E}
    if kind == "sw":
        g.swendsen_wang(s.ctx, s.lattices[0], _sw_beta(case), case["updates"], s.E, s.M)
        return {"spins": s.spins[0], "E": s.E, "M": s.M}
    g.mlp_grad(s.ctx, s.params, s.X[: case["batch"]], s.T[: case["batch"]], s.grad, s.loss)
    g.mlp_forward(s.ctx, s.params, s.X[: case["points"]], s.Y)
    return {"grad": s.grad, "loss": s.loss, "Y": s.Y}


def work(case):
    """Bytes: each configuration read and written once, results written once. Operations: a
    quarter of a Philox4x32-10 call (20 integer operations) per site update or, for cluster
    updates, two thirds of one per bond and site; multiply-adds of the network."""
    kind = case["kind"]
    if kind == "mlp":
        n = MLP_IN * MLP_HIDDEN + MLP_HIDDEN * MLP_HIDDEN + MLP_HIDDEN
        params = n + 2 * MLP_HIDDEN + 1
        return {"bytes": 4 * (2 * params + 1 + (MLP_IN + 1) * (case["batch"] + case["points"])),
                "flops": 2 * n * (3 * case["batch"] + case["points"])}
    if kind in ("pa", "bisect"):
        sites = sum(case.get("L" + k, 0) ** case.get("dim", 2) * case.get("R" + k, 0) for k in ("", "2", "3"))
        sites *= case.get("instances", 1)
        steps = case.get("steps", 50)
        return {"bytes": sites * (1 + 2 * steps), "flops": 20 * sites * case["theta"] * steps}
    copies = case["instances"] * case["temps"] if kind == "pt" else case["copies"]
    sites = copies * case["L"] ** case["dim"]
    n = {"series": "sweeps", "sweeps": "sweeps", "pt": "rounds", "sw": "updates"}[kind]
    n = case[n]
    if kind == "pt":
        n *= case["theta"]
    moved = sites // (8 if case.get("layout") == "bitpack" else 1)
    if kind == "sw":
        return {"bytes": 2 * moved + 8 * copies * n, "flops": 20 * case["dim"] * sites * n}
    return {"bytes": 2 * moved + (8 * copies * n if kind == "series" or case.get("series") else 8 * copies),
            "flops": 20 * sites * n}


# ---- the schedule network in 64 bits ----


def _mlp_inputs(case, seed):
    """Parameters as after a short training, inputs with the spread of real schedule features."""
    gen = torch.Generator().manual_seed(seed)
    H = MLP_HIDDEN
    def uniform(n, fan):
        return (torch.rand(n, generator=gen, dtype=torch.float64) * 2 - 1) / math.sqrt(fan)
    p = torch.cat([uniform(H * MLP_IN, MLP_IN), uniform(H, MLP_IN), uniform(H * H, H), uniform(H, H), uniform(H, H),
                   uniform(1, H)])
    n = max(case["batch"], case["points"])
    lo = torch.tensor([-1.9, -2.0, -1.0, 0.0, 3.4, 6.9], dtype=torch.float64)
    hi = torch.tensor([-0.1, 1.5, 1.0, 1.0, 5.6, 11.5], dtype=torch.float64)
    X = lo + (hi - lo) * torch.rand(n, MLP_IN, generator=gen, dtype=torch.float64)
    T = -0.7 + 0.3 * torch.randn(n, generator=gen, dtype=torch.float64)
    return p.float().double(), X.float().double(), T.float().double()


def exact(case, seed):
    """The network's gradient, loss and outputs in 64 bits (weights rounded to bf16, as the network
    defines them). The other kinds return whole numbers, and statistics of them after a random walk
    of integers that plain code could only repeat word for word: none."""
    if case["kind"] != "mlp":
        return None
    p, X, T = _mlp_inputs(case, seed)
    H = MLP_HIDDEN
    w = p.float().bfloat16().double().requires_grad_()
    at = np.cumsum([0, H * MLP_IN, H, H * H, H, H, 1])
    W1, b1, W2, b2, W3, b3 = (w[a:b] for a, b in zip(at[:-1], at[1:]))

    def net(x):
        h1 = torch.tanh(x @ W1.view(H, MLP_IN).T + b1)
        h2 = torch.tanh(h1 @ W2.view(H, H).T + b2)
        return h2 @ W3 + b3

    B = case["batch"]
    loss = 0.5 * ((net(X[:B]) - T[:B]) ** 2).mean()
    (grad,) = torch.autograd.grad(loss, w)
    with torch.no_grad():
        Y = net(X[: case["points"]])
    return {"grad": grad, "loss": loss.detach().reshape(1), "Y": Y}
