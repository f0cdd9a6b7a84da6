"""The work a user of this library has it do, as measurable cases.

A case is a dict of plain values; ``kind`` names the entry point it goes through
(an SA sample, a whole multi-start solve, an SQA or PTICM sample, the
persistence pass, the request server) and the rest are its sizes and options.
Problem classes and sizes are the ones the benchmark and the tests use (3D +-J
lattices, Chimera, weak-strong Chimera, the U_10 class), and a 3D lattice with
Gaussian couplers stored as integers, which is how a real-valued problem is
passed.  Every output of the library is a whole number.
"""
import math
import random

import numpy as np
import torch

from paper_1706_07826_gb300 import instances, spvar


# ------------------------------------------------------------------ cases
def listed():
    return [
        # a first look at a small problem: one short anneal, where launch and latency are all there is
        dict(name="sample_l4", kind="sample", problem="cubic", size=4, samples=64, sweeps=100),
        # a sample of the largest served size, as a user with their own outer loop draws it
        dict(name="sample_l20", kind="sample", problem="cubic", size=20, samples=1000, sweeps=1000),
        # small integer couplers with biases (reduced degeneracy, U_10) on a full Chimera C8
        dict(name="sample_u10_c8", kind="sample", problem="u10", size=8, samples=2000, sweeps=1000),
        # a real-valued (Gaussian) lattice, scaled to integers: general couplers, odd size
        dict(name="sample_gauss_l9", kind="sample", problem="gauss100", size=9, samples=1000, sweeps=1000),
        # the benchmark's headline as its users call it: edge list in, host arrays out
        dict(name="solve_chimera_c8", kind="solve", problem="chimera", size=8, starts=10, fixing=1000, solving=1000,
             sweeps=1000, elite=0.1),
        # weak-strong clusters on Chimera C12: one large coupler magnitude, biases, a tiny solving phase
        dict(name="plan_weak_strong_c12", kind="plan", problem="weak_strong", size=12, starts=32, fixing=250,
             solving=250, sweeps=1000, elite=0.2),
        # a batch of 64 lattices of uneven size (L 6 .. 12) in one plan: the largest amount of work
        dict(name="plan_uneven_3d", kind="batch", problem="cubic", size=12, count=64, starts=1, fixing=2000,
             solving=2000, sweeps=1000, elite=0.1),
        # ISPVAR to exhaustion on L = 4: many short dependent phases
        dict(name="plan_ispvar_l4", kind="plan", problem="cubic", size=4, starts=1, fixing=256, solving=256,
             sweeps=1000, elite=0.2, phases=16),
        # the second sampler in every phase of the multi-start loop
        dict(name="plan_sqa_c8", kind="sqa", problem="chimera", size=8, starts=10, fixing=500, solving=500,
             sweeps=500, slices=16, elite=0.1),
        # the third sampler on its own: one run per resident block, 32 temperatures
        dict(name="pticm_l10", kind="pticm", problem="cubic", size=10, runs=304, temps=32, sweeps=500, keep=10),
        # Alg. 1 by hand on an existing sample: elite, counts, fixings, reduced problem
        dict(name="persistence_l20", kind="reduce", problem="cubic", size=20, samples=2000, elite=0.1, noalloc=False),
        # requests of mixed size submitted together to the server and stepped until all are done
        dict(name="serve_l8_l20", kind="serve", problem="cubic", size=20, small=8, count=6, starts=20, fixing=250,
             solving=250, sweeps=1000, step=500, elite=0.2),
    ]


def _log_int(rng, lo, hi):
    """A whole number spread over [lo, hi] by its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["sample", "sample", "sample", "solve", "plan", "plan", "batch", "sqa", "pticm", "reduce",
                       "serve"])
    if kind == "sample":
        problem = rng.choice(["cubic", "cubic", "chimera", "u10", "gauss10", "gauss100", "weak_strong"])
        size = rng.randint(4, 20) if problem == "cubic" else rng.randint(4, 12)
        return dict(kind=kind, problem=problem, size=size, samples=_log_int(rng, 30, 2000),
                    sweeps=_log_int(rng, 100, 1000))
    if kind in ("solve", "plan"):
        problem = rng.choice(["cubic", "chimera", "weak_strong", "u10"])
        phases = rng.choice([1, 1, 1, 8])
        return dict(kind=kind, problem=problem, size=rng.randint(4, 12), starts=_log_int(rng, 1, 40),
                    fixing=_log_int(rng, 50, 1000), solving=_log_int(rng, 50, 1000), sweeps=_log_int(rng, 100, 1000),
                    elite=rng.choice([0.1, 0.2]), phases=phases)
    if kind == "batch":
        return dict(kind=kind, problem="cubic", size=rng.randint(8, 12), count=_log_int(rng, 4, 64),
                    starts=rng.randint(1, 2), fixing=_log_int(rng, 100, 1000), solving=_log_int(rng, 100, 1000),
                    sweeps=_log_int(rng, 100, 1000), elite=rng.choice([0.1, 0.2]))
    if kind == "sqa":
        return dict(kind=kind, problem=rng.choice(["chimera", "cubic"]), size=rng.randint(4, 8),
                    starts=rng.randint(1, 10), fixing=_log_int(rng, 50, 500), solving=_log_int(rng, 50, 500),
                    sweeps=_log_int(rng, 50, 500), slices=rng.choice([4, 8, 16]), elite=rng.choice([0.1, 0.2]))
    if kind == "pticm":
        return dict(kind=kind, problem=rng.choice(["cubic", "cubic", "u10"]), size=rng.randint(4, 10),
                    runs=_log_int(rng, 10, 304), temps=rng.choice([8, 13, 16, 24, 30]), sweeps=_log_int(rng, 50, 500),
                    keep=rng.randint(1, 12))
    if kind == "reduce":
        return dict(kind=kind, problem=rng.choice(["cubic", "chimera", "u10", "weak_strong"]),
                    size=rng.randint(5, 20), samples=_log_int(rng, 50, 4000), elite=rng.choice([0.05, 0.1, 0.2]),
                    noalloc=rng.random() < 0.3)
    return dict(kind="serve", problem="cubic", size=rng.randint(12, 20), small=rng.randint(4, 10),
                count=rng.randint(2, 6), starts=rng.randint(4, 20), fixing=_log_int(rng, 50, 250),
                solving=_log_int(rng, 50, 250), sweeps=_log_int(rng, 200, 1000), step=rng.choice([0, 200, 500]),
                elite=0.2)


# ----------------------------------------------------------------- inputs
def _instance(problem, size, seed):
    if problem == "cubic":
        return instances.cubic3d(size, seed)
    if problem == "chimera":
        return instances.chimera(size, seed)
    if problem == "u10":
        return instances.chimera_u10(size, seed)
    if problem == "weak_strong":
        return instances.weak_strong(size, seed)
    # Gaussian couplers and a weak random field, rounded to integers at the given scale
    scale = int(problem[len("gauss"):])
    inst = instances.cubic3d(size, seed)
    g = np.random.default_rng([seed, scale])
    j = np.clip(np.rint(scale * g.standard_normal(inst.m)), -4 * scale, 4 * scale).astype(np.int32)
    inst.J = np.where(j == 0, 1, j).astype(np.int32)
    inst.h = np.rint(0.1 * scale * g.standard_normal(inst.n)).astype(np.int32)
    inst.scale = scale
    return inst


def _sizes(case):
    """The lattice sizes of a case with several problems: spread evenly over its range, the largest last."""
    n, hi = case["count"], case["size"]
    lo = case.get("small", max(4, hi // 2))
    return [lo + round((hi - lo) * i / max(n - 1, 1)) for i in range(n)]


def _params(case, **more):
    phases = case.get("phases", 1)
    return spvar.make_params(num_starts=case["starts"], fixing_sample_size=case["fixing"],
                             solving_sample_size=case["solving"], num_sweeps=case["sweeps"], beta0=0.1, beta1=3.0,
                             elite_threshold=case["elite"], iterate=phases > 1, max_fix_phases=phases, **more)


def prepare(case, seed):
    rng = random.Random(seed)
    kind = case["kind"]
    s = dict(kind=kind, case=case, seed=rng.randrange(1 << 62))
    iseed = rng.randrange(1 << 31)
    if kind in ("batch", "serve"):
        s["inst"] = [_instance(case["problem"], n, iseed + i) for i, n in enumerate(_sizes(case))]
        s["seeds"] = [rng.randrange(1 << 62) for _ in s["inst"]]
    else:
        s["inst"] = _instance(case["problem"], case["size"], iseed)
    if kind in ("sample", "pticm", "reduce"):
        s["problem"] = spvar.Problem.from_instance(s["inst"])
    if kind in ("sample", "reduce"):
        sweeps = case.get("sweeps", 200)
        dmax = s["problem"].info().dmax
        thr = spvar.thresholds(spvar.beta_geometric(sweeps, 0.1, 3.0), dmax, s["inst"].scale)
        s["thr"], s["stride"] = spvar.thresholds_device(thr), dmax + 1
    if kind == "solve":
        s["params"] = _params(case)
    elif kind == "plan":
        s["plan"] = spvar.Plan([spvar.Problem.from_instance(s["inst"])], _params(case))
    elif kind == "batch":
        s["plan"] = spvar.Plan([spvar.Problem.from_instance(i) for i in s["inst"]], _params(case))
    elif kind == "sqa":
        prm = _params(case, sampler=spvar.SAMPLER_SQA, sqa_slices=case["slices"], sqa_beta=3.0, sqa_gamma0=3.0,
                      sqa_gamma1=0.01)
        s["plan"] = spvar.Plan([spvar.Problem.from_instance(s["inst"])], prm)
    elif kind == "pticm":
        s["betas"], s["dx"] = np.geomspace(0.2, 3.0, case["temps"]), spvar.energy_range(s["inst"])
    elif kind == "reduce":
        # the sample an anneal leaves behind, not random states
        s["spins"], s["energies"] = spvar.sample(s["problem"], s["thr"], s["stride"], 200, case["samples"], s["seed"])
        if case["noalloc"]:
            info = s["problem"].info()
            new = lambda n, t=torch.int32: torch.zeros(max(n, 1), dtype=t, device="cuda")  # noqa: E731
            s["buffers"] = dict(row_ptr=new(info.n + 1), col=new(info.nnz), val=new(info.nnz), h=new(info.n),
                                offset=new(1, torch.int64), old_of_new=new(info.n), n_out=new(1))
    elif kind == "serve":
        n = max(i.n for i in s["inst"])
        s["server"] = spvar.Server(_params(case, sweep_kernel=spvar.SWEEP_PM1), 2 << 30, max_n=n, max_nnz=6 * n,
                                   max_degree=6, max_dmax=12, max_requests=case["count"],
                                   sweeps_per_step=case["step"])
    return s


# ------------------------------------------------------------------- pass
def _recorded(out):
    """A solve's outputs; energies past a phase's recorded count carry nothing and read as 0."""
    if isinstance(out.energies, np.ndarray):
        seen = np.arange(out.energies.shape[2]) < out.counts[:, :, None]
        energies = np.where(seen, out.energies, 0)
    else:
        seen = torch.arange(out.energies.shape[2], device="cuda") < out.counts[:, :, None]
        energies = torch.where(seen, out.energies, 0)
    return dict(energies=energies, counts=out.counts, nfree=out.nfree, fixed=out.fixed,
                best_energy=out.best_energy, best_state=out.best_state)


def run(s):
    case, kind = s["case"], s["kind"]
    if kind == "sample":
        return spvar.sample(s["problem"], s["thr"], s["stride"], case["sweeps"], case["samples"], s["seed"])
    if kind == "solve":
        return _recorded(spvar.solve(spvar.Problem.from_instance(s["inst"]), s["params"], s["seed"]))
    if kind in ("plan", "sqa"):
        return _recorded(s["plan"].run([s["seed"]], device=True))
    if kind == "batch":
        return _recorded(s["plan"].run(s["seeds"], device=True))
    if kind == "pticm":
        return spvar.pticm_sample(s["problem"], s["betas"], case["sweeps"], s["dx"], K=case["keep"],
                                  num_runs=case["runs"], seed=s["seed"])
    if kind == "reduce":
        elite, counts, fixed, nfixed, k = spvar.persistence(s["problem"], case["samples"], s["spins"], s["energies"],
                                                            case["elite"])
        out = dict(elite=elite, counts=counts, fixed=fixed, nfixed=nfixed, k=k)
        if case["noalloc"]:
            spvar.reduce_noalloc(s["problem"], fixed, **s["buffers"])
            out.update(s["buffers"])
        else:
            red, out["old_of_new"] = spvar.reduce(s["problem"], fixed)
            info = red.info()
            out.update(n=info.n, nnz=info.nnz, ncol=info.ncol, dmax=info.dmax, offset=int(info.offset))
        return out
    server = s["server"]
    ids = [server.submit(i, r) for i, r in zip(s["inst"], s["seeds"])]
    while server.step() > 0:
        pass
    out = []
    for rid in ids:
        out.append(_recorded(server.result(rid)))
        server.release(rid)
    return out


# ------------------------------------------------------------------- work
def _shape(problem, size):
    """Spins and couplers of one problem."""
    if problem in ("cubic",) or problem.startswith("gauss"):
        return size ** 3, 3 * size ** 3
    return 8 * size * size, 16 * size * size + 8 * size * (size - 1)


def work(case):
    """Bytes: the problems (couplers once, biases) and the samples, energies and states
    returned.  Operations: 18 integer operations and one per neighbour for every spin-flip
    attempt (a quarter of a ten-round Philox4x32 block is 15 of them, the acceptance 3), with
    one fixing and one solving phase at the problem's own size."""
    kind, prob = case["kind"], case["problem"]
    sizes = _sizes(case) if kind in ("batch", "serve") else [case["size"]]
    total_b = total_f = 0.0
    for size in sizes:
        n, m = _shape(prob, size)
        w = (n + 31) // 32 * 4
        problem_b = 12 * m + 4 * n
        per = 18 + 2 * m / n
        if kind == "sample":
            b = problem_b + case["samples"] * (w + 8)
            f = case["samples"] * case["sweeps"] * n * per
        elif kind == "pticm":
            reps = 2 * case["temps"]
            kept = 2 * (case["temps"] - case["temps"] // 2) * case["keep"]
            b = problem_b + case["runs"] * (reps + kept) * (w + 8)
            f = case["runs"] * reps * case["sweeps"] * n * per
        elif kind == "reduce":
            k = max(1, math.ceil(case["elite"] * case["samples"]))
            b = 8 * case["samples"] + k * w + 2 * problem_b + 13 * n
            f = case["samples"] + k * n + 4 * m
        else:
            s = case["fixing"] + case["solving"]
            slices = case.get("slices", 1)
            b = problem_b + case["starts"] * (8 * s + 2 * n + 8)
            f = case["starts"] * s * case["sweeps"] * slices * n * (per + (2 if slices > 1 else 0))
        total_b += b
        total_f += f
    return dict(bytes=total_b, flops=total_f)


def exact(case, seed):
    """None: every output is a whole number (spins, energies, counts, fixings), which has to stay the same."""
    return None
