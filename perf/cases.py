"""Performance cases of the pilot-assignment library: the work its users have
it do, through the public entry points of paper_2511_20511_gb300.binding.

Four kinds of case:
  eval    fitness of n device-resident chromosomes (Context.eval_population);
  solve   one whole solve (Context.solve): K-means seeding, G generations,
          final evaluation, best member -- plain (Alg. 1) or with islands
          (Alg. 2);
  batch   many uneven instances solved together (Batch.solve), tuned once;
  serve   a burst of requests submitted to the continuous-batching server and
          drained (Server.submit, Server.run_until_idle).
Instances are seeded hexagonal layouts (inputs.instance) cut to L cells;
populations are uniformly random permutations, as a GA's first generation has
them.
"""
import random

import numpy as np
import torch

from paper_2511_20511_gb300 import binding as B
from paper_2511_20511_gb300 import inputs

RINGS = (7, 19, 37, 61)
DEV = "cuda"


def listed():
    return [
        # one generation's population of the smallest configured layout: a
        # user who composes the GA from its steps calls this per generation
        {"name": "eval_7x4_n32", "kind": "eval", "L": 7, "K": 4, "n": 32, "prec": "fp32",
         "mode": "asymptotic", "objective": "sum_se", "M": 128.0},
        # one population of the paper-scale layout, the finite-antenna SINR
        {"name": "eval_19x10_n256", "kind": "eval", "L": 19, "K": 10, "n": 256, "prec": "fp32",
         "mode": "finite_m", "objective": "sum_se", "M": 256.0},
        # throughput: scoring a large set of candidate assignments (the
        # benchmark's batch)
        {"name": "eval_19x10_n1048576", "kind": "eval", "L": 19, "K": 10, "n": 1 << 20,
         "prec": "fp32", "mode": "finite_m", "objective": "sum_se", "M": 256.0},
        # three rings, an odd number of users, a ragged count, the max-min objective
        {"name": "eval_37x13_n50021", "kind": "eval", "L": 37, "K": 13, "n": 50021,
         "prec": "fp32", "mode": "asymptotic", "objective": "min_sinr", "M": 256.0},
        # more than 16 users per cell with the table still on chip
        {"name": "eval_19x24_n100003", "kind": "eval", "L": 19, "K": 24, "n": 100003,
         "prec": "fp32", "mode": "finite_m", "objective": "sum_se", "M": 256.0},
        # four rings x 32 users: the table exceeds one SM and is tiled
        {"name": "eval_61x32_n131072", "kind": "eval", "L": 61, "K": 32, "n": 1 << 17,
         "prec": "fp32", "mode": "finite_m", "objective": "sum_se", "M": 512.0},
        # the double-precision evaluation (reproducible, checked against the oracle)
        {"name": "eval64_19x10_n4096", "kind": "eval", "L": 19, "K": 10, "n": 4096,
         "prec": "fp64", "mode": "finite_m", "objective": "sum_se", "M": 256.0},
        # one scheduling decision: the headline whole solve
        {"name": "solve_19x10_N256_G200", "kind": "solve", "L": 19, "K": 10, "N": 256, "G": 200,
         "islands": 0, "mode": "finite_m", "objective": "sum_se", "M": 256.0},
        # the large single instance, population 2048
        {"name": "solve_61x32_N2048_G500", "kind": "solve", "L": 61, "K": 32, "N": 2048, "G": 500,
         "islands": 0, "mode": "finite_m", "objective": "sum_se", "M": 512.0},
        # the island GA, five islands re-clustered every three generations
        {"name": "islands_19x10_N256_G200_C5", "kind": "solve", "L": 19, "K": 10, "N": 256,
         "G": 200, "islands": 5, "mode": "finite_m", "objective": "sum_se", "M": 256.0},
        # a network's instances of mixed size solved in one go
        {"name": "batch_512_N128_G100", "kind": "batch", "n": 512, "Lmax": 37, "shapes": 0,
         "N": 128, "G": 100, "mode": "finite_m", "M": 256.0},
        # scheduling requests that arrive together at the server
        {"name": "serve_64_N64_G40", "kind": "serve", "n": 64, "Lmax": 19, "shapes": 0, "N": 64,
         "G": 40, "tick": 40, "mode": "finite_m", "M": 256.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))


def draw(rng):
    mode = rng.choice(["asymptotic", "finite_m", "finite_m"])
    objective = rng.choice(["sum_se", "sum_se", "min_sinr"])
    kind = rng.choice(["eval"] * 6 + ["solve"] * 3 + ["batch", "serve"])
    if kind == "eval":
        prec = rng.choice(["fp32"] * 5 + ["fp64"])
        if rng.random() < 0.6:  # full layouts, 4 to 16 users: the scheduler's sizes
            L, K = rng.choice([7, 19, 37]), rng.randint(4, 16)
        else:                   # anything up to four rings and 32 users
            L, K = rng.randint(2, 61), rng.randint(2, 32)
        # at most a quarter of the largest listed evaluation's gathers (a
        # hundredth in double precision), at most 2^20 chromosomes
        most = (61 * 61 * 32 << 17) // (4 if prec == "fp32" else 400)
        n = _log_int(rng, 16, max(64, min(1 << 20, most // (L * L * K))))
        return {"kind": "eval", "L": L, "K": K, "n": n, "prec": prec, "mode": mode,
                "objective": objective, "M": rng.choice([64.0, 128.0, 256.0, 512.0])}
    if kind == "solve":
        islands = rng.choice([0, 0, rng.randint(2, 8)])
        return {"kind": "solve", "L": rng.choice([7, 19, 37]), "K": rng.randint(4, 16),
                "N": _log_int(rng, 32, 512), "G": _log_int(rng, 20, 200), "islands": islands,
                "mode": mode, "objective": objective, "M": 256.0}
    if kind == "batch":
        return {"kind": "batch", "n": _log_int(rng, 8, 200), "Lmax": rng.choice([19, 37]),
                "shapes": rng.randint(1, 1 << 20), "N": rng.choice([32, 64, 100, 128]),
                "G": rng.randint(20, 100), "mode": mode, "M": 256.0}
    G = rng.randint(20, 60)
    return {"kind": "serve", "n": _log_int(rng, 4, 128), "Lmax": rng.choice([7, 19]),
            "shapes": rng.randint(1, 1 << 20), "N": rng.choice([32, 64, 96]), "G": G,
            "tick": rng.choice([G, G, 10]), "mode": mode, "M": 256.0}


# ------------------------------------------------------------------ inputs
def _instance(L, K, seed):
    """Gains and positions of the first L cells of the smallest full layout
    holding L (a full layout when L is one)."""
    full = next(r for r in RINGS if r >= L)
    inst = inputs.instance(full, K, seed=seed, dtype=np.float32)
    if full != L:
        inst["beta"] = np.ascontiguousarray(inst["beta"][:L, :L])
        inst["user_xy_mm"] = np.ascontiguousarray(inst["user_xy_mm"][:L])
        inst["bs_xy_mm"] = np.ascontiguousarray(inst["bs_xy_mm"][:L])
    return inst


def _config(L, K, rho, mode, M, seed, **kw):
    return B.pa_config_default(
        L, K, rho=rho, M=M, seed=seed, tau_p=K,
        mode=B.PA_SINR_FINITE_M if mode == "finite_m" else B.PA_SINR_ASYMPTOTIC, **kw)


def _objective(case):
    return B.PA_OBJ_MIN_SINR if case.get("objective") == "min_sinr" else B.PA_OBJ_SUM_SE


def _shapes(case):
    """(L, K) of a batch's or burst's instances: full layouts up to Lmax."""
    rng = random.Random(case["shapes"])
    Ls = [r for r in RINGS if r <= case["Lmax"]]
    Ks = list(range(4, 17)) if case["kind"] == "batch" else [8, 16]
    return [(rng.choice(Ls), rng.choice(Ks)) for _ in range(case["n"])]


def _population(case, seed):
    return inputs.random_population_torch(case["n"], case["L"], case["K"], seed, DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "eval":
        inst = _instance(case["L"], case["K"], seed)
        cfg = _config(case["L"], case["K"], inst["rho"], case["mode"], case["M"], seed,
                      prec=B.PA_FP64 if case["prec"] == "fp64" else B.PA_FP32,
                      objective=_objective(case))
        ctx = B.Context(cfg, inst["beta"], inst["user_xy_mm"], inst["bs_xy_mm"])
        pop = _population(case, seed)
        fit = torch.empty(case["n"], dtype=ctx.torch_fit_dtype(), device=DEV)
        return {"kind": kind, "ctx": ctx, "pop": pop, "fit": fit}
    if kind == "solve":
        inst = _instance(case["L"], case["K"], seed)
        cfg = _config(case["L"], case["K"], inst["rho"], case["mode"], case["M"], seed,
                      N=case["N"], objective=_objective(case), islands=case["islands"])
        ctx = B.Context(cfg, inst["beta"], inst["user_xy_mm"], inst["bs_xy_mm"])
        return {"kind": kind, "ctx": ctx, "G": case["G"], "views": {}}
    shapes = _shapes(case)
    insts = [_instance(L, K, seed * 1000003 + i) for i, (L, K) in enumerate(shapes)]
    if kind == "batch":
        items = [dict(cfg=_config(L, K, inst["rho"], case["mode"], case["M"], seed + i,
                                  N=case["N"]),
                      beta=inst["beta"], user_xy_mm=inst["user_xy_mm"],
                      bs_xy_mm=inst["bs_xy_mm"])
                 for i, ((L, K), inst) in enumerate(zip(shapes, insts))]
        batch = B.Batch(items)
        batch.tune(case["G"])
        return {"kind": kind, "batch": batch, "G": case["G"]}
    base = _config(shapes[0][0], shapes[0][1], insts[0]["rho"], case["mode"], case["M"], 0,
                   N=case["N"])
    server = B.Server(base, case["G"], case["tick"], 40 << 30)
    requests = [(i, L, K, seed + i, inst["beta"], inst["user_xy_mm"], inst["bs_xy_mm"])
                for i, ((L, K), inst) in enumerate(zip(shapes, insts))]
    return {"kind": kind, "server": server, "requests": requests}


class _DeviceBytes:
    """The context's resident population, seen by torch without a copy."""

    def __init__(self, ptr, shape):
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "|u1", "data": (ptr, False),
                                         "version": 2}


def run(state):
    kind = state["kind"]
    if kind == "eval":
        return state["ctx"].eval_population(state["pop"], state["fit"])
    if kind == "solve":
        ctx = state["ctx"]
        best, fitness = ctx.solve(state["G"])
        ptr, _ = B.pa_population_device(ctx.handle)
        if ptr not in state["views"]:
            state["views"][ptr] = torch.as_tensor(_DeviceBytes(ptr, (ctx.N, ctx.L, ctx.K)),
                                                  device=DEV)
        return {"best": best, "fitness": fitness, "population": state["views"][ptr]}
    if kind == "batch":
        rows, fit = state["batch"].solve(state["G"])
        return {"best": np.concatenate([r.reshape(-1) for r in rows]), "fitness": fit}
    server = state["server"]
    for r in state["requests"]:
        server.submit(*r)
    done = sorted(server.run_until_idle(), key=lambda d: d[0])
    return {"ids": np.array([d[0] for d in done]), "fitness": np.array([d[2] for d in done]),
            "best": np.concatenate([d[1][:r[1] * r[2]]
                                    for d, r in zip(done, state["requests"])])}


# ------------------------------------------------------------------ work
def _eval_work(L, K, n, fin, fsz):
    # table in, chromosomes in, fitness out; per gathered gain a multiply-add
    # (and an add for the finite-M sum), per user about a dozen operations
    return (8 * L * L * K + n * L * K + fsz * n, n * (L * L * K * (3 if fin else 2) + 12 * L * K))


def work(case):
    fin = case["mode"] == "finite_m"
    if case["kind"] == "eval":
        b, f = _eval_work(case["L"], case["K"], case["n"], fin, 8 if case["prec"] == "fp64" else 4)
        return {"bytes": b, "flops": f}
    shapes = [(case["L"], case["K"])] if case["kind"] == "solve" else _shapes(case)
    b = f = 0
    for L, K in shapes:
        # gains and positions in; best member, its fitness and the final
        # population out; every generation's members evaluated once
        b += 8 * L * L * K + 8 * L * K + 8 * L + (case["N"] + 1) * L * K + 8
        f += (case["G"] + 1) * _eval_work(L, K, case["N"], fin, 4)[1]
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ exact values
def exact(case, seed):
    """Fitness of an evaluation case in 64 bits (Eq. 3-6 by gathers); a GA
    run's outputs have no value apart from its own trajectory."""
    if case["kind"] != "eval":
        return None
    L, K, n = case["L"], case["K"], case["n"]
    inst = _instance(L, K, seed)
    beta = torch.from_numpy(inst["beta"]).to(DEV)
    rho, sigma2 = inst["rho"], 1.0
    bn = beta.sum(dim=(1, 2)) + sigma2 / rho
    pop = _population(case, seed)
    own = torch.diagonal(beta, dim1=0, dim2=1).t().contiguous()  # [L][K]
    cells = torch.arange(L, device=DEV)
    out = torch.empty(n, dtype=torch.float64, device=DEV)
    step = max(1, (64 << 20) // (L * L * K))
    flat = beta.reshape(L, L * K)
    for n0 in range(0, n, step):
        inv = torch.argsort(pop[n0:n0 + step].long(), dim=-1)       # user of each pilot
        m = inv.shape[0]
        idx = (inv + cells[None, :, None] * K).reshape(-1)          # (m, l, p)
        g = flat[:, idx].reshape(L, m, L, K)                        # gains at BS j
        b = torch.gather(own[None].expand(m, L, K), 2, inv)         # own gain of (j, p)
        s1 = g.sum(dim=2)
        g[cells, :, cells, :] = 0.0
        s2 = g.square().sum(dim=2)
        s1, s2 = s1.permute(1, 0, 2), s2.permute(1, 0, 2)           # (m, j, p)
        if case["mode"] == "finite_m":
            sinr = case["M"] * b * b / (case["M"] * s2 + bn[None, :, None] *
                                        (s1 + sigma2 / (K * rho)))
        else:
            sinr = b * b / s2
        out[n0:n0 + step] = (sinr.amin(dim=(1, 2)) if case["objective"] == "min_sinr" else
                             torch.log2(1.0 + sinr).sum(dim=(1, 2)))
    return out.cpu()
