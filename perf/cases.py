"""Performance cases: the solves a user of the library runs, through its public entry points.

listed() holds the standing cases, draw() gives more of the same ranges.  A case is a dict:

  path     "1d" (Solver.step), "2d" (Solver2D.step), "batch" (Batch.run) or
           "adjoint" (Solver.forward_ckpt, then Solver.adjoint)
  scheme   "heat", "ks" or "euler" (1d, adjoint); 2D is heat, a batch mixes heat and KS
  dtype    "f32" or "f64"
  bc       "periodic" or "reflective" (insulated heat, Euler walls)
  n / nx, ny / count, log2_hi    the grid, or the batch's number and largest size of problems
  nsteps   timesteps of one pass (a batch draws its own per problem, up to 5 nsteps)
  tile_w, threads, persistent, cluster, warp_tiles   the plan; 0 is the library's choice

Every pass starts again from its initial state, as a parameter study or an ensemble does.
"""
import math

import numpy as np
import torch

from paper_1612_02495_gb300 import inputs
from paper_1612_02495_gb300 import swept as S

SCHEMES = {"heat": S.HEAT, "ks": S.KS, "euler": S.EULER}
RADIUS = {"heat": 1, "ks": 2, "euler": 2}
STAGES = {"heat": 1, "ks": 2, "euler": 2}
COMPONENTS = {"heat": 1, "ks": 1, "euler": 3}
# floating-point operations of one point (cell) per sub-timestep, fma = 2, division and root 1
FLOPS = {"heat": 4, "ks": 18, "euler": 82}
FLOPS_2D = 6


def _case(path, scheme, dtype, bc, nsteps, tile_w=0, threads=0, persistent=0, cluster=0, warp_tiles=0, **size):
    return dict(path=path, scheme=scheme, dtype=dtype, bc=bc, nsteps=nsteps, tile_w=tile_w, threads=threads,
                persistent=persistent, cluster=cluster, warp_tiles=warp_tiles, **size)


def listed():
    def c(name, *a, **k):
        return dict(_case(*a, **k), name=name)

    return [
        # the shortest call: a few steps of a small insulated rod of odd size (output every few
        # steps, coupling to another solver); launches and latency are all of it
        c("heat_1009_f64_short", "1d", "heat", "f64", "reflective", 16, n=1009),
        # the paper's smallest grid for a whole run, as a program that sets no plan gets it
        c("heat_1k_f32", "1d", "heat", "f32", "periodic", 10000, n=1 << 10),
        # the same run in double precision with the plan the tuner keeps for it
        c("heat_1k_f64_warp", "1d", "heat", "f64", "periodic", 10000, n=1 << 10, tile_w=32, threads=32, warp_tiles=1),
        # a mid-sized KS run, tuned plan: too small to fill the GPU
        c("ks_16k_f64", "1d", "ks", "f64", "periodic", 2000, n=1 << 14, tile_w=128, threads=256),
        # the headline workload (fewer steps): the largest of the paper's KS grids, double precision
        c("ks_1m_f64_persist", "1d", "ks", "f64", "periodic", 1000, n=1 << 20, tile_w=1024, threads=256,
          persistent=1),
        # a grid no tile divides, single precision, no plan set
        c("ks_65537_f32", "1d", "ks", "f32", "periodic", 2000, n=65537),
        # the largest KS grid in single precision, tuned plan
        c("ks_1m_f32", "1d", "ks", "f32", "periodic", 5000, n=1 << 20, tile_w=1024, threads=128),
        # the Sod tube between walls, tuned plan
        c("euler_64k_f64_persist", "1d", "euler", "f64", "reflective", 500, n=1 << 16, tile_w=128, threads=256,
          persistent=1),
        # two dimensions, single precision, tuned plan
        c("heat2d_1k_f32", "2d", "heat", "f32", "periodic", 1000, nx=1024, ny=1024, tile_w=128, threads=1024),
        # two dimensions, insulated, double precision, not square, no plan set
        c("heat2d_768x512_f64", "2d", "heat", "f64", "reflective", 300, nx=768, ny=512),
        # a batch of unequal problems in one launch (the batched workload, fewer problems and steps)
        c("batch_128_f32", "batch", "mixed", "f32", "periodic", 400, count=128, log2_hi=16),
        # a gradient: checkpointing forward solve and adjoint sweep
        c("ks_64k_adjoint", "adjoint", "ks", "f64", "periodic", 400, n=1 << 16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _plan_1d(rng, scheme, n, dtype):
    """No plan, or one of those the tuner tries: a power-of-two tile, threads, a mode."""
    if rng.random() < 0.5:
        return {}
    r = RADIUS[scheme]
    tiles = [w for w in (32, 64, 128, 256, 512, 1024) if w % (4 * r) == 0 and n // w >= 2]
    if scheme == "euler":
        tiles = [w for w in tiles if w <= 512]
    w = rng.choice(tiles)
    mode = rng.choice(("pass", "pass", "persistent", "warp"))
    if mode == "warp" and scheme != "euler" and w <= 256 and n % w == 0:
        return dict(tile_w=w, threads=32, warp_tiles=1, persistent=rng.choice((0, 1)))
    return dict(tile_w=w, threads=rng.choice([t for t in (32, 64, 128, 256, 512) if t <= max(32, 2 * w)]),
                persistent=int(mode == "persistent"))


def _size_1d(rng, lo, hi):
    """Log-uniform; half of them powers of two or multiples of 1024, half whatever comes."""
    n = _log_int(rng, lo, hi)
    kind = rng.random()
    if kind < 0.25:
        return 1 << max(10, int(round(math.log2(n))))
    if kind < 0.5:
        return max(1024, n // 1024 * 1024)
    return n


def draw(rng):
    path = rng.choice(("1d", "1d", "1d", "1d", "2d", "2d", "batch", "adjoint"))
    dtype = rng.choice(("f32", "f64"))
    if path == "1d":
        scheme = rng.choice(("heat", "ks", "ks", "euler"))
        n = _size_1d(rng, 1000, 1 << 20)
        bc = "periodic" if scheme == "ks" else rng.choice(("periodic", "reflective"))
        # point-substeps of a pass, below the largest listed case's
        budget = (1 << 28) if dtype == "f64" else (1 << 31)
        most = budget / (n * STAGES[scheme]) / (10 if scheme == "euler" else 1)
        nsteps = _log_int(rng, 8, max(16, min(5000, most)))
        return _case("1d", scheme, dtype, bc, nsteps, n=n, **_plan_1d(rng, scheme, n, dtype))
    if path == "2d":
        q = rng.choice((16, 32, 64))  # a side is a multiple of its tile width
        nx, ny = (max(4, _log_int(rng, 256, 2048) // q) * q for _ in range(2))
        nsteps = _log_int(rng, 16, max(32, min(1000, (1 << 28) / (nx * ny))))
        plan = {} if rng.random() < 0.5 else dict(tile_w=q, threads=rng.choice((256, 512, 1024)),
                                                  persistent=rng.choice((0, 1)))
        return _case("2d", "heat", dtype, rng.choice(("periodic", "reflective")), nsteps, nx=nx, ny=ny, **plan)
    if path == "batch":
        return _case("batch", "mixed", dtype, "periodic", _log_int(rng, 20, 80 if dtype == "f64" else 400),
                     threads=rng.choice((0, 64, 128)), count=_log_int(rng, 8, 128), log2_hi=rng.choice((14, 15, 16)))
    scheme = rng.choice(("heat", "ks"))
    n = _size_1d(rng, 1 << 12, 1 << 17)
    return _case("adjoint", scheme, "f64", "periodic", _log_int(rng, 50, min(800, (1 << 25) / n)), n=n)


def _problem(case, seed):
    """The case's 1D problem: initial state and the constants of its scheme."""
    npd = np.float32 if case["dtype"] == "f32" else np.float64
    if case["scheme"] == "heat":
        p = inputs.heat_problem(n=case["n"], seed=seed, dtype=npd)
        return p["u0"], p["dx"], p["dt"], p["alpha"]
    if case["scheme"] == "ks":
        p = inputs.ks_problem(n=case["n"], seed=seed, dtype=npd)
        return p["u0"], p["dx"], p["dt"], p["nu"]
    p = inputs.euler_problem(n=case["n"], seed=seed, dtype=npd)
    return p["U0"], p["dx"], p["dt"], p["gamma"]


def _problem_2d(case, seed):
    return inputs.heat2d_problem(nx=case["nx"], ny=case["ny"], seed=seed,
                                 dtype=np.float32 if case["dtype"] == "f32" else np.float64)


def _batch(case, seed):
    lo, hi = case["nsteps"], 5 * case["nsteps"]
    # the sizes, kinds and step counts belong to the case; the seed draws the initial states
    spec = inputs.batch_problems(count=case["count"], seed=case["count"], log2_hi=case["log2_hi"], steps_lo=lo,
                                 steps_hi=hi)
    return inputs.batch_instances(spec, dtype=np.float32 if case["dtype"] == "f32" else np.float64, seed=seed % 99991)


def _cotangent(case, seed):
    return np.random.Generator(np.random.Philox(seed + 1)).standard_normal(case["n"])


def prepare(case, seed):
    dt = S.F32 if case["dtype"] == "f32" else S.F64
    bc = S.BC_REFLECTIVE if case["bc"] == "reflective" else S.BC_PERIODIC
    plan = {k: case[k] for k in ("tile_w", "threads", "persistent", "cluster", "warp_tiles")}
    st = {"path": case["path"], "nsteps": case["nsteps"]}
    if case["path"] == "batch":
        probs = _batch(case, seed)
        st["sol"] = S.Batch(probs, dt, threads=case["threads"])
        st["u0"] = st["sol"].pack([q["u0"] for q in probs])
    elif case["path"] == "2d":
        p = _problem_2d(case, seed)
        st["sol"] = S.Solver2D(dt, case["nx"], case["ny"], p["dx"], p["dt"], p["alpha"], tile_w=case["tile_w"],
                               threads=case["threads"], bc=bc, persistent=case["persistent"])
        st["u0"] = torch.from_numpy(p["u0"]).cuda()
    else:
        u0, dx, step, param = _problem(case, seed)
        st["sol"] = S.Solver(SCHEMES[case["scheme"]], dt, case["n"], dx, step, param, bc=bc, **plan)
        st["u0"] = torch.from_numpy(np.ascontiguousarray(u0)).cuda()
        if case["path"] == "adjoint":
            st["ckpt"] = torch.empty(st["sol"].ckpt_size(case["nsteps"]), dtype=torch.uint8, device="cuda")
            st["gT"] = torch.from_numpy(_cotangent(case, seed)).cuda()
            st["g_u0"] = torch.empty_like(st["u0"])
            st["g_param"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    st["u"] = torch.empty_like(st["u0"])
    return st


def run(st):
    u, sol = st["u"], st["sol"]
    u.copy_(st["u0"])
    if st["path"] == "batch":
        return {"u": sol.run(u)}
    if st["path"] == "adjoint":
        sol.forward_ckpt(u, st["nsteps"], st["ckpt"])
        g, gp = sol.adjoint(st["gT"], st["nsteps"], st["ckpt"], g_u0=st["g_u0"], g_param=st["g_param"])
        return {"u": u, "g_u0": g, "g_param": gp}
    return {"u": sol.step(u, st["nsteps"])}


def work(case):
    vb = 4 if case["dtype"] == "f32" else 8
    if case["path"] == "2d":
        n = case["nx"] * case["ny"]
        return {"bytes": 2 * n * vb, "flops": FLOPS_2D * n * case["nsteps"]}
    if case["path"] == "batch":
        # the mean over the problems' distribution: sizes 2^U(10, log2_hi), half heat and half KS,
        # steps U(nsteps, 5 nsteps)
        hi, lo = case["log2_hi"], 10
        n = case["count"] * (2.0 ** hi - 2.0 ** lo) / ((hi - lo) * math.log(2.0))
        return {"bytes": 2 * n * vb, "flops": n * 3 * case["nsteps"] * (FLOPS["heat"] + 2 * FLOPS["ks"]) / 2}
    s = case["scheme"]
    units = case["n"] * STAGES[s] * case["nsteps"]
    if case["path"] == "adjoint":
        # forward once, then the transposed sweep with the parameter's derivative (as many operations again and
        # 6 more); in: u0 and the cotangent; out: the final state and the gradient
        return {"bytes": 4 * case["n"] * vb, "flops": (2 * FLOPS[s] + 6) * units}
    return {"bytes": 2 * case["n"] * COMPONENTS[s] * vb, "flops": FLOPS[s] * units}


# ---- the same solves in 64 bits, in plain torch ----
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _t64(x):
    return torch.from_numpy(np.ascontiguousarray(np.asarray(x, dtype=np.float64))).to(_device())


def _pad(u, r, bc):
    if bc == "periodic":
        return torch.cat((u[-r:], u, u[:r]))
    return torch.cat((u[:r].flip(0), u, u[-r:].flip(0)))


def _ks_rhs(a, b, c, d, e, dx, nu):
    return -((d * d - b * b) / (4 * dx) + (d - 2 * c + b) / dx ** 2 + nu * (e - 4 * d + 6 * c - 4 * b + a) / dx ** 4)


def _ks_steps(u, dx, dt, nu, nsteps):
    def f(v):
        p = _pad(v, 2, "periodic")
        return _ks_rhs(p[:-4], p[1:-3], v, p[3:-1], p[4:], dx, nu)

    for _ in range(nsteps):
        u = u + dt * f(u + 0.5 * dt * f(u))
    return u


def _heat_steps(u, dx, dt, alpha, nsteps, bc):
    fo = alpha * dt / dx ** 2
    for _ in range(nsteps):
        p = _pad(u, 1, bc)
        u = u + fo * (p[2:] - 2 * u + p[:-2])
    return u


def _heat2d_steps(u, fo, nsteps, bc):
    for _ in range(nsteps):
        py = _pad(u, 1, bc)
        px = _pad(u.t(), 1, bc).t()
        u = u + fo * (py[2:] + py[:-2] + px[:, 2:] + px[:, :-2] - 4 * u)
    return u


def _euler_steps(U, dx, dt, gamma, nsteps, bc):
    def minmod(a, b):
        return torch.where(a * b > 0, torch.where(a.abs() <= b.abs(), a, b), torch.zeros_like(a))

    def advance(V):
        q = [_pad(c, 2, bc) for c in V]
        if bc == "reflective":  # the momentum turns its sign in the mirror cells
            q[1] = torch.cat((-q[1][:2], q[1][2:-2], -q[1][-2:]))
        r, u = q[0], q[1] / q[0]
        w = torch.stack((r, u, (gamma - 1) * (q[2] - 0.5 * q[1] * u)))
        d = w[:, 1:] - w[:, :-1]
        h = 0.5 * minmod(d[:, :-1], d[:, 1:])
        sides = []
        for x in (w[:, 1:-2] + h[:, :-1], w[:, 2:-1] - h[:, 1:]):
            m = x[0] * x[1]
            E = 0.5 * m * x[1] + x[2] / (gamma - 1)
            sides.append((torch.stack((x[0], m, E)), torch.stack((m, m * x[1] + x[2], x[1] * (E + x[2]))),
                          x[1].abs() + torch.sqrt(gamma * x[2] / x[0])))
        (ul, fl, sl), (ur, fr, sr) = sides
        F = 0.5 * (fl + fr) - 0.5 * torch.maximum(sl, sr) * (ur - ul)
        return V - dt / dx * (F[:, 1:] - F[:, :-1])

    for _ in range(nsteps):
        U = 0.5 * (U + advance(advance(U)))
    return U


def _batch_exact(probs):
    """All problems of one kind at once, neighbours by index; a finished problem is left as it is."""
    out = [None] * len(probs)
    for kind in (0, 1):
        ids = [i for i, q in enumerate(probs) if q["scheme"] == kind]
        if not ids:
            continue
        starts = np.cumsum([0] + [probs[i]["n"] for i in ids])
        dev = _device()

        def per_point(values, dtype=torch.float64):
            return torch.cat([torch.full((probs[i]["n"],), v, dtype=dtype, device=dev) for i, v in zip(ids, values)])

        def shifted(k):
            return torch.from_numpy(np.concatenate([s + (np.arange(probs[i]["n"]) + k) % probs[i]["n"]
                                                    for i, s in zip(ids, starts)])).to(dev)

        at = {k: shifted(k) for k in ((-1, 1) if kind == 0 else (-2, -1, 1, 2))}
        u = torch.cat([_t64(probs[i]["u0"]) for i in ids])
        dx, dt = (per_point([probs[i][k] for i in ids]) for k in ("dx", "dt"))
        param = per_point([probs[i]["param"] for i in ids])
        last = per_point([probs[i]["nsteps"] for i in ids], torch.int64)
        fo = param * dt / dx ** 2

        def f(v):
            return _ks_rhs(v[at[-2]], v[at[-1]], v, v[at[1]], v[at[2]], dx, param)

        for k in range(int(last.max())):
            v = u + fo * (u[at[1]] - 2 * u + u[at[-1]]) if kind == 0 else u + dt * f(u + 0.5 * dt * f(u))
            u = torch.where(last > k, v, u)
        for j, i in enumerate(ids):
            out[i] = u[starts[j]:starts[j + 1]]
    return torch.cat(out)


def exact(case, seed):
    if _device() == "cpu" and work(case)["flops"] > 1e9:
        return None
    if case["path"] == "batch":
        return {"u": _batch_exact(_batch(case, seed))}
    if case["path"] == "2d":
        p = _problem_2d(case, seed)
        return {"u": _heat2d_steps(_t64(p["u0"]), p["alpha"] * p["dt"] / p["dx"] ** 2, case["nsteps"], case["bc"])}
    u0, dx, dt, param = _problem(case, seed)
    u = _t64(u0)
    if case["path"] == "adjoint":
        u.requires_grad_()
        q = torch.tensor([float(param)], dtype=torch.float64, device=u.device, requires_grad=True)
        if case["scheme"] == "heat":
            v = _heat_steps(u, dx, dt, q, case["nsteps"], case["bc"])
        else:
            v = _ks_steps(u, dx, dt, q, case["nsteps"])
        g, gq = torch.autograd.grad(v, (u, q), _t64(_cotangent(case, seed)))
        return {"u": v.detach(), "g_u0": g, "g_param": gq}
    if case["scheme"] == "heat":
        return {"u": _heat_steps(u, dx, dt, param, case["nsteps"], case["bc"])}
    if case["scheme"] == "ks":
        return {"u": _ks_steps(u, dx, dt, param, case["nsteps"])}
    return {"u": _euler_steps(u, dx, dt, param, case["nsteps"], case["bc"])}
