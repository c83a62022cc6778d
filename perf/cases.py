"""The work a user has this planner do, as measurable cases.

Every case goes through the package's public entry points: plan (build a model
and solve it), csr (build it and export P and R in the paper's layout), solve
(value iteration on a model that is kept), plan3d (the 3-D build and solve),
batch (many uneven MDPs in one call), serve (a burst of replanning requests)
and rollout (a policy flown through every flow realization).  Sizes are those
of the repository's own workloads (inputs.py, bench.py) and odd sizes between
them.  Fields are the synthetic double gyre with sinusoidal modes of inputs.py;
the seed changes the flow (its unsteadiness and phase), the coefficients'
spread and their draw, and the target.
"""
from __future__ import annotations

import dataclasses
import functools
import math
import random

import numpy as np
import torch

from paper_2109_00857_gb300 import inputs, mdp

TIME, ENERGY, NET = inputs.OBJ_TIME, inputs.OBJ_ENERGY, inputs.OBJ_NET_ENERGY
OBJECTIVES = {1: (TIME,), 2: (TIME, NET), 3: (TIME, ENERGY, NET)}
METHODS = {"jacobi": mdp.MDP_SOLVE_JACOBI, "layered": mdp.MDP_SOLVE_LAYERED}


def listed():
    return [
        # the plain method on the smallest grid (an interactive replan: latency and launches)
        dict(name="plan_tiny", kind="plan", nx=20, ny=20, nt=10, K=2, N=200, headings=16, speeds=1, L=7,
             n_obj=1, method="jacobi", tol=0.0, amplitude=0.5, sigma0=0.2),
        # an odd, non-square coastal grid with an odd mode count, the sub-grid sized by the
        # library, solved exactly by the backward pass
        dict(name="plan_ragged", kind="plan", nx=77, ny=45, nt=37, K=5, N=1234, headings=16, speeds=1, L=0,
             n_obj=1, method="layered", tol=0.0, amplitude=2.0, sigma0=0.3),
        # the energy-harvesting mission: net energy, value iteration to residual 1e-6
        dict(name="plan_energy", kind="plan", nx=100, ny=100, nt=60, K=4, N=1000, headings=16, speeds=2, L=15,
             n_obj=-1, method="jacobi", tol=1e-6, amplitude=2.5, sigma0=0.3),
        # the large instance: three objectives from one build, solved together to the fixed point
        dict(name="plan_large", kind="plan", nx=200, ny=200, nt=120, K=8, N=5000, headings=16, speeds=2, L=21,
             n_obj=3, method="jacobi", tol=0.0, amplitude=2.5, sigma0=0.3),
        # P and R handed to another solver, in arrays it keeps: a build and the paper-layout export
        dict(name="csr_mid", kind="csr", nx=90, ny=90, nt=40, K=6, N=800, headings=16, speeds=1, L=21,
             n_obj=2, amplitude=2.0, sigma0=0.3),
        # value iteration alone on a kept model, 16 actions (two states per slice)
        dict(name="solve_a16", kind="solve", nx=160, ny=160, nt=80, K=3, N=500, headings=16, speeds=1, L=21,
             n_obj=1, method="jacobi", tol=0.0, amplitude=2.0, sigma0=0.3),
        # the backward pass alone on the large instance's shape, three objectives
        dict(name="solve_large", kind="solve", nx=200, ny=200, nt=120, K=4, N=600, headings=16, speeds=2, L=21,
             n_obj=3, method="layered", tol=0.0, amplitude=2.5, sigma0=0.3),
        # the 3-D instance: build and fused solve
        dict(name="plan3d_cube", kind="plan3d", nx=64, ny=64, nz=16, nt=40, K=4, N=1000, n_obj=3),
        # uneven MDPs (sides 40-160, nt 20-80, K 2-6, N 500-2000, 16 or 32 actions) in one call
        dict(name="batch_16", kind="batch", first=0, members=16),
        # a burst of replanning requests on two resident environments
        dict(name="serve_burst", kind="serve", side=96, nt=40, K=6, N=1500, requests=8),
        # a policy flown through every realization from a set of starts
        dict(name="rollout_64", kind="rollout", nx=200, ny=200, nt=120, K=8, N=5000, starts=64, n_obj=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["plan", "plan", "plan", "csr", "solve", "solve", "plan3d", "batch", "serve", "rollout"])
    headings, speeds = rng.choice([(16, 1), (16, 2), (16, 2), (8, 3), (12, 1), (8, 1)])
    if kind in ("plan", "csr", "solve"):
        while True:
            c = dict(kind=kind, nx=_log_int(rng, 20, 200), ny=_log_int(rng, 20, 200), nt=_log_int(rng, 8, 120),
                     K=rng.randint(1, 8), N=_log_int(rng, 200, 5000), headings=headings, speeds=speeds,
                     L=rng.choice([0, 21, 21]), n_obj=rng.choice([1, 1, -1, 2, 3]), amplitude=rng.uniform(0.5, 2.5),
                     sigma0=rng.uniform(0.15, 0.3))
            A = headings * speeds
            if kind == "csr" and c["nx"] * c["ny"] * c["nt"] * A > 20_000_000:
                continue
            if c["nx"] * c["ny"] * c["nt"] * A * c["N"] <= 2e11:
                break
        if kind != "csr":
            c["method"] = rng.choice(["jacobi", "jacobi", "layered"])
            c["tol"] = 0.0 if c["method"] == "layered" else rng.choice([0.0, 1e-6, 1e-3])
        return c
    if kind == "plan3d":
        return dict(kind=kind, nx=_log_int(rng, 16, 64), ny=_log_int(rng, 16, 64), nz=rng.randint(4, 16),
                    nt=_log_int(rng, 8, 40), K=rng.randint(2, 6), N=_log_int(rng, 200, 1000),
                    n_obj=rng.choice([1, 2, 3]))
    if kind == "batch":
        return dict(kind=kind, first=rng.randint(16, 58), members=rng.randint(3, 6))
    if kind == "serve":
        return dict(kind=kind, side=rng.randint(30, 120), nt=rng.randint(20, 60), K=rng.randint(1, 6),
                    N=_log_int(rng, 500, 2000), requests=rng.randint(2, 12))
    return dict(kind=kind, nx=_log_int(rng, 40, 200), ny=_log_int(rng, 40, 200), nt=_log_int(rng, 20, 120),
                K=rng.randint(2, 8), N=_log_int(rng, 500, 5000), starts=_log_int(rng, 4, 64),
                n_obj=rng.choice([1, 2, 3]))


# ------------------------------------------------------------------ inputs --
@functools.lru_cache(maxsize=24)
def _base(nx, ny, nt, K):
    """What depends on the sizes alone: the modes and the mean scalar field."""
    return inputs.do_modes(nx, ny, nt, K), inputs.solar_field(nx, ny, nt, np.random.default_rng(nx + ny))


def _env2d(c, seed):
    nx, ny, nt, K = c["nx"], c["ny"], c["nt"], c["K"]
    rng = np.random.default_rng(seed)
    modes, gbar = _base(nx, ny, nt, K)
    vbar = inputs.double_gyre(nx, ny, nt, c["amplitude"], eps=float(rng.uniform(0.1, 0.3)),
                              phase=float(rng.uniform(0, 2 * math.pi)))
    sigma = c["sigma0"] * float(rng.uniform(0.9, 1.0)) * 2.0 ** (-np.arange(K) / 2.0)
    square = max(3, min(nx, ny) // 10)
    obstacle = inputs.moving_squares(nx, ny, nt, square, rows=(float(rng.uniform(0.3, 0.4)), float(rng.uniform(0.6, 0.7))))
    target = inputs.target_block(nx, ny, int(rng.integers(nx // 4, 3 * nx // 4)), int(rng.integers(ny // 2, ny - 3)))
    n_obj = c.get("n_obj", 1)
    return inputs.Environment(
        nx=nx, ny=ny, nt=nt, K=K, N=c["N"], L=c.get("L", 21), vbar=vbar, modes=modes, sigma=sigma,
        seed=int(rng.integers(1, 2 ** 62)), obstacle=obstacle, target=target,
        actions=inputs.action_table(c.get("headings", 16), c.get("speeds", 2), 1.0), gbar=gbar,
        r_outbound=-10.0 * nt, objectives=(NET,) if n_obj == -1 else OBJECTIVES[n_obj], name=c["kind"])


@functools.lru_cache(maxsize=4)
def _base3d(nx, ny, nz, nt, K):
    return inputs.make_env3d(nx, ny, nz, nt, K, N=1, L=9, sigma=[0.15 * 2.0 ** (-q / 2.0) for q in range(K)],
                             seed=61, amplitude=0.8, with_gbar=True)


def _env3d(c, seed):
    b = _base3d(c["nx"], c["ny"], c["nz"], c["nt"], c["K"])
    rng = np.random.default_rng(seed)
    target = np.zeros_like(b.target)
    i, j = int(rng.integers(b.nx // 4, 3 * b.nx // 4)), int(rng.integers(b.ny // 2, b.ny - 3))
    target[b.nz - 2:, j:j + 2, i:i + 2] = 1
    return dataclasses.replace(b, N=c["N"], vbar=b.vbar * float(rng.uniform(0.85, 1.0)),
                               sigma=b.sigma * float(rng.uniform(0.75, 0.9)), seed=int(rng.integers(1, 2 ** 62)),
                               target=target, objectives=OBJECTIVES[c["n_obj"]])


@functools.lru_cache(maxsize=80)
def _member(i):
    return inputs.batch_member(i)


def _members(c, seed):
    out = []
    for i in range(c["first"], c["first"] + c["members"]):
        b = _member(i)
        rng = np.random.default_rng([seed, i])
        vbar = inputs.double_gyre(b.nx, b.ny, b.nt, 2.0, eps=float(rng.uniform(0.1, 0.3)),
                                  phase=float(rng.uniform(0, 2 * math.pi)))
        out.append(dataclasses.replace(b, vbar=vbar, sigma=b.sigma * float(rng.uniform(0.9, 1.0)),
                                       seed=int(rng.integers(1, 2 ** 62))))
    return out


def _serve_envs(c, seed):
    sides = (c["side"], max(30, (2 * c["side"]) // 3))
    return [_env2d(dict(kind="serve", nx=s, ny=s, nt=c["nt"], K=c["K"], N=c["N"], L=21, speeds=1 + q, n_obj=1,
                        amplitude=1.5, sigma0=0.25), seed * 2 + q) for q, s in enumerate(sides)]


def _requests(c, seed, envs):
    """Replanning requests: new start, target, coefficient spread, seed and N."""
    rng = np.random.default_rng([seed, 7])
    out = []
    for r in range(c["requests"]):
        e = envs[r % 2]
        out.append(dict(env=r % 2, start=(int(rng.integers(0, e.nx)), int(rng.integers(0, e.ny // 2))),
                        target=(int(rng.integers(0, e.nx - 2)), int(rng.integers(e.ny // 2, e.ny - 2))),
                        sigma_scale=float(rng.uniform(0.5, 1.5)), seed=int(rng.integers(1, 2 ** 62)),
                        N=max(500, c["N"] - 117 * r), start_t=(r % 3) * (c["nt"] // 4)))
    return out


def _heading_policy(e):
    """Steer at the target against the mean flow: the action whose mean step ends nearest to it."""
    j0, i0 = np.argwhere(e.target)[0]
    vb = torch.as_tensor(e.vbar).cuda()
    gx = i0 - torch.arange(e.nx, device="cuda", dtype=torch.float64)[None, None, :] - vb[..., 0]
    gy = j0 - torch.arange(e.ny, device="cuda", dtype=torch.float64)[None, :, None] - vb[..., 1]
    best = torch.full(gx.shape, math.inf, device="cuda", dtype=torch.float64)
    pol = torch.zeros(gx.shape, device="cuda", dtype=torch.int16)
    for a in range(e.A):
        d = (gx - e.actions[a, 0]) ** 2 + (gy - e.actions[a, 1]) ** 2
        pol[d < best] = a
        best = torch.minimum(best, d)
    fixed = torch.as_tensor(e.obstacle != 0).cuda() | torch.as_tensor(e.target != 0).cuda()[None]
    pol[fixed] = -1
    return pol.reshape(-1).contiguous()


def _starts(c, seed, e):
    rng = np.random.default_rng([seed, 9])
    return [(int(rng.integers(0, e.nx)), int(rng.integers(0, e.ny))) for _ in range(c["starts"])]


def prepare(case, seed):
    mdp.load()
    c, kind = case, case["kind"]
    s = {"case": c, "kind": kind}
    if kind in ("plan", "csr", "solve"):
        env = _env2d(c, seed)
        s["denv"], s["objs"] = mdp.DeviceEnv(env), env.objectives
        if kind == "solve":
            s["model"] = mdp.mdp_build(s["denv"], objs=s["objs"])
            s["V"] = [torch.empty(env.nS + 1, device="cuda") for _ in s["objs"]]
            s["pi"] = [torch.empty(env.nS, dtype=torch.int16, device="cuda") for _ in s["objs"]]
            del s["denv"]
        elif kind == "csr":   # the other solver's arrays, with room for any model of these sizes
            s["col"] = torch.zeros(env.nS * env.A * 16, dtype=torch.int64, device="cuda")
            s["count"] = torch.zeros(env.nS * env.A * 16, dtype=torch.int32, device="cuda")
    elif kind == "plan3d":
        env = _env3d(c, seed)
        s["denv"], s["objs"] = mdp.DeviceEnv3D(env), env.objectives
    elif kind == "batch":
        s["batch"] = mdp.Batch([mdp.DeviceEnv(e) for e in _members(c, seed)])
    elif kind == "serve":
        envs = _serve_envs(c, seed)
        s["server"] = mdp.Server(24 << 30, 8)
        s["ids"] = [s["server"].register(mdp.DeviceEnv(e)) for e in envs]
        s["requests"] = _requests(c, seed, envs)
    else:
        env = _env2d(dict(c, amplitude=1.5, sigma0=0.25), seed)
        s["denv"], s["objs"] = mdp.DeviceEnv(env), env.objectives
        s["policy"], s["starts"] = _heading_policy(env), _starts(c, seed, env)
    return s


# --------------------------------------------------------------------- run --
def _solve(model, c, n, V=None, pi=None):
    method, tol = METHODS[c.get("method", "jacobi")], c.get("tol", 0.0)
    if n == 1:
        V, pi, _ = mdp.mdp_solve(model, 0, method=method, tol=tol, V=V and V[0], policy=pi and pi[0])
        return {"V": [V], "policy": [pi]}
    V, pi, _ = mdp.mdp_solve_multi(model, tuple(range(n)), method=method, tol=tol, V=V, policy=pi)
    return {"V": V, "policy": pi}


def run(state):
    c, kind = state["case"], state["kind"]
    if kind == "plan":
        model = mdp.mdp_build(state["denv"], objs=state["objs"])
        out = _solve(model, c, len(state["objs"]))
        model.free()
        return out
    if kind == "csr":
        model = mdp.mdp_build(state["denv"], objs=state["objs"])
        rowptr, col, count, R0 = mdp.mdp_export_csr(model, 0)
        R = [R0] + [mdp.mdp_export_csr(model, o, with_entries=False)[3] for o in range(1, len(state["objs"]))]
        model.free()
        state["col"][:col.numel()].copy_(col)
        state["count"][:count.numel()].copy_(count)
        return {"rowptr": rowptr, "col": state["col"], "count": state["count"], "R": R}
    if kind == "solve":
        return _solve(state["model"], c, len(state["objs"]), V=state["V"], pi=state["pi"])
    if kind == "plan3d":
        model = mdp.mdp_build3d(state["denv"], objs=state["objs"])
        out = _solve(model, c, len(state["objs"]))
        model.free()
        return out
    if kind == "batch":
        state["batch"].run()
        return {"V": state["batch"].V, "policy": state["batch"].policy}
    if kind == "serve":
        server, ids = state["server"], state["ids"]
        tickets = [server.submit(ids[r["env"]], r["start"], r["target"], sigma_scale=r["sigma_scale"], seed=r["seed"],
                                 N=r["N"], start_t=r["start_t"]) for r in state["requests"]]
        out = []
        for t, r in zip(tickets, state["requests"]):
            got = server.poll(t, timeout_ms=60000, env_id=ids[r["env"]], want_V=True)
            out.append({"V": got[1], "policy": got[2]})
        return out
    ret, steps, status, _ = mdp.mdp_rollout(state["denv"], state["policy"], state["starts"], objs=state["objs"])
    return {"ret": ret, "steps": steps, "status": status}


# -------------------------------------------------------------------- work --
# Successors kept per row: about 6.5 on the large instance, between 4 and 8 on the others.
_SUCC = 6.5


def _plan_work(nS, A, K, N, n_obj, dims=2, entries=False):
    """A build and a solve: the fields in, V and the policy out (P stays inside); the velocity
    of every realization, one multiply-add per mode and component, and one backup."""
    fields = nS * (4 * dims * (K + 1) + 4 + 1)
    out = nS * n_obj * 6
    flops = nS * N * 2 * dims * (K + 1) + 2 * _SUCC * nS * A * n_obj
    if entries:
        out = nS * A * (8 + 4 * n_obj + 12 * _SUCC)
    return {"bytes": fields + out, "flops": flops}


def work(case):
    c, kind = case, case["kind"]
    n_obj = abs(c.get("n_obj", 1))
    if kind in ("plan", "csr"):
        return _plan_work(c["nx"] * c["ny"] * c["nt"], c["headings"] * c["speeds"], c["K"], c["N"], n_obj,
                          entries=kind == "csr")
    if kind == "solve":   # P and R once, V and the policy out
        nS, A = c["nx"] * c["ny"] * c["nt"], c["headings"] * c["speeds"]
        return {"bytes": nS * A * 4 * (_SUCC + n_obj) + nS * n_obj * 6, "flops": 2 * _SUCC * nS * A * n_obj}
    if kind == "plan3d":
        return _plan_work(c["nx"] * c["ny"] * c["nz"] * c["nt"], 24, c["K"], c["N"], n_obj, dims=3)
    if kind == "batch":
        ws = [_plan_work(e.nS, e.A, e.K, e.N, 1) for e in (_member(i) for i in range(c["first"], c["first"] + c["members"]))]
    elif kind == "serve":
        ws = []
        for r in range(c["requests"]):
            side = c["side"] if r % 2 == 0 else max(30, (2 * c["side"]) // 3)
            nt = c["nt"] - (r % 3) * (c["nt"] // 4)
            ws.append(_plan_work(side * side * nt, 16 * (1 + r % 2), c["K"], max(500, c["N"] - 117 * r), 1))
    else:
        # a path flies at most nt steps, each reading its modes and coefficients (half of nt on average)
        steps = c["starts"] * c["N"] * c["nt"] / 2
        return {"bytes": c["nt"] * c["N"] * c["K"] * 4 + c["starts"] * c["N"] * (4 * n_obj + 5), "flops": steps * 4 * (c["K"] + 1)}
    return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}


# ------------------------------------------------------- the same in 64 bits --
def _mulhi(a, b):
    m = np.uint64(0xFFFFFFFF)
    s = np.uint64(32)
    a0, a1, b0, b1 = a & m, a >> s, b & m, b >> s
    t = a0 * b0
    u = a1 * b0 + (t >> s)
    v = a0 * b1 + (u & m)
    return a1 * b1 + (u >> s) + (v >> s)


def _philox(c, key):
    """Philox4x64-10 (Salmon et al. 2011) on arrays of counters."""
    c0, c1, c2, c3 = c
    k0, k1 = np.uint64(key[0]), np.uint64(key[1])
    M0, M1 = np.uint64(0xD2E7470EE14C6C93), np.uint64(0xCA5A826395121157)
    with np.errstate(over="ignore"):
        for r in range(10):
            if r:
                k0, k1 = k0 + np.uint64(0x9E3779B97F4A7C15), k1 + np.uint64(0xBB67AE8584CAA73B)
            c0, c1, c2, c3 = _mulhi(M1, c2) ^ c1 ^ k0, M1 * c2, _mulhi(M0, c0) ^ c3 ^ k1, M0 * c0
    return c0, c1


def _coefficients(nt, N, K, sigma, seed, mdp_id=0):
    """Y[t][w][k] = sigma_k z: polar pairs (Marsaglia & Bray) on the counters (t, w, pair, attempt)."""
    pairs = (K + 1) // 2
    t, w, j = (x.reshape(-1).astype(np.uint64) for x in np.meshgrid(np.arange(nt), np.arange(N), np.arange(pairs), indexing="ij"))
    z = np.zeros((t.size, 2))
    left = np.arange(t.size)
    for att in range(64):
        if not left.size:
            break
        a, b = _philox((t[left], w[left], j[left], np.full(left.size, att, np.uint64)), (seed, mdp_id))
        v1 = 2.0 * ((a >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1.0
        v2 = 2.0 * ((b >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1.0
        q = v1 * v1 + v2 * v2
        ok = (q < 1.0) & (q > 0.0)
        f = np.sqrt(-2.0 * np.log(q[ok]) / q[ok])
        z[left[ok], 0], z[left[ok], 1] = v1[ok] * f, v2[ok] * f
        left = left[~ok]
    return z.reshape(nt, N, 2 * pairs)[:, :, :K] * np.asarray(sigma)[None, None, :]


def _plan64(e, objs, Y, want_R=False, target=None):
    """Backward induction over the realizations themselves: Q(s,a) = mean over w of r + V(s'_w),
    the landing cell floor(1/2 + (v + a) dt/dx) per axis.  dims 2 or 3; fields [nt][..., axes]."""
    f64 = dict(device="cuda", dtype=torch.float64)
    three = hasattr(e, "nz")
    size = (e.nz, e.ny, e.nx) if three else (e.ny, e.nx)
    dims, Nc, A = len(size), int(np.prod(size)), e.A
    target = torch.as_tensor((e.target if target is None else target).reshape(-1) != 0).cuda()
    obstacle = torch.as_tensor(e.obstacle.reshape(e.nt, Nc) != 0).cuda()
    act = torch.as_tensor(e.actions, **f64)
    F = act[:, dims]
    gb = torch.as_tensor(e.gbar.reshape(e.nt, Nc), **f64) if e.gbar is not None else None
    n = len(objs)
    V = torch.zeros(n, e.nt, Nc, **f64)
    R = torch.zeros(n, A, e.nt, Nc, **f64) if want_R else None
    Yd = torch.as_tensor(Y, **f64) if e.K else None
    chunk = max(1, int(4e7) // e.N)
    h = 12   # border of sink cells around the grid: no landing of these flows goes further
    shape = [s + 2 * h for s in size]
    strides = [int(np.prod(shape[d + 1:])) for d in range(dims)]
    for t in range(e.nt - 1, -1, -1):
        sink_all = obstacle[t] | (t == e.nt - 1)
        V[:, t] = torch.where(target, 0.0, torch.where(sink_all, e.r_outbound, 0.0))
        if want_R:
            R[:, :, t] = V[:, t][:, None, :]
        cells = torch.nonzero(~target & ~sink_all).reshape(-1)
        if not cells.numel():
            continue
        free = ~obstacle[t + 1]
        tab = torch.zeros((n + 1 + (n if want_R else 0), Nc), **f64)   # per objective V' (and reward parts), then "free"
        for o, ob in enumerate(objs):
            g = torch.where(target, e.r_term, 0.0) + (0.5 * e.c_r * gb[t + 1] * e.dt if ob == NET else 0.0)
            tab[o] = torch.where(free, V[o, t + 1] + g, 0.0)
            if want_R:
                tab[n + 1 + o] = torch.where(free, g, 0.0)
        tab[n] = free.to(torch.float64)
        pad = torch.zeros([tab.shape[0]] + shape, **f64)
        pad[(slice(None),) + tuple(slice(h, h + s) for s in size)] = tab.reshape([-1] + list(size))
        pad = pad.reshape(tab.shape[0], -1)
        vb = torch.as_tensor(np.ascontiguousarray(e.vbar[t]), **f64).reshape(Nc, dims)
        ph = torch.as_tensor(np.ascontiguousarray(e.modes[t]), **f64).reshape(e.K, Nc, dims) if e.K else None
        lam = e.dt / e.dx
        for lo in range(0, cells.numel(), chunk):
            cc = cells[lo:lo + chunk]
            pos, rest = [], cc
            for s in reversed(size):
                pos.insert(0, rest % s)
                rest = rest // s
            u = []
            for x in range(dims):   # x, y (, z)
                w = vb[cc, x][:, None].expand(-1, e.N)
                if e.K:
                    w = w + ph[:, cc, x].T @ Yd[t].T
                u.append(0.5 + w * lam)
            base = sum((p + h) * st for p, st in zip(pos, strides)).to(torch.float64)[:, None]
            best = torch.full((n, cc.numel()), -math.inf, **f64)
            for a in range(A):
                idx = base
                for x in range(dims):
                    idx = idx + torch.floor(u[x] + act[a, x] * lam) * strides[dims - 1 - x]
                idx = idx.to(torch.int64)
                mean = [pad[r][idx].mean(1) for r in range(pad.shape[0])]
                p = mean[n]
                for o, ob in enumerate(objs):
                    step = -e.dt if ob == TIME else -e.c_f * float(F[a]) ** 2 * e.dt
                    b = p * step + (1.0 - p) * e.r_outbound
                    if ob == NET:
                        b = b + p * 0.5 * e.c_r * gb[t, cc] * e.dt
                    if want_R:
                        R[o, a, t, cc] = b + mean[n + 1 + o]
                    best[o] = torch.maximum(best[o], b + mean[o])
            V[:, t, cc] = best
    Vs = [torch.cat([V[o].reshape(-1), torch.zeros(1, **f64)]) for o in range(n)]
    return (Vs, [R[o].reshape(-1) for o in range(n)]) if want_R else Vs


def _rollout64(e, objs, Y, policy, starts):
    f64 = dict(device="cuda", dtype=torch.float64)
    i = torch.tensor([s[0] for s in starts], device="cuda")[:, None].expand(-1, e.N).reshape(-1).clone()
    j = torch.tensor([s[1] for s in starts], device="cuda")[:, None].expand(-1, e.N).reshape(-1).clone()
    w = torch.arange(e.N, device="cuda").repeat(len(starts))
    ret = torch.zeros(i.numel(), len(objs), **f64)
    live = torch.ones(i.numel(), dtype=torch.bool, device="cuda")
    target, act = torch.as_tensor(e.target.reshape(-1) != 0).cuda(), torch.as_tensor(e.actions, **f64)
    pol = policy.reshape(e.nt, -1).long()
    for t in range(e.nt):
        c = j * e.nx + i
        live &= ~target[c]
        at = torch.nonzero(live).reshape(-1)
        if not at.numel():
            break
        ca, obs = c[at], torch.as_tensor(e.obstacle[t].reshape(-1) != 0).cuda()
        a = pol[t, ca]
        out = obs[ca] | (a < 0) | (t == e.nt - 1)
        vb = torch.as_tensor(np.ascontiguousarray(e.vbar[t]), **f64).reshape(-1, 2)
        ph = torch.as_tensor(np.ascontiguousarray(e.modes[t]), **f64).reshape(e.K, -1, 2)
        y = torch.as_tensor(Y[t], **f64)[w[at]]
        v = vb[ca] + torch.einsum("pk,kpx->px", y, ph[:, ca])
        d = act[a.clamp(min=0)]
        ip = i[at] + torch.floor(0.5 + (v[:, 0] + d[:, 0]) * e.dt / e.dx).long()
        jp = j[at] + torch.floor(0.5 + (v[:, 1] + d[:, 1]) * e.dt / e.dx).long()
        out |= (ip < 0) | (ip >= e.nx) | (jp < 0) | (jp >= e.ny)
        cp = torch.where(out, torch.zeros_like(ip), jp * e.nx + ip)
        nxt = min(t + 1, e.nt - 1)
        out |= torch.as_tensor(e.obstacle[nxt].reshape(-1) != 0).cuda()[cp]
        for o, ob in enumerate(objs):
            if ob == TIME:
                r = torch.full_like(d[:, 2], -e.dt)
            else:
                r = -e.c_f * d[:, 2] ** 2 * e.dt
            if ob == NET:
                g0, g1 = (torch.as_tensor(e.gbar[k].reshape(-1), **f64) for k in (t, nxt))
                r = r + 0.5 * e.c_r * (g0[ca] + g1[cp]) * e.dt
            r = r + torch.where(target[cp], e.r_term, 0.0)
            ret[at, o] += torch.where(out, e.r_outbound, r)
        live[at[out]] = False
        i[at], j[at] = torch.where(out, i[at], ip), torch.where(out, j[at], jp)
    return ret.reshape(len(starts), e.N, len(objs))


# landings above which the 64-bit reference takes too long
_MOST = 8e10


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("plan", "csr", "solve"):
        e = _env2d(c, seed)
        if e.samples() * len(e.objectives) > _MOST:
            return None
        Y = _coefficients(e.nt, e.N, e.K, e.sigma, e.seed, e.mdp_id)
        if kind == "csr":
            _, R = _plan64(e, e.objectives, Y, want_R=True)
            return {"rowptr": None, "col": None, "count": None, "R": R}
        V = _plan64(e, e.objectives, Y)
        return {"V": V, "policy": [None] * len(V)}
    if kind == "plan3d":
        e = _env3d(c, seed)
        if e.samples() * len(e.objectives) > 2 * _MOST:
            return None
        V = _plan64(e, e.objectives, _coefficients(e.nt, e.N, e.K, e.sigma, e.seed, e.mdp_id))
        return {"V": V, "policy": [None] * len(V)}
    if kind == "batch":   # the smallest members, as many as the time allows
        envs, left = _members(c, seed), _MOST
        V = [None] * len(envs)
        for q in sorted(range(len(envs)), key=lambda q: envs[q].samples()):
            e = envs[q]
            left -= e.samples()
            if left < 0:
                break
            V[q] = _plan64(e, e.objectives[:1], _coefficients(e.nt, e.N, e.K, e.sigma, e.seed, e.mdp_id))[0]
        return {"V": V, "policy": [None] * len(V)}
    if kind == "serve":
        envs, left = _serve_envs(c, seed), _MOST
        out = []
        for r in _requests(c, seed, envs):
            b, t0 = envs[r["env"]], r["start_t"]
            e = dataclasses.replace(b, nt=b.nt - t0, vbar=b.vbar[t0:], modes=b.modes[t0:], gbar=b.gbar[t0:],
                                    obstacle=b.obstacle[t0:], sigma=b.sigma * r["sigma_scale"], seed=r["seed"], N=r["N"],
                                    target=inputs.target_block(b.nx, b.ny, r["target"][0], r["target"][1]))
            left -= e.samples()
            V = _plan64(e, (TIME,), _coefficients(e.nt, e.N, e.K, e.sigma, e.seed))[0] if left >= 0 else None
            out.append({"V": V, "policy": None})
        return out
    e = _env2d(dict(c, amplitude=1.5, sigma0=0.25), seed)
    Y = _coefficients(e.nt, e.N, e.K, e.sigma, e.seed, e.mdp_id)
    return {"ret": _rollout64(e, e.objectives, Y, _heading_policy(e), _starts(c, seed, e)), "steps": None, "status": None}
