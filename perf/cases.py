"""The workloads whose speed is tracked: what a user of this library has it do.

Sizes are those of ``workloads`` (the 2-D point mass, the 7-link arm, the
16-link legged robot, the uneven batch, the serving fleet) and of the tests'
ragged problems.  A case is a dict of plain values; ``prepare`` makes what a
program holds before the call (handles, plans, start states, candidates),
``run`` makes the call, ``work`` states the bytes and flops it cannot do
without and ``exact`` gives its result in 64 bits from the formulas of the
paper, written here in plain torch.

Kinds:

* ``rollout``   mtp_rollout_cost: all candidates of one problem through the
  dynamics, to their costs (Alg. 2, Eq. 2).
* ``generate``  mtp_generate_candidates: local samples, graph paths and the
  mean row of one iteration (Defs. 1-3, Alg. 1).
* ``elite``     mtp_elite_update: selection and the update of mean and spread.
* ``plan``      mtp_plan_step: whole planner iterations of one problem.
* ``batch``     mtp_batch_plan_step: one iteration of many uneven problems.
* ``serve``     one cycle of a re-plan loop: the robots that asked are filled
  into a reserved batch, planned, and their warm start shifted.
"""
import math

import numpy as np
import torch

from paper_2505_01059_gb300 import mtp
from paper_2505_01059_gb300 import workloads as W

DEV = "cuda:0"
ITER = 3  # the planner iteration whose draws a single step uses


def listed():
    return [
        # one robot re-planning by itself with the default 2-D problem: ten
        # iterations of very small kernels, where latency and launches count
        {"name": "plan_pointmass2", "kind": "plan", "dyn": "pointmass", "dim": 2, "B": 512, "H": 64,
         "M": 4, "N": 8, "E": 32, "interp": "bspline", "degree": 3, "iters": 10},
        # the vectorised planner: 256 uneven problems, point masses and arms
        # mixed, one iteration (the library's headline workload)
        {"name": "batch_256", "kind": "batch", "count": 256, "mix": 3},
        # a serving cycle: the robots with a waiting request, other ones each
        # time, so the batch is refilled and its kernels launched directly
        {"name": "serve_cycle_48", "kind": "serve", "count": 48, "mix": 4},
        # rollouts of the 7-link arm: one warp's chain per 32 candidates
        {"name": "rollout_arm7", "kind": "rollout", "dyn": "chain", "dim": 7, "B": 4096, "H": 128, "dr": "per_sample"},
        # rollouts of the 16-link legged robot with ground contact: the largest problem
        {"name": "rollout_legged16", "kind": "rollout", "dyn": "legged", "dim": 16, "B": 16384, "H": 256,
         "dr": "per_sample"},
        # rollouts of a many-axis point mass at the batch's largest size
        {"name": "rollout_pointmass12", "kind": "rollout", "dyn": "pointmass", "dim": 12, "B": 8192, "H": 256,
         "dr": "none"},
        # a ragged arm problem whose cost is averaged over shared models
        {"name": "rollout_arm5_shared", "kind": "rollout", "dyn": "chain", "dim": 5, "B": 1000, "H": 50,
         "dr": "shared", "R": 4},
        # the legged robot's candidates: B-splines with bfloat16 operands on the
        # tensor cores, most rows drawn locally; the largest tensor written
        {"name": "generate_legged16", "kind": "generate", "n": 15, "B": 16384, "H": 256, "M": 16, "N": 64,
         "beta": 0.3, "interp": "bspline", "degree": 2, "bf16": True},
        # the arm's candidates: Akima paths, half of the rows
        {"name": "generate_arm7", "kind": "generate", "n": 7, "B": 4096, "H": 128, "M": 8, "N": 32,
         "beta": 0.5, "interp": "akima", "degree": 2, "bf16": False},
        # a small odd-sized problem with straight-line paths
        {"name": "generate_ragged", "kind": "generate", "n": 3, "B": 333, "H": 33, "M": 7, "N": 13,
         "beta": 0.37, "interp": "linear", "degree": 2, "bf16": False},
        # the arm's elite selection and softmax update
        {"name": "elite_arm7", "kind": "elite", "B": 4096, "E": 64, "H": 128, "n": 7, "rule": "softmax"},
        # many candidates (two-stage selection), many elites, plain CEM
        {"name": "elite_wide", "kind": "elite", "B": 65536, "E": 512, "H": 64, "n": 12, "rule": "plain_cem"},
    ]


def _between(rng, lo, hi):
    """A whole number in lo..hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rollout", "rollout", "rollout", "generate", "generate", "elite", "plan", "batch", "serve"])
    if kind == "rollout":
        dyn = rng.choice(["pointmass", "chain", "chain", "legged"])
        case = {"kind": kind, "dyn": dyn}
        if dyn == "pointmass":
            case.update(dim=rng.randint(2, 12), B=_between(rng, 300, 8192), H=_between(rng, 30, 256))
        elif dyn == "chain":
            case.update(dim=rng.randint(3, 9), B=_between(rng, 300, 8192), H=_between(rng, 30, 128))
        else:
            case.update(dim=rng.randint(4, 16), B=_between(rng, 200, 16384), H=_between(rng, 30, 256))
        case["dr"] = rng.choice(["none", "per_sample", "per_sample", "shared"]) if dyn != "legged" else "per_sample"
        if case["dr"] == "shared":
            case["R"] = rng.randint(2, 8)
            case["B"] = max(64, case["B"] // case["R"])
        return case
    if kind == "generate":
        interp = rng.choice(["bspline", "bspline", "akima", "linear"])
        n = rng.randint(2, 15)
        M = rng.randint(4, 16)
        return {"kind": kind, "n": n, "B": _between(rng, 300, 16384), "H": _between(rng, 30, 256), "M": M,
                "N": rng.choice([8, 13, 16, 32, 64]), "beta": rng.choice([0.3, 0.5, 0.9]), "interp": interp,
                "degree": rng.randint(2, 3), "bf16": interp == "bspline" and rng.random() < 0.5}
    if kind == "elite":
        B = _between(rng, 300, 65536)
        n = rng.randint(2, 12)
        return {"kind": kind, "B": B, "E": min(B, rng.choice([16, 32, 50, 64, 128, 512])),
                "H": _between(rng, 30, 128) if B > 8192 else _between(rng, 30, 256), "n": n,
                "rule": rng.choice(["softmax", "softmax", "plain_cem"])}
    if kind == "plan":
        return {"kind": kind, "dyn": "pointmass", "dim": rng.randint(2, 4), "B": _between(rng, 256, 2048),
                "H": _between(rng, 32, 128), "M": rng.randint(4, 8), "N": rng.choice([8, 16, 32]), "E": 32,
                "interp": rng.choice(["bspline", "akima"]), "degree": 3, "iters": rng.randint(1, 10)}
    return {"kind": kind, "count": rng.randint(16, 200) if kind == "batch" else rng.randint(8, 96),
            "mix": rng.randint(10, 1000000)}


# ---------------------------------------------------------------------------
# what a program holds before the call
# ---------------------------------------------------------------------------

def _f(x):
    """The float32 value a problem field holds, as a double."""
    return float(np.float32(x))


def _rollout_spec(case, seed):
    extra = dict(B=case["B"], H=case["H"], E=1, beta=0.5, seed=seed)
    if case["dyn"] == "pointmass":
        spec = W.pointmass(k=case["dim"], degree=2, **extra)
    elif case["dyn"] == "chain":
        spec = W.chain(links=case["dim"], **extra)
    else:
        spec = W.legged(links=case["dim"], **extra)
    if case["dr"] == "none":
        spec.update(dr_mode="none")
    else:
        spec.update(dr_mode=case["dr"], R=case.get("R", 1), dr_lo=0.8, dr_hi=1.2)
    return spec


def _start(spec, gen):
    """A start state near the problem's own: small joint angles and rates; the
    legged robot's base a little above the ground."""
    x = np.array(spec["x0"], np.float64)
    e = gen.uniform(-1.0, 1.0, size=x.shape)
    if spec["dyn"] == "legged":
        x[0] += 0.1 * e[0]
        x[1] += 0.02 * (1.0 + e[1])
        x[2:spec["n_links"] + 2] += 0.005 * e[2:spec["n_links"] + 2]
    else:
        x += 0.1 * e
    return x.astype(np.float32)


def _controls(B, H, n, lo, hi, seed, half_gauss=0.5):
    """Candidate controls as a planner makes them: Gaussian rows around a
    smooth mean, and straight lines through random knots, in the box."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    lo = torch.tensor(lo, dtype=torch.float32, device=DEV)
    hi = torch.tensor(hi, dtype=torch.float32, device=DEV)
    U = torch.empty(B, H, n, device=DEV)
    L = int(B * half_gauss)
    U[:L] = torch.randn(L, H, n, generator=g, device=DEV) * (0.5 * (hi - lo)) + 0.5 * (hi + lo)
    M = 8
    K = lo + (hi - lo) * torch.rand(B - L, M, n, generator=g, device=DEV)
    t = torch.linspace(0, M - 1, H, device=DEV)
    k = t.floor().clamp(max=M - 2).long()
    w = (t - k)[:, None]
    U[L:] = K[:, k] * (1 - w) + K[:, k + 1] * w
    return torch.minimum(torch.maximum(U, lo), hi).contiguous()


def _generate_spec(case, seed):
    spec = W.pointmass(k=case["n"], H=case["H"], M=case["M"], N=case["N"], B=case["B"], beta=case["beta"],
                       interp=case["interp"], degree=case["degree"], E=1, seed=seed,
                       u_min=[-2.0] * case["n"], u_max=[2.0] * case["n"])
    spec["flags"] = 0x4 if case["bf16"] else 0
    return spec


def _state_before(case, seed):
    """Mean and spread of a run that is under way."""
    gen = np.random.default_rng(seed + 77)
    mu = gen.uniform(-1.0, 1.0, size=(case["H"], case["n"]))
    sigma = gen.uniform(0.1, 1.0, size=(case["H"], case["n"]))
    return mu, sigma


def _elite_inputs(case, seed):
    """Costs with a spread of a few temperatures among the best, one in a
    hundred of them a rollout that diverged, and the candidates' controls."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    cost = 40.0 * torch.exp(0.5 * torch.randn(case["B"], generator=g, device=DEV))
    bad = torch.rand(case["B"], generator=g, device=DEV) < 0.01
    cost = torch.where(bad, torch.full_like(cost, float("inf")), cost)
    return cost, _controls(case["B"], case["H"], case["n"], [-2.0] * case["n"], [2.0] * case["n"], seed + 1)


def _many_specs(case, seed):
    specs = W.batch(seed=case["mix"], count=case["count"], bf16=True) if case["kind"] == "batch" else \
        W.robots(seed=case["mix"], count=case["count"])
    for i, s in enumerate(specs):
        s["seed"] = seed * 4096 + i
    return specs


def _views(h, names):
    """The handle's own device buffers as tensors, which keep the handle."""
    buf = mtp.mtp_get_buffers(h)
    views = [torch.as_tensor(buf[k], device=DEV) for k in names]
    for v in views:
        v.owner = h
    return views


def prepare(case, seed):
    kind = case["kind"]
    if kind == "rollout":
        spec = _rollout_spec(case, seed)
        x0 = torch.tensor(_start(spec, np.random.default_rng(seed)), device=DEV)
        U = _controls(case["B"], case["H"], spec["n"], spec["u_min"], spec["u_max"], seed)
        return {"kind": kind, "h": mtp.mtp_create(spec), "x0": x0, "U": U,
                "cost": torch.empty(case["B"], device=DEV)}
    if kind == "generate":
        h = mtp.mtp_create(_generate_spec(case, seed))
        mtp.mtp_set_state(h, *_state_before(case, seed), 0)
        return {"kind": kind, "h": h, "U": torch.empty(case["B"], case["H"], case["n"], device=DEV)}
    if kind == "elite":
        spec = W.pointmass(k=case["n"], H=case["H"], B=case["B"], E=case["E"], degree=2, seed=seed,
                           update_rule=case["rule"])
        spec["lambda"] = 5.0
        h = mtp.mtp_create(spec)
        cost, U = _elite_inputs(case, seed)
        mu, sigma = _views(h, ("mu", "sigma"))
        return {"kind": kind, "h": h, "cost": cost, "U": U,
                "elite": torch.empty(case["E"], dtype=torch.int32, device=DEV),
                "ustar": torch.empty(case["n"], device=DEV), "mu": mu, "sigma": sigma}
    if kind == "plan":
        spec = W.pointmass(k=case["dim"], H=case["H"], M=case["M"], N=case["N"], B=case["B"], E=case["E"],
                           interp=case["interp"], degree=case["degree"], seed=seed)
        h = mtp.mtp_create(spec)
        cost, mu, sigma = _views(h, ("cost", "mu", "sigma"))
        return {"kind": kind, "h": h, "iters": case["iters"],
                "x0": torch.tensor(_start(spec, np.random.default_rng(seed)), device=DEV),
                "ustar": torch.empty(case["dim"], device=DEV), "cost": cost, "mu": mu, "sigma": sigma}
    specs = _many_specs(case, seed)
    gen = np.random.default_rng(seed)
    x0 = torch.tensor(np.concatenate([_start(s, gen) for s in specs]), device=DEV)
    hs = [mtp.mtp_create(s) for s in specs]
    if kind == "batch":
        b = mtp.mtp_batch_create(hs)
        mtp.mtp_batch_autotune(b)
    else:
        b = mtp.mtp_batch_reserve(len(hs))
    us = torch.empty(sum(s["n"] for s in specs), device=DEV)
    costs = [_views(h, ("cost",))[0] for h in hs]
    return {"kind": kind, "b": b, "hs": hs, "x0": x0, "us": us, "costs": costs}


def run(s):
    kind = s["kind"]
    if kind == "rollout":
        mtp.mtp_rollout_cost(s["h"], ITER, s["x0"], s["U"], s["cost"])
        return s["cost"]
    if kind == "generate":
        mtp.mtp_generate_candidates(s["h"], ITER, s["U"])
        return s["U"]
    if kind == "elite":
        mtp.mtp_elite_update(s["h"], s["cost"], s["U"], s["elite"], s["ustar"])
        return [s["elite"], s["ustar"], s["mu"], s["sigma"]]
    if kind == "plan":
        mtp.mtp_plan_step(s["h"], s["x0"], s["iters"], s["ustar"])
        return [s["ustar"], s["cost"], s["mu"], s["sigma"]]
    if kind == "serve":
        mtp.mtp_batch_fill(s["b"], s["hs"])
    mtp.mtp_batch_plan_step(s["b"], s["x0"], 1, s["us"])
    if kind == "serve":
        mtp.mtp_batch_shift(s["b"], 1)
    return [s["us"], torch.cat(s["costs"])]


# ---------------------------------------------------------------------------
# the least work
# ---------------------------------------------------------------------------

def _step_flops(dyn, dim, obstacles=5):
    """Flops of one rollout step of one candidate, in forms linear in the
    number of links: cost, forces, velocity terms, the structured solve, Euler."""
    if dyn == "pointmass":
        return 9 * dim + 8 + obstacles * (3 * dim + 3)
    return (76 if dyn == "chain" else 97) * dim


def work(case):
    kind = case["kind"]
    if kind == "rollout":
        n = case["dim"] - 1 if case["dyn"] == "legged" else case["dim"]
        return {"bytes": 4 * case["B"] * (case["H"] * n + 1),
                "flops": case["B"] * case["H"] * case.get("R", 1) * _step_flops(case["dyn"], case["dim"])}
    if kind == "generate":
        out = case["B"] * case["H"] * case["n"]
        return {"bytes": 4 * out + 8 * case["H"] * case["n"], "flops": 10 * out}
    if kind == "elite":
        hn = case["H"] * case["n"]
        return {"bytes": 4 * case["B"] + 4 * case["E"] * (hn + 1) + 16 * hn, "flops": 5 * case["E"] * hn}
    if kind == "plan":
        # the candidates of all iterations but the last need not leave the chip
        hn = case["H"] * case["dim"]
        return {"bytes": 4 * case["B"] + 16 * hn + 4 * case["iters"] * 2 * hn,
                "flops": case["iters"] * case["B"] * case["H"] * (_step_flops("pointmass", case["dim"]) + 10 * case["dim"])}
    total = {"bytes": 0, "flops": 0}
    for s in _many_specs(case, 1):
        hn = s["H"] * s["n"]
        total["bytes"] += 4 * s["B"] + 16 * hn + 8 * hn
        total["flops"] += s["B"] * s["H"] * (_step_flops(s["dyn"], s["n"]) + 10 * s["n"])
    return total


# ---------------------------------------------------------------------------
# the results in 64 bits
# ---------------------------------------------------------------------------

def _mul_hi_lo(m, x):
    """High and low 32 bits of m * x for a 32-bit m and 32-bit values x."""
    p0, p1 = (x & 0xFFFF) * m, (x >> 16) * m
    t = (p0 >> 16) + p1
    return t >> 16, ((t & 0xFFFF) << 16) | (p0 & 0xFFFF)


def _philox(c, seed):
    """Philox4x32-10 (Salmon et al., SC'11) of the counters c (four int64
    tensors of 32-bit values) under a 64-bit key."""
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    x, y, z, w = c
    for _ in range(10):
        h0, l0 = _mul_hi_lo(0xD2511F53, x)
        h1, l1 = _mul_hi_lo(0xCD9E8D57, z)
        x, y, z, w = h1 ^ y ^ k0, l1, h0 ^ w ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return x, y, z, w


def _words(units, slots, tag, seed):
    """The 32-bit draws (units, slots) of one stream: word slot % 4 of the
    generator call (unit, slot / 4, iteration, tag)."""
    a = torch.arange(units, dtype=torch.int64, device=DEV)[:, None]
    q = torch.arange((slots + 3) // 4, dtype=torch.int64, device=DEV)[None, :]
    a, q = torch.broadcast_tensors(a, q)
    r = _philox((a, q, torch.full_like(a, ITER), torch.full_like(a, tag)), seed)
    return torch.stack(r, dim=2).reshape(units, -1)[:, :slots]


def _unit(w):
    return (w >> 8).double() * 2.0 ** -24


def _scales(spec, slots):
    """Model scales per model: (B or R, slots)."""
    if spec["dr_mode"] == "none":
        return torch.ones(1, slots, dtype=torch.float64, device=DEV)
    shared = spec["dr_mode"] == "shared"
    w = _words(spec["R"] if shared else spec["B"], slots, 5 if shared else 4, spec["seed"])
    lo, hi = _f(spec["dr_lo"]), _f(spec["dr_hi"])
    return lo + float(np.float32(hi) - np.float32(lo)) * _unit(w)


def _t64(v):
    return torch.tensor(np.asarray(v, np.float32), device=DEV).double()


def _roll_pointmass(spec, x0, U, scale):
    k, dt = spec["n"], _f(spec["dt"])
    target, oc, orad = _t64(spec["target"]), _t64(spec["obs_c"]), _t64(spec["obs_r"])

    def cost(p):
        pen = (orad - (p[:, None] - oc).norm(dim=2)).clamp(min=0).sum(1)
        return _f(spec["w_target"]) * (p - target).square().sum(1) + _f(spec["w_obs"]) * pen

    p, v = x0[:k].expand(U.shape[0], k), x0[k:].expand(U.shape[0], k)
    J = torch.zeros(U.shape[0], dtype=torch.float64, device=DEV)
    for t in range(spec["H"]):
        u = U[:, t].double()
        J = J + cost(p) + _f(spec["w_ctrl"]) * u.square().sum(1)
        v = v + dt * scale * u
        p = p + dt * v
    return J + _f(spec["w_term"]) * cost(p)


def _inertia(mass, length):
    """First moments lb_j and the constants D_jk of uniform thin rods in a chain
    (masses (rows, L)): D_jj = l_j^2 (m_j / 3 + sum of the masses beyond j),
    D_jk = l_k lb_j for k < j."""
    beyond = mass.flip(1).cumsum(1).flip(1) - mass
    lb = length * (0.5 * mass + beyond)
    D = length[None, None, :] * lb[:, :, None]
    D = D.tril(-1)
    return lb, D + D.transpose(1, 2) + torch.diag_embed(length ** 2 * (mass / 3 + beyond))


def _roll_chain(spec, x0, U, scale):
    L, dt, g = spec["n_links"], _f(spec["dt"]), _f(spec["gravity"])
    length, target = _t64(spec["length"]), _t64(spec["target"])
    lb, D = _inertia(_t64(spec["mass"]) * scale, length)
    B = U.shape[0]
    phi, w = x0[:L].cumsum(0).expand(B, L), x0[L:].cumsum(0).expand(B, L)

    def reach(phi):
        x, y = (length * phi.cos()).sum(1), (length * phi.sin()).sum(1)
        return _f(spec["w_target"]) * ((x - target[0]) ** 2 + (y - target[1]) ** 2)

    J = torch.zeros(B, dtype=torch.float64, device=DEV)
    for t in range(spec["H"]):
        u = U[:, t].double()
        J = J + reach(phi) + _f(spec["w_ctrl"]) * u.square().sum(1)
        diff = phi[:, :, None] - phi[:, None, :]
        force = u - torch.nn.functional.pad(u[:, 1:], (0, 1)) - g * lb * phi.cos()
        force = force - ((D * diff.sin()) @ (w * w)[:, :, None])[:, :, 0]
        acc = torch.cholesky_solve(force[:, :, None], torch.linalg.cholesky_ex(D * diff.cos())[0])[:, :, 0]
        w = w + dt * acc
        phi = phi + dt * w
    return J + _f(spec["w_term"]) * reach(phi)


def _roll_legged(spec, x0, U, scale):
    L, dt, g = spec["n_links"], _f(spec["dt"]), _f(spec["gravity"])
    length, target = _t64(spec["length"]), _t64(spec["target"])
    mass = _t64(spec["mass"]) * scale[:, :L]
    friction = _f(spec["mu_friction"]) * scale[:, L:]
    lb, D = _inertia(mass, length)
    B, nq = U.shape[0], L + 2
    m = mass.sum(1, keepdim=True)
    S = D - lb[:, :, None] * lb[:, None, :] / m[:, :, None]
    base, vel = x0[:2].expand(B, 2), x0[nq:nq + 2].expand(B, 2)
    phi, w = x0[2:nq].cumsum(0).expand(B, L), x0[nq + 2:].cumsum(0).expand(B, L)

    def cost():
        return (_f(spec["w_height"]) * (base[:, 1] - target[0]) ** 2 + _f(spec["w_vel"]) * (vel[:, 0] - target[1]) ** 2 +
                _f(spec["w_pitch"]) * (phi[:, 0] - target[2]) ** 2)

    J = torch.zeros(B, dtype=torch.float64, device=DEV)
    for t in range(spec["H"]):
        u = U[:, t].double()
        J = J + cost() + _f(spec["w_ctrl"]) * u.square().sum(1)
        c, s = phi.cos(), phi.sin()
        pad = torch.nn.functional.pad
        y = pad((length * s).cumsum(1), (1, 0)) + base[:, 1:]
        vx = pad((-length * w * s).cumsum(1), (1, 0)) + vel[:, :1]
        vy = pad((length * w * c).cumsum(1), (1, 0)) + vel[:, 1:]
        normal = torch.where(y < 0, (-_f(spec["k_contact"]) * y - _f(spec["c_contact"]) * vy).clamp(min=0),
                             torch.zeros_like(y))
        tangent = -friction * normal * (vx / _f(spec["v_slip"])).tanh()
        beyond_x = tangent.flip(1).cumsum(1).flip(1)[:, 1:]
        beyond_y = normal.flip(1).cumsum(1).flip(1)[:, 1:]
        diff = phi[:, :, None] - phi[:, None, :]
        force = pad(u, (1, 0)) - pad(u, (0, 1)) - g * lb * c + length * (c * beyond_y - s * beyond_x)
        force = force - ((D * diff.sin()) @ (w * w)[:, :, None])[:, :, 0]
        rx = tangent.sum(1, keepdim=True) + (lb * c * w * w).sum(1, keepdim=True)
        ry = normal.sum(1, keepdim=True) - m * g + (lb * s * w * w).sum(1, keepdim=True)
        force = force - lb / m * (-s * rx + c * ry)
        acc = torch.cholesky_solve(force[:, :, None], torch.linalg.cholesky_ex(S * diff.cos())[0])[:, :, 0]
        ax = (rx + (lb * s * acc).sum(1, keepdim=True)) / m
        ay = (ry - (lb * c * acc).sum(1, keepdim=True)) / m
        vel = vel + dt * torch.cat([ax, ay], 1)
        base = base + dt * vel
        w = w + dt * acc
        phi = phi + dt * w
    return J + _f(spec["w_term"]) * cost()


def _exact_rollout(case, seed):
    spec = _rollout_spec(case, seed)
    x0 = torch.tensor(_start(spec, np.random.default_rng(seed)), device=DEV).double()
    U = _controls(case["B"], case["H"], spec["n"], spec["u_min"], spec["u_max"], seed)
    roll = {"pointmass": _roll_pointmass, "chain": _roll_chain, "legged": _roll_legged}[spec["dyn"]]
    scale = _scales(spec, {"pointmass": spec["n"], "chain": spec["n_links"], "legged": spec["n_links"] + 1}[spec["dyn"]])
    if spec["dr_mode"] == "shared":
        J = sum(roll(spec, x0, U, scale[r:r + 1]) for r in range(spec["R"])) / spec["R"]
    else:
        J = roll(spec, x0, U, scale)
    return torch.where(J.isfinite(), J, torch.full_like(J, float("inf")))


def _bspline_basis(p, x):
    """The cardinal B-spline of degree p on the knots 0..p+1 (Def. 2)."""
    if p == 0:
        return ((x >= 0) & (x < 1)).astype(np.float64)
    return (x * _bspline_basis(p - 1, x) + (p + 1 - x) * _bspline_basis(p - 1, x - 1)) / p


def _interpolated(spec, C):
    """Rows (P, H, n) of the waypoints C (P, M, n): Def. 2, Def. 3 or straight lines."""
    H, M, p = spec["H"], spec["M"], spec["degree"]
    if spec["interp"] == "bspline":
        x = p + (M - p) * np.arange(H) / (H - 1)
        basis = np.stack([_bspline_basis(p, x - m) for m in range(M)], axis=1)
        basis = torch.tensor(basis, device=DEV)
        if spec["flags"] & 0x4:
            basis, C = basis.float().bfloat16().double(), C.float().bfloat16().double()
        return torch.einsum("tm,pmi->pti", basis, C)
    tau = torch.arange(H, dtype=torch.float64, device=DEV) / (H - 1)
    k = torch.clamp((torch.arange(H, device=DEV) * (M - 1)) // (H - 1), max=M - 2)
    h = 1.0 / (M - 1)
    d = (tau - k * h)[None, :, None]
    slope = (C[:, 1:] - C[:, :-1]) / h
    if spec["interp"] == "linear":
        return C[:, k] + d * slope[:, k]
    s = torch.empty_like(C)
    s[:, 0], s[:, -1] = slope[:, 0], slope[:, -1]
    s[:, 1], s[:, -2] = 0.5 * (slope[:, 0] + slope[:, 1]), 0.5 * (slope[:, -1] + slope[:, -2])
    if M > 4:
        w1 = (slope[:, 3:] - slope[:, 2:-1]).abs()
        w2 = (slope[:, 1:-2] - slope[:, :-3]).abs()
        s[:, 2:-2] = (w1 * slope[:, 1:-2] + w2 * slope[:, 2:-1]) / (w1 + w2)
    c2 = (3 * slope - 2 * s[:, :-1] - s[:, 1:]) / h
    c3 = (s[:, :-1] + s[:, 1:] - 2 * slope) / h ** 2
    return C[:, k] + d * (s[:, k] + d * (c2[:, k] + d * c3[:, k]))


def _exact_generate(case, seed):
    spec = _generate_spec(case, seed)
    B, H, n, M, N = (spec[k] for k in ("B", "H", "n", "M", "N"))
    P = min(int(math.floor(case["beta"] * B)), B - 1)
    L = B - P - 1
    lo, hi = _t64(spec["u_min"]), _t64(spec["u_max"])
    mu, sigma = (torch.tensor(a, device=DEV).float().double() for a in _state_before(case, seed))
    out = torch.empty(B, H, n, dtype=torch.float64, device=DEV)
    # local rows: standard normal pairs by Box-Muller
    w = _words(L, 4 * ((H * n + 3) // 4), 3, seed).reshape(L, -1, 2)
    radius = (-2.0 * (_unit(w[:, :, 0]) + 2.0 ** -24).log()).sqrt()
    angle = 2.0 * math.pi * _unit(w[:, :, 1])
    eps = torch.stack([radius * angle.cos(), radius * angle.sin()], dim=2).reshape(L, -1)[:, :H * n]
    out[:L] = mu + sigma * eps.reshape(L, H, n)
    del w, radius, angle, eps
    # graph rows: knots uniform in the box, one node per layer and path
    Z = lo + (hi - lo) * _unit(_words(M * N, n, 1, seed))
    j = (_words(P, M, 2, seed) * N) >> 32
    C = Z.reshape(M, N, n)[torch.arange(M, device=DEV)[None, :], j]
    out[L:L + P] = _interpolated(spec, C)
    out[B - 1] = mu
    return torch.minimum(torch.maximum(out, lo), hi)


def _exact_elite(case, seed):
    cost, U = _elite_inputs(case, seed)
    order = torch.argsort(cost.double(), stable=True)[:case["E"]]
    c = cost.double()[order]
    u = U[order].double()
    w = torch.exp(-(c - c[0]) / 5.0)
    if case["rule"] == "plain_cem":
        w = torch.ones_like(w)
    w = (w / w.sum())[:, None, None]
    mu = (w * u).sum(0)
    var = (w * (u - mu).square()).sum(0)
    if case["rule"] == "plain_cem":
        sigma = (var * (case["E"] / (case["E"] - 1.0))).sqrt()
    else:
        sigma = var.sqrt().clamp(min=0.1)
    return [None, U[order[0], 0].double(), mu, sigma]


def exact(case, seed):
    """In 64 bits; none for whole planner iterations, where one rounding
    decides between two elites."""
    kinds = {"rollout": _exact_rollout, "generate": _exact_generate, "elite": _exact_elite}
    return kinds[case["kind"]](case, seed) if case["kind"] in kinds else None
