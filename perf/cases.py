"""The workloads the simulator is timed on: whole calls through the public entry points
(`mpm.Simulator`, `mass_spring.MassSprings`), inputs made on the GPU from a seed.

A case is a dict of plain values:
  kind      "mpm" or "springs"
  mpm       body ("box": elastic boxes, "rects": uneven 2D rectangles, "robot": actuated boxes,
            "liquid": a standing column, "pool": an actuated robot in a liquid), dim, n_grid,
            scenes, the particle lattice nx, ny, nz (2D: nx, ny; "rects": the largest scene's
            particle count n_max), material, steps, ckpt_every, grad (backward too),
            deterministic, hidden (units of the closed-loop controller, 0: open loop or none)
  springs   dim, masses, springs, systems, states

One pass of an mpm case is one iteration of an optimisation loop: load the initial state and
parameters, run the steps, take the final state, and with grad seed the reverse pass and take
every gradient.  One pass of a springs case records the states and runs the reverse pass.
"""
import math

import numpy as np
import torch

from paper_1910_00935_gb300 import mass_spring, mpm

FCR, NH, LIQ, MIX = (mpm.MPM_FIXED_COROTATED, mpm.MPM_NEO_HOOKEAN, mpm.MPM_LIQUID, mpm.MPM_MIXED)
GROUPS, BASIS, PERIOD = 8, 4, 50.0
CTRL_SCALE = 50.0
MAX_MASSES = 8  # MS_MAX_MASSES of include/mass_spring.h
STIFFNESS, DAMPING, SPRING_DT, MASS = 100.0, 10.0, 2e-3, 1.0


def _mpm(name, body, dim, n_grid, scenes, n, material, steps, ckpt_every, grad, deterministic=False, hidden=0):
    c = {"name": name, "kind": "mpm", "body": body, "dim": dim, "n_grid": n_grid, "scenes": scenes,
         "material": material, "steps": steps, "ckpt_every": ckpt_every, "grad": grad,
         "deterministic": deterministic, "hidden": hidden}
    c.update(zip(("nx", "ny", "nz"), n))
    return c


def _springs(name, dim, masses, springs, systems, states):
    return {"name": name, "kind": "springs", "dim": dim, "masses": masses, "springs": springs,
            "systems": systems, "states": states}


def listed():
    return [
        # a preview of one small 2D body (the paper's 2D elastic object): a rollout, no gradients;
        # 32 blocks, so launches and latency count
        _mpm("square2d", "box", 2, 128, 1, (64, 64), FCR, 128, 32, False),
        # gradients of one small, oddly sized 2D body: the inner loop of an inverse problem
        _mpm("square2d_grad", "box", 2, 128, 1, (61, 57), FCR, 384, 32, True),
        # a batch of 64 uneven 2D rectangles trained together (ragged scenes, 1K to 16K particles)
        _mpm("rects2d_grad", "rects", 2, 128, 64, (16384, 0), FCR, 192, 32, True),
        # one 3D elastic cube, 262,144 particles: a rollout for validation
        _mpm("cube3d", "box", 3, 128, 1, (64, 64, 64), NH, 256, 64, False),
        # the same cube, forward and reverse: the headline workload, at a quarter of its length
        _mpm("cube3d_grad", "box", 3, 128, 1, (64, 64, 64), NH, 256, 64, True),
        # an oddly sized body on an odd grid in the bitwise reproducible mode, automatic checkpoints
        _mpm("cube3d_repro", "box", 3, 100, 1, (45, 39, 51), NH, 48, 0, True, deterministic=True),
        # 16 actuated soft robots of 65,536 particles, the open-loop weights being trained
        _mpm("robots3d_grad", "robot", 3, 64, 16, (64, 32, 32), FCR, 128, 64, True),
        # 4 robots of 27,648 particles driven by a neural controller, its parameters being trained
        _mpm("robots_nn_grad", "robot", 3, 64, 4, (48, 24, 24), FCR, 192, 64, True, hidden=32),
        # a dam break of weakly compressible liquid, 49,152 particles
        _mpm("liquid3d_grad", "liquid", 3, 64, 1, (32, 48, 32), LIQ, 256, 32, True),
        # an actuated robot standing in a pool of liquid: two materials in one grid
        _mpm("pool3d_grad", "pool", 3, 64, 1, (96, 12, 48), MIX, 192, 32, True),
        # the mass-spring triangle, 1,048,576 copies, its rest lengths being optimised
        _springs("triangles", 2, 3, 3, 1 << 20, 256),
        # a larger mass-spring network in 3D, an odd number of copies
        _springs("networks", 3, 8, 14, 100003, 128),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    which = rng.choice(["box2", "rects", "box3", "box3", "robot", "robot_nn", "liquid", "pool", "springs", "springs"])
    if which == "springs":
        masses = rng.randint(2, MAX_MASSES)
        springs = rng.randint(masses - 1, min(2 * masses, masses * (masses - 1) // 2))
        states = _log(rng, 32, 256)
        most = (1 << 28) // (states * max(springs, masses))
        return {k: v for k, v in _springs("", rng.choice([2, 3]), masses, springs,
                                          min(_log(rng, 1000, 1 << 20), most), states).items() if k != "name"}
    grad = rng.random() < 0.75
    det = rng.random() < 0.2 and which in ("box2", "rects", "box3")
    ckpt = rng.choice([0, 16, 32, 64])
    if which == "box2":
        nx = _log(rng, 16, 140)
        c = _mpm("", "box", 2, rng.choice([96, 128, 160, 250]), 1, (nx, max(8, min(140, int(nx * rng.uniform(0.6, 1.6))))),
                 rng.choice([FCR, NH]), _log(rng, 32, 384), ckpt, grad, det)
    elif which == "rects":
        c = _mpm("", "rects", 2, 128, _log(rng, 4, 64), (_log(rng, 3000, 16384), 0), rng.choice([FCR, FCR, NH]),
                 _log(rng, 24, 128), ckpt, grad, det)
    elif which == "box3":
        n = [_log(rng, 10, 64) for _ in range(3)]
        c = _mpm("", "box", 3, rng.choice([96, 100, 128]), 1, n, rng.choice([NH, NH, FCR]), _log(rng, 24, 192), ckpt, grad, det)
    elif which in ("robot", "robot_nn"):
        nx = _log(rng, 24, 64)
        scenes = _log(rng, 1, 16 if which == "robot" else 4)
        c = _mpm("", "robot", 3, 64, scenes, (nx, max(10, nx // 2 + rng.randint(-3, 3)), max(10, nx // 2 + rng.randint(-3, 3))),
                 FCR, _log(rng, 24, 96), ckpt, grad, False, 0 if which == "robot" else rng.choice([8, 16, 32, 64]))
    elif which == "liquid":
        if rng.random() < 0.4:
            c = _mpm("", "liquid", 2, 128, 1, (_log(rng, 24, 96), _log(rng, 24, 128)), LIQ, _log(rng, 32, 256), ckpt, grad)
        else:
            c = _mpm("", "liquid", 3, 64, 1, (_log(rng, 12, 40), _log(rng, 12, 60), _log(rng, 12, 40)), LIQ, _log(rng, 24, 192),
                     ckpt, grad)
    else:
        c = _mpm("", "pool", 3, 64, 1, (_log(rng, 40, 96), rng.randint(6, 14), _log(rng, 20, 60)), MIX, _log(rng, 24, 160), ckpt, grad)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1000003 + 17)


def _u(g, shape, lo, hi):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _lattice(n, corner, h):
    ax = [corner[a] + (torch.arange(n[a], device="cuda", dtype=torch.float64) + 0.5) * h for a in range(len(n))]
    grids = torch.meshgrid(*ax, indexing="ij")
    return torch.stack([x.reshape(-1) for x in grids])


def _octants(n):
    ax = [(torch.arange(m, device="cuda") >= m // 2).to(torch.int32) << a for a, m in enumerate(n)]
    grids = torch.meshgrid(*ax, indexing="ij")
    return sum(x.reshape(-1) for x in grids).to(torch.int32)


def _body(g, x, strain, drift):
    """A body taken up in mid-motion: its lattice under a small affine deformation about its
    centre (the deformation gradient to match), a drift with a velocity gradient, noise."""
    d, n = x.shape
    c = x.mean(1, keepdim=True)
    A = torch.eye(d, device="cuda", dtype=torch.float64) + _u(g, (d, d), -strain, strain)
    L = _u(g, (d, d), -1.0, 1.0)
    v = torch.tensor(drift, device="cuda", dtype=torch.float64)[:, None] + L @ (x - c) + _u(g, (d, n), -0.05, 0.05)
    F = A.reshape(d * d, 1).expand(d * d, n) + _u(g, (d * d, n), -1e-3, 1e-3)
    C = L.reshape(d * d, 1).expand(d * d, n)
    return c + A @ (x - c), v, C, F


def _controller(g, dim, hidden):
    n_in = BASIS + 2 * dim * GROUPS
    W1 = _u(g, (hidden, n_in), -1.0, 1.0) * math.sqrt(3.0 / n_in)
    W1[:, BASIS:] *= 10.0
    W2 = _u(g, (GROUPS, hidden), -1.0, 1.0) * math.sqrt(3.0 / hidden)
    z = torch.zeros(hidden + GROUPS, device="cuda", dtype=torch.float64)
    return torch.cat([W1.reshape(-1), z[:hidden], W2.reshape(-1), z[hidden:]])


def _scene_counts(case):
    """Particle lattice of every scene (the uneven rectangles come from the case alone, so that
    two seeds differ in their values and not in their sizes)."""
    d = case["dim"]
    n = tuple(case[k] for k in ("nx", "ny", "nz")[:d])
    if case["body"] != "rects":
        return [n] * case["scenes"]
    out, rng = [], np.random.RandomState(case["scenes"] * 7919 + case["nx"])
    for _ in range(case["scenes"]):
        target = math.exp(rng.uniform(math.log(1024), math.log(case["nx"])))
        a = max(1, int(round(math.sqrt(target * rng.uniform(0.5, 2.0)))))
        out.append((a, max(1, int(round(target / a)))))
    return out


def _inputs(case, seed):
    """Initial state, parameters and reverse-pass seeds, in 64 bits on values that 32 bits hold."""
    g, d, ng = _gen(seed), case["dim"], case["n_grid"]
    dx = 1.0 / ng
    h, body = 0.5 * dx, case["body"]
    parts, dt = [], 1e-4 * min(1.0, 128.0 / ng)  # the stable step shrinks with the cell
    for n in _scene_counts(case):
        p = {}
        size = [k * h for k in n]
        if body in ("box", "rects"):
            lo = [0.1 + 0.8 * float(u) * max(0.0, 1.0 - s / 0.8) for u, s in zip(_u(g, (d,), 0.2, 0.8).tolist(), size)]
            x, v, C, F = _body(g, _lattice(n, lo, h), 0.01, [1.0] + [0.0] * (d - 1))
            E = 10 ** float(_u(g, (1,), 2.7, 3.5)) if d == 2 else 4e3
            p.update(E=E, nu=0.2 if d == 2 else 0.3, material=case["material"])
        elif body == "robot":
            lo = [0.1 + float(_u(g, (1,), 0.0, dx)), 3.5 * dx, 0.5 - size[2] / 2 + float(_u(g, (1,), 0.0, dx))]
            x, v, C, F = _body(g, _lattice(n, lo, h), 0.005, [0.0] * d)
            p.update(E=5e3, nu=0.3, material=FCR, group=_octants(n))
        else:
            lo = [0.1, 4.0 * dx] + ([0.5 - size[2] / 2] if d == 3 else [])
            x, v, C, F = _body(g, _lattice(n, lo, h), 0.003, [0.0] * d)
            p.update(E=500.0, nu=0.3, material=LIQ)
        p.update(x=x, v=v, C=C, F=F)
        if body == "pool":  # the robot stands in the pool, its lower half wet
            m = (32, 16, 16)
            lo_r = [0.1 + 2 * h, 4.0 * dx + size[1] / 2, 0.5 - m[2] * h / 2]
            xr, vr, Cr, Fr = _body(g, _lattice(m, lo_r, h), 0.005, [0.0] * d)
            nr, nl = xr.shape[1], x.shape[1]
            p = {"x": torch.cat([xr, x], 1), "v": torch.cat([vr, v], 1), "C": torch.cat([Cr, C], 1), "F": torch.cat([Fr, F], 1),
                 "E": torch.cat([torch.full((nr,), 5e3), torch.full((nl,), 500.0)]).cuda().double(), "nu": 0.3,
                 "group": torch.cat([_octants(m), torch.full((nl,), -1, dtype=torch.int32, device="cuda")]),
                 "material": torch.cat([torch.full((nr,), FCR), torch.full((nl,), LIQ)]).to("cuda", torch.int32)}
        parts.append(p)
    counts = [p["x"].shape[1] for p in parts]
    N = sum(counts)

    def rows(key, dtype=torch.float64):
        return torch.cat([p[key] if isinstance(p[key], torch.Tensor) else torch.full((k,), p[key], device="cuda", dtype=dtype)
                          for p, k in zip(parts, counts)], -1).to(dtype)

    a = {k: rows(k) for k in ("x", "v", "C", "F", "E", "nu")}
    a["E"] = a["E"] * _u(g, (N,), 0.9, 1.0)  # a material that varies from particle to particle
    if body in ("robot", "pool"):
        a["group"] = rows("group", torch.int32)
        w = [_controller(g, d, case["hidden"]) if case["hidden"] else _u(g, (GROUPS, BASIS), -50.0, 50.0) for _ in counts]
        a["w"] = torch.stack(w)
    a["material"] = rows("material", torch.int32)
    # the loss: a random functional of the final state (weights of a shape-matching loss)
    s = {"dL_dx": _u(g, (d, N), -1.0, 1.0), "dL_dv": _u(g, (d, N), -0.1, 0.1),
         "dL_dC": _u(g, (d * d, N), -1e-4, 1e-4), "dL_dF": _u(g, (d * d, N), -0.1, 0.1)}
    f32 = lambda t: t.float() if t.is_floating_point() else t  # noqa: E731
    desc = {"dim": d, "n_grid": ng, "n_particles": counts, "dt": dt, "gravity": (0.0, -9.8, 0.0), "wall_cells": 3,
            "material": case["material"], "rho": 1.0, "ckpt_every": case["ckpt_every"],
            "n_groups": GROUPS if "group" in a else 0, "n_basis": BASIS if "group" in a else 0, "act_period": PERIOD,
            "act_phase": 0.0, "deterministic_p2g": int(case["deterministic"]), "ctrl_hidden": case["hidden"],
            "ctrl_scale": CTRL_SCALE}
    return desc, {k: f32(t).contiguous() for k, t in a.items()}, {k: f32(t).contiguous() for k, t in s.items()}


def _network(case):
    n = case["masses"]
    pairs = [(i, i + s) for s in range(1, n) for i in range(n - s)]
    return pairs[:case["springs"]]


def _spring_inputs(case, seed):
    g, d, n, S = _gen(seed), case["dim"], case["masses"], case["systems"]
    # masses on a ring (3D: alternately raised), so that no two start close together
    at = 2.0 * math.pi * (torch.arange(n, device="cuda", dtype=torch.float64) / n) + float(_u(g, (1,), 0.0, 1.0))
    up = 0.08 * (torch.arange(n, device="cuda", dtype=torch.float64) % 2)
    base = torch.stack([0.15 * torch.cos(at), 0.15 * torch.sin(at), up][:d], 1)[:, :, None]
    x0 = (base + _u(g, (n, d, S), -0.01, 0.01)).reshape(n * d, S)
    v0 = _u(g, (n * d, S), -0.2, 0.2)
    pairs = _network(case)
    rest = torch.stack([(x0.view(n, d, S)[i] - x0.view(n, d, S)[j]).norm(dim=0) for i, j in pairs]) * _u(g, (len(pairs), S), 0.85, 1.15)
    seeds = _u(g, (2, n * d, S), -1.0, 1.0)
    return pairs, [t.float().contiguous() for t in (x0, v0, rest, seeds[0], seeds[1])]


def prepare(case, seed):
    if case["kind"] == "springs":
        pairs, t = _spring_inputs(case, seed)
        sim = mass_spring.MassSprings(case["dim"], case["masses"], pairs, case["systems"], STIFFNESS, DAMPING, SPRING_DT, MASS,
                                      steps=case["states"])
        return {"case": case, "sim": sim, "inputs": t[:3], "seeds": t[3:]}
    desc, a, s = _inputs(case, seed)
    return {"case": case, "sim": mpm.Simulator(desc, case["steps"]), "inputs": a, "seeds": s}


def run(state):
    case, sim, a = state["case"], state["sim"], state["inputs"]
    if case["kind"] == "springs":
        sim.forward(*a, case["states"])
        x, v = sim.state()
        gx, gv, gl = sim.backward(*state["seeds"])
        return {"x": x, "v": v, "gx0": gx, "gv0": gv, "grest": gl}
    sim.set_initial(a["x"], a["v"], a["C"], a["F"], a["E"], a["nu"], a.get("group"), a.get("w"),
                    a["material"] if case["material"] == MIX else None)
    sim.forward(case["steps"])
    out = dict(zip(("x", "v", "C", "F"), sim.state()))
    if case["grad"]:
        g = sim.backward(**state["seeds"])
        out.update((k, t) for k, t in g.items() if t.numel())
    return out


def work(case):
    """Bytes: inputs read once, outputs written once (a springs case records its states, which
    are part of what it returns).  FLOPs: one particle's arithmetic for a step and its reverse
    (weights, two transfers over 3^d nodes, the stress), per particle and step."""
    d = case["dim"]
    if case["kind"] == "springs":
        rows, S, m, T = case["masses"] * d, case["systems"], case["springs"], case["states"]
        return {"bytes": 4 * S * (2 * rows * T + rows * T + 8 * rows + 2 * m),
                "flops": float(S) * (T - 1) * (m * (7 * d + 12) + 6 * rows + m * (12 * d + 24) + 4 * rows)}
    counts = _scene_counts(case)
    N = sum(math.prod(n) for n in counts) + (32 * 16 * 16 if case["body"] == "pool" else 0)
    state = 2 * d + 2 * d * d
    nodes = 3 ** d
    fwd = nodes * (2 * d + 3 * d * d + 2 + 4 * d + 2 * d) + 120 * (d - 1)
    bwd = nodes * (2 * (2 * d + 3 * d * d) + 8 * d + 12 * d) + 240 * (d - 1)
    floats = (state + 2) + state + (state + state + 2 if case["grad"] else 0)
    return {"bytes": 4 * N * floats, "flops": float(N) * case["steps"] * (fwd + (bwd if case["grad"] else 0))}


# ---------------------------------------------------------------------------
# the same, plainly, in 64 bits
# ---------------------------------------------------------------------------

def _cof(F):
    d = F.shape[0]
    if d == 2:
        return torch.stack([torch.stack([F[1, 1], -F[1, 0]]), torch.stack([-F[0, 1], F[0, 0]])])
    r = []
    for i in range(3):
        i1, i2 = (i + 1) % 3, (i + 2) % 3
        r.append(torch.cross(F[i1], F[i2], dim=0))
    return torch.stack(r)


def _mm(A, B):
    return torch.stack([torch.stack([sum(A[i, k] * B[k, j] for k in range(A.shape[1])) for j in range(B.shape[1])])
                        for i in range(A.shape[0])])


def _rotation(F):
    """Polar factor of F [d, d, n], differentiable: Newton's iteration for the value, the
    linearised W S + S W = R^T dF - dF^T R for the derivative."""
    d = F.shape[0]
    with torch.no_grad():
        R = F.detach().clone()
        for _ in range(40):
            c = _cof(R)
            Rn = 0.5 * (R + c / (R[0] * c[0]).sum(0))
            done = (Rn - R).abs().max() < 1e-15
            R = Rn
            if done:
                break
        S = _mm(R.transpose(0, 1), F.detach())
        S = 0.5 * (S + S.transpose(0, 1))
        tr = sum(S[i, i] for i in range(d))
    M = _mm(R.transpose(0, 1), F - F.detach())
    if d == 2:
        w = (M[1, 0] - M[0, 1]) / tr
        W = torch.stack([torch.stack([torch.zeros_like(w), -w]), torch.stack([w, torch.zeros_like(w)])])
    else:
        b = torch.stack([M[2, 1] - M[1, 2], M[0, 2] - M[2, 0], M[1, 0] - M[0, 1]])
        with torch.no_grad():
            G = -S + tr * torch.eye(3, device=F.device, dtype=F.dtype)[:, :, None]
            c = _cof(G)
            inv = c.transpose(0, 1) / (G[0] * c[0]).sum(0)
        w = torch.stack([sum(inv[i, k] * b[k] for k in range(3)) for i in range(3)])
        z = torch.zeros_like(w[0])
        W = torch.stack([torch.stack([z, -w[2], w[1]]), torch.stack([w[2], z, -w[0]]), torch.stack([-w[1], w[0], z])])
    return R + _mm(R, W)


class _Plain:
    """MLS-MPM steps as plain torch in 64 bits."""

    def __init__(self, desc, a):
        self.d, self.ng, self.S = desc["dim"], desc["n_grid"], len(desc["n_particles"])
        f = lambda v: float(np.float32(v))  # noqa: E731  (the entry points take these as 32-bit values)
        self.dt, self.dx, self.rho = f(desc["dt"]), 1.0 / desc["n_grid"], f(desc["rho"])
        self.gravity = [f(v) for v in desc["gravity"]][:self.d]
        self.V0 = (0.5 * self.dx) ** self.d
        self.m = self.rho * self.V0
        self.hidden, self.scale = desc["ctrl_hidden"], f(desc["ctrl_scale"])
        self.scene = torch.repeat_interleave(torch.arange(self.S, device="cuda"), torch.tensor(desc["n_particles"], device="cuda"))
        self.mat, self.group = a["material"], a.get("group")
        self.kinds = sorted(set(self.mat.unique().tolist()))
        ax = torch.arange(self.ng, device="cuda")
        free = (ax >= desc["wall_cells"]) & (ax < self.ng - desc["wall_cells"])
        inside = free
        for _ in range(self.d - 1):
            inside = inside[..., None] & free
        self.inside = inside.reshape(-1).repeat(self.S)
        o = torch.stack(torch.meshgrid(*[torch.arange(3, device="cuda")] * self.d, indexing="ij")).reshape(self.d, -1)
        self.offsets = o

    def stencil(self, x):
        X = x * self.ng
        base = (X.detach() - 0.5).floor()
        f = X - base
        w = torch.stack([0.5 * (1.5 - f) ** 2, 0.75 - (f - 1.0) ** 2, 0.5 * (f - 0.5) ** 2])  # [3, d, n]
        W = w[self.offsets[0], 0]
        idx = self.scene * 1
        for a in range(self.d):
            if a:
                W = W * w[self.offsets[a], a]
            idx = idx * self.ng + base[a].long().clamp(0, self.ng - 3)  # (a body that left the grid is not indexed outside it)
        step = sum(self.offsets[a] * self.ng ** (self.d - 1 - a) for a in range(self.d))
        dp = [(self.offsets[a][:, None] - f[a]) * self.dx for a in range(self.d)]  # each [3^d, n]
        return W, dp, (idx[None] + step[:, None]).reshape(-1)

    def actuation(self, x, v, w, t):
        """Actuation of every particle at step t (0 outside the groups)."""
        if self.group is None:
            return None
        basis = torch.tensor([math.sin(2 * math.pi * k * t / PERIOD) for k in range(1, BASIS + 1)], device="cuda", dtype=torch.float64)
        g = self.group.long()
        if not self.hidden:
            act = w.reshape(self.S, GROUPS, BASIS) @ basis
        else:
            d, H, n_in = self.d, self.hidden, BASIS + 2 * self.d * GROUPS
            slot = self.scene * GROUPS + g
            one = torch.zeros(self.S * GROUPS, device="cuda", dtype=torch.float64).index_add(0, slot, torch.ones_like(x[0]))
            mean = lambda q: torch.zeros_like(one).index_add(0, slot, q) / one  # noqa: E731
            n_s = torch.zeros(self.S, device="cuda", dtype=torch.float64).index_add(0, self.scene, torch.ones_like(x[0]))
            com = [torch.zeros_like(n_s).index_add(0, self.scene, x[a]) / n_s for a in range(d)]
            sens = [mean(x[a]).reshape(self.S, GROUPS) - com[a][:, None] for a in range(d)]
            sens += [mean(v[a]).reshape(self.S, GROUPS) for a in range(d)]
            u = torch.cat([basis.expand(self.S, BASIS), torch.stack(sens, 2).reshape(self.S, -1)], 1)
            W1, b1, W2, b2 = torch.split(w, [H * n_in, H, GROUPS * H, GROUPS], dim=1)
            hid = torch.tanh((W1.reshape(self.S, H, n_in) @ u[:, :, None])[..., 0] + b1)
            act = self.scale * torch.tanh((W2.reshape(self.S, GROUPS, H) @ hid[:, :, None])[..., 0] + b2)
        return torch.where(g >= 0, act[self.scene, g.clamp(min=0)], torch.zeros_like(x[0]))

    def stress(self, F, mu, la, act):
        d = self.d
        eye = torch.eye(d, device="cuda", dtype=torch.float64)[:, :, None]
        J = (F[0] * _cof(F)[0]).sum(0)
        tau = torch.zeros_like(F)
        for k in self.kinds:
            on = (self.mat == k).to(torch.float64)
            if k == FCR:
                t = 2 * mu * _mm(F - _rotation(F), F.transpose(0, 1)) + la * (J - 1) * J * eye
            elif k == NH:
                t = mu * (_mm(F, F.transpose(0, 1)) - eye) + la * torch.log(J) * eye
            else:
                t = (la + 2 * mu / d) * (J - J ** -6) * eye
            tau = tau + on * t
        if act is not None:
            e = torch.remainder(self.group.clamp(min=0).long(), d)
            fe = torch.stack([sum(F[i, j] * (e == j) for j in range(d)) for i in range(d)])
            tau = tau + act * fe[:, None] * fe[None]
        return tau

    def step(self, x, v, C, F, mu, la, w, t):
        d, nn = self.d, self.S * self.ng ** self.d
        W, dp, idx = self.stencil(x)
        tau = self.stress(F, mu, la, self.actuation(x, v, w, t))
        A = (-self.dt * self.V0 * 4.0 / self.dx ** 2) * tau + self.m * C
        zero = torch.zeros(nn, device="cuda", dtype=torch.float64)
        gm = zero.index_add(0, idx, (self.m * W).reshape(-1))
        touched = gm > 0
        keep = touched & self.inside
        u = []
        for a in range(d):
            q = self.m * v[a] + sum(A[a, b] * dp[b] for b in range(d))
            p = zero.index_add(0, idx, (W * q).reshape(-1))
            va = p / torch.where(touched, gm, torch.ones_like(gm)) + self.dt * self.gravity[a]
            u.append(torch.where(keep, va, torch.zeros_like(va))[idx].reshape(W.shape))
        v2 = torch.stack([(W * u[a]).sum(0) for a in range(d)])
        C2 = torch.stack([torch.stack([(W * u[a] * dp[b]).sum(0) for b in range(d)]) for a in range(d)]) * (4.0 / self.dx ** 2)
        return x + self.dt * v2, v2, C2, F + self.dt * _mm(C2, F)


def _exact_mpm(case, seed):
    from torch.utils.checkpoint import checkpoint
    desc, a, s = _inputs(case, seed)
    P, d, N = _Plain(desc, a), case["dim"], a["x"].shape[1]
    leaf = {k: a[k].double().requires_grad_(case["grad"]) for k in ("x", "v", "C", "F", "E", "nu", "w") if k in a}
    mu = leaf["E"] / (2 * (1 + leaf["nu"]))
    la = leaf["E"] * leaf["nu"] / ((1 + leaf["nu"]) * (1 - 2 * leaf["nu"]))
    x, v, C, F = leaf["x"], leaf["v"], leaf["C"].reshape(d, d, N), leaf["F"].reshape(d, d, N)
    for t in range(case["steps"]):
        args = (x, v, C, F, mu, la, leaf.get("w"), t)
        x, v, C, F = checkpoint(P.step, *args, use_reentrant=False) if case["grad"] else P.step(*args)
    out = {"x": x, "v": v, "C": C.reshape(d * d, N), "F": F.reshape(d * d, N)}
    if case["grad"]:
        L = sum((out[k] * s["dL_d" + k].double()).sum() for k in out)
        names = {"x": "gx0", "v": "gv0", "C": "gC0", "F": "gF0", "E": "gE", "nu": "gnu", "w": "gw"}
        for k, g in zip(leaf, torch.autograd.grad(L, list(leaf.values()))):
            out[names[k]] = g
    return {k: t.detach() for k, t in out.items()}


def _exact_springs(case, seed):
    from torch.utils.checkpoint import checkpoint
    pairs, t = _spring_inputs(case, seed)
    d, n, S = case["dim"], case["masses"], case["systems"]
    x0, v0, rest = (q.double().requires_grad_(True) for q in t[:3])
    k, dt, m = STIFFNESS, float(np.float32(SPRING_DT)), MASS
    decay = math.exp(-dt * DAMPING)

    def steps(x, v, rest, count):
        for _ in range(count):
            f = [0.0] * n
            for j, (a, b) in enumerate(pairs):
                dd = x[a * d:a * d + d] - x[b * d:b * d + d]
                length = dd.norm(dim=0) + 1e-4
                q = k * (length - rest[j]) / length * dd
                f[a], f[b] = f[a] - q, f[b] + q
            f = torch.cat([q if isinstance(q, torch.Tensor) else torch.zeros(d, S, device="cuda", dtype=torch.float64) for q in f])
            v = decay * v + dt * f / m
            x = x + dt * v
        return x, v

    x, v, left = x0, v0, case["states"] - 1
    while left:
        x, v = checkpoint(steps, x, v, rest, min(8, left), use_reentrant=False)
        left -= min(8, left)
    L = (x * t[3].double()).sum() + (v * t[4].double()).sum()
    gx, gv, gl = torch.autograd.grad(L, [x0, v0, rest])
    return {k: q.detach() for k, q in zip(("x", "v", "gx0", "gv0", "grest"), (x, v, gx, gv, gl))}


def exact(case, seed):
    if case["kind"] == "springs":
        return _exact_springs(case, seed)
    return _exact_mpm(case, seed)
