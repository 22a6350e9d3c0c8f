"""The workloads whose speed is followed: what a user of this framework has it do.

Each case is one pass of a control or planning loop through the public entry
points: the particle state and the bodies of an episode are handed to the
context (device tensors), some rigid time steps run, and the new state, the
bodies and the contact impulses come back. The scenes are those of
``paper_2503_05046_gb300.scenes`` at the sizes of the tests and of the
benchmark, taken in mid-motion: a smooth velocity field with its gradient in C,
strains of a fraction of a percent to one percent in F, and bodies already
touching the particles where the scene is about contact.

Kinds of case (``case["kind"]``):
  flight    a cube of elastic material or sand away from every body: the
            transfers alone, on a dense or a block-sparse grid
  cube      an elastic cube at touch-down on the ground, beside a moving sphere
  squeeze   a cube held between two force-controlled panels (dynamic bodies)
  sand      randomly sampled sand on the ground
  scoop     granular scooping: a bin of sand with two moving paddles
  mixed     elastic and sand objects on a floor with a gripper and obstacles
  batch     many independent scenes of uneven size advanced together
  cradle    the pinned cloth sheet with a dynamic box on it
  push      a differentiable rollout, forward and backward
"""
import math

import numpy as np
import torch

from paper_2503_05046_gb300 import autograd, native, scenes

DEV = "cuda"


def listed():
    return [
        # one substep per step, dynamic bodies: the shortest call, as an
        # interactive controller makes it (the panel squeeze of Fig. 2)
        {"name": "squeeze_1728", "kind": "squeeze", "n_side": 12, "steps": 5},
        # the 8,000-particle cube in free flight: launch latency
        {"name": "flight_8k", "kind": "flight", "material": "elastic", "n_side": 20, "steps": 2,
         "substeps": 10, "sparse": False},
        # the same cube at touch-down: a small contact solve every substep
        {"name": "cube_8k_contact", "kind": "cube", "n_side": 20, "steps": 1},
        # cloth, pins and a dynamic box: the box-bagging cradle
        {"name": "cradle_900", "kind": "cradle", "n_side": 30, "steps": 10},
        # sand in a large domain kept block-sparse, an odd size
        {"name": "flight_sparse_79k", "kind": "flight", "material": "sand", "n_side": 43, "steps": 1,
         "substeps": 10, "sparse": True},
        # several particles per cell at random, ground contact, an odd size
        {"name": "sand_250k", "kind": "sand", "n": 250_007, "ppc": 4.0, "steps": 1},
        # one million elastic particles in flight: the transfers at size
        {"name": "flight_1M", "kind": "flight", "material": "elastic", "n_side": 100, "steps": 1,
         "substeps": 10, "sparse": False},
        # granular scooping at the benchmark's size, with the P2G form that
        # the tuner picks at about one particle per cell
        {"name": "scoop_1M", "kind": "scoop", "n": 1_000_000, "steps": 1, "form": 1, "chunk": 256},
        # the headline workload: 4M particles in 32 objects, 12 bodies, with
        # the P2G form the tuner picks for it
        {"name": "mixed_4M", "kind": "mixed", "objects": 32, "per_object": 125_000, "steps": 1,
         "form": 0, "chunk": 1024},
        # batched scenes of uneven size
        {"name": "batch_24", "kind": "batch", "scenes": 24, "n_min": 2000, "n_max": 64000, "steps": 1,
         "substeps": 4},
        # the differentiable push: 25 substeps forward, and back
        {"name": "push_65536", "kind": "push", "n": 65_536, "steps": 1, "substeps": 25},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["squeeze", "flight", "flight", "cube", "sand", "scoop", "mixed", "batch", "cradle", "push"])
    if kind == "squeeze":
        return {"kind": kind, "n_side": rng.randint(6, 18), "steps": rng.randint(2, 8)}
    if kind == "flight":
        return {"kind": kind, "material": rng.choice(["elastic", "sand"]), "n_side": _log(rng, 12, 100),
                "steps": 1, "substeps": rng.randint(3, 10), "sparse": rng.random() < 0.3}
    if kind == "cube":
        return {"kind": kind, "n_side": rng.randint(10, 32), "steps": 1}
    if kind == "sand":
        return {"kind": kind, "n": _log(rng, 20_000, 1_000_000), "ppc": round(rng.uniform(1.0, 8.0), 2), "steps": 1}
    if kind == "scoop":
        return {"kind": kind, "n": _log(rng, 300_000, 1_000_000), "steps": 1, "form": rng.randint(0, 1),
                "chunk": 256}
    if kind == "mixed":
        return {"kind": kind, "objects": rng.choice([8, 16, 24]), "per_object": _log(rng, 20_000, 125_000),
                "steps": 1, "form": 0, "chunk": rng.choice([256, 1024])}
    if kind == "batch":
        return {"kind": kind, "scenes": rng.randint(4, 32), "n_min": 2000, "n_max": _log(rng, 8_000, 64_000),
                "steps": 1, "substeps": rng.randint(2, 4)}
    if kind == "cradle":
        return {"kind": kind, "n_side": rng.randint(22, 30), "steps": rng.randint(7, 10)}
    return {"kind": kind, "n": _log(rng, 8_000, 65_536), "steps": 1, "substeps": rng.randint(5, 25)}


# ------------------------------------------------------------------ inputs

def _sand_near(x, coord, wall, band, sign, rng):
    """Sand within `band` of a wall rests against it: up to 4e-6 m inside
    (a column's weight over 1e4 N/m)."""
    near = np.abs(x[:, coord] - wall) < band
    x[near, coord] = wall + sign * 4e-6 * rng.random(int(near.sum()), dtype=np.float32)


def _scene(case, seed):
    """(scene, dynamics {body: dict}) of a single-scene case."""
    kind = case["kind"]
    rng = np.random.default_rng(seed)
    if kind == "squeeze":
        # (10 N over the face's contacts of 1e4 N/m: 7e-6 m deep)
        sc, dyn = scenes.panel_squeeze(n_side=case["n_side"], overlap=7e-6)
        return sc, {0: dyn[0], 1: dyn[1]}
    if kind == "flight":
        mat = scenes.elastic() if case["material"] == "elastic" else dict(scenes.SAND)
        n, dx = case["n_side"], 0.01
        g = scenes.cube_group(n, dx / 2, (0.0, 0.0, 0.0), (0.0, 0.0, -0.5), mat, jitter=0.05 * dx, rng=rng)
        res = 256 if case["sparse"] else 4 * math.ceil((n / 2 + 14) / 4)
        grid = {"dx": dx, "res": (res, res, res), "origin": (-res * dx / 2,) * 3,
                "gravity": (0.0, 0.0, -9.81), "bc_layers": 3}
        if case["sparse"]:
            grid["max_blocks"] = (math.ceil(n / 8) + 4) ** 3
        return {"name": "flight", "grid": grid, "groups": [g],
                "bodies": [scenes.body(scenes.HALFSPACE, p=(0.0, 0.0, -res * dx / 2))], "h": 1e-4,
                "substeps": case["substeps"]}, {}
    if kind == "cube":
        return scenes.cube_contact(n_side=case["n_side"], seed=seed, penetration=4e-6,
                                   sphere_overlap=2e-5), {}
    if kind == "sand":
        return scenes.sand_random(case["n"], case["ppc"], seed=seed, penetration=2e-5), {}
    if kind == "scoop":
        # the sand has settled: its outermost particles rest on floor, walls
        # and paddles
        sc = scenes.granular_scoop(case["n"], seed=seed)
        x = sc["groups"][0]["x"]
        _sand_near(x, 2, 0.0, 5e-4, -1, rng)
        for axis in (0, 1):
            for s in (-1, 1):
                _sand_near(x, axis, s * 0.15, 1e-4, s, rng)
        for b in sc["bodies"][5:]:
            b["p"] = b["p"] + np.array([1e-5, 0.0, 0.0])
        return sc, {}
    if kind == "mixed":
        sc = scenes.mixed_manipulation(case["objects"], case["per_object"], seed=seed)
        for g in sc["groups"]:  # the objects stand on the floor
            low = g["x"][:, 2] < 1e-5
            g["x"][low, 2] = -2e-8 * rng.random(int(low.sum()), dtype=np.float32)
        for b, s in zip(sc["bodies"][1:3], (-1, 1)):  # the jaws are about to touch theirs
            b["p"] = b["p"] + np.array([s * 2.1e-5, 0.0, 0.0])
        return sc, {}
    if kind == "cradle":
        sc, dyn = scenes.box_bagging(n_side=case["n_side"], sink=-2e-4)
        return sc, {1: dyn}  # (the box is about to land on the sheet)
    raise ValueError(kind)


def _motion(x, v, gen, speed, strain, cloth):
    """Velocities, their gradients (C) and deformation gradients (F) of a body
    in motion: sums of three plane waves of about the body's size."""
    n = x.shape[0]
    x64 = x.double()
    size = float((x64.max(0).values - x64.min(0).values).max()) + 1e-6
    vv, C = v.double(), torch.zeros(n, 3, 3, dtype=torch.float64, device=DEV)
    F = torch.eye(3, dtype=torch.float64, device=DEV).repeat(n, 1, 1)
    for _ in range(3):
        k = torch.randn(3, generator=gen, device=DEV, dtype=torch.float64) * (3.0 / size)
        a = torch.randn(3, generator=gen, device=DEV, dtype=torch.float64) * (speed / 2)
        b = torch.randn(3, 3, generator=gen, device=DEV, dtype=torch.float64) * (strain / 3)
        ph = torch.rand(2, generator=gen, device=DEV, dtype=torch.float64) * (2 * math.pi)
        arg = x64 @ k
        vv = vv + torch.sin(arg + ph[0])[:, None] * a
        C += torch.cos(arg + ph[0])[:, None, None] * (a[:, None] * k[None, :])
        if not cloth:
            F += torch.sin(arg + ph[1])[:, None, None] * b
    if not cloth:  # on average slightly compressed, as under its own weight
        F -= 0.3 * strain * torch.eye(3, dtype=torch.float64, device=DEV)
        vv = vv + 0.02 * speed * torch.randn(n, 3, generator=gen, device=DEV, dtype=torch.float64)
    return vv.float().contiguous(), C.float().contiguous(), F.float().contiguous()


def _state(sc, seed, speed, strain):
    """The episode's particle state on the device: x, v, C, F in id order."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    parts = []
    for g in sc["groups"]:
        x = torch.from_numpy(np.ascontiguousarray(g["x"])).to(DEV)
        v = torch.from_numpy(np.ascontiguousarray(g["v"])).to(DEV)
        parts.append((x,) + _motion(x, v, gen, speed, strain, "tris" in g))
    return tuple(torch.cat(f).contiguous() for f in zip(*parts))


# speed (m/s) and strain of the motion: brisk in flight, a settled body's
# where the bodies hold it
MOTION = {"flight": (0.02, 5e-3), "cradle": (0.02, 0.0)}
SETTLED = (5e-3, 1e-3)


def _inputs(case, seed):
    sc, dyn = _scene(case, seed)
    return sc, dyn, _state(sc, seed, *MOTION.get(case["kind"], SETTLED))


def _outputs(n):
    return {"x": torch.empty(n, 3, device=DEV), "v": torch.empty(n, 3, device=DEV),
            "C": torch.empty(n, 3, 3, device=DEV), "F": torch.empty(n, 3, 3, device=DEV)}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        # sizes and materials by the scenes' own seed, motion by this one
        scs = [scenes.batch_scene(i, n_min=case["n_min"], n_max=case["n_max"], penetration=2e-6)
               for i in range(case["scenes"])]
        for sc in scs:  # landed
            sc["groups"][0]["v"][:, 2] = np.float32(-0.005)
        bt = native.Batch(scs)
        ins = [_state(sc, seed * 1009 + i, *SETTLED) for i, sc in enumerate(scs)]
        out = _outputs(sum(i[0].shape[0] for i in ins))
        views, at = [], 0
        for i in ins:
            n = i[0].shape[0]
            views.append({k: t[at:at + n] for k, t in out.items()})
            at += n
        bodies = [[native.make_body(b) for b in sc["bodies"]] for sc in scs]
        return {"case": case, "batch": bt, "ins": ins, "out": out, "views": views, "bodies": bodies,
                "h": scs[0]["h"], "solver": native.solver_params()}
    if kind == "push":
        sc, target = scenes.push_cube(case["n"], seed=seed, substeps=case["substeps"],
                                      sink=1e-5, box_overlap=1e-5)
        x, v, _, _ = _state(sc, seed, *SETTLED)
        sim = native.Sim(sc)

        def leaf(a, dev="cpu"):
            return torch.as_tensor(np.asarray(a), dtype=torch.float32, device=dev).requires_grad_()

        return {"case": case, "sim": sim, "x": x.requires_grad_(), "v": v.requires_grad_(),
                "E": leaf([sc["groups"][0]["material"]["E"]]), "nu": leaf([sc["groups"][0]["material"]["nu"]]),
                "mu": leaf([b["mu"] for b in sc["bodies"]]),
                "target": torch.as_tensor(target, dtype=torch.float32, device=DEV), "bodies": sc["bodies"],
                "solver": native.solver_params(eps_r=1e-5)}
    sc, dyn, ins = _inputs(case, seed)
    sim = native.Sim(sc)
    if "form" in case:
        native.mpm_set_option(sim.ctx, native.OPT_P2G_FORM, case["form"])
        native.mpm_set_option(sim.ctx, native.OPT_P2G_CHUNK, case["chunk"])
    return {"case": case, "sim": sim, "ins": ins, "out": _outputs(ins[0].shape[0]), "dyn": dyn,
            "bodies": [native.make_body(b) for b in sc["bodies"]], "solver": native.solver_params()}


# --------------------------------------------------------------------- run

def _bodies(sims):
    """A row per body, as an observation holds it: pose, velocities, and the
    impulse and moment it took in this pass."""
    rows = []
    for s in sims:
        imp = s.impulses(reset=True)
        rows += [np.concatenate([b["p"], b["R"].ravel(), b["v"], b["omega"], i]) for b, i in zip(s.bodies(), imp)]
    return np.asarray(rows, np.float32)


def run(state):
    case = state["case"]
    if case["kind"] == "push":
        sim, leaves = state["sim"], [state[k] for k in ("x", "v", "E", "nu", "mu")]
        xf, vf = autograd.rollout(sim, case["steps"], *leaves, solver=state["solver"], eps_r=1e-5,
                                  bodies=state["bodies"])
        loss = ((xf.mean(0) - state["target"]) ** 2).sum() + 1e-2 * (vf ** 2).sum(1).mean()
        grads = torch.autograd.grad(loss, leaves)
        return {"x": xf.detach(), "v": vf.detach(), "loss": loss.detach(),
                "grads": dict(zip(("x", "v", "E", "nu", "mu"), grads))}
    if case["kind"] == "batch":
        bt = state["batch"]
        for sim, ins, bodies in zip(bt.sims, state["ins"], state["bodies"]):
            sim.set_particles(*ins)
            sim.set_bodies(bodies)
        bt.sort()
        for _ in range(case["steps"]):
            bt.step(state["h"], case["substeps"], state["solver"])
        bt.synchronize(stats=False)
        for sim, view in zip(bt.sims, state["views"]):
            sim.read_particles(view["x"], view["v"], view["C"], view["F"])
        return dict(state["out"], bodies=_bodies(bt.sims))
    sim, out = state["sim"], state["out"]
    sim.set_particles(*state["ins"])
    sim.set_bodies(state["bodies"])
    for i, d in state["dyn"].items():
        sim.set_dynamics(i, d)
    for _ in range(case["steps"]):
        sim.step(solver=state["solver"], stats=False)
    sim.read_particles(out["x"], out["v"], out["C"], out["F"])
    return dict(out, bodies=_bodies([sim]))


# -------------------------------------------------------------------- work

def _particle_substeps(case):
    """(particles, substeps) of a pass."""
    kind = case["kind"]
    if kind in ("squeeze", "flight", "cube"):
        n = case["n_side"] ** 3
    elif kind == "cradle":
        n = case["n_side"] ** 2
    elif kind == "mixed":
        n = case["objects"] * case["per_object"]
    elif kind == "batch":
        n = case["scenes"] * (case["n_min"] + case["n_max"]) // 2
    else:
        n = case["n"]
    return n, case["steps"] * (1 if kind == "squeeze" else case.get("substeps", 10))


def work(case):
    """Bytes: the state (x, v, C, F: 96 B) read and written once per substep,
    since a substep's grid depends on all particles of it, and handed in and
    out once. Arithmetic: per particle and substep 27 nodes x 20 (P2G) and
    x 24 (G2P), and about 500 for the stress and the plasticity. The contact
    solve, whose iterations depend on the state, is left out; the backward
    pass repeats the forward one and takes twice its transfers."""
    n, sub = _particle_substeps(case)
    back = 4 if case["kind"] == "push" else 1
    return {"bytes": 192 * n * (sub * back + 2), "flops": 1700 * n * sub * back}


# ------------------------------------------------------------------- exact

def _invert(A):
    """Inverse transpose of 3x3 matrices by cofactors, and determinants."""
    c = torch.stack([torch.linalg.cross(A[:, 1], A[:, 2]), torch.linalg.cross(A[:, 2], A[:, 0]),
                     torch.linalg.cross(A[:, 0], A[:, 1])], 1)
    det = (A[:, 0] * c[:, 0]).sum(-1)
    return c / det[:, None, None], det


def _eigen(A):
    """Eigenvalues and eigenvectors (columns) of symmetric 3x3 matrices by
    Jacobi's rotations."""
    A = A.clone()
    V = torch.eye(3, dtype=A.dtype, device=A.device).repeat(A.shape[0], 1, 1)
    for p, q in [(0, 1), (0, 2), (1, 2)] * 8:
        th = 0.5 * torch.atan2(2 * A[:, p, q], A[:, q, q] - A[:, p, p])
        G = torch.eye(3, dtype=A.dtype, device=A.device).repeat(A.shape[0], 1, 1)
        G[:, p, p] = G[:, q, q] = torch.cos(th)
        G[:, p, q], G[:, q, p] = torch.sin(th), -torch.sin(th)
        A = G.transpose(1, 2) @ A @ G
        V = V @ G
    return A.diagonal(dim1=1, dim2=2), V


def _kirchhoff(F, m, sand):
    """Plastic projection of F (sand) and the Kirchhoff stress of the result."""
    mu, lam = m["E"] / (2 * (1 + m["nu"])), m["E"] * m["nu"] / ((1 + m["nu"]) * (1 - 2 * m["nu"]))
    eye = torch.eye(3, dtype=torch.float64, device=F.device)
    R = F
    for _ in range(8):  # Newton's iteration for the polar factor
        R = 0.5 * (R + _invert(R)[0])
    if not sand:
        J = _invert(F)[1]
        return F, 2 * mu * (F - R) @ F.transpose(1, 2) + (lam * J * (J - 1))[:, None, None] * eye
    lw, V = _eigen(F.transpose(1, 2) @ F)
    e = 0.5 * torch.log(lw)
    tr = e.sum(1, keepdim=True)
    dev = e - tr / 3
    nh = dev.norm(dim=1, keepdim=True)
    s = math.sin(math.radians(m["friction_angle_deg"]))
    alpha = math.sqrt(2.0 / 3.0) * 2 * s / (3 - s)
    dg = nh + (3 * lam + 2 * mu) / (2 * mu) * tr * alpha
    en = torch.where(dg > 0, e - dg * dev / nh.clamp_min(1e-300), e)
    en = torch.where(tr >= 0, torch.zeros_like(e), en)
    S = V @ torch.diag_embed(torch.exp(en)) @ V.transpose(1, 2)
    U = R @ V
    tau = U @ torch.diag_embed(2 * mu * en + lam * en.sum(1, keepdim=True)) @ U.transpose(1, 2)
    return R @ S, tau


def exact(case, seed):
    """The flight cases in 64 bits: quadratic B-spline MLS-MPM without contact.
    A contact solve stops anywhere within its tolerance, so the other cases
    have no value of their own."""
    if case["kind"] != "flight":
        return None
    sc, _, ins = _inputs(case, seed)
    x, v, C, F = (t.double() for t in ins)
    g, m = sc["grid"], sc["groups"][0]["material"]
    dx, res = g["dx"], g["res"][0]
    o = torch.tensor(g["origin"], dtype=torch.float64, device=DEV)
    grav = torch.tensor(g["gravity"], dtype=torch.float64, device=DEV)
    h, vol = float(np.float32(sc["h"])), float(np.float32(sc["groups"][0]["vol"]))
    mass, dinv = vol * m["rho"], 4.0 / dx ** 2
    sand = case["material"] == "sand"
    lo = ((x.min(0).values - o) / dx).floor().long() - 3
    ext = (((x.max(0).values - o) / dx).floor().long() + 5 - lo).tolist()
    assert int(lo.min()) >= 3 and max(int(a) + b for a, b in zip(lo, ext)) <= res - 3
    # (the stress of the given F, without a projection of it)
    tau = _kirchhoff(F, m, False)[1] if not sand else _hencky(F, m)
    for _ in range(case["steps"] * case["substeps"]):
        xc = (x - o) / dx
        base = (xc - 0.5).floor()
        f = xc - base
        w = torch.stack([0.5 * (1.5 - f) ** 2, 0.75 - (f - 1) ** 2, 0.5 * (f - 0.5) ** 2])
        b = base.long() - lo
        A = mass * C - h * dinv * vol * tau
        grid = torch.zeros(ext[0] * ext[1] * ext[2], 4, dtype=torch.float64, device=DEV)
        nodes = []
        for c in range(27):
            off = torch.tensor([c % 3, c // 3 % 3, c // 9], device=DEV)
            wt = w[c % 3, :, 0] * w[c // 3 % 3, :, 1] * w[c // 9, :, 2]
            node = ((b[:, 2] + off[2]) * ext[1] + b[:, 1] + off[1]) * ext[0] + b[:, 0] + off[0]
            d = (off - f) * dx
            q = torch.cat([torch.full_like(wt, mass)[:, None], mass * v + (A @ d[:, :, None])[:, :, 0]], 1)
            grid.index_add_(0, node, wt[:, None] * q)
            nodes.append((wt, node, d))
        gv = torch.where(grid[:, :1] > 0, grid[:, 1:] / grid[:, :1].clamp_min(1e-300) + h * grav, 0.0)
        v, B = torch.zeros_like(v), torch.zeros_like(C)
        for wt, node, d in nodes:
            wv = wt[:, None] * gv[node]
            v += wv
            B += wv[:, :, None] * d[:, None, :]
        C = dinv * B
        x = x + h * v
        F, tau = _kirchhoff(F + h * C @ F, m, sand)
    return {"x": x, "v": v, "C": C, "F": F, "bodies": np.asarray(
        [np.concatenate([b["p"], b["R"].ravel(), b["v"], b["omega"], np.zeros(6)]) for b in sc["bodies"]])}


def _hencky(F, m):
    """Kirchhoff stress of Hencky elasticity, no projection."""
    mu, lam = m["E"] / (2 * (1 + m["nu"])), m["E"] * m["nu"] / ((1 + m["nu"]) * (1 - 2 * m["nu"]))
    lw, U = _eigen(F @ F.transpose(1, 2))
    e = 0.5 * torch.log(lw)
    return U @ torch.diag_embed(2 * mu * e + lam * e.sum(1, keepdim=True)) @ U.transpose(1, 2)
