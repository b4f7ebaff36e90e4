"""What this framework is used for, as cases that can be timed and checked.

A case is a dict of plain values.  `listed()` gives the standing ones, `draw`
more of the same ranges; `prepare` makes from a seed what a user's program has
in hand before the call, `run` is one pass through the public entry points,
`work` the bytes and operations such a pass cannot do without and `exact` its
result in 64 bits, written with torch alone.

Kinds of case:
  coupled  `steps` whole time steps of a lattice with particles: the driver
           hands over the particles' poses (page-locked host memory), steps,
           and takes back the poses, the populations of the fluid nodes and
           the node classes
  bed      `substeps` DEM substeps (contact detection, contact forces, rigid
           bodies) of a packed bed without the fluid
  train    one training step of the contact network: forward, loss, backward,
           AdamW
  ga       contour capture by the Genetic Algorithm on one hull
  gs       Gradient Search refinement of many models
  shape    shape descriptors of many models
"""
import math

import numpy as np
import torch

from paper_2209_10411_gb300 import _binding as B
from paper_2209_10411_gb300 import scenes

STORAGE = {"f32": B.STORE_F32, "f16": B.STORE_F16_DEV, "bf16": B.STORE_BF16_DEV}
ELEMENT = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1)]
W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]
GRAVITY = (0.0, 0.0, -1e-5)
DENSITY, SKIN = 2.5, 1.0


def _coupled(name, nx, ny, nz, storage, particles, shape, balls, radii, steps, bb="ibb", periodic="", force=0.0,
             substeps=1):
    c = {"kind": "coupled", "nx": nx, "ny": ny, "nz": nz, "storage": storage, "particles": particles, "shape": shape,
         "balls_lo": balls[0], "balls_hi": balls[1], "r_lo": radii[0], "r_hi": radii[1], "steps": steps, "bb": bb,
         "periodic": periodic, "force": force, "substeps": substeps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest simulation: one four-ball particle in a 64^3 box; launches and latency
        _coupled("box64_f32", 64, 64, 64, "f32", 1, "blob", (4, 4), (6.0, 6.0), 20),
        # a forced channel with odd sizes, periodic along x, halfway links
        _coupled("channel_ragged_ladd_f32", 141, 83, 119, "f32", 4, "clustered", (8, 32), (6.0, 9.0), 20, bb="ladd",
                 periodic="x", force=2e-6),
        # the settling tank, in both storages it is run with
        _coupled("tank_f32", 256, 256, 512, "f32", 3, "cobble", (24, 40), (12.0, 20.0), 20),
        _coupled("tank_f16", 256, 256, 512, "f16", 3, "cobble", (24, 40), (12.0, 20.0), 20),
        # the suspension of 300 particles: the largest lattice
        _coupled("suspension_f32", 512, 512, 512, "f32", 300, "clustered", (8, 64), (8.0, 16.0), 10),
        _coupled("suspension_bf16", 512, 512, 512, "bf16", 300, "clustered", (8, 64), (8.0, 16.0), 10),
        # a pair of grains in a channel with the paper's 100 DEM substeps per lattice step
        _coupled("pair_substeps_f32", 128, 128, 256, "f32", 2, "clustered", (16, 32), (9.0, 12.0), 5, substeps=100),
        # the packed bed: contacts alone
        {"name": "bed_contacts", "kind": "bed", "particles": 3000, "balls_lo": 4, "balls_hi": 128, "spacing": 18.7,
         "substeps": 10},
        # training of the contact network
        {"name": "train_step", "kind": "train", "batch": 4096},
        # fitting of particle shapes: capture, refinement, descriptors
        {"name": "capture", "kind": "ga", "individuals": 1200, "genes": 32, "points": 2048, "generations": 20,
         "mutate": 0.05},
        {"name": "refine", "kind": "gs", "fits": 300, "balls_lo": 8, "balls_hi": 64, "points": 2048, "epochs": 100},
        {"name": "descriptors", "kind": "shape", "models": 300, "balls_lo": 8, "balls_hi": 64, "r_lo": 8.0,
         "r_hi": 16.0, "h": 0.25},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["coupled", "coupled", "coupled", "coupled", "bed", "train", "ga", "gs", "shape"])
    if kind == "coupled":
        nodes = math.exp(rng.uniform(math.log(2e5), math.log(3e7)))
        ax, ay = math.exp(rng.uniform(-0.7, 0.7)), math.exp(rng.uniform(-0.7, 0.7))
        nx = int(round(nodes ** (1 / 3) * ax))
        ny = int(round(nodes ** (1 / 3) * ay))
        nz = max(24, int(nodes / (nx * ny)))
        if rng.random() < 0.4:
            nx = nx // 4 * 4
        r = rng.uniform(4.0, 0.11 * min(nx, ny, nz) + 4.0)
        r = min(r, 16.0, 0.3 * (min(nx, ny, nz) - 8))
        # a grid of places that far apart that no two particles touch
        most = math.prod(int((n - 8) / (3.0 * r + 5.0)) for n in (nx, ny, nz))
        particles = 0 if most == 0 else min(most, _log_int(rng, 1, 300))
        lo = rng.randint(1, 24)
        return _coupled(None, nx, ny, nz, rng.choice(["f32", "f32", "f16", "bf16"]), particles, "clustered",
                        (lo, rng.randint(lo, 64)), (round(0.6 * r, 3), round(r, 3)), 20 if nodes < 2e6 else 8,
                        bb=rng.choice(["ibb", "ibb", "ladd"]), periodic=rng.choice(["", "", "x", "y", "z"]),
                        force=rng.choice([0.0, 0.0, 1e-6]),
                        substeps=rng.choice([1, 1, 1, 10, 100]) if 0 < particles <= 64 else 1)
    if kind == "bed":
        lo = rng.randint(4, 16)
        return {"kind": "bed", "particles": _log_int(rng, 70, 3000), "balls_lo": lo, "balls_hi": rng.randint(lo, 128),
                "spacing": round(rng.uniform(18.7, 26.0), 2), "substeps": rng.choice([1, 5, 10])}
    if kind == "train":
        return {"kind": "train", "batch": _log_int(rng, 256, 16384)}
    if kind == "ga":
        return {"kind": "ga", "individuals": _log_int(rng, 64, 1200), "genes": rng.randint(4, 100),
                "points": _log_int(rng, 200, 2048), "generations": rng.randint(5, 20),
                "mutate": rng.choice([0.02, 0.05, 0.2])}
    if kind == "gs":
        lo = rng.randint(1, 16)
        return {"kind": "gs", "fits": _log_int(rng, 1, 300), "balls_lo": lo, "balls_hi": rng.randint(lo, 64),
                "points": _log_int(rng, 100, 4096), "epochs": rng.randint(10, 100)}
    lo = rng.randint(4, 16)
    return {"kind": "shape", "models": _log_int(rng, 1, 300), "balls_lo": lo, "balls_hi": rng.randint(lo, 64),
            "r_lo": 6.0, "r_hi": round(rng.uniform(6.0, 16.0), 2), "h": rng.choice([0.25, 0.4, 0.5, 1.0])}


# ---------------------------------------------------------------------------
# Inputs, all from the seed alone.  Positions, shapes and poses are rounded to
# float32 values, as the scenes of this repository are.
# ---------------------------------------------------------------------------
def _rng(case, seed):
    return np.random.default_rng([abs(int(seed)), len(case["kind"])])


def _f32(a):
    return np.asarray(a, dtype=np.float64).astype(np.float32).astype(np.float64)


def _in_ball(rng, n, radius):
    u = rng.normal(size=(n, 3))
    return u / np.linalg.norm(u, axis=1, keepdims=True) * radius * rng.random((n, 1)) ** (1 / 3)


def _clustered(rng, n, R):
    """n control points in a ball of 0.5 R with sum k = R^2."""
    c = _in_ball(rng, n, 0.5 * R)
    c -= c.mean(axis=0)
    k = rng.uniform(0.5, 1.5, n)
    return _f32(c), _f32(k / k.sum() * R * R)


def _cobble(rng, n, lo, hi):
    """n control points, Gaussian inside a random ellipsoid of semi-axes in [lo, hi]."""
    a = rng.uniform(lo, hi, 3)
    p = rng.normal(size=(16 * n, 3)) * a / 2.0
    c = p[((p / a) ** 2).sum(axis=1) <= 1.0][:n]
    return _f32(c - c.mean(axis=0)), _f32(np.exp(rng.uniform(math.log(9.0), math.log(36.0), n)))


def _quaternions(rng, n):
    q = rng.normal(size=(n, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    return _f32(q * np.where(q[:, :1] < 0, -1.0, 1.0))


def _sphere_mass(k):
    """Mass, volume and moment of inertia of the sphere of radius sqrt(sum k), given as the particle's own."""
    r = math.sqrt(float(k.sum()))
    vol = 4.0 / 3.0 * math.pi * r ** 3
    return DENSITY * vol, vol, 0.4 * DENSITY * vol * r * r


def _places(rng, n, size, r):
    """n places on a jittered grid inside the box, no two within about 2.6 r of each other."""
    best = None
    for cz in range(1, n + 1):
        for cy in range(1, -(-n // cz) + 1):
            cx = -(-n // (cz * cy))
            pitch = min((size[0] - 8) / cx, (size[1] - 8) / cy, (size[2] - 8) / cz)
            if best is None or pitch > best[0]:
                best = (pitch, (cx, cy, cz))
    cells = best[1]
    pick = rng.permutation(math.prod(cells))[:n]
    ijk = np.stack([pick % cells[0], pick // cells[0] % cells[1], pick // (cells[0] * cells[1])], axis=1)
    pitch = np.array([(size[a] - 8) / cells[a] for a in range(3)])
    room = np.maximum(pitch / 2 - 1.3 * r - 1.5, 0.0)
    return 4.0 + (ijk + 0.5) * pitch + rng.uniform(-1.0, 1.0, (n, 3)) * room


def _scene(case, rng):
    """Shapes [(centers, k)] and states (n, 13): position, quaternion, velocity, angular velocity."""
    n, size = case["particles"], (case["nx"], case["ny"], case["nz"])
    shapes = []
    for _ in range(n):
        balls = int(rng.integers(case["balls_lo"], case["balls_hi"] + 1))
        if case["shape"] == "cobble":
            shapes.append(_cobble(rng, balls, case["r_lo"], case["r_hi"]))
        elif case["shape"] == "blob":
            shapes.append((_f32(_in_ball(rng, balls, case["r_lo"])), _f32(rng.uniform(4.0, 9.0, balls))))
        else:
            shapes.append(_clustered(rng, balls, rng.uniform(case["r_lo"], case["r_hi"])))
    st = np.zeros((n, 13))
    if n:
        st[:, :3] = _places(rng, n, size, 1.45 * case["r_hi"] if case["shape"] == "cobble" else case["r_hi"])
        st[:, 3:7] = _quaternions(rng, n)
        st[:, 7:10] = rng.uniform(-0.02, 0.02, (n, 3))
        st[:, 10:13] = rng.uniform(-0.002, 0.002, (n, 3))
    return shapes, _f32(st)


def _flow(case, rng, each):
    """The populations of a smooth flow, a few per cent off equilibrium: each(i, f_i - w_i as float32 (nz, ny, nx))."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    wave, phase = rng.integers(1, 4, (3, 3)), rng.uniform(0.0, 2.0 * math.pi, (3, 3))
    axes = [torch.arange(n, device="cuda", dtype=torch.float32) for n in (nx, ny, nz)]
    u = []
    for a in range(3):
        x, y, z = (torch.sin(2.0 * math.pi * float(wave[a, b]) / axes[b].numel() * axes[b] + float(phase[a, b]))
                   for b in range(3))
        u.append(0.03 * z[:, None, None] * y[None, :, None] * x[None, None, :])
    usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    for i in range(19):
        eu = E[i][0] * u[0] + E[i][1] * u[1] + E[i][2] * u[2]
        ne = 0.02 * u[i % 3] * (1.0 if i % 2 else -1.0)
        each(i, W[i] * (3.0 * eu + 4.5 * eu * eu - 1.5 * usq + ne))


def _stored(case, i, dev):
    """The value the lattice holds: f in float32, f - w in 16 bits."""
    return dev + W[i] if case["storage"] == "f32" else dev.to(ELEMENT[case["storage"]])


def _bed(case, rng):
    n, d = case["particles"], case["spacing"]
    side = max(1, round((n * 2.8) ** (1 / 3)))
    high = -(-n // (side * side))
    shapes = []
    for _ in range(n):
        balls = int(round(math.exp(rng.uniform(math.log(case["balls_lo"]), math.log(case["balls_hi"])))))
        shapes.append(_clustered(rng, balls, rng.uniform(8.0, 16.0)))
    pick = rng.permutation(side * side * high)[:n]
    ijk = np.stack([pick % side, pick // side % side, pick // (side * side)], axis=1)
    st = np.zeros((n, 13))
    st[:, :3] = 14.0 + (ijk + 0.5) * d + rng.uniform(-0.35, 0.35, (n, 3)) * d
    st[:, 3:7] = _quaternions(rng, n)
    st[:, 7:10] = rng.uniform(-0.01, 0.01, (n, 3))
    st[:, 10:13] = rng.uniform(-0.001, 0.001, (n, 3))
    return shapes, _f32(st), (int(28 + side * d), int(28 + side * d), int(28 + high * d))


def _models(case, rng, n):
    return [_clustered(rng, int(rng.integers(case["balls_lo"], case["balls_hi"] + 1)),
                       rng.uniform(case["r_lo"], case["r_hi"])) for _ in range(n)]


def _gs_inputs(case, rng):
    hulls, planes, kinds = [], [], min(case["fits"], 12)
    for _ in range(kinds):
        semi = rng.uniform(8.0, 14.0, 3)
        h = scenes.ellipsoid_hull(rng, case["points"], semi, bumps=0.05)
        hulls.append((h, semi))
        planes.append(scenes.hull_planes(h))
    models = []
    counts = rng.permutation(np.linspace(case["balls_lo"], case["balls_hi"], case["fits"]).round().astype(int))
    for f, n in enumerate(counts):
        semi = hulls[f % kinds][1]
        k = np.full(n, float(np.prod(semi)) ** (2.0 / 3.0) / n)
        models.append((_f32(_in_ball(rng, n, 0.5) * semi), _f32(k)))
    return ([hulls[f % kinds][0] for f in range(case["fits"])], models,
            [planes[f % kinds] for f in range(case["fits"])])


def _train_inputs(case, rng):
    parts = []
    for a, b in ((64, 256), (256, 256), (256, 4)):
        parts += [rng.uniform(-1.0, 1.0, a * b) * math.sqrt(6.0 / a), rng.normal(0.0, 0.05, b)]
    p = np.concatenate(parts)
    # in the middle of training: the moments of earlier gradients
    v = rng.uniform(0.5, 1.5, p.size) * 1e-4
    m = rng.normal(0.0, 3e-3, p.size)
    X = rng.normal(size=(case["batch"], 64))
    T = 0.3 * X[:, :4] + 0.1 * np.sin(2.0 * X[:, 4:8])
    return [torch.as_tensor(a.astype(np.float32), device="cuda") for a in (p, m, v, X, T)]


# ---------------------------------------------------------------------------
def _add(sim, shapes, st):
    for (c, k), s in zip(shapes, st):
        mass, vol, inertia = _sphere_mass(k)
        sim.add_particle(c, k, DENSITY, SKIN, s[:3], s[3:7], s[7:10], s[10:13],
                         mass_props={"mass": mass, "volume": vol, "inertia": np.eye(3) * inertia})


def _view(ptr, shape, typestr):
    return torch.as_tensor(B.CudaArray(ptr, shape, typestr), device="cuda")


def _populations(sim, case):
    v = sim.device_view()
    t = _view(v.populations, (19, v.plane_stride), "<f4" if case["storage"] == "f32" else "<i2")
    return t.view(ELEMENT[case["storage"]])[:, :sim.ncell].unflatten(1, sim.shape), v


def _hold_states(state, st):
    state["given"] = torch.from_numpy(st.copy()).pin_memory()
    state["taken"] = torch.zeros_like(state["given"]).pin_memory()


def prepare(case, seed):
    rng, kind = _rng(case, seed), case["kind"]
    state = {"case": case}
    if kind == "coupled":
        shapes, st = _scene(case, rng)
        sim = B.Simulation(case["nx"], case["ny"], case["nz"], tau=0.8, gravity=GRAVITY,
                           storage=STORAGE[case["storage"]], bb_mode=B.BB_LADD if case["bb"] == "ladd" else B.BB_IBB,
                           periodic=tuple(a in case["periodic"] for a in "xyz"),
                           fluid_body_force=(case["force"], 0.0, 0.0), dem_substeps=case["substeps"],
                           max_particles=max(16, len(shapes)))
        pop, _ = _populations(sim, case)
        _flow(case, rng, lambda i, dev: pop[i].copy_(_stored(case, i, dev)))
        _add(sim, shapes, st)
        _hold_states(state, st)
        state["zero"] = torch.zeros((), dtype=ELEMENT[case["storage"]], device="cuda")
        torch.cuda.synchronize()
        state["sim"] = sim
    elif kind == "bed":
        shapes, st, size = _bed(case, rng)
        # the box gives the walls; without the fluid its lattice is never stepped
        sim = B.Simulation(*size, tau=0.8, gravity=GRAVITY, storage=B.STORE_F16_DEV, dem_substeps=case["substeps"],
                           max_particles=len(shapes), max_balls=sum(len(k) for _, k in shapes) + 16, eta_n=0.1,
                           eta_t=0.1)
        _add(sim, shapes, st)
        _hold_states(state, st)
        state["sim"] = sim
    elif kind == "train":
        state["tensors"], state["t"] = _train_inputs(case, rng), 1000
    elif kind == "ga":
        semi = rng.uniform(9.0, 13.0, 3)
        hull = scenes.ellipsoid_hull(rng, case["points"], semi, bumps=0.03)
        r = float(np.prod(semi)) ** (1.0 / 3.0)
        state["args"] = (hull, scenes.hull_planes(hull), np.concatenate([hull.min(axis=0), hull.max(axis=0)]),
                         (0.05 * r * r / case["genes"], 2.0 * r * r / case["genes"]), case["individuals"],
                         case["genes"], case["generations"], case["mutate"], 0.5, int(rng.integers(1 << 40)))
    elif kind == "gs":
        state["args"] = _gs_inputs(case, rng) + (case["epochs"], 0.2 / case["points"])
    else:
        state["args"] = (_models(case, rng, case["models"]), case["h"])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("coupled", "bed"):
        sim, n = state["sim"], state["given"].shape[0]
        if n:
            sim.set_particle_states_ptr(state["given"].data_ptr(), n)
        if kind == "bed":
            sim.step_phases(B.PHASE_CONTACT | B.PHASE_INTEGRATE)
        else:
            sim.step(case["steps"])
        out = {}
        if n:
            sim.get_particle_states_ptr(state["taken"].data_ptr(), n)
            out["states"] = state["taken"]
        if kind == "coupled":
            pop, v = _populations(sim, case)
            with torch.cuda.stream(sim.torch_stream):
                if n:
                    # values at solid nodes are unspecified: the fluid's alone
                    owner = _view(v.owner, sim.shape, "<i4")
                    fluid, masked = owner == -1, torch.empty(pop.shape, dtype=pop.dtype, device="cuda")
                    for i in range(19):  # plane by plane: contiguous, without an index per element
                        torch.where(fluid, pop[i], state["zero"], out=masked[i])
                    out["populations"] = masked
                    out["owner"] = owner.clone()
                    out["classes"] = _view(v.node_class, sim.shape, "|u1").clone()
                else:
                    out["populations"] = pop.clone()
        return out
    if kind == "train":
        p, m, v, X, T = state["tensors"]
        state["t"] += 1
        Y, acts = B.mlp_forward(p, X)
        loss, dY = B.mlp_mse(Y, T)
        grads = B.mlp_backward(p, X, acts, dY)
        B.mlp_adamw(p, grads, m, v, state["t"], lr=1e-3)
        return {"Y": Y, "loss": loss, "grads": grads, "params": p, "m": m, "v": v}
    if kind == "ga":
        pop, fit, off, fit_off = B.ga_run(*state["args"])
        return {"population": pop, "fitness": fit, "children": off, "children_fitness": fit_off}
    if kind == "gs":
        models, loss = B.gs_fit(*state["args"])
        return {"centers": np.concatenate([c for c, _, _ in models]), "k": np.concatenate([k for _, k, _ in models]),
                "active": np.concatenate([a for _, _, a in models]), "loss": loss}
    rows = B.shape_descriptors(*state["args"])
    out = {f: np.array([r[f] for r in rows]) for f in B.SHAPE_FIELDS if f != "cells"}
    out["cells"] = np.array([int(r["cells"]) for r in rows])
    return out


def work(case):
    kind = case["kind"]
    if kind == "coupled":
        # every stored population read and written once a step; BGK about 300 operations a node;
        # per particle the field at the nodes of its ball (10 a ball and node)
        nodes = case["nx"] * case["ny"] * case["nz"]
        size = 4 if case["storage"] == "f32" else 2
        balls = 0.5 * (case["balls_lo"] + case["balls_hi"])
        r = 0.5 * (case["r_lo"] + case["r_hi"])
        return {"bytes": case["steps"] * (38.0 * size * nodes + 13 * 16.0 * case["particles"]),
                "flops": case["steps"] * (300.0 * nodes + case["particles"] * 10.0 * balls * 4.2 * r ** 3)}
    if kind == "bed":
        # about 16 candidate pairs a particle, four Newton steps of 35 operations a ball; the poses and balls once
        balls = (case["balls_hi"] - case["balls_lo"]) / max(1e-9, math.log(case["balls_hi"] / case["balls_lo"])) \
            if case["balls_hi"] > case["balls_lo"] else case["balls_lo"]
        pairs = case["particles"] * 16.0 * (18.7 / case["spacing"]) ** 3
        return {"bytes": case["substeps"] * case["particles"] * (208.0 + 16.0 * balls),
                "flops": case["substeps"] * pairs * 4 * (35 * 2 * balls + 60)}
    if kind == "train":
        macs = 64 * 256 + 256 * 256 + 256 * 4
        return {"bytes": 4.0 * (case["batch"] * 72 + 7 * 83460), "flops": 2.0 * case["batch"] * (3 * macs - 64 * 256)}
    if kind == "ga":
        cells = case["individuals"] * case["genes"] * (case["generations"] + 1.0)
        return {"bytes": 32.0 * case["individuals"] * case["genes"] + 12.0 * case["points"],
                "flops": 9.0 * cells * case["points"]}
    if kind == "gs":
        balls = 0.5 * (case["balls_lo"] + case["balls_hi"])
        return {"bytes": case["fits"] * (12.0 * case["points"] + 32 * balls),
                "flops": case["fits"] * 2.0 * case["epochs"] * 27 * balls * case["points"]}
    # the field once in every cell of the solid's bounding cube, on both grids
    balls, r = 0.5 * (case["balls_lo"] + case["balls_hi"]), 0.5 * (case["r_lo"] + case["r_hi"])
    return {"bytes": case["models"] * (16.0 * balls + 124), "flops": case["models"] * 2.0 * (2.2 * r / case["h"]) ** 3
            * 9 * balls}


# ---------------------------------------------------------------------------
# The same in 64 bits, torch alone
# ---------------------------------------------------------------------------
F64 = {"dtype": torch.float64, "device": "cuda"}


def _rotation(q):
    q = q / q.norm(dim=-1, keepdim=True)
    w, x, y, z = q.unbind(-1)
    rows = [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
            1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
            1 - 2 * (x * x + y * y)]
    return torch.stack(rows, -1).unflatten(-1, (3, 3))


def _rigid(st, body, F, T, dt):
    """Semi-implicit Euler of all particles: velocity, position, Euler's equations in body axes."""
    mass, vol, inertia = body
    g = torch.tensor(GRAVITY, **F64)
    v = st[:, 7:10] + dt * (F + (mass - vol)[:, None] * g) / mass[:, None]
    Rt = _rotation(st[:, 3:7]).transpose(1, 2)
    wb = (Rt @ st[:, 10:13, None])[..., 0]
    wb = wb + dt * (Rt @ T[..., None])[..., 0] / inertia[:, None]  # equal moments: no gyroscopic term
    th = wb * dt
    t = th.norm(dim=1, keepdim=True).clamp_min(1e-300)
    e = torch.cat([torch.cos(0.5 * t), torch.sin(0.5 * t) / t * th], 1)
    a = st[:, 3:7] / st[:, 3:7].norm(dim=1, keepdim=True)
    aw, ax, ay, az = a.unbind(1)
    bw, bx, by, bz = e.unbind(1)
    q = torch.stack([aw * bw - ax * bx - ay * by - az * bz, aw * bx + ax * bw + ay * bz - az * by,
                     aw * by - ax * bz + ay * bw + az * bx, aw * bz + ax * by - ay * bx + az * bw], 1)
    q = q / q.norm(dim=1, keepdim=True)
    w = (_rotation(q) @ wb[..., None])[..., 0]
    return torch.cat([st[:, :3] + dt * v, q, v, w], 1)


def _bodies(shapes):
    return tuple(torch.tensor(x, **F64) for x in zip(*(_sphere_mass(k) for _, k in shapes))) if shapes else None


def _field_at(x, c, k):
    f = torch.zeros(x.shape[0], **F64)
    for j in range(len(k)):
        f += k[j] / ((x - c[j]) ** 2).sum(1)
    return f


def _source(t, e, periodic):
    """t at x - e for every node of the last three axes, and where that lies outside the box."""
    shifts = (e[2], e[1], e[0])
    s = torch.roll(t, shifts, (-3, -2, -1)) if any(e) else t
    out = None
    for a, d in enumerate(e):
        if d and not periodic[a]:
            face = torch.zeros(t.shape[-3:], dtype=torch.bool, device="cuda")
            face.select(2 - a, 0 if d > 0 else -1).fill_(True)
            out = face if out is None else out | face
    return s, out


def _exact_coupled(case, seed):
    rng = _rng(case, seed)
    shapes, st = _scene(case, rng)
    n, size = len(shapes), (case["nz"], case["ny"], case["nx"])
    nodes = math.prod(size)
    if nodes > 5e7 or n * case["steps"] > 400:
        return None
    periodic = [a in case["periodic"] for a in "xyz"]
    f = torch.empty((19,) + size, **F64)

    def each(i, dev):
        s = _stored(case, i, dev)
        f[i] = s.double() if case["storage"] == "f32" else s.double() + W[i]
    _flow(case, rng, each)
    st = torch.tensor(st, **F64)
    C = [torch.tensor(c, **F64) for c, _ in shapes]
    K = [torch.tensor(k, **F64) for _, k in shapes]
    ev = torch.tensor(E, **F64)
    wv = torch.tensor(W, **F64)
    g = torch.zeros(3, **F64)
    g[0] = case["force"]
    om = 1.0 / 0.8
    before = torch.full(size, -1, dtype=torch.int64, device="cuda")
    body = _bodies(shapes)
    contacts = _Contacts(shapes, size[::-1], periodic, 0.0) if n else None

    def equilibrium(rho, u, w, e):
        eu = (u * e).sum(-1)
        return w * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(-1))

    def moments(cells):
        h = f.flatten(1)[:, cells]
        rho = h.sum(0)
        return rho, (ev.T @ h).T / rho[:, None]

    def neighbour(cells, e):
        x, y, z = cells % size[2], cells // size[2] % size[1], cells // (size[1] * size[2])
        ok = torch.ones_like(cells, dtype=torch.bool)
        to = []
        for a, (v, length) in enumerate(((x, size[2]), (y, size[1]), (z, size[0]))):
            v = v + e[..., a]
            if periodic[a]:
                v = v % length
            else:
                ok &= (v >= 0) & (v < length)
                v = v.clamp(0, length - 1)
            to.append(v)
        return (to[2] * size[1] + to[1]) * size[2] + to[0], ok

    def xyz(cells):
        return torch.stack([cells % size[2], cells // size[2] % size[1], cells // (size[1] * size[2])], 1).double()

    ei = torch.tensor(E, device="cuda")
    opp = torch.tensor(OPP, device="cuda")
    for step in range(case["steps"]):
        R = _rotation(st[:, 3:7]) if n else None
        owner = torch.full(size, -1, dtype=torch.int64, device="cuda")
        for p in reversed(range(n)):  # overlaps: the lowest index last
            reach = float(C[p].norm(dim=1).max() + K[p].sum().sqrt()) + 1.0
            lo = [max(0, math.floor(float(st[p, a]) - reach)) for a in range(3)]
            hi = [min(size[2 - a], math.ceil(float(st[p, a]) + reach) + 1) for a in range(3)]
            ax = [torch.arange(lo[a], hi[a], device="cuda") for a in range(3)]
            if min(len(a) for a in ax) == 0:
                continue
            zz, yy, xx = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
            x = torch.stack([xx, yy, zz], -1).reshape(-1, 3).double() - st[p, :3]
            inside = _field_at(x @ R[p], C[p], K[p]) >= 1.0
            box = owner[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
            box[inside.reshape(box.shape)] = p
        solid = owner >= 0
        if n:
            # uncovered nodes
            flat, was = owner.flatten(), before.flatten()
            new = ((flat < 0) & (was >= 0)).nonzero()[:, 0]
            if len(new):
                p = was[new]
                u = st[p, 7:10] + torch.linalg.cross(st[p, 10:13], xyz(new) - st[p, :3])
                vals = []
                for i in range(19):
                    nb, ok = neighbour(new, ei[i].expand(len(new), 3))
                    ok = ok & (flat[nb] < 0) & (was[nb] < 0)
                    vals.append(torch.where(ok, f[OPP[i]].flatten()[nb] + 6 * W[i] * (u * ev[i]).sum(1),
                                            equilibrium(1.0, u, W[i], ev[i])))
                f.flatten(1)[:, new] = torch.stack(vals)
            cells, dirs = [], []
            for d in range(1, 19):
                nb, out = _source(owner, tuple(-x for x in E[d]), periodic)
                m = (owner < 0) & (nb >= 0)
                if out is not None:
                    m &= ~out
                c = m.flatten().nonzero()[:, 0]
                cells.append(c)
                dirs.append(torch.full_like(c, d))
            cells, dirs = torch.cat(cells), torch.cat(dirs)
            own = flat[neighbour(cells, ei[dirs])[0]]
            q = torch.full((len(cells),), 0.5, **F64)
            if case["bb"] == "ibb":
                for p in range(n):
                    m = (own == p).nonzero()[:, 0]
                    a, b = (xyz(cells[m]) - st[p, :3]) @ R[p], ev[dirs[m]] @ R[p]
                    lo, hi = torch.zeros(len(m), **F64), torch.ones(len(m), **F64)
                    for _ in range(50):
                        mid = 0.5 * (lo + hi)
                        d = (a + mid[:, None] * b)[:, None, :] - C[p]
                        inside = (K[p] / (d * d).sum(-1)).sum(1) >= 1.0
                        hi, lo = torch.where(inside, mid, hi), torch.where(inside, lo, mid)
                    q[m] = 0.5 * (lo + hi)
            qc, ed, j = q[:, None], ev[dirs], opp[dirs]
            arm = xyz(cells) + qc * ed - st[own, :3]
            uw = st[own, 7:10] + torch.linalg.cross(st[own, 10:13], arm)
            fd = f.flatten(1)[dirs, cells]
            G = fd + 6 * wv[dirs] * (-ed * uw).sum(1)
            if case["bb"] == "ibb":
                rho, uf = moments(cells)
                ff, ok = neighbour(cells, -ei[dirs])
                ok = ok & (flat[ff] < 0)
                uff = torch.where(ok[:, None], moments(ff)[1], uf)
                us = torch.where(qc <= 0.5, 2 * qc * uf + (1 - 2 * qc) * uff, ((1 - qc) * uf + (2 * qc - 1) * uw) / qc)
                ud = us / 3 + 2 / 3 * ((1 - qc) * uff + 2 * qc * uw) / (1 + qc)
                G = G + equilibrium(rho, ud, wv[dirs], ed) - equilibrium(rho, uf, wv[dirs], ed)
            dP = (ed - uw) * fd[:, None] - (-ed - uw) * G[:, None]
            F = torch.zeros((n, 3), **F64).index_add_(0, own, dP)
            T = torch.zeros((n, 3), **F64).index_add_(0, own, torch.linalg.cross(arm, dP))
        h = torch.empty_like(f)
        for i in range(19):
            s, out = _source(f[i], E[i], periodic)
            h[i] = s if out is None else torch.where(out, f[OPP[i]], s)
        if n:
            h.flatten(1)[j, cells] = G
        rho = h.sum(0)
        u = [(torch.tensordot(ev[:, a], h, 1) + 0.5 * g[a]) / rho for a in range(3)]
        usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        ug = u[0] * g[0]
        for i in range(19):
            eu = E[i][0] * u[0] + E[i][1] * u[1] + E[i][2] * u[2]
            h[i] += om * (W[i] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * usq) - h[i])
            if case["force"]:
                eg = E[i][0] * g[0]
                h[i] += (1 - 0.5 * om) * W[i] * (3 * (eg - ug) + 9 * eu * eg)
        f = h
        if n:
            for _ in range(case["substeps"]):
                dt = 1.0 / case["substeps"]
                Fc, Tc = contacts.forces(st, dt)
                st = _rigid(st, body, F + Fc, T + Tc, dt)
            before = owner
    if case["storage"] != "f32":
        f -= wv[:, None, None, None]
    out = {}
    if n:
        out = {"states": st.cpu(), "owner": None, "classes": None}
        f.masked_fill_(before >= 0, 0.0)
    out["populations"] = f
    return out


class _Contacts:
    """Contact forces between the particles and with the walls, one DEM substep after another."""

    def __init__(self, shapes, size, periodic, eta):
        self.n, self.size, self.periodic, self.eta, self.springs = len(shapes), size, periodic, eta, {}
        nb = max(len(k) for _, k in shapes)
        self.C, self.K = torch.full((self.n, nb, 3), 1e6, **F64), torch.zeros((self.n, nb), **F64)
        for p, (c, k) in enumerate(shapes):
            self.C[p, :len(k)], self.K[p, :len(k)] = torch.tensor(c, **F64), torch.tensor(k, **F64)
        re = self.K.sum(1).sqrt()
        self.s = ((re - SKIN) / re) ** 2
        self.real = self.K > 0
        self.Rb = torch.where(self.real, self.C.norm(dim=-1), torch.zeros((), **F64)).amax(1) + re

    def start(self, a, b):
        """The plain start: between the closest two spheres of a pair."""
        C, K = self.C, self.K
        ca = torch.einsum("mij,mbj->mbi", self.R[a], C[a]) + self.st[a, None, :3]
        cb = torch.einsum("mij,mbj->mbi", self.R[b], C[b]) + self.st[b, None, :3]
        gap = torch.cdist(ca, cb, compute_mode="donot_use_mm_for_euclid_dist")
        gap = gap - K[a].sqrt()[:, :, None] - K[b].sqrt()[:, None, :]
        gap = torch.where(self.real[a][:, :, None] & self.real[b][:, None, :], gap, torch.full((), math.inf, **F64))
        at = gap.flatten(1).argmin(1)
        i, j, r = at // C.shape[1], at % C.shape[1], torch.arange(len(a), device="cuda")
        u = cb[r, j] - ca[r, i]
        u = u / u.norm(dim=1, keepdim=True)
        return 0.5 * (ca[r, i] + K[a, i].sqrt()[:, None] * u + cb[r, j] - K[b, j].sqrt()[:, None] * u)

    def core(self, p, x):
        """g = s f of particles p at x, its gradient and Hessian."""
        R, s, K = self.R[p], self.s[p], self.K[p]
        d = torch.einsum("mji,mj->mi", R, x - self.st[p, :3])[:, None, :] - self.C[p]
        r2 = (d * d).sum(-1)
        b = K / (r2 * r2)
        G = -2 * (b[..., None] * d).sum(1)
        H = 8 * torch.einsum("mb,mbi,mbj->mij", b / r2, d, d) - 2 * b.sum(1)[:, None, None] * torch.eye(3, **F64)
        return (s * (K / r2).sum(1), s[:, None] * torch.einsum("mij,mj->mi", R, G),
                s[:, None, None] * (R @ H @ R.transpose(1, 2)))

    def pairs(self, a, b):
        x = self.start(a, b)
        tol = 1e-5 * torch.maximum(self.Rb[a], self.Rb[b])
        done = torch.zeros(len(a), dtype=torch.bool, device="cuda")
        dead = done.clone()

        def newton(w):
            _, ga, Ha = self.core(a[w], x[w])
            _, gb, Hb = self.core(b[w], x[w])
            return torch.linalg.solve_ex(Ha + Hb, (ga + gb)[..., None])[0][..., 0]

        for _ in range(50):
            w = (~(done | dead)).nonzero()[:, 0]
            if not len(w):
                break
            dx = newton(w)
            bad = ~torch.isfinite(dx).all(1)
            x[w] = torch.where(bad[:, None], x[w], x[w] - dx)
            dead[w] |= bad
            done[w] |= ~bad & (dx.norm(dim=1) <= tol[w])
        w = (done & ~dead).nonzero()[:, 0]
        for _ in range(2):  # to the last bits
            x[w] -= newton(w)
        ga, da, _ = self.core(a, x)
        gb, db, _ = self.core(b, x)
        ok = done & ~dead & (ga < 1) & (gb < 1) & (ga >= 1e-6) & (gb >= 1e-6)
        xa = x + ((1 - ga) / (da * da).sum(1))[:, None] * da
        xb = x + ((1 - gb) / (db * db).sum(1))[:, None] * db
        d = xa - xb
        dist = d.norm(dim=1)
        nrm = d / dist.clamp_min(1e-300)[:, None]
        delta = 2 * SKIN - dist
        return ok & (delta > 0), delta, nrm, xa - (SKIN - 0.5 * delta)[:, None] * nrm

    def wall(self, a, axis, sign, level):
        nw = torch.zeros(3, **F64)
        nw[axis] = sign
        ca = torch.einsum("mij,mbj->mbi", self.R[a], self.C[a]) + self.st[a, None, :3]
        rs = (self.s[a, None] * self.K[a]).sqrt()
        depth = torch.where(self.real[a], ca @ nw - rs, torch.full((), math.inf, **F64))
        i, r = depth.argmin(1), torch.arange(len(a), device="cuda")
        x = ca[r, i] - rs[r, i][:, None] * nw
        lam = self.core(a, x)[1].norm(dim=1)
        ok = torch.zeros(len(a), dtype=torch.bool, device="cuda")
        for _ in range(50):
            g, G, H = self.core(a, x)
            J = torch.zeros((len(a), 4, 4), **F64)
            J[:, :3, :3], J[:, :3, 3], J[:, 3, :3] = H, -nw, G
            dz = torch.linalg.solve_ex(J, torch.cat([G - lam[:, None] * nw, g[:, None] - 1], 1)[..., None])[0][..., 0]
            dz = torch.where(torch.isfinite(dz), dz, torch.zeros((), **F64))
            x, lam = x - dz[:, :3], lam - dz[:, 3]
            ok |= dz[:, :3].norm(dim=1) <= 1e-5 * self.Rb[a]
        dist = (x * nw).sum(1) - sign * level
        delta = SKIN - dist
        return ok & (delta > 0), delta, nw.expand(len(a), 3), x + (0.5 * delta - dist)[:, None] * nw

    def push(self, name, key, got, a, b, F, T, dt):
        kt, mu, st = 2.0 / 7.0, 0.4, self.st
        old = self.springs.pop(name, None)
        i = got[0].nonzero()[:, 0]
        if not len(i):
            return
        a, key, delta, nrm, xc = a[i], key[i], got[1][i, None], got[2][i], got[3][i]
        va = st[a, 7:10] + torch.linalg.cross(st[a, 10:13], xc - st[a, :3])
        vb = torch.zeros_like(va)
        if b is not None:
            b = b[i]
            vb = st[b, 7:10] + torch.linalg.cross(st[b, 10:13], xc - st[b, :3])
        vn = ((vb - va) * nrm).sum(1, keepdim=True)
        vt = vb - va - vn * nrm
        Fn = (1.0 * delta + self.eta * vn).clamp_min(0.0)
        xi = torch.zeros_like(vt)
        if old is not None:
            k = torch.searchsorted(old[0], key).clamp_max(len(old[0]) - 1)
            xi = torch.where((old[0][k] == key)[:, None], old[1][k], xi)
        xi = xi - (xi * nrm).sum(1, keepdim=True) * nrm + vt * dt
        Ft = kt * xi + self.eta * vt
        nt = Ft.norm(dim=1, keepdim=True)
        slip = nt > mu * Fn
        Ft = torch.where(slip, Ft * (mu * Fn / nt.clamp_min(1e-300)), Ft)
        xi = torch.where(slip, (Ft - self.eta * vt) / kt, xi)
        f = Fn * nrm + Ft
        F.index_add_(0, a, f)
        T.index_add_(0, a, torch.linalg.cross(xc - st[a, :3], f))
        if b is not None:
            F.index_add_(0, b, -f)
            T.index_add_(0, b, -torch.linalg.cross(xc - st[b, :3], f))
        order = key.argsort()
        self.springs[name] = key[order], xi[order]

    def forces(self, st, dt):
        self.st, self.R = st, _rotation(st[:, 3:7])
        F, T = torch.zeros((self.n, 3), **F64), torch.zeros((self.n, 3), **F64)
        near = torch.cdist(st[:, :3], st[:, :3], compute_mode="donot_use_mm_for_euclid_dist")
        near = (near <= self.Rb[:, None] + self.Rb[None, :] + 1.0).triu(1)
        a, b = near.nonzero().unbind(1)
        if len(a):
            got = [self.pairs(a[k:k + 4096], b[k:k + 4096]) for k in range(0, len(a), 4096)]
            self.push("pairs", a * self.n + b, [torch.cat(v) for v in zip(*got)], a, b, F, T, dt)
        for axis in range(3):
            for sign, level in ((1.0, -0.5), (-1.0, self.size[axis] - 0.5)):
                w = (sign * (st[:, axis] - level) <= self.Rb + 1.0).nonzero()[:, 0]
                if len(w) and not self.periodic[axis]:
                    self.push((axis, sign), w, self.wall(w, axis, sign, level), w, None, F, T, dt)
        return F, T


def _exact_bed(case, seed):
    shapes, st, size = _bed(case, _rng(case, seed))
    contacts, body, st = _Contacts(shapes, size, (False,) * 3, 0.1), _bodies(shapes), torch.tensor(st, **F64)
    for _ in range(case["substeps"]):
        dt = 1.0 / case["substeps"]
        st = _rigid(st, body, *contacts.forces(st, dt), dt)
    return {"states": st.cpu()}


def _exact_train(case, seed):
    p, m, v, X, T = (t.double() for t in _train_inputs(case, _rng(case, seed)))
    sizes = [(64, 256), (256,), (256, 256), (256,), (256, 4), (4,)]
    W1, b1, W2, b2, W3, b3 = (t.view(s) for t, s in zip(p.split([math.prod(s) for s in sizes]), sizes))
    H1 = (X @ W1 + b1).relu()
    H2 = (H1 @ W2 + b2).relu()
    Y = H2 @ W3 + b3
    loss = ((Y - T) ** 2).sum() / len(X)
    dY = 2 * (Y - T) / len(X)
    d2 = (dY @ W3.T) * (H2 > 0)
    d1 = (d2 @ W2.T) * (H1 > 0)
    g = torch.cat([t.flatten() for t in (X.T @ d1, d1.sum(0), H1.T @ d2, d2.sum(0), H2.T @ dY, dY.sum(0))])
    t = 1001
    m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
    p = p - 1e-3 * (m / (1 - 0.9 ** t) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8) + 1e-4 * p)
    return {"Y": Y, "loss": loss[None], "grads": g, "params": p, "m": m, "v": v}


def _exact_gs(case, seed):
    hulls, models, planes, epochs, lr = _gs_inputs(case, _rng(case, seed)) + (case["epochs"], 0.2 / case["points"])
    n, nb, many = len(models), max(len(k) for _, k in models), max(len(h) for h in hulls)
    H = torch.tensor(np.stack(hulls), **F64)
    C, K = torch.full((n, nb, 3), 1e6, **F64), torch.zeros((n, nb), **F64)
    live = torch.zeros((n, nb), dtype=torch.bool, device="cuda")
    for f, (c, k) in enumerate(models):
        C[f, :len(k)], K[f, :len(k)], live[f, :len(k)] = torch.tensor(c, **F64), torch.tensor(k, **F64), True
    there = live.clone()

    def terms(a, z):
        d = H[a:z, :, None, :] - C[a:z, None, :, :]
        r2 = (d * d).sum(-1)
        return d, r2, (K[a:z, None, :] / r2).sum(-1)

    def loss_of():
        out = []
        for a in range(0, n, 64):
            f = terms(a, a + 64)[2]
            out.append(torch.where(f >= 2, (f - 1) ** 2, torch.where(f >= 1, f - 1, (f - 1) ** 2 + 1 / f - 1)).sum(1))
        return torch.cat(out)

    def descend():
        for _ in range(epochs):
            for a in range(0, n, 64):
                z = min(n, a + 64)
                d, r2, f = terms(a, z)
                w = torch.where(f >= 2, 2 * (f - 1), torch.where(f >= 1, torch.ones_like(f), 2 * (f - 1) - 1 / (f * f)))
                gk = (w[..., None] / r2).sum(1)
                gc = torch.einsum("fmb,fmbi->fbi", w[..., None] * 2 * K[a:z, None, :] / (r2 * r2), d)
                K[a:z] -= torch.where(live[a:z], lr * gk, torch.zeros_like(gk))
                C[a:z] -= torch.where(live[a:z, :, None], lr * gc, torch.zeros_like(gc))

    descend()
    first = loss_of()
    for f in range(n):
        pl = torch.tensor(planes[f], dtype=torch.float32, device="cuda")
        c = C[f].float()
        out = (c[:, :1] * pl[:, 0] + c[:, 1:2] * pl[:, 1] + c[:, 2:] * pl[:, 2] > pl[:, 3]).any(1)
        live[f] &= ~(out | (K[f] < 0))
    K[~live] = 0.0
    descend()
    loss = torch.stack([first, loss_of()], 1).cpu()
    return {"centers": C[there].cpu(), "k": K[there].cpu(), "active": None, "loss": loss}


def _exact_shape(case, seed):
    models, h, eps = _models(case, _rng(case, seed), case["models"]), case["h"], 0.1
    rows = {f: [] for f in B.SHAPE_FIELDS if f != "cells"}
    for c, k in models:
        rg = float(np.float32(np.sqrt((c * c).sum(1)).max() + np.sqrt(k.sum() / (1.0 - eps))))
        n = math.ceil(2.0 * rg / h)
        C, K = torch.tensor(c, **F64), torch.tensor(k, **F64)

        def grid(m, lo, axes, origin):
            """The field on the m^3 cells, the axes' coordinates along dimensions 0, 1, 2."""
            u = lo + (torch.arange(m, **F64) + 0.5) * h
            f = torch.zeros((m, m, m), **F64)
            rel = (C - origin) @ axes.T
            for j in range(len(K)):
                d = [(u - rel[j, a]) ** 2 for a in range(3)]
                f += K[j] / (d[0][:, None, None] + d[1][None, :, None] + d[2][None, None, :])
            return u, f

        u, f = grid(n, -rg, torch.eye(3, **F64), torch.zeros(3, **F64))
        x = u[(f >= 1).nonzero()]
        mean = x.mean(0)
        cov = (x.T @ x) / len(x) - mean[:, None] * mean[None, :]
        val, vec = torch.linalg.eigh(cov)
        axes = vec.T.flip(0)
        xb = u[((f - 1).abs() < eps).nonzero()]
        G = torch.zeros_like(xb)
        for j in range(len(K)):
            d = xb - C[j]
            G -= 2 * K[j] * d / (d * d).sum(1, keepdim=True) ** 2
        area = float(G.norm(dim=1).sum()) * h ** 3 / (2 * eps)
        u, f = grid(n + 4, -(rg + 2 * h), axes, mean)
        inside = f >= 1
        L = []
        for a in range(3):
            at = inside.any(dim=tuple(b for b in range(3) if b != a)).nonzero()[:, 0]
            L.append(float(u[at[-1]] - u[at[0]]) + h)
        flat = float(inside.any(dim=2).sum()) * h * h
        vol = len(x) * h ** 3
        dn = (6 * vol / math.pi) ** (1 / 3)
        for key, value in zip(rows, (vol, area, *L, flat, math.pi * dn * dn / area, dn, math.sqrt(4 * flat / math.pi),
                                     L[2] / math.sqrt(L[1] * L[0]))):
            rows[key].append(value)
    return {**{f: np.array(v) for f, v in rows.items()}, "cells": None}


def exact(case, seed):
    kind = case["kind"]
    if kind == "ga":
        return None  # which individuals are kept turns on comparisons of float32 sums
    return {"coupled": _exact_coupled, "bed": _exact_bed, "train": _exact_train, "gs": _exact_gs,
            "shape": _exact_shape}[kind](case, seed)
