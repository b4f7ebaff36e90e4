"""Writes tests/golden/states_16bit.json: what 16-bit population storages give for
a few light particles, to the bit of every stored population.

A 16-bit value that lies near the middle of two representable ones moves by a
whole unit when its FP32 value moves by one ulp, and the bounce-back hands such
units on to the particles: the states of a light particle then differ by 1e-7
after 20 steps.  The figures fix the result: the FP64 states after the run and,
for each direction, the sum of the raw bits of the populations of all fluid nodes
(a checksum).  The recorded ones were written on a GB300 with the library of
revision f69cc36 of this repository.

The inputs take only exactly rounded operations (+, *, /, sqrt and the uniform
generator), so that they are the same on every machine.  Run on a GPU:
    python tests/golden/make_states_16bit.py
"""
import json
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

OUT = os.path.join(os.path.dirname(os.path.abspath(__file__)), "states_16bit.json")
SHAPE = (40, 42, 44)
STEPS = 16

# name: (bounce-back, radius, control points, body force, periodic in x, DEM substeps, cover/uncover, speed)
SCENES = {
    "light spheres": ("ibb", 2.5, 1, 0.0, False, 1, False, 0.02),
    "clusters": ("ibb", 4.0, 7, 0.0, False, 1, False, 0.02),
    "clusters, forced, periodic": ("ibb", 4.0, 6, 2e-5, True, 1, False, 0.02),
    "halfway": ("ladd", 3.0, 3, 0.0, False, 1, False, 0.02),
    "halfway, forced": ("ladd", 3.0, 4, 2e-5, False, 1, False, 0.02),
    "substeps": ("ibb", 3.0, 5, 0.0, False, 20, False, 0.02),
    "cover and uncover": ("ibb", 3.0, 5, 0.0, False, 1, True, 0.2),
}
E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
     (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
     (0, -1, 1)]
W = np.array([1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12)


def flow(seed):
    """f_i of a smooth flow with one per cent of noise, float32."""
    rng = np.random.default_rng(seed)
    nx, ny, nz = SHAPE
    bump = [4.0 * x * (1.0 - x) for x in (np.arange(n) / n for n in (nz, ny, nx))]
    amp = (rng.random(3) - 0.5) * 0.08
    u = [amp[a] * bump[0][:, None, None] * bump[1][None, :, None] * bump[2][None, None, :] for a in range(3)]
    usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
    f = np.empty((19, nz, ny, nx), dtype=np.float32)
    for i in range(19):
        eu = E[i][0] * u[0] + E[i][1] * u[1] + E[i][2] * u[2]
        f[i] = W[i] * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * usq) * (1.0 + 0.02 * (rng.random((nz, ny, nx)) - 0.5))
    return f


def particles(scene):
    """(centers, k, position, quaternion, velocity, angular velocity, mass properties) of five particles."""
    bb, r, balls, _, _, _, _, speed = SCENES[scene]
    rng = np.random.default_rng(list(SCENES).index(scene))
    out = []
    for p in range(5):
        R = r * (1.0 - 0.1 * p / 4.0)
        c = (rng.random((balls, 3)) - 0.5) * (0.7 * R if balls > 1 else 0.0)
        c = (c - c.sum(axis=0) / balls).astype(np.float32).astype(np.float64)
        k = np.full(balls, R * R / balls).astype(np.float32).astype(np.float64)
        q = rng.random(4) - 0.5
        q = q / np.sqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2] + q[3] * q[3])
        at = np.array([(11.0, 11.0, 11.0), (29.0, 12.0, 30.0), (12.0, 30.0, 31.0), (30.0, 30.0, 12.0),
                       (20.0, 21.0, 21.5)][p]) + rng.random(3) - 0.5
        vel, om = (rng.random(3) - 0.5) * 2.0 * speed, (rng.random(3) - 0.5) * 0.01
        vol = 4.0 / 3.0 * 3.14159265358979 * R * R * R
        mp = {"mass": 2.5 * vol, "volume": vol, "inertia": np.eye(3) * (0.4 * 2.5 * vol * R * R)}
        out.append((c, k, at, q, vel, om, mp))
    return out


def run(B, scene, storage):
    """(states (5, 13), checksum of each direction) after STEPS steps."""
    bb, _, _, force, periodic, substeps, cover, _ = SCENES[scene]
    with B.Simulation(*SHAPE, tau=0.8, storage=storage, bb_mode=B.BB_LADD if bb == "ladd" else B.BB_IBB,
                      gravity=(0.0, 0.0, -1e-5), fluid_body_force=(force, 0.0, 0.0), periodic=(periodic, False, False),
                      dem_substeps=substeps, max_particles=8) as sim:
        sim.set_populations(flow(3))
        for c, k, at, q, vel, om, mp in particles(scene):
            sim.add_particle(c, k, 2.5, 0.6, at, q, vel, om, mass_props=mp)
        if cover:
            sim.set_momentum_rules(cover_uncover=True)
        sim.step(STEPS)
        sim.synchronize()
        states = np.array([np.concatenate([s[key] for key in ("pos", "quat", "vel", "omega")])
                           for s in (sim.get_particle_state(p) for p in range(5))])
        _, owner = sim.node_classes()
        raw = sim.get_raw_populations().astype(np.int64)
        return states, [int(raw[i][owner == 0xFFFFFFFF].sum()) for i in range(19)]


def main():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2209_10411_gb300 import _binding as B
    out = {}
    for scene in SCENES:
        for name, storage in (("f16", B.STORE_F16_DEV), ("bf16", B.STORE_BF16_DEV)):
            states, sums = run(B, scene, storage)
            out["%s, %s" % (scene, name)] = {"states": [[v.hex() for v in row] for row in states.tolist()], "sums": sums}
    with open(OUT, "w") as f:
        json.dump(out, f, indent=1)
    print("wrote", OUT)


if __name__ == "__main__":
    main()
