"""16-bit population storages with light particles.

test_recorded: the states and the stored populations of tests/golden/states_16bit.json.
The populations are compared to the bit.  The states: the same sums of
forces enter an FP64 update of about 50 roundings per substep, whose order may differ: at most
320 substeps x 50 x 2^-53 relative to the largest entry (44), 8e-11.

test_against_oracle: the velocities of spheres against the FP64 oracle, bounded by
what the storage alone explains.  A stored value is off by at most half a unit, u
|h| with u = 2^-9 (BF16) or 2^-12 (FP16, whose subnormals round to 2^-25), of
either sign: a standard deviation of u h_max / sqrt(3), h_max the largest deviation
of a moving direction.  A value that reaches a link in step s has been rounded s
times at most (the collision does not amplify), a link's momentum takes two of
them, and a bounce-back population is formed with weights of at most 2.  So the
velocity's variance after n steps is at most sum_s links * 2 * 4 * s * (u h_max /
sqrt(3) + 2^-25)^2 / mass^2; six standard deviations are allowed.
"""
import json
import os

import numpy as np
import pytest

from oracle import step as ostep
from tests.golden import make_states_16bit as mk
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu

with open(mk.OUT) as _f:
    RECORDED = json.load(_f)


@pytest.mark.parametrize("name", list(RECORDED))
def test_recorded(name):
    B = binding()
    scene, storage = name.rsplit(", ", 1)
    states, sums = mk.run(B, scene, B.STORE_F16_DEV if storage == "f16" else B.STORE_BF16_DEV)
    want = np.array([[float.fromhex(v) for v in row] for row in RECORDED[name]["states"]])
    assert sums == RECORDED[name]["sums"]
    assert np.abs(states - want).max() < 8e-11, np.abs(states - want).max()


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("radius", [2.5, 4.0, 6.0])
@pytest.mark.parametrize("seed", [1, 2])
def test_against_oracle(storage, radius, seed):
    B = binding()
    rng = np.random.default_rng(seed)
    shape, steps = (26, 25, 24), 6
    f0 = mk.flow(seed)[:, :shape[2], :shape[1], :shape[0]]
    vol = 4.0 / 3.0 * np.pi * radius ** 3
    P = {"centers": np.zeros((1, 3)), "k": np.array([radius * radius]), "pos": 12.0 + rng.random(3),
         "quat": np.array([1.0, 0.0, 0.0, 0.0]), "vel": (rng.random(3) - 0.5) * 0.04, "omega": np.zeros(3),
         "density": 2.5, "skin": 0.6, "mass": 2.5 * vol, "volume": vol, "inertia": np.eye(3) * vol * radius ** 2}
    with B.Simulation(*shape, tau=0.8, storage=B.STORE_F16_DEV if storage == "f16" else B.STORE_BF16_DEV) as sim:
        sim.set_populations(f0)
        S = ostep.OracleState(shape, sim.get_populations().astype(np.float64), [P], tau=0.8)
        sim.add_particle(P["centers"], P["k"], 2.5, 0.6, P["pos"], P["quat"], P["vel"], P["omega"],
                         mass_props={"mass": P["mass"], "volume": vol, "inertia": P["inertia"]})
        links, var, hmax = 0, 0.0, 0.0
        u = 2.0 ** -12 if storage == "f16" else 2.0 ** -9
        for s in range(1, steps + 1):
            ostep.step(S)
            sim.step(1)
            links = max(links, len(sim.links()["q"]))
            dev = S.f[1:, np.isfinite(S.f).all(axis=0)] - mk.W[1:, None]
            hmax = max(hmax, float(np.abs(dev).max()))
            var += links * 8.0 * s * (u * hmax / np.sqrt(3.0) + 2.0 ** -25) ** 2 / P["mass"] ** 2
            bound = 6.0 * np.sqrt(var)
            err = np.abs(sim.get_particle_state(0)["vel"] - S.particles[0]["vel"]).max()
            assert err < bound, (s, err, bound)
    print("STATES16", storage, radius, seed, "velocity error %.2e, bound %.2e" % (err, bound))
