"""Wall fractions of links that graze the surface (FP32 storage): a sphere moved so
that lattice nodes lie a depth d below its surface and links reach them along the
tangent, d from 1e-7 to 3e-2 lu; against the sphere's intersection in FP64.

Bound per link as for ordinary ones: 1e-7 of Newton's remainder, 3e-8 of FP32 at 1,
and the residual's error, 14 * 2^-24 grid spacings / R + 2^-42, over the slope of
f along the link, which goes to 0 with d; q is at least 1e-6."""
import numpy as np
import pytest

from oracle.d3q19 import E
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu
R, NX = 5.3, 40
SPACING = 2.0 ** -8  # 4096 times it is the first power of two above 2 R_b + 4 = 14.6


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("shift", [0.0, 0.003, 0.02, -0.01])
def test_grazing_links(axis, shift):
    B = binding()
    with B.Simulation(NX, NX, NX, tau=0.8) as sim:
        sim.add_particle(np.zeros((1, 3)), np.array([R * R]), 2.5, 0.5, (20.0, 20.0, 20.0), (1, 0, 0, 0),
                         mass_props={"mass": 1000.0, "volume": 400.0, "inertia": np.eye(3) * 5000.0})
        flat = 1.0
        for depth in 10.0 ** np.linspace(-7.0, -1.5, 23):
            pos = np.array([20.0, 20.0, 20.0])
            pos[axis] += R - depth
            pos[(axis + 1) % 3] += shift
            sim.set_particle_state(0, pos=pos)
            sim.step_phases(B.PHASE_FLAG | B.PHASE_LINKS)
            sim.synchronize()
            g = sim.links()
            cell = g["cell"].astype(np.int64)
            x = np.stack([cell % NX, cell // NX % NX, cell // NX ** 2], axis=1)
            e = np.asarray(E, dtype=np.float64)[g["dir"].astype(np.int64)]
            a = x - pos
            ee, ae = (e * e).sum(1), (a * e).sum(1)
            q = (-ae - np.sqrt(np.maximum(ae * ae - ee * ((a * a).sum(1) - R * R), 0.0))) / ee
            slope = np.abs(2.0 * ((a + q[:, None] * e) * e).sum(1)) / (R * R)
            noise = 14.0 * 2.0 ** -24 * SPACING / R + 2.0 ** -42
            err = np.abs(g["q"].astype(np.float64) - np.clip(q, 1e-6, 1.0))
            bound = 1.3e-7 + noise / np.maximum(slope, 1e-12)
            assert (err < bound).all(), (depth, err.max(), slope[err.argmax()])
            flat = min(flat, slope.min())
        assert flat < 3e-3  # some links did graze
