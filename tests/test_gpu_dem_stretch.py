"""The fused DEM kernel's stretches without candidates (rigid-body updates
alone) against one launch sequence per substep: the same bits, from particles
that no test could pair through the substep in which they first can be, and for
the counts at which the lanes' groups and warps fill."""
import numpy as np
import pytest

from tests.gpu_helpers import binding
from tests.test_gpu_contact import _assert_same_bits, _compact, _dem_snapshot, _particle, _sim
from paper_2209_10411_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 5, 17, 64])
@pytest.mark.parametrize("substeps", [2, 7, 100])
def test_stretches_equal_per_substep_launches(n, substeps):
    """Particles on a grid, every second one moving towards its neighbour and
    the first towards the wall, over steps that begin without a candidate and
    end with contacts (checked)."""
    B = binding()
    rng = np.random.default_rng(100 * n + substeps)
    side = int(np.ceil(n ** (1 / 3)))
    pitch = 15.0
    shape = (int(side * pitch) + 4,) * 3
    parts = []
    for k in range(n):
        at = np.array([k % side, k // side % side, k // side ** 2]) * pitch + 9.5
        c, kk = _compact(rng)
        v = np.array([0.35 if k % 2 == 0 else -0.35, 0.02, -0.01])
        if k == 0 and n == 1:
            v[0] = -0.35
        parts.append(_particle(c, kk, at, scenes.random_unit_quaternion(rng), vel=v, omega=rng.uniform(-0.05, 0.05, 3)))
    runs = []
    for unfused in (False, True):
        sim = _sim(B, shape, parts, dem_substeps=substeps, gravity=(0, 0, -1e-4))
        sim.set_schedule(unfused_dem=unfused)
        snaps = []
        for _ in range(16):
            sim.step_phases(B.PHASE_CONTACT | B.PHASE_INTEGRATE)
            snaps.append(_dem_snapshot(sim, n))
        runs.append(snaps)
        sim.close()
    assert not runs[0][0][1] and any(s[1] for s in runs[0])  # none at first, some later
    for a, b in zip(*runs):
        _assert_same_bits(a, b)


def test_fast_rotation_takes_the_long_series():
    """Angular velocities above 1/32 a substep leave the short series; the
    quaternion handed in is off its norm by 1e-3 and is normalised."""
    B = binding()
    rng = np.random.default_rng(3)
    c, k = _compact(rng)
    snaps = []
    for unfused in (False, True):
        sim = _sim(B, (40, 40, 40), [_particle(c, k, [20.0, 20.0, 20.0], [1, 0, 0, 0], omega=(0.3, -0.2, 0.25))],
                   dem_substeps=2)
        sim.set_schedule(unfused_dem=unfused)
        sim.set_particle_state(0, quat=np.array([1.001, 0.02, -0.03, 0.01]))
        for _ in range(5):
            sim.step_phases(B.PHASE_CONTACT | B.PHASE_INTEGRATE)
        snaps.append(_dem_snapshot(sim, 1))
        sim.close()
    _assert_same_bits(*snaps)
    assert abs(np.linalg.norm(snaps[0][0][0]["quat"]) - 1.0) < 1e-15
