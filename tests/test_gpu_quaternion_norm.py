"""A quaternion that is handed in a little off unit norm is a rotation all the same:
the angular velocity of a freely turning sphere stays what it is.

omega goes to the body frame and back, R' R^T omega with equal moments, where R is
formed from the given quaternion and R' from the normalised new one: an error of the
norm left in R is an error of omega.  Bound: what is left of the norm, 8 ulps, and
three roundings in each of the two rotations' entries and sums, 12 more of
2^-53; the given ones are 30 to 60 ulps off."""
import numpy as np
import pytest

from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("substeps", [1, 10])
@pytest.mark.parametrize("off", [60, 30, -30, -50])
def test_norm(substeps, off):
    import torch
    B = binding()
    n = 24
    rng = np.random.default_rng(3)
    st = np.zeros((n, 13))
    for p in range(n):
        q = rng.random(4) - 0.5
        st[p, :3] = 12.0 + 20.0 * np.array([p % 3, p // 3 % 3, p // 9])
        st[p, 3:7] = q / np.sqrt((q * q).sum()) * (1.0 + 0.5 * off * 2.0 ** -52)
        st[p, 10:13] = (rng.random(3) - 0.5) * 0.02
    with B.Simulation(64, 64, 64, tau=0.8, max_particles=n, dem_substeps=substeps) as sim:
        for p in range(n):
            sim.add_particle(np.zeros((1, 3)), np.array([9.0]), 2.5, 0.5, st[p, :3], st[p, 3:7], (0, 0, 0), st[p, 10:13],
                             mass_props={"mass": 300.0, "volume": 120.0, "inertia": np.eye(3) * 1024.0})
        given, taken = torch.from_numpy(st.copy()).pin_memory(), torch.zeros((n, 13), dtype=torch.float64).pin_memory()
        sim.set_particle_states_ptr(given.data_ptr(), n)
        sim.step_phases(B.PHASE_CONTACT | B.PHASE_INTEGRATE)
        sim.get_particle_states_ptr(taken.data_ptr(), n)
        sim.synchronize()
    err = np.linalg.norm(taken.numpy()[:, 10:] - st[:, 10:], axis=1) / np.linalg.norm(st[:, 10:], axis=1)
    assert np.linalg.norm(taken.numpy()[:, 10:]) > 0.0
    assert err.max() < 8 * 2.0 ** -52 + substeps * 12 * 2.0 ** -53, (err.max() / 2.0 ** -53)
