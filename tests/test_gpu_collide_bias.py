"""The collision adds no momentum of its own: the fluid's summed momentum over
a periodic lattice after one step, against before.

Bound: the exact collision conserves it, so the change is the sum of the
rounding errors of 18 N stored populations.  Each is a handful of independent
roundings of values below 1/18 (1 + 0.3) and at most 2^-25 relative, the store
itself the largest: a standard deviation of at most 2^-25 * 0.072 / sqrt(3) *
2 per population.  Six standard deviations of the sum are allowed; a relative
error of 2.4e-8 common to all nodes (a rounded omega w_i) is an order of
magnitude more."""
import numpy as np
import pytest

from oracle.d3q19 import E, W
from paper_2209_10411_gb300 import scenes
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu

SHAPE = (48, 33, 31)


@pytest.mark.parametrize("tau", [0.6, 0.8, 1.0, 2.6])
@pytest.mark.parametrize("seed", [1, 2])
def test_momentum_is_kept(tau, seed):
    B = binding()
    noise = scenes.lattice_noise(SHAPE, seed).astype(np.float64)
    u = np.array([0.06, -0.05, 0.04])
    eu = np.asarray(E, dtype=np.float64) @ u
    f0 = (W * (1.0 + 3.0 * eu)).reshape(19, 1, 1, 1) * (1.0 + 0.05 * noise)
    f0 = f0.astype(np.float32)
    with B.Simulation(*SHAPE, tau=tau, periodic=(True, True, True)) as sim:
        sim.set_populations(f0)
        sim.step(1)
        f1 = sim.get_populations()
    e = np.asarray(E, dtype=np.float64)
    j0 = e.T @ f0.astype(np.float64).sum(axis=(1, 2, 3))
    j1 = e.T @ f1.astype(np.float64).sum(axis=(1, 2, 3))
    n = np.prod(SHAPE)
    tol = 6.0 * np.sqrt(18.0 * n) * 2.0 ** -25 * 0.072 / np.sqrt(3.0) * 2.0
    assert np.abs(j1 - j0).max() < tol, (j1 - j0, tol)
