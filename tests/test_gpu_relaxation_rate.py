"""The relaxation rate of FP32 storage for large tau: the decay of a stress.

The pattern s_i = +1 on (1, 1, 0) and (-1, -1, 0), -1 on (1, -1, 0) and (-1, 1, 0)
has no density and no momentum; the sum over the lattice of s_i f_i loses the
share 1 / tau a step, whatever the streaming does, but for the small equilibrium
stress, which the FP64 oracle follows.

Bound: the sum takes 4 N stored values a step, each off by at most half a unit in
the last place (2^-28 for f below 1/16) from the store and as much again from
the arithmetic before it, of either sign: six standard deviations of that,
2e-8 of the sum after eight steps.  The noise of the initial values makes the
roundings independent as long as the steps of 1 / tau of it are well above an ulp, which
holds up to tau = 1000 (at 10,000 every value moves by the same fraction of an ulp
and exact arithmetic stored in FP32 is 4e-8 a step off).  1 - 1 / tau rounded to FP32 is
off by 0.5 to 1.3e-8 a step at these tau, 4e-8 to 1e-7 in all."""
import numpy as np
import pytest

from oracle import lbm
from oracle.d3q19 import E, W
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [20.0, 200.0, 1000.0])
def test_stress_decay(tau):
    B = binding()
    steps, side = 8, 32
    s = np.array([e[0] * e[1] for e in np.asarray(E)], dtype=np.float64)
    rng = np.random.default_rng(5)
    f0 = W[:, None, None, None] + 0.005 * s[:, None, None, None]
    f0 = (f0 + 1e-3 * np.asarray(W)[:, None, None, None] * (rng.random((19,) + (side,) * 3) - 0.5)).astype(np.float32)
    with B.Simulation(side, side, side, tau=tau, periodic=(True, True, True)) as sim:
        sim.set_populations(f0)
        sim.step(steps)
        got = sim.get_populations().astype(np.float64)
    ref = f0.astype(np.float64)
    start = np.tensordot(s, ref, 1).sum()
    for _ in range(steps):
        ref = lbm.step_bulk(ref, tau, periodic=(True, True, True))
    off = (np.tensordot(s, got, 1).sum() - np.tensordot(s, ref, 1).sum()) / start
    tol = 6.0 * np.sqrt(steps * 4.0 * side ** 3) * 2.0 * 2.0 ** -28 / np.sqrt(12.0) / start
    assert abs(off) < tol, (off, tol)
