"""Gradient Search in very small and very large units: lengths scaled by s, k by s^2
(the field and the loss stay as they are), the centres' gradients scale by 1 / s.

Large: with a learning rate of s^2 / (64 points) the centres' steps scale by s, while k moves
by less than 2^-24 of itself; so the moves at s = 2^34 are those at 2^14 in other
units, but for k's last bits (1e-5 of the largest move allowed).  Small: at a learning rate of 0 the model stays as it is
(a gradient that is not a finite number would make it NaN)."""
import numpy as np
import pytest

from paper_2209_10411_gb300 import scenes
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


def _case(balls, points):
    rng = np.random.default_rng(balls)
    hull = scenes.f32(scenes.ellipsoid_hull(rng, points, np.array([9.0, 8.0, 7.0]), bumps=0.05))
    c = scenes.f32(rng.uniform(-3.0, 3.0, (balls, 3)))
    inside = np.array([[1.0, 0.0, 0.0, 3e38]], dtype=np.float32)  # a facet plane with everything inside
    return hull, c, scenes.f32(np.full(balls, 60.0 / balls)), inside


@pytest.mark.parametrize("balls,points", [(1, 64), (7, 301), (16, 2048)])
def test_large(balls, points):
    B = binding()
    hull, c, k, inside = _case(balls, points)
    moves = []
    for s in (2.0 ** 14, 2.0 ** 34):
        ((got, _, active),), _ = B.gs_fit([hull * s], [(c * s, k * s * s)], [inside], 1, s * s / (64.0 * points))
        assert active.all()
        moves.append(got / s - c)
    assert np.abs(moves[0]).max() > 1e-4  # hundreds of ulps of a centre
    assert np.abs(moves[1] - moves[0]).max() <= 1e-5 * np.abs(moves[0]).max()


@pytest.mark.parametrize("balls,points", [(1, 64), (7, 301), (16, 2048)])
@pytest.mark.parametrize("power", [-38, -30])
def test_small(balls, points, power):
    B = binding()
    hull, c, k, inside = _case(balls, points)
    s = 2.0 ** power
    ((got, gk, _),), loss = B.gs_fit([hull * s], [(c * s, k * s * s)], [inside], 2, 0.0)
    assert np.isfinite(loss).all()
    assert np.array_equal(got, (c * s).astype(np.float32)) and np.array_equal(gk, (k * s * s).astype(np.float32))
