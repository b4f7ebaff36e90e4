"""One epoch of each descent of the Gradient Search at the edges of its units (odd and
even counts of hull points and control points, one of each), with moves far above
the bar.

The learning rate makes the largest move a thousandth of the largest value.  Bar: 1e-4
of the largest move (FP32 sums of up to 5000 terms of one sign differ by at most
5000 2^-24 = 3e-4 of the sum of their sizes; the sums here cancel to no less than a
tenth of it on average) plus the rounding of the values.  The bar tells: a model that
does not move at all, and one whose last hull point counts twice (an odd last point
shares its pair with a copy of itself), lie outside it; both are made here from the
oracle."""
import numpy as np
import pytest

from oracle import gs
from paper_2209_10411_gb300 import scenes
from tests.gpu_helpers import binding

P = np.array([[1.0, 0, 0, 1e6]])  # a plane nothing lies outside of


def _clear(f):
    """All hull points 2e-5 away from the kinks of the loss, where the branch is a coin toss in FP32."""
    return np.all((np.abs(f - 1.0) > 2e-5) & (np.abs(f - 2.0) > 2e-5))


def _problem(m, n):
    """Hull, model, learning rate, the oracle's model after the two epochs and the bar."""
    semi = (9.0, 7.0, 8.0)
    for seed in range(300):
        rng = np.random.default_rng(1000 * m + n + 10 ** 7 * seed)
        H = scenes.ellipsoid_hull(rng, m, semi, bumps=0.1)
        c, k = scenes.gs_start_model(rng, n, semi)
        gc, gk = gs.gradient(H, c, k)
        vals = max(np.abs(c).max(), np.abs(k).max())
        lr = float(np.float32(1e-3 * vals / max(np.abs(gc).max(), np.abs(gk).max())))
        c1, k1 = gs.descend(H, c, k, 1, lr)
        if k1.min() > 0.0 and _clear(gs.field(H, c, k)) and _clear(gs.field(H, c1, k1)):
            break
    else:
        raise AssertionError("no seed whose hull points keep away from the kinks")
    moved = _move(gs.descend(H, c1, k1, 1, lr), c, k)
    tol = 1e-4 * np.abs(moved).max() + 4e-7 * vals
    return H, c, k, lr, moved, tol


def _move(model, c, k):
    return np.concatenate([(model[0] - c).ravel(), model[1] - k])


M, N = [1, 2, 3, 64, 65, 1023, 1025, 5000], [1, 2, 3, 33, 256]


@pytest.mark.parametrize("m", M)
@pytest.mark.parametrize("n", N)
def test_the_bar_tells(m, n):
    H, c, k, lr, moved, tol = _problem(m, n)
    assert np.abs(moved).max() > 100.0 * tol  # not moving at all
    if m % 2 and m < 1000:
        twice = np.concatenate([H, H[-1:]])
        again = gs.descend(twice, *gs.descend(twice, c, k, 1, lr), 1, lr)
        assert np.abs(_move(again, c, k) - moved).max() > 2.0 * tol


@pytest.mark.gpu
@pytest.mark.parametrize("m", M)
@pytest.mark.parametrize("n", N)
def test_one_epoch(m, n):
    B = binding()
    H, c, k, lr, moved, tol = _problem(m, n)
    (cg, kg, act), = B.gs_fit([H], [(c, k)], [P], 1, lr)[0]
    assert act.all()
    got = _move((cg, kg), c, k)
    assert np.abs(got - moved).max() <= tol, (np.abs(got - moved).max(), tol, np.abs(moved).max())
