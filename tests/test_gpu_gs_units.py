"""The Gradient Search kernel's units at their edges: odd and even counts of
hull points (pairs), of control points (two to a unit), one of each, and counts
below and above the threads' and the chunks' strides.

Bar: one descent of one epoch moves every model value as the FP64 gradient does,
within 1e-4 of the largest move (FP32 sums of up to 5000 terms of one sign
differ by at most 5000 2^-24 = 3e-4 of the sum of their sizes; the sums here
cancel to no less than a tenth of it on average) plus the rounding of the
values; an escaped control point (1e25 away) adds nothing and takes no value of
the others with it."""
import numpy as np
import pytest

from oracle import gs
from paper_2209_10411_gb300 import scenes
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


def _problem(m, n):
    """The first of a series of seeds whose hull points all lie 1e-5 away from
    the kinks of the loss (f = 1, f = 2), where the branch is a coin toss in FP32."""
    for seed in range(1000 * m + n, 1000 * m + n + 100000, 1000):
        rng = np.random.default_rng(seed)
        semi = (9.0, 7.0, 8.0)
        H = scenes.ellipsoid_hull(rng, m, semi, bumps=0.1)
        c, k = scenes.gs_start_model(rng, n, semi)
        f = gs.field(H, c, k)
        if np.all((np.abs(f - 1.0) > 1e-5) & (np.abs(f - 2.0) > 1e-5)):
            break
    P = np.array([[1.0, 0, 0, 1e6]])  # a plane nothing lies outside of
    return H, c, k, P


@pytest.mark.parametrize("m", [1, 2, 3, 64, 1023, 1025, 5000])
@pytest.mark.parametrize("n", [1, 2, 3, 33, 256])
def test_one_epoch(m, n):
    B = binding()
    H, c0, k0, P = _problem(m, n)
    lr = 1e-6
    (c, k, act), = B.gs_fit([H], [(c0, k0)], [P], 1, lr)[0]
    c1, k1 = gs.descend(H, c0, k0, 1, lr)
    c2, k2 = gs.descend(H, c1, k1, 1, lr)
    dg, do = np.concatenate([(c - c0).ravel(), k - k0]), np.concatenate([(c2 - c0).ravel(), k2 - k0])
    vals = np.abs(np.concatenate([c2.ravel(), k2])).max()
    assert act.all()
    assert np.abs(dg - do).max() <= 1e-4 * np.abs(do).max() + 4e-7 * vals


def test_escaped_control_point():
    B = binding()
    H, c0, k0, P = _problem(500, 6)
    P = np.array([[1.0, 0, 0, 1e30]])
    c1 = np.concatenate([c0, [[1e25, 0.0, 0.0]]])
    k1 = np.concatenate([k0, [1.0]])
    (ca, ka, _), = B.gs_fit([H], [(c0, k0)], [P], 5, 1e-5)[0]
    (cb, kb, _), = B.gs_fit([H], [(c1, k1)], [P], 5, 1e-5)[0]
    assert np.allclose(ca, cb[:6], rtol=0, atol=1e-6) and np.allclose(ka, kb[:6], rtol=0, atol=1e-6)
    assert kb[6] == 1.0 and cb[6, 0] == np.float32(1e25)
