"""Wall fractions q of the boundary links against FP64, over the forms of the
coordinate split: small, ordinary and large grid spacings with exactly summed
squares (bounding radius below 1000) and squares summed as float pairs
(beyond), one ball, odd and even ball counts.

Bound per link: 1e-7 of Newton's quadratic remainder, half a unit of FP32 at 1
(3e-8), and the residual's error over |f'(q)|.  The residual's: r^2 = |u|^2 +
m . (2 u + m) with |u|^2 exact and |m| per axis at most one grid spacing, the
second term rounded in FP32 with six roundings: 14 * 2^-24 spacing / r of a
ball's term k / r^2 covers it, and 2^-42 the sums."""
import numpy as np
import pytest

from oracle import coupling, metaball
from oracle.d3q19 import E
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


def _spacing(rb):
    g = 2.0 ** -7
    if rb < 1000.0:
        g = 2.0 ** -12
        while g * 4096.0 < 2.0 * rb + 4.0:
            g *= 2.0
    return g


def _cluster(n, r, seed):
    rng = np.random.default_rng(seed)
    c = rng.normal(size=(n, 3))
    c *= (0.6 * r * rng.random(n) ** (1.0 / 3.0) / np.linalg.norm(c, axis=1))[:, None]
    return c, rng.uniform(0.5, 1.5, n) * r * r / n


def _pair(half, r):
    return np.array([[-half, 0.3, 0.1], [half, -0.2, 0.4]]), np.array([r * r, 1.1 * r * r])


Q = np.array([0.9, 0.1, -0.3, 0.2]) / np.linalg.norm([0.9, 0.1, -0.3, 0.2])
QX = np.array([1.0, 0.0, 0.0004, 0.0003]) / np.linalg.norm([1.0, 0.0, 0.0004, 0.0003])
CASES = {
    "tiny": ((20, 19, 18), _cluster(1, 1.6, 0), Q),
    "one": ((24, 25, 26), _cluster(1, 5.3, 1), Q),
    "odd": ((40, 39, 38), _cluster(5, 9.0, 2), Q),
    "even": ((72, 70, 68), _cluster(64, 20.0, 3), Q),
    "long, exact": ((2010, 24, 26), _pair(985.0, 6.0), QX),
    "long, pairs": ((2090, 24, 26), _pair(1020.0, 6.0), QX),
}


@pytest.mark.parametrize("name", list(CASES))
def test_wall_fractions(name):
    B = binding()
    shape, (c, k), quat = CASES[name]
    c, k = c.astype(np.float32).astype(np.float64), k.astype(np.float32).astype(np.float64)
    pos = np.array([0.5 * n + d for n, d in zip(shape, (0.137, -0.241, 0.318))])
    with B.Simulation(*shape, tau=0.8) as sim:
        sim.add_particle(c, k, 2.5, 0.5, pos, quat,
                         mass_props={"mass": 1000.0, "volume": 400.0, "inertia": np.eye(3) * 5000.0})
        sim.step(1)
        g = sim.links()
    assert len(g["q"]) > 50
    nx, ny, _ = shape
    cell = g["cell"].astype(np.int64)
    x = np.stack([cell % nx, (cell // nx) % ny, cell // (nx * ny)], axis=1)
    d = g["dir"].astype(np.int64)
    P = {"pos": pos, "quat": quat, "centers": c, "k": k}
    ref = coupling.wall_fraction(x, d, P)
    R = metaball.quat_to_matrix(quat)
    e = np.asarray(E, dtype=np.float64)[d]
    p = metaball.to_body(x + ref[:, None] * e, pos, R)
    a = p[:, None, :] - c[None]
    r2 = (a * a).sum(-1)
    t = k / r2
    slope = np.abs((-2.0 * t / r2 * (a * (e @ R)[:, None, :]).sum(-1)).sum(-1))
    rb = np.linalg.norm(c, axis=1).max() + np.sqrt(k.sum())
    noise = (t * 14.0 * 2.0 ** -24 * _spacing(rb) / np.sqrt(r2)).sum(-1) + 2.0 ** -42
    err = np.abs(g["q"].astype(np.float64) - ref)
    assert (err < 1.3e-7 + noise / slope).all(), (err.max(), (err / (1.3e-7 + noise / slope)).max())
