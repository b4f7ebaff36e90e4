"""The column walk of the shape descriptors where nothing changes and where one cell shows.

A ball of k = 0 or -0.0 inside the model changes neither the field nor the grid, so
every figure is the same bits, whichever table (staged or in place) it fits.

The surface counts every band cell once: on a grid so coarse that the least of the
band's gradients is above twice the bar, against the FP64 sum over the same cells.
Bar, relative: a gradient is a sum of n terms of about 8 roundings each, the terms'
lengths adding up to at most four times their sum's, and the cells' sum adds about a
hundred positive terms in turn in FP32 (threads, block): (4 (n + 8) + 96) 2^-24."""
import numpy as np
import pytest

from oracle import shape
from paper_2209_10411_gb300 import scenes
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


def _model(n, seed):
    rng = np.random.default_rng(seed)
    c = scenes.uniform_in_ball(rng, n, 3.0) * np.array([1.6, 1.0, 0.6])
    k = rng.uniform(0.5, 1.5, n)
    return scenes.f32(c), scenes.f32(k / k.sum() * 36.0)


@pytest.mark.parametrize("n", [1, 2, 64, 510, 511, 512, 600])
@pytest.mark.parametrize("zero", [0.0, -0.0])
def test_ball_without_weight(n, zero):
    B = binding()
    c, k = _model(n, n)
    one = B.shape_descriptors([(c, k)], 0.3)[0]
    more = B.shape_descriptors([(np.concatenate([c, [[0.11, 0.07, -0.13]]]), np.append(k, zero))], 0.3)[0]
    for f in B.SHAPE_FIELDS:
        assert more[f] == one[f], f
    assert np.array_equal(more["axes"], one["axes"])


@pytest.mark.parametrize("n", [1, 2, 3, 64, 511, 512, 600])
@pytest.mark.parametrize("h,eps", [(1.0, 0.1), (1.3, 0.3)])
def test_every_band_cell_once(n, h, eps):
    B = binding()
    c, k = _model(n, 5 * n + 1)
    R = np.float32(shape.grid_radius(c, k, eps))
    ax = shape._axis(int(np.ceil(2.0 * float(R) / float(np.float32(h)))), -R, h)
    points = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), axis=-1).reshape(-1, 3)
    f = shape.field_f32(points, c, k)
    g = shape.grad_norm(points[np.abs(f - np.float32(1.0)) < np.float32(eps)], c, k)
    bar = (4.0 * (n + 8) + 96.0) * 2.0 ** -24
    assert len(g) > 20 and g.min() > 2.0 * bar * g.sum()
    want = g.sum() * float(np.float32(h)) ** 3 / (2.0 * float(np.float32(eps)))
    assert B.shape_descriptors([(c, k)], h, eps)[0]["surface"] == pytest.approx(want, rel=bar)
