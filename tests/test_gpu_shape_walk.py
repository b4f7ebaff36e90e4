"""The column walk of the shape descriptors against a table that turns it off:
the same particle with one more ball of k = 0 far away keeps its field, and
with one of k = -0.0 keeps it too; a ball of negative k takes the cell-by-cell
path (its bounds do not hold), so a pair of opposite balls in one place, whose
terms cancel exactly, gives the cell-by-cell result of the same field: counts,
volume, extents and projected area equal, sums within the float32 rounding of
their order-free parts (the same terms in the same order: 1e-12).  Ball counts
at the staging limit, odd and even, thin and thick bands, coarse and fine grids."""
import numpy as np
import pytest

from tests.gpu_helpers import binding
from paper_2209_10411_gb300 import scenes

pytestmark = pytest.mark.gpu


def _model(n, seed):
    rng = np.random.default_rng(seed)
    c = scenes.uniform_in_ball(rng, n, 4.0) * np.array([1.6, 1.0, 0.6])
    k = rng.uniform(0.5, 1.5, n)
    return scenes.f32(c), scenes.f32(k / k.sum() * 36.0)


def _cellwise(c, k):
    """The model with two opposite balls appended in one place: the fields'
    two terms are equal and of opposite sign in every cell, added last."""
    at = np.array([[0.1, 0.2, 0.3]])
    return np.concatenate([c, at, at]), np.concatenate([k, [2.0 ** -20], [-2.0 ** -20]])


@pytest.mark.parametrize("n", [1, 2, 3, 64, 509, 510, 511, 600])
@pytest.mark.parametrize("h,eps", [(0.5, 0.1), (0.23, 0.01), (1.1, 0.9)])
def test_walk_equals_cell_by_cell(n, h, eps):
    B = binding()
    c, k = _model(n, 7 * n + 1)
    walked, cellwise = B.shape_descriptors([(c, k)], h, eps)[0], B.shape_descriptors([_cellwise(c, k)], h, eps)[0]
    # appending the cancelling pair leaves R_g and so both grids as they are
    for f in ("cells", "volume", "l_long", "l_int", "l_short", "projected_area", "d_n", "d_s", "csf"):
        assert walked[f] == cellwise[f], f
    assert walked["surface"] == pytest.approx(cellwise["surface"], rel=1e-12 if n == 1 else 1e-5)
    assert np.array_equal(walked["axes"], cellwise["axes"])
