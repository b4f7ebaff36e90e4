"""Shape descriptors of one model in other units: scaling lengths by a power of two
and k by its square scales every operation of the field exactly, so the cells
are the same ones and the lengths and the area are scaled to the bit, also where
products of squared distances would leave FP32."""
import numpy as np
import pytest

from paper_2209_10411_gb300 import scenes
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 33, 600])
@pytest.mark.parametrize("power", [-39, -38, -37, -36, -20, 12, 28, 29, 30])
def test_units(n, power):
    B = binding()
    rng = np.random.default_rng(n)
    c = scenes.f32(scenes.uniform_in_ball(rng, n, 4.0) * np.array([1.6, 1.0, 0.6]))
    k = scenes.f32(np.full(n, 36.0 / n))
    s = 2.0 ** power
    one, other = (B.shape_descriptors([(c * f, k * f * f)], 0.2 * f)[0] for f in (1.0, s))
    assert one["cells"] > 1000 and other["cells"] == one["cells"]
    assert other["volume"] == one["volume"] * s ** 3
    for f in ("l_long", "l_int", "l_short"):
        assert other[f] == one[f] * s, f
    assert other["projected_area"] == one["projected_area"] * s * s
