"""Gene counts around the default shared-memory limit (48 KB holds 3008 genes beside
the reduction's 1 KB, 3072 alone): every count runs, and the fitness of parents and
children is the FP64 sum to FP32 rounding: 64 points' squares of f - 1, each f a sum
of n terms with an error of at most n 2^-24 f."""
import numpy as np
import pytest

from paper_2209_10411_gb300 import scenes
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("genes", [3007, 3008, 3009, 3072, 3073])
def test_shared_memory_limit(genes):
    B = binding()
    rng = np.random.default_rng(1)
    hull = scenes.ellipsoid_hull(rng, 64, np.array([9.0, 8.0, 7.0]), bumps=0.0)
    planes = scenes.hull_planes(hull)
    box = np.concatenate([hull.min(axis=0), hull.max(axis=0)])
    pop, fit, off, fit_off = B.ga_run(hull, planes, box, (0.01, 0.05), 2, genes, 1, 0.01, 0.5, 7)
    H = np.asarray(hull, dtype=np.float32).astype(np.float64)
    for members, values in ((pop, fit), (off, fit_off)):
        m = np.asarray(members.cpu() if hasattr(members, "cpu") else members, dtype=np.float64).reshape(2, genes, 4)
        v = np.asarray(values.cpu() if hasattr(values, "cpu") else values, dtype=np.float64)
        for g, got in zip(m, v):
            f = (g[:, 3] / ((H[:, None, :] - g[None, :, :3]) ** 2).sum(axis=2)).sum(axis=1)
            want, err = ((f - 1.0) ** 2).sum(), (2.0 * np.abs(f - 1.0) * genes * 2.0 ** -24 * f).sum()
            assert abs(got - want) <= err + 1e-5 * want, (got, want, err)
