"""Owners, classes and links of the flagging and classification against the
oracle, exactly, on a lattice large enough for cubes of nodes and four rows a
warp and on a small one (node by node, row by row): odd extents, boxes cut by the
domain's faces and corners, one ball and many, a field far from spherical, and
boxes of several particles over the same nodes."""
import numpy as np
import pytest

from oracle import coupling, metaball
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu

LARGE, SMALL = (131, 129, 127), (45, 43, 41)


def _cluster(n, r, seed, squeeze=(1.0, 1.0, 1.0)):
    rng = np.random.default_rng(seed)
    c = rng.normal(size=(n, 3))
    c *= (0.7 * r * rng.random(n) ** (1.0 / 3.0) / np.linalg.norm(c, axis=1))[:, None]
    return c * np.asarray(squeeze), rng.uniform(0.3, 1.7, n) * 0.5 * r * r / n


def _scene(kind, shape):
    far = np.array(shape, dtype=float) - 1.0
    if kind == "middle":
        return [(_cluster(7, 8.0, 1), 0.5 * far + [0.3, -0.2, 0.4])]
    if kind == "one ball":
        return [((np.zeros((1, 3)), np.array([30.25])), 0.5 * far + [0.5, 0.5, 0.0])]
    if kind == "many balls":
        return [(_cluster(83, 11.0, 2, (1.5, 0.4, 0.8)), 0.5 * far + [0.1, 0.7, -0.6])]
    if kind == "corners":
        return [(_cluster(5, 7.0, 3), np.array([2.2, 3.4, 1.7])), (_cluster(6, 7.0, 4), far - [3.1, 1.2, 2.6])]
    # boxes over one another, surfaces a few nodes apart
    return [(_cluster(4, 6.0, 5), 0.5 * far - [7.4, 0.0, 0.0]), (_cluster(9, 6.0, 6), 0.5 * far + [6.6, 1.0, 0.5]),
            (_cluster(3, 5.0, 7), 0.5 * far + [0.0, 9.3, 1.2])]


@pytest.mark.parametrize("shape", [LARGE, SMALL], ids=["large", "small"])
@pytest.mark.parametrize("kind", ["middle", "one ball", "many balls", "corners", "neighbours"])
def test_owners_classes_links(kind, shape):
    B = binding()
    parts = []
    with B.Simulation(*shape, tau=0.8, max_particles=4) as sim:
        for i, ((c, k), pos) in enumerate(_scene(kind, shape)):
            c, k = c.astype(np.float32).astype(np.float64), k.astype(np.float32).astype(np.float64)
            quat = np.array([0.8, 0.3 - 0.2 * i, 0.1, -0.4])
            quat /= np.linalg.norm(quat)
            sim.add_particle(c, k, 2.5, 0.5, pos, quat,
                             mass_props={"mass": 1000.0, "volume": 400.0, "inertia": np.eye(3) * 5000.0})
            parts.append({"centers": c, "k": k, "pos": pos, "quat": quat})
        sim.step_phases(B.PHASE_FLAG | B.PHASE_LINKS)
        cls, own = sim.node_classes()
        g = sim.links()
    ref = metaball.flag_nodes(shape, parts)
    own = own.astype(np.int64)
    own[own == 0xFFFFFFFF] = -1
    assert (ref >= 0).sum() > 20
    assert np.array_equal(own, ref), int((own != ref).sum())
    cell, d, p = coupling.find_links(ref)
    lin = (cell[:, 2] * shape[1] + cell[:, 1]) * shape[0] + cell[:, 0]
    want = {tuple(v) for v in np.stack([lin, d, p], axis=1).tolist()}
    have = list(zip(g["cell"].astype(np.int64).tolist(), g["dir"].tolist(), g["particle"].tolist()))
    assert len(have) == len(want) and set(have) == want
    boundary = np.zeros(ref.size, dtype=bool)
    boundary[lin] = True
    assert np.array_equal((cls.reshape(-1) & 2) != 0, boundary)
    assert np.array_equal((cls & 1) != 0, ref >= 0)
