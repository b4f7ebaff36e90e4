"""Launch shapes are kept where they are not set, and shapes that were tuned for other
kernels are not read back."""
import json

import numpy as np
import pytest

from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu


def test_what_is_not_given_stays():
    B = binding()
    with B.Simulation(192, 192, 192, tau=0.8, storage=B.STORE_F16_DEV) as sim:
        first = sim.get_tuning()
        sim.set_tuning()
        assert sim.get_tuning() == first
        sim.set_tuning(list_blocks_per_sm=16)
        assert sim.get_tuning() == dict(first, list_blocks_per_sm=16)
        sim.set_tuning(bulk_block_x=32)
        assert sim.get_tuning() == dict(first, list_blocks_per_sm=16, bulk_block_x=32)
        # more than 128 threads and paired nodes exclude each other
        sim.set_tuning(bulk_block_x=256)
        assert sim.get_tuning() == dict(first, list_blocks_per_sm=16, bulk_block_x=256, bulk_pairs=0)
        sim.set_tuning(bulk_pairs=True)
        assert sim.get_tuning() == dict(first, list_blocks_per_sm=16, bulk_block_x=128, bulk_pairs=1)
        with pytest.raises(B.MiDelbmError):
            sim.set_tuning(bulk_block_x=256, bulk_pairs=1)


def test_lines_of_other_kernels_miss(tmp_path):
    B = binding()
    cache = str(tmp_path / "tune.json")

    def tuned():
        with B.Simulation(48, 40, 32, tau=0.8) as sim:
            sim.add_particle(np.zeros((1, 3)), np.array([36.0]), 2.5, 0.5, (20.0, 20.0, 16.0), (1, 0, 0, 0))
            sim.step(2)
            return sim.autotune(cache)

    tuned()
    with open(cache) as f:
        line = json.loads(f.read())
    revision, rest = line["key"].split("/", 1)
    assert revision.startswith("kernels")
    # the same device, lattice and particles as an earlier library wrote them
    stale = [dict(line, key=k, bulk_block_x=256, list_blocks_per_sm=61) for k in (rest, "kernels1/" + rest)]
    with open(cache, "w") as f:
        f.write("".join(json.dumps(s) + "\n" for s in stale))
    assert tuned()["list_blocks_per_sm"] != 61
    with open(cache) as f:
        lines = [json.loads(s) for s in f]
    assert len(lines) == 3 and lines[2]["key"] == line["key"]
    assert tuned()["list_blocks_per_sm"] == lines[2]["list_blocks_per_sm"]
    with open(cache) as f:
        assert len(f.readlines()) == 3  # read back, nothing appended
