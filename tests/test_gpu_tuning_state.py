"""Launch shapes are kept where they are not set."""
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
