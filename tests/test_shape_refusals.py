"""Models that have no grid are refused before anything reaches the device: each
beside a good one, whose cell count alone would size the call.  (Without a GPU: the
refusal comes first.)"""
import numpy as np
import pytest

from tests.gpu_helpers import binding

GOOD = (np.zeros((1, 3)), np.array([9.0]))
NAN = (np.array([[0.0, np.nan, 0.0]]), np.array([9.0]))
NEGATIVE = (np.zeros((2, 3)), np.array([1.0, -9.0]))
ESCAPED = (np.array([[0.0, 0.0, 0.0], [1e25, 0.0, 0.0]]), np.array([9.0, 1.0]))
INFINITE = (np.zeros((1, 3)), np.array([np.inf]))


@pytest.mark.filterwarnings("ignore::RuntimeWarning")
@pytest.mark.parametrize("bad,error", [(NAN, ValueError), (NEGATIVE, ValueError), (ESCAPED, OverflowError),
                                       (INFINITE, OverflowError)])
def test_no_grid(bad, error):
    B = binding()
    with pytest.raises(error):
        B.shape_descriptors([GOOD, bad], 0.25)


@pytest.mark.filterwarnings("ignore::RuntimeWarning")
@pytest.mark.parametrize("h,eps,error", [(0.0, 0.1, ZeroDivisionError), (1e-9, 0.1, OverflowError),
                                         (0.25, 1.0, OverflowError), (0.25, 1.5, ValueError)])
def test_no_spacing_or_band(h, eps, error):
    B = binding()
    with pytest.raises(error):
        B.shape_descriptors([GOOD, GOOD], h, eps)


@pytest.mark.gpu
def test_counts_outside_the_bound():
    """The C entry is bounded by its own argument: counts outside 1 .. max_n give NaN, the others their values."""
    import torch
    B = binding()
    n = 34
    counts = [n, 0, -5, n + 1, 2 ** 31 - 1, -2 ** 31, n]
    balls = torch.tensor([[0.0, 0.0, 0.0, 9.0]] * len(counts), dtype=torch.float32, device="cuda")
    off = torch.arange(len(counts) + 1, dtype=torch.int32, device="cuda")
    R = torch.full((len(counts),), 3.2, dtype=torch.float32, device="cuda")
    N = torch.tensor(counts, dtype=torch.int32, device="cuda")
    out = torch.empty((len(counts), len(B.SHAPE_FIELDS)), dtype=torch.float64, device="cuda")
    scratch = torch.empty(int(B.lib.mi_shape_scratch_bytes(len(counts), n)), dtype=torch.uint8, device="cuda")
    st = B.lib.mi_shape_descriptors(len(counts), B._tp(off), B._tp(balls), B._tp(R), B._tp(N), n, 0.2, 0.1, B._tp(out),
                                    None, B._tp(scratch), B._cur_stream())
    assert st == 0
    got = out.cpu().numpy()
    cells = B.SHAPE_FIELDS.index("cells")
    assert got[0][cells] > 100 and np.array_equal(got[0], got[-1])
    others = np.delete(got[1:-1], cells, axis=1)
    assert np.isnan(others).all()
