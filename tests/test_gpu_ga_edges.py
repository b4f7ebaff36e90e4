"""Genetic Algorithm at the edges of its launches: two individuals, counts and
genes that fill no block, few facet planes (fewer than a round of planes in
flight), more individuals than the selection stages in shared memory, and facet planes
off their 16-byte alignment.  Integer decisions and copies: exact; the selection of the
oracle fed the GPU's fitness values: the same individuals in the same order."""
import ctypes

import numpy as np
import pytest

from oracle import ga
from paper_2209_10411_gb300 import scenes
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu

KR = (1.0, 6.0)


def _hull(m):
    rng = np.random.default_rng(m)
    H = scenes.ellipsoid_hull(rng, m, (6.0, 4.0, 3.0), bumps=0.1)
    return H, scenes.hull_planes(H), np.concatenate([H.min(0), H.max(0)]).astype(np.float32)


@pytest.mark.parametrize("n_ind,genes,points", [(2, 1, 12), (6, 5, 33), (30, 7, 130), (130, 3, 257)])
def test_one_generation(n_ind, genes, points):
    B = binding()
    H, P, bbox = _hull(points)
    pop0, fit0, _, _ = B.ga_run(H, P, bbox, KR, n_ind, genes, 0, 0.3, 0.4, 9)
    assert np.array_equal(pop0, ga.initial_population(9, n_ind, genes, bbox, KR, P))
    pop1, fit1, off, fo = B.ga_run(H, P, bbox, KR, n_ind, genes, 1, 0.3, 0.4, 9, pop=pop0)
    assert np.array_equal(off, ga.offspring(pop0, 9, 0, 0.3, 0.4, bbox, KR, P))
    sel, sf, _ = ga.select(pop0, fit0.astype(np.float64), off, fo.astype(np.float64))
    assert np.array_equal(pop1, sel) and np.array_equal(fit1, sf.astype(np.float32))


@pytest.mark.parametrize("n_ind", [4096, 4098])
def test_selection_of_many(n_ind):
    B = binding()
    H, P, bbox = _hull(20)
    pop0, fit0, _, _ = B.ga_run(H, P, bbox, KR, n_ind, 2, 0, 0.2, 0.5, 3)
    pop1, fit1, off, fo = B.ga_run(H, P, bbox, KR, n_ind, 2, 1, 0.2, 0.5, 3, pop=pop0)
    sel, sf, _ = ga.select(pop0, fit0.astype(np.float64), off, fo.astype(np.float64))
    assert np.array_equal(pop1, sel) and np.array_equal(fit1, sf.astype(np.float32))


def test_unaligned_planes():
    import torch
    B = binding()
    H, P, bbox = _hull(70)
    n_ind, genes, gens = 40, 6, 3
    want = B.ga_run(H, P, bbox, KR, n_ind, genes, gens, 0.3, 0.5, 21)
    hull = torch.as_tensor(np.asarray(H, dtype=np.float32).reshape(-1, 3), device="cuda").contiguous()
    planes = np.asarray(P, dtype=np.float32).reshape(-1, 4)
    shifted = torch.zeros(planes.size + 1, dtype=torch.float32, device="cuda")
    shifted[1:] = torch.as_tensor(planes.reshape(-1), device="cuda")
    assert shifted[1:].data_ptr() % 16 == 4
    pop, off = (torch.empty((n_ind, genes, 4), dtype=torch.float32, device="cuda") for _ in range(2))
    fit, fo = (torch.empty(n_ind, dtype=torch.float32, device="cuda") for _ in range(2))
    scratch = torch.empty(int(B.lib.mi_ga_scratch_bytes(n_ind, genes)), dtype=torch.uint8, device="cuda")
    bb, kr = (ctypes.c_float * 6)(*bbox.tolist()), (ctypes.c_float * 2)(*KR)
    p = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    torch.cuda.synchronize()
    st = B.lib.mi_ga_run(n_ind, genes, p(hull), int(hull.shape[0]), p(shifted[1:]), len(planes),
                         ctypes.cast(bb, ctypes.c_void_p), ctypes.cast(kr, ctypes.c_void_p), 0.3, 0.5, 21, gens, 1, p(pop),
                         p(fit), p(off), p(fo), p(scratch), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    torch.cuda.synchronize()
    for a, b in zip((pop, fit, off, fo), want):
        assert np.array_equal(a.cpu().numpy(), b)
