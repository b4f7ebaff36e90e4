"""The training kernels at the edges of their tiles (32 rows a tile, one tile
per SM then several, 64 rows a stage of the gradients, six ahead) and on
arrays that are not 16-byte aligned.

Bars: as for the other batch sizes against the oracle fed BF16-rounded operands
(2e-4 forward, 2e-3 backward); aligned and unaligned arrays give the same
bits; the loss of one cluster (up to 2^16 rows) and of two launches within 1e-6
of the FP64 sum (a float32 result)."""
import numpy as np
import pytest

from tests.gpu_helpers import binding
from tests.test_gpu_mlp import KEYS, _flat, _oracle_bf16, _rel, _unflat
from oracle import mlp

pytestmark = pytest.mark.gpu


def _inputs(n):
    rng = np.random.default_rng(n)
    p = _unflat(_flat(mlp.init_params(3)))
    f = lambda *s: rng.normal(size=s).astype(np.float32).astype(np.float64)
    return p, f(n, 64), f(n, 4)


def _step(B, torch, p, X, T, shift):
    """Forward, loss and gradients; every array starts `shift` floats into its allocation."""
    n = len(X)

    def place(a):
        t = torch.zeros(a.size + shift, dtype=torch.float32, device="cuda")[shift:]
        return t.copy_(torch.as_tensor(a.ravel(), dtype=torch.float32))

    dp, dX, dT = place(_flat(p)), place(X), place(T)
    Y, acts, dY, G = (place(np.zeros(k)) for k in (4 * n, 512 * n, 4 * n, _flat(p).size))
    work = place(np.zeros(512 * n))
    loss = torch.empty(1, device="cuda")
    s64 = torch.empty(64, dtype=torch.float64, device="cuda")
    P, S = B._tp, B._cur_stream()
    assert B.lib.mi_mlp_forward(P(dp), P(dX), n, P(Y), P(acts), S) == 0
    assert B.lib.mi_mlp_mse(P(Y), P(dT), n, P(dY), P(loss), P(s64), S) == 0
    assert B.lib.mi_mlp_backward(P(dp), P(dX), P(acts), P(dY), n, P(G), P(work), S) == 0
    torch.cuda.synchronize()
    return [t.cpu().numpy() for t in (Y, acts, dY, G, loss)]


@pytest.mark.parametrize("n", [2, 31, 32, 33, 64, 65, 384, 385, 4863, 4865, 9800])
def test_tile_edges(n):
    B = binding()
    import torch
    p, X, T = _inputs(n)
    Y, acts, dY, G, loss = _step(B, torch, p, X, T, 0)
    Yb, Gb, cache = _oracle_bf16(p, X, T)
    assert _rel(Y.reshape(n, 4), Yb) <= 2e-4
    acts = acts.reshape(2, n, 256)
    assert _rel(acts[0], cache["H1"]) <= 2e-4 and _rel(acts[1], cache["H2"]) <= 2e-4
    G = _unflat(G)
    for k in KEYS:
        assert _rel(G[k], Gb[k]) <= 2e-3, (k, _rel(G[k], Gb[k]))


@pytest.mark.parametrize("n", [1, 33, 300])
def test_unaligned_arrays_give_the_same_bits(n):
    B = binding()
    import torch
    p, X, T = _inputs(n)
    for a, b in zip(_step(B, torch, p, X, T, 0), _step(B, torch, p, X, T, 1)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("n", [1, 65536, 65537])
def test_loss_either_way(n):
    B = binding()
    import torch
    rng = np.random.default_rng(n)
    Y, T = (rng.normal(size=(n, 4)).astype(np.float32) for _ in range(2))
    loss, dY = B.mlp_mse(torch.as_tensor(Y, device="cuda"), torch.as_tensor(T, device="cuda"))
    d = Y.astype(np.float64) - T
    assert abs(float(loss.item()) - (d * d).sum() / n) <= 1e-6 * (d * d).sum() / n
    assert _rel(dY.cpu().numpy(), 2.0 * d / n) <= 1e-6
