"""The collision of 16-bit storages to the bit: one step of a periodic lattice
against the same operations in the same order, each rounded once, in numpy.

A 16-bit value near the middle of two representable ones turns on the last bit of
its FP32 value, so the order and the fused operations are part of the result.
The reference writes them out; a fused multiply-add is formed from the exact
product and the sum rounded to odd in FP64 (53 bits, more than 24 + 2), whose
rounding to FP32 is then the single rounding of the exact value.  No
tolerance."""
import numpy as np
import pytest

from oracle.d3q19 import E
from tests.gpu_helpers import binding

pytestmark = pytest.mark.gpu
F = np.float32
WF = [F(1) / F(3)] + [F(1) / F(18)] * 6 + [F(1) / F(36)] * 12


def fma(a, b, c):
    a, b, c = np.broadcast_arrays(*(np.asarray(v, dtype=np.float64) for v in (a, b, c)))
    p = a * b                       # exact: 24 x 24 bits
    s = p + c
    t = s - p
    e = (p - (s - t)) + (c - t)     # the sum's rounding error, exact
    i = np.ascontiguousarray(s).view(np.int64)
    odd = np.where((e > 0) == (s > 0), i + 1, i - 1)
    return np.where((e != 0) & (i & 1 == 0), odd, i).view(np.float64).astype(F)


def collide(h, omega, force):
    drho = h[0]
    for i in range(1, 19):
        drho = drho + h[i]
    d = [None] + [h[2 * k - 1] - h[2 * k] for k in range(1, 10)]
    j = [(((d[1] + d[4]) + d[5]) + d[6]) + d[7], (((d[2] + d[4]) - d[5]) + d[8]) + d[9],
         (((d[3] + d[6]) - d[7]) + d[8]) - d[9]]
    rho = F(1) + drho
    inv = F(1) / rho
    g = [F(v) for v in force]
    forced = any(g)
    u = [((j[a] + F(0.5) * g[a]) if forced else j[a]) * inv for a in range(3)]
    usq = fma(u[2], u[2], fma(u[0], u[0], u[1] * u[1]))
    ug = fma(u[2], g[2], fma(u[0], g[0], u[1] * g[1]))
    out = []
    for i in range(19):
        eu = np.zeros_like(rho)
        eg = F(0)
        for a in range(3):
            eu = eu + F(E[i][a]) * u[a]
            eg = F(eg + F(E[i][a]) * g[a])
        n = fma(F(-1.5), usq, fma(F(3), eu, (F(4.5) * eu) * eu))
        v = fma(omega, fma(WF[i], fma(rho, n, drho), -h[i]), h[i])
        if forced:
            v = fma(F(F(F(1) - F(0.5) * omega) * WF[i]), fma(F(9) * eu, eg, F(3) * (eg - ug)), v)
        out.append(v)
    return np.stack(out)


@pytest.mark.parametrize("storage", ["f16", "bf16"])
@pytest.mark.parametrize("nx", [64, 38, 35])  # four, two and one node per thread
@pytest.mark.parametrize("tau,force", [(0.8, (0.0, 0.0, 0.0)), (0.8, (0.02, -0.01, 0.004)), (0.53, (0.0, 0.0, 0.0)),
                                       (200.0, (0.0, 0.0, 0.0)), (20.0, (1e-5, 0.0, -2e-5))])
def test_bits(storage, nx, tau, force):
    import torch
    B = binding()
    kind = torch.float16 if storage == "f16" else torch.bfloat16
    rng = np.random.default_rng(nx)
    shape = (18, 34, nx)
    u = 0.08 * (rng.random(3) - 0.5)
    eu = (np.asarray(E, dtype=np.float64) @ u)[:, None, None, None]
    w = np.asarray(WF, dtype=np.float64)[:, None, None, None]
    dev = w * (3.0 * eu + 4.5 * eu * eu + 0.1 * (rng.random((19,) + shape) - 0.5))
    stored = torch.from_numpy(dev.astype(F)).to(kind)
    with B.Simulation(nx, 34, 18, tau=tau, storage=B.STORE_F16_DEV if storage == "f16" else B.STORE_BF16_DEV,
                      periodic=(True, True, True), fluid_body_force=force) as sim:
        for pairs, block in ((0, 64), (1, 64), (3, 32)):
            sim.set_tuning(bulk_block_x=block, bulk_pairs=pairs)
            sim.set_raw_populations(stored.view(torch.int16).numpy().view(np.uint16))
            sim.step(1)
            got = sim.get_raw_populations()
            h = stored.float().numpy()
            h = np.stack([np.roll(h[i], (E[i][2], E[i][1], E[i][0]), (0, 1, 2)) for i in range(19)])
            want = torch.from_numpy(collide(h, F(1.0 / tau), force)).to(kind).view(torch.int16).numpy().view(np.uint16)
            assert np.array_equal(got, want), (pairs, (got != want).sum(), got.size)
