"""Moments of nodes whose populations differ by many orders of magnitude."""
import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "bf16"])
@pytest.mark.parametrize("spread", [20, 34, 36, 45, 70])
def test_small_momentum_beside_a_large_population(storage, spread):
    """Moving populations 2^-spread of the one at rest: the momentum does not hold the latter, and keeps
    the precision of FP64 additions of its own terms (6 roundings, 1 of the reciprocal, 1 of the product)."""
    n = 32
    rng = np.random.default_rng(spread)
    d = np.empty((9, n * n))
    d[0] = rng.uniform(0.5, 1.0, n * n) * rng.choice([-1.0, 1.0], n * n)
    d[1:] = np.ldexp(rng.uniform(-1.0, 1.0, (8, n * n)), -spread)
    d[1:, ::7] = 0.0
    raw = d.astype(np.float32)
    if storage == "bf16":
        raw = (raw.view(np.uint32) & 0xffff0000).view(np.float32)
    d = raw.astype(np.float64)
    with lbm.Lattice("d2q9", [(n, n)], 0.1, "periodic", compute="f32", storage=storage, rho0=2.0) as lat:
        lat.init(np.ones(n * n))
        state = lat.save_state()
        data = raw if storage == "f32" else (raw.view(np.uint32) >> 16).astype(np.uint16)
        state[144:144 + data.nbytes] = np.ascontiguousarray(data).view(np.uint8).ravel()
        lat.load_state(state)
        rho, ux, uy = lat.moments(allow_unstable=True)
    big = d.astype(np.longdouble)
    r = 2.0 + big.sum(axis=0)
    a57, a86 = big[5] - big[7], big[8] - big[6]
    scale = np.abs(d[1:]).sum(axis=0) / r
    assert np.abs(rho - r).max() <= 8 * 2.0 ** -53 * 4
    assert (np.abs(ux - (big[1] - big[3] + a57 + a86) / r) <= 8 * 2.0 ** -53 * scale).all()
    assert (np.abs(uy - (big[2] - big[4] + a57 - a86) / r) <= 8 * 2.0 ** -53 * scale).all()
