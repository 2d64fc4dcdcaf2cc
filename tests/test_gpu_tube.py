"""The D1Q3 kernel that takes several steps per launch: any split of a run into calls gives the same
bits as one step per call, at segment edges, tube ends and every storage type."""
import numpy as np
import pytest

import oracle
from paper_1801_03863_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu

# one node, shorter than a lane's chunk, around one segment's useful nodes, several segments, odd
SIZES = [1, 2, 3, 7, 8, 9, 31, 48, 112, 113, 240, 241, 1001, 2305]


def _fields(seed):
    rng = np.random.default_rng(seed)
    n = sum(SIZES)
    return 1.0 + 0.2 * rng.random(n), 0.05 * (rng.random(n) - 0.5)


@pytest.mark.parametrize("bc", ["periodic", "zero_gradient"])
@pytest.mark.parametrize("compute,storage,shape", [
    ("f64", "f64", None), ("f64", "f64", "1,128,1"), ("f64", "f64", "2,128,1"), ("f64", "f64", "4,32,1"),
    ("f32", "f32", None), ("f32", "f32", "2,128,1"), ("f32", "f32", "4,256,1"), ("f32", "f32", "8,64,1"),
    ("f32", "f16", "4,128,1"), ("f32", "f16", "8,128,1"), ("f32", "bf16", None)])
def test_any_split_into_calls(bc, compute, storage, shape, monkeypatch):
    if shape:
        monkeypatch.setenv("LBM_SHAPE", shape)
    dims = [(n, 1) for n in SIZES]
    rho, u = _fields(3)
    got = []
    for calls in ([1] * 75, [75], [50, 1, 7, 17]):
        with lbm.Lattice("d1q3", dims, 0.01, bc, compute=compute, storage=storage) as lat:
            lat.init(rho, u)
            for k in calls:
                lat.step(k)
            got.append((lat.populations(), lat.status()))
    for f, st in got[1:]:
        assert np.array_equal(f, got[0][0])
        assert st == got[0][1] and st["steps"] == 75


@pytest.mark.parametrize("bc", ["periodic", "zero_gradient"])
@pytest.mark.parametrize("n", SIZES)
def test_against_oracle(bc, n):
    rng = np.random.default_rng(n)
    rho, u = 1.0 + 0.2 * rng.random((1, n)), 0.05 * (rng.random((1, n)) - 0.5)
    sim = oracle.Sim(oracle.D1Q3, n, 1, oracle.tau_from_nu(0.01),
                     oracle.BC_PERIODIC if bc == "periodic" else oracle.BC_ZERO_GRADIENT)
    sim.init(rho, u)
    sim.step(60)
    with lbm.Lattice("d1q3", [(n, 1)], 0.01, bc) as lat:
        lat.init(rho, u)
        lat.step(60)
        f = lat.populations().reshape(3, 1, n)
        st = lat.status()
    assert np.abs(f - sim.get_f()).max() <= 1e-12 * np.abs(f).max()
    assert st["unstable"] == sim.counters()["unstable"] == 0


@pytest.mark.parametrize("compute", ["f64", "f32"])
def test_unstable_nodes_counted_once(compute):
    """Negative populations inside the halo of a neighbouring segment: each node-step counts once, as
    with one step per call."""
    n = 700
    rho, u = np.ones((1, n)), np.zeros((1, n))
    u[0, 90:130] = 0.9  # f^eq_- = W (1 - 3 u + 3 u^2) > 0 at first, over-relaxed below 0 later
    rho[0, 100] = 0.01
    got = []
    for calls in ([30], [1] * 30):
        with lbm.Lattice("d1q3", [(n, 1)], 1e-4, "zero_gradient", compute=compute) as lat:
            lat.init(rho, u)
            for k in calls:
                lat.step(k)
            got.append(lat.status())
    assert got[0] == got[1] and got[0]["unstable"] > 0
