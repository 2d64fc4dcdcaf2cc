"""Variants of the step kernels that only some sizes reach, against another kernel or the oracle."""
import numpy as np
import pytest

import oracle
from paper_1801_03863_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu


def _state(dims, eps):
    return np.concatenate([wl.random_populations(9, ny, nx, eps=eps, seed=7 * i).ravel()
                           for i, (nx, ny) in enumerate(dims)])


def _run(dims, bc, storage, rule, shape, calls, f0, monkeypatch):
    monkeypatch.setenv("LBM_SHAPE", shape)
    with lbm.Lattice("d2q9", dims, 0.02, bc, u_lid=0.08, compute="f32", storage=storage, collision=rule) as lat:
        lat.set_populations(f0)
        for k in calls:
            lat.step(k)
        return lat.populations(), lat.status(), lat.launch_shape()


@pytest.mark.parametrize("bc", ["periodic", "zero_gradient", "cavity"])
@pytest.mark.parametrize("storage,rule", [("f32", "minxent4"), ("f16", "mrt"), ("bf16", "minxent2")])
def test_regions_of_eight_warps(bc, storage, rule, monkeypatch):
    """More than 152 regions whose buffers fit an SM twice: CTAs of 8 warps."""
    dims = [(700, 300), (61, 33)]
    f0 = _state(dims, 0.2)
    ref, st, _ = _run(dims, bc, storage, rule, "smems", [14], f0, monkeypatch)
    for shape in ("block,4,24", "block,2,13"):
        got, sg, sh = _run(dims, bc, storage, rule, shape, [14], f0, monkeypatch)
        assert sh["kind"] == "block" and sh["grid"] > 152
        assert np.array_equal(got, ref) and sg == st


@pytest.mark.parametrize("bc", ["periodic", "zero_gradient", "cavity"])
@pytest.mark.parametrize("storage,rule", [("f16", "minxent4"), ("bf16", "srt")])
@pytest.mark.parametrize("K,rows", [(6, 62), (8, 95), (2, 96)])
def test_tall_regions(bc, storage, rule, K, rows, monkeypatch):
    """16-bit storage: regions of more than 48 rows."""
    dims = [(300, 310), (70, 96), (64, 5), (50, 97)]
    f0 = _state(dims, 0.2)
    ref, st, _ = _run(dims, bc, storage, rule, "smems", [19], f0, monkeypatch)
    got, sg, sh = _run(dims, bc, storage, rule, f"block,{K},{rows}", [19], f0, monkeypatch)
    assert sh["th"] == rows and np.array_equal(got, ref) and sg == st


@pytest.mark.parametrize("bc", ["periodic", "cavity"])
@pytest.mark.parametrize("shape,tile", [("smem", 1792), ("smemw", 2304)])
@pytest.mark.parametrize("storage,rule", [("f16", "minxent4"), ("bf16", "minxent2"), ("bf16", "trt")])
def test_drawn_tiles_of_16_bit_storage(bc, shape, tile, storage, rule, monkeypatch):
    """More tiles than the CTAs' first two, whatever their width: at least nodes / tile of them."""
    dims = [(1400, 1100), (513, 900)]
    f0 = _state(dims, 0.1)
    ref, st, _ = _run(dims, bc, storage, rule, "smemd", [9], f0, monkeypatch)
    got, sg, sh = _run(dims, bc, storage, rule, shape, [4, 5], f0, monkeypatch)
    assert sum(-(-a * b // tile) for a, b in dims) > 2 * sh["grid"]
    assert np.array_equal(got, ref) and sg == st


@pytest.mark.parametrize("bc", ["periodic", "zero_gradient"])
def test_tube_counts_against_the_oracle(bc):
    """Unstable node-steps of a tube cut into many segments, which recompute each other's halos."""
    n, steps = 700, 13
    rho, u = np.ones((1, n)), np.zeros((1, n))
    u[0, 90:130] = 0.6
    u[0, 400:440:3] = -0.5
    sim = oracle.Sim(oracle.D1Q3, n, 1, oracle.tau_from_nu(1e-4),
                     oracle.BC_PERIODIC if bc == "periodic" else oracle.BC_ZERO_GRADIENT)
    sim.init(rho, u)
    sim.step(steps)
    with lbm.Lattice("d1q3", [(n, 1)], 1e-4, bc) as lat:
        lat.init(rho, u)
        lat.step(steps)
        assert lat.step_launches(steps)["launches"] < steps
        st = lat.status()
    assert st["unstable"] == sim.counters()["unstable"] > 0
