"""The FP64 kernel with one node per thread: node numbering (fluid nodes first, ring last), entries of
more than one warp, and the table logarithm away from equilibrium."""
import numpy as np
import pytest

import oracle
from paper_1801_03863_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu

RULES = {"minxent4": oracle.MINXENT4, "minxent2": oracle.MINXENT2, "srt": oracle.SRT,
         "mrt": oracle.MRT, "trt": oracle.TRT}
BCS = {"periodic": oracle.BC_PERIODIC, "zero_gradient": oracle.BC_ZERO_GRADIENT,
       "cavity": oracle.BC_CAVITY}


@pytest.mark.parametrize("bc", list(BCS))
@pytest.mark.parametrize("rule", list(RULES))
def test_flat_kernel_agrees_with_chunks(bc, rule, monkeypatch):
    """Same collision code in two kernels: 6 steps of contraction-free differences stay within 6 x 16
    roundings of the largest population."""
    dims = [(3, 3), (33, 7), (5, 34), (301, 61)]
    f0 = np.concatenate([wl.random_populations(9, ny, nx, eps=0.1, seed=i).ravel()
                         for i, (nx, ny) in enumerate(dims)])
    got = []
    for shape in ("1,32,1", "2,16,8"):
        monkeypatch.setenv("LBM_SHAPE", shape)
        with lbm.Lattice("d2q9", dims, [0.02, 0.03, 0.05, 0.01], bc, u_lid=0.08,
                         collision=rule) as lat:
            assert lat.launch_shape()["V"] == int(shape[0])
            lat.set_populations(f0)
            lat.step(6)
            got.append((lat.populations(), lat.status()))
    (a, sa), (b, sb) = got
    assert np.abs(a - b).max() <= 6 * 16 * 2.0 ** -53 * np.abs(b).max()
    assert sa == sb


@pytest.mark.parametrize("bc", list(BCS))
@pytest.mark.parametrize("rule", ["minxent4", "minxent2"])
def test_one_step_far_from_equilibrium(bc, rule):
    """Velocities up to 0.5 a component: p / W from about 0.02 to 5, so logarithms inside and outside the
    table and skipped Newton steps.  The Newton system's condition grows as 1 / min(p / W)^2 <= 1e4 on
    the nodes that take the step: 1e4 x 2^-53 x 10 on the largest population."""
    nx, ny = 61, 47
    rng = np.random.default_rng(5)
    ux, uy = rng.uniform(-0.5, 0.5, (2, ny, nx))
    rho = rng.uniform(0.4, 2.5, (ny, nx))
    with lbm.Lattice("d2q9", [(nx, ny)], 0.3, bc, u_lid=0.08, collision=rule) as lat:
        lat.init(rho, ux, uy)
        f0 = lat.populations().reshape(9, ny, nx)
        lat.step(1)
        f1 = lat.populations().reshape(9, ny, nx)
        st = lat.status()
    sim = oracle.Sim(oracle.D2Q9, nx, ny, oracle.tau_from_nu(0.3), BCS[bc], collision=RULES[rule],
                     u_lid=0.08)
    sim.set_f(f0)
    sim.step(1)
    co = sim.counters()
    assert np.abs(f1 - sim.get_f()).max() <= 1e5 * 2.0 ** -53 * np.abs(f1).max()
    assert 0 < st["newton_skipped"] == co["newton_skipped"]
    assert st["unstable"] == co["unstable"]


def test_thin_cavities_share_out_their_ring():
    """More ring nodes than lanes of the colliding warps, and the smallest fluid regions."""
    dims = [(3, 90), (90, 3), (4, 4), (3, 3), (200, 4)]
    nus, uls = [0.02, 0.03, 0.04, 0.05, 0.02], [0.05, 0.06, 0.07, 0.08, 0.09]
    with lbm.Lattice("d2q9", dims, nus, "cavity", u_lid=uls) as lat:
        lat.init(np.ones(sum(a * b for a, b in dims)))
        lat.step(25)
        f = lat.populations()
    k = 0
    for (nx, ny), nu, ul in zip(dims, nus, uls):
        sim = oracle.Sim(oracle.D2Q9, nx, ny, oracle.tau_from_nu(nu), oracle.BC_CAVITY, u_lid=ul)
        sim.init(np.ones((ny, nx)), np.zeros((ny, nx)), np.zeros((ny, nx)))
        sim.step(25)
        g = f[k:k + 9 * nx * ny].reshape(9, ny, nx)
        assert np.abs(g - sim.get_f()).max() <= 1e-12 * np.abs(g).max()
        k += 9 * nx * ny
