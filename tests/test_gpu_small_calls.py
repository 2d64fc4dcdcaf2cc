"""Programs that step in small calls: the region kernel takes a launch only where it pays."""
import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,bc,storage,rule", [(512, 512, "periodic", "f32", "minxent4"),
                                                   (600, 601, "cavity", "f16", "minxent2"),
                                                   (97, 140, "zero_gradient", "bf16", "mrt")])
def test_calls_of_any_length_agree(nx, ny, bc, storage, rule, monkeypatch):
    """Single steps and regions in turn, bit for bit the TMA kernel's steps."""
    f0 = wl.random_populations(9, ny, nx, eps=0.1, seed=nx).ravel()
    got = []
    for shape, calls in (("smems", [26]), (None, [26]), (None, [1] * 26), (None, [2, 3, 4, 5, 1, 11]), (None, [7, 13, 6])):
        if shape:
            monkeypatch.setenv("LBM_SHAPE", shape)
        else:
            monkeypatch.delenv("LBM_SHAPE", raising=False)
        with lbm.Lattice("d2q9", [(nx, ny)], 0.02, bc, u_lid=0.08, compute="f32", storage=storage,
                         collision=rule) as lat:
            lat.set_populations(f0)
            for k in calls:
                lat.step(k)
            got.append((lat.populations(), lat.status()))
    for f, st in got[1:]:
        assert np.array_equal(f, got[0][0]) and st == got[0][1]


def test_short_calls_do_not_pay_for_regions():
    """700 x 700: a region launch takes 20 us for one step and 36 for three, a step of the TMA kernel 11 us;
    six steps take 57 us in one launch."""
    with lbm.Lattice("d2q9", [(700, 700)], 0.02, "periodic", compute="f32", storage="f32") as lat:
        lat.init(np.ones(700 * 700))
        assert lat.launch_shape()["kind"] == "block"
        assert lat.step_launches(0) == {"launches": 0, "of_several_steps": 0}
        assert lat.step_launches(1) == {"launches": 1, "of_several_steps": 0}  # the first collision
        lat.step(1)
        k = lat.launch_shape()["tw"]
        for n in (1, 2):
            assert lat.step_launches(n) == {"launches": n, "of_several_steps": 0}
        assert lat.step_launches(5 * k) == {"launches": 5, "of_several_steps": 5}
        assert lat.step_launches(5 * k + 1) == {"launches": 6, "of_several_steps": 5}

@pytest.mark.parametrize("bc", ["periodic", "zero_gradient"])
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_tube_calls_of_any_length_agree(bc, storage):
    """Single steps and several steps per launch are different kernels: the same bits and counters, a
    nearly inviscid tube's unstable nodes among them."""
    dims = [(n, 1) for n in (1, 2, 3, 7, 64, 511, 513, 800, 4097)]
    f0 = np.concatenate([wl.random_populations(3, 1, nx, eps=0.6, seed=nx).ravel() for nx, _ in dims])
    got = []
    for calls in ([30], [1] * 30, [2, 1, 5, 1, 1, 20], [29, 1]):
        with lbm.Lattice("d1q3", dims, [1e-4] * len(dims), bc, compute="f32", storage=storage) as lat:
            lat.set_populations(f0)
            for k in calls:
                lat.step(k)
            got.append((lat.populations(), lat.status()))
    assert got[0][1]["unstable"] > 0
    for f, st in got[1:]:
        assert np.array_equal(f, got[0][0]) and st == got[0][1]



def test_single_steps_of_tubes_take_their_own_kernel():
    """16 M nodes in FP16, one step: a launch of the tube kernel takes 73 us, the kernel for single steps 50;
    in FP64 the tube kernel is ahead."""
    for storage, several in (("f16", 0), ("f64", 1)):
        with lbm.Lattice("d1q3", [(4000, 1)] * 64, 0.02, "zero_gradient",
                         compute="f64" if storage == "f64" else "f32", storage=storage) as lat:
            lat.init(np.ones(4000 * 64))
            assert lat.step_launches(1) == {"launches": 1, "of_several_steps": 1}
            lat.step(1)
            assert lat.step_launches(1) == {"launches": 1, "of_several_steps": several}
            assert lat.step_launches(2) == {"launches": 1, "of_several_steps": 1}
