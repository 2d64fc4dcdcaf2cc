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
