"""Tiles drawn from a counter on two-stage rings: the same bits as the fixed deal, launch after launch
(the counter is back at zero after every one), and a lost drawn tile times out like any other."""
import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu

# more than two tiles per CTA of the 8- and 10-warp geometries (304 CTAs)
DIMS = [(1000, 900), (513, 700)]


def _state():
    return np.concatenate([wl.random_populations(9, ny, nx, eps=0.1, seed=i).ravel()
                           for i, (nx, ny) in enumerate(DIMS)])


@pytest.mark.parametrize("bc", ["periodic", "cavity", "zero_gradient"])
@pytest.mark.parametrize("storage,rule", [("f32", "minxent4"), ("f32", "mrt"), ("f16", "srt"), ("bf16", "minxent2")])
def test_drawn_and_dealt_tiles_agree(bc, storage, rule, monkeypatch):
    f0, got = _state(), []
    for shape, calls in (("smemd", [40]), ("smem", [40]), ("smem", [1, 2, 5, 32]), ("smemw", [7, 33])):
        monkeypatch.setenv("LBM_SHAPE", shape)
        with lbm.Lattice("d2q9", DIMS, [0.02, 0.05], bc, u_lid=0.08, compute="f32", storage=storage,
                         collision=rule) as lat:
            lat.set_populations(f0)
            for k in calls:
                lat.step(k)
            got.append((lat.populations(), lat.status()))
    for f, st in got[1:]:
        assert np.array_equal(f, got[0][0]) and st == got[0][1]


@pytest.mark.parametrize("shape", ["smem", "smemw"])
def test_lost_drawn_tile_times_out(shape, monkeypatch):
    monkeypatch.setenv("LBM_SHAPE", shape)
    monkeypatch.setenv("LBM_SPIN_LIMIT", "65536")
    monkeypatch.setenv("LBM_TEST_LOST_TILE", "640")  # 2 x 304 tiles are dealt
    n = sum(a * b for a, b in DIMS)
    with lbm.Lattice("d2q9", DIMS, 0.02, "cavity", u_lid=0.05, compute="f32", storage="f32") as lat:
        lat.init(np.ones(n))
        lat.step(3)
        lat.stream.synchronize()
        with pytest.raises(lbm.LBMError) as e:
            lat.status()
        assert e.value.code == lbm.LBM_ERR_TIMEOUT
