"""The kernel that takes several steps per launch on overlapping regions gives the bits of the other
step kernels: region edges, lattice edges, any split of a run into calls, every rule and storage."""
import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu

DIMS = {"periodic": [(1, 1), (2, 3), (5, 9), (63, 7), (64, 64), (131, 50), (57, 97)],
        "zero_gradient": [(1, 1), (2, 3), (5, 9), (64, 7), (65, 30), (131, 50), (57, 97)],
        "cavity": [(3, 3), (4, 9), (64, 40), (65, 33), (131, 50), (57, 97), (17, 17)]}


def _run(dims, bc, storage, rule, shape, calls, f0, monkeypatch):
    monkeypatch.setenv("LBM_SHAPE", shape)
    with lbm.Lattice("d2q9", dims, [0.02 + 0.01 * i for i in range(len(dims))], bc, u_lid=0.08,
                     compute="f32", storage=storage, collision=rule) as lat:
        lat.set_populations(f0)
        for k in calls:
            lat.step(k)
        return lat.populations(), [lat.status_instance(i) for i in range(len(dims))], lat.launch_shape()


def _state(dims, eps):
    return np.concatenate([wl.random_populations(9, ny, nx, eps=eps, seed=7 * i).ravel()
                           for i, (nx, ny) in enumerate(dims)])


@pytest.mark.parametrize("bc", list(DIMS))
@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("rule", ["minxent4", "minxent2", "srt", "mrt", "trt"])
@pytest.mark.parametrize("K,rows", [(2, 7), (6, 40), (4, 48)])
def test_same_bits_as_the_tma_kernel(bc, storage, rule, K, rows, monkeypatch):
    dims = DIMS[bc]
    f0 = _state(dims, 0.2)
    ref, st, _ = _run(dims, bc, storage, rule, "smems", [13], f0, monkeypatch)
    got, sg, shape = _run(dims, bc, storage, rule, f"block,{K},{rows}", [1, 9, 3], f0, monkeypatch)
    assert shape["kind"] == "block" and shape["tw"] == K and shape["th"] == rows
    assert np.array_equal(got, ref)
    assert sg == st


@pytest.mark.parametrize("storage", ["f32", "f16"])
def test_unstable_nodes_counted_once(storage, monkeypatch):
    """Over-relaxed random states: skipped and unstable node-steps inside the margins that several
    regions recompute."""
    dims = [(140, 90), (60, 30)]
    f0 = _state(dims, 0.9)
    ref, st, _ = _run(dims, "cavity", storage, "minxent4", "smemd", [11], f0, monkeypatch)
    for calls in ([11], [1] * 11):
        got, sg, _ = _run(dims, "cavity", storage, "minxent4", "block,4,30", calls, f0, monkeypatch)
        assert np.array_equal(got, ref, equal_nan=True)
        assert sg == st
    assert sum(s["newton_skipped"] + s["unstable"] for s in st) > 0


def test_uncut_regions_take_many_steps(monkeypatch):
    dims = [(17, 17)] * 5 + [(64, 48), (33, 5)]
    f0 = _state(dims, 0.1)
    ref, st, _ = _run(dims, "cavity", "f32", "minxent4", "smem", [70], f0, monkeypatch)
    got, sg, shape = _run(dims, "cavity", "f32", "minxent4", "block,32,48", [70], f0, monkeypatch)
    assert shape["tw"] == 32 and np.array_equal(got, ref) and sg == st


@pytest.mark.parametrize("shape", ["block,3,40", "block,4,8", "block,32,40", "block,2,0", "block,2,200"])
def test_shapes_that_do_not_fit_are_refused(shape, monkeypatch):
    monkeypatch.setenv("LBM_SHAPE", shape)
    with pytest.raises(lbm.LBMError) as e:
        lbm.Lattice("d2q9", [(200, 200)], 0.02, "periodic", compute="f32", storage="f16")
    assert e.value.code == lbm.LBM_ERR_ARG


def test_same_bits_from_a_small_lattice_choice(monkeypatch):
    """The autotuner's own choice on a small lattice, whichever it is."""
    monkeypatch.delenv("LBM_SHAPE", raising=False)
    f0 = _state([(100, 80)], 0.1)
    ref = None
    for shape in (None, "smem", "block,4,24"):
        if shape:
            monkeypatch.setenv("LBM_SHAPE", shape)
        with lbm.Lattice("d2q9", [(100, 80)], 0.02, "periodic", compute="f32") as lat:
            lat.set_populations(f0)
            lat.step(37)
            f = lat.populations()
        ref = f if ref is None else ref
        assert np.array_equal(f, ref)
