"""Stream function of lattices whose rows share a warp."""
import numpy as np
import pytest

import oracle
from paper_1801_03863_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("compute,storage", [("f64", "f64"), ("f32", "f32"), ("f32", "f16")])
@pytest.mark.parametrize("steps", [0, 3])
def test_stream_function_of_narrow_lattices(compute, storage, steps):
    """Against the oracle's rule on the library's own velocities (both add at most 33 terms: 64 roundings
    of the largest sum), and the same bits from a call for one instance."""
    dims = [(1, 5), (2, 71), (3, 9), (4, 1000), (5, 33), (7, 2), (8, 130), (9, 9), (15, 40), (16, 17), (17, 17),
            (31, 31), (32, 64), (33, 20), (64, 3)]
    f0 = np.concatenate([wl.random_populations(9, ny, nx, eps=0.1, seed=nx).ravel() for nx, ny in dims])
    with lbm.Lattice("d2q9", dims, 0.05, "periodic", compute=compute, storage=storage) as lat:
        lat.set_populations(f0)
        lat.step(steps)
        uy = lat.moments()[2]
        psi = lat.stream_function()
        k = 0
        for i, (nx, ny) in enumerate(dims):
            want = oracle.stream_function(np.asarray(uy).ravel()[k:k + nx * ny].reshape(ny, nx))
            got = np.asarray(psi).ravel()[k:k + nx * ny].reshape(ny, nx)
            assert np.abs(got - want).max() <= 64 * 2.0 ** -53 * max(np.abs(want).max(), 1e-3)
            assert np.array_equal(np.asarray(lat.stream_function_instance(i)).reshape(ny, nx), got)
            k += nx * ny
