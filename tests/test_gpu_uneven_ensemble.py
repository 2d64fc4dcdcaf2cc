"""One large lattice beside small ones: blocks of more than 2048 nodes in the kernels around the step."""
import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f16", "f32"])
def test_large_lattice_beside_small_ones(storage):
    """Fields in and out of the ensemble as of each lattice alone."""
    dims = [(5, 7), (4097, 2500), (33, 2), (64, 64)]
    rng = np.random.default_rng(1)
    rho = [1.0 + 1e-3 * rng.random(a * b) for a, b in dims]
    u = [0.01 * rng.random((2, a * b)) for a, b in dims]

    def run(members):
        with lbm.Lattice("d2q9", [dims[i] for i in members], 0.05, "periodic", compute="f32",
                         storage=storage) as lat:
            lat.init(np.concatenate([rho[i] for i in members]), *(np.concatenate([u[i][c] for i in members])
                                                                 for c in range(2)))
            lat.step(2)
            return lat.moments(), lat.conservation().reshape(-1, 3)
    fields, totals = run(range(len(dims)))
    k = 0
    for i, (nx, ny) in enumerate(dims):
        alone, total = run([i])
        for a, b in zip(fields, alone):
            assert np.array_equal(a[k:k + nx * ny], b)
        assert np.array_equal(totals[i], total[0])
        k += nx * ny
