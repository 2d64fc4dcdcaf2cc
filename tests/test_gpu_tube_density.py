"""The tube kernel's quick test of a node's stability does not depend on the unit of density."""
import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm

pytestmark = pytest.mark.gpu


def test_densities_take_the_same_time():
    """The populations of rho = 4 at rest lie on both sides of 2, those of rho = 1 below 1: timed in turn,
    the best of 12."""
    import torch
    stream = torch.cuda.Stream()
    lats, best = {}, {}
    for rho in (1.0, 4.0):
        lats[rho] = lbm.Lattice("d1q3", [(4000, 1)] * 1024, 0.02, "zero_gradient", compute="f32",
                                storage="f32", rho0=rho, stream=stream)
        lats[rho].init(np.full(4000 * 1024, rho))
        lats[rho].step(64)
    for _ in range(12):
        for rho, lat in lats.items():
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record(stream)
            lat.step(320)
            b.record(stream)
            b.synchronize()
            best[rho] = min(best.get(rho, float("inf")), a.elapsed_time(b))
    for lat in lats.values():
        lat.close()
    assert best[4.0] <= 1.25 * best[1.0]


@pytest.mark.parametrize("scale", [1e-3, 1.0, 4.0, 1e4, 2.0 ** 70])
def test_counts_do_not_depend_on_the_density_unit(scale):
    """The rule is linear in (f, rho0): scaled by a power of two or not, the same nodes are counted."""
    rng = np.random.default_rng(3)
    n, count = 3000, {}
    rho = 1.0 + 0.3 * (np.arange(n) < n // 2) + 0.05 * rng.random(n)
    ux = 0.6 * rng.uniform(-1, 1, n)
    for s in (1.0, 2.0 ** np.round(np.log2(scale))):
        with lbm.Lattice("d1q3", [(n, 1)], 2e-4, "periodic", compute="f32", storage="f32", rho0=s) as lat:
            lat.init(s * rho, ux)
            lat.step(3)
            count[s] = lat.status()["unstable"]
    assert len(set(count.values())) == 1 and count[1.0] > 0
