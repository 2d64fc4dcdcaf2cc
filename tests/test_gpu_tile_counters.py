"""The counters that tiles are drawn from start at zero wherever a state is set afresh."""
import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm

pytestmark = pytest.mark.gpu

DIMS = [(1000, 900), (513, 700)]  # more than two tiles per CTA


@pytest.mark.parametrize("fresh", ["init", "init_instance", "set_populations", "load_state"])
def test_left_over_draws_are_cleared(fresh, monkeypatch):
    """A draw that a timed-out launch left behind would make the next one skip tiles."""
    import torch
    monkeypatch.setenv("LBM_SHAPE", "smem")
    n = sum(a * b for a, b in DIMS)
    rho = 1.0 + 1e-3 * np.random.default_rng(1).random(n)
    got = []
    for left in (0, 3):
        with lbm.Lattice("d2q9", DIMS, 0.02, "cavity", u_lid=0.05, compute="f32", storage="f32") as lat:
            lat.init(rho)
            state, f = lat.save_state(), lat.populations()
            # the error block is the last 256 bytes of the library's memory, the counters its words 8 and 9
            at = -lat._mem.data_ptr() % 256 + int(lat.opts.device_mem_bytes) - 256 + 32
            lat._mem[at:at + 4].view(torch.int32).fill_(left)
            torch.cuda.synchronize()
            if fresh == "init":
                lat.init(rho)
            elif fresh == "load_state":
                lat.load_state(state)
            elif fresh == "set_populations":
                lat.set_populations(f)
            else:
                k = 0
                for i, (nx, ny) in enumerate(DIMS):
                    lat.init_instance(i, rho[k:k + nx * ny])
                    k += nx * ny
            lat.step(4)
            got.append(lat.populations())
    assert np.array_equal(got[0], got[1])
