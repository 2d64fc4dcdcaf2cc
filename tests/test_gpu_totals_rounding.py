"""Totals that FP64 holds exactly must come out exactly."""
import math

import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", ["periodic", "zero_gradient"])
def test_f32_totals_add_threads_in_f64(bc):
    """Positive multiples of 2^-30 below 2^-12 and a 2^17 in every 64th node: a thread's few nodes fit an
    FP32 pair and every partial sum of the lattice fits 53 bits, a warp's needs more than a pair's 48."""
    n = 64
    rng = np.random.default_rng(2)
    d = np.ldexp(rng.integers(1, 1 << 18, (9, n * n)).astype(np.float64), -30)
    d[rng.integers(0, 9, n), np.arange(n) * n + rng.integers(0, n, n)] = 2.0 ** 17
    with lbm.Lattice("d2q9", [(n, n)], 0.1, bc, compute="f32", storage="f32") as lat:
        lat.init(np.ones(n * n))
        state = lat.save_state()
        state[144:].view(np.float32)[:d.size] = d.ravel()  # header, counters; then planes without padding
        lat.load_state(state)
        mass, jx, jy = lat.conservation().ravel()
    assert mass == n * n + math.fsum(d.ravel())
    assert jx == math.fsum((d[1] - d[3]) + (d[5] - d[7]) + (d[8] - d[6]))
    assert jy == math.fsum((d[2] - d[4]) + (d[5] - d[7]) - (d[8] - d[6]))


def test_f16_totals_of_the_widest_row(monkeypatch):
    """A row of 2^26 nodes, every population FP16's largest: a warp's 2^20 nodes add up to more than 63
    bits in units of 2^-24."""
    import torch
    n = 1 << 26
    if torch.cuda.mem_get_info()[0] < 20 << 30:
        pytest.skip("needs 20 GB")
    monkeypatch.setenv("LBM_NO_AUTOTUNE", "1")
    with lbm.Lattice("d2q9", [(n, 1)], 0.1, "periodic", compute="f32", storage="f16") as lat:
        lat.init_device(torch.ones(n, device="cuda", dtype=torch.float64))
        lat.stream.synchronize()
        at = -lat._mem.data_ptr() % 256  # the state is the first buffer of the library's memory
        lat._mem[at:at + 18 * n].view(torch.float16).fill_(65504.0)
        torch.cuda.synchronize()
        mass, jx, jy = lat.conservation().ravel()
    assert mass == n * (1.0 + 9 * 65504.0)
    assert jx == 0.0 and jy == 0.0
