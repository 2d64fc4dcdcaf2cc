"""Read-out and load kernels: conversions by bits, exact FP16 sums, the conservation reduction over
stored planes with its ring weights, and the stream function's stretches."""
import math

import numpy as np
import pytest

import oracle
from paper_1801_03863_gb300 import lbm, workloads as wl

pytestmark = pytest.mark.gpu

W9 = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)


def _bf16(x):
    """Nearest BF16 (ties to even) of FP64 values, from the value itself."""
    m, e = np.frexp(x)
    q = np.maximum(e - 8, -133)  # weight of the last place (FP32's exponent range)
    return np.ldexp(np.round(np.ldexp(m, e - q)), q)


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
def test_loads_round_to_nearest(storage):
    """At rest f - W rho0 = W (rho - rho0) in one FP64 product, rounded once to the storage type:
    normal, subnormal and vanishing magnitudes, ties, both signs."""
    rng = np.random.default_rng(1)
    n = 4096
    dr = np.ldexp(rng.uniform(0.5, 1.0, n), rng.integers(-50, 0, n)) * rng.choice([-1.0, 1.0], n)
    dr[:64] = np.ldexp(np.arange(64) + 0.5, -30) * 9.0  # ties after the product with 1/9
    dr[64] = 0.0
    rho = 1.0 + dr
    d = W9[:, None] * (rho - 1.0)[None]
    want = {"f32": lambda v: v.astype(np.float32).astype(np.float64),
            "f16": lambda v: v.astype(np.float16).astype(np.float64), "bf16": _bf16}[storage](d)
    with lbm.Lattice("d2q9", [(64, 64)], 0.1, "periodic", compute="f32", storage=storage) as lat:
        lat.init(rho)
        f = lat.populations().reshape(9, n)
        # the same values as full populations: f - W rho0 loses W rho0's rounding, no more
        lat.set_populations(W9[:, None] + want)
        g = lat.populations().reshape(9, n)
    assert np.array_equal(f, W9[:, None] + want)
    assert np.array_equal(f, g)


@pytest.mark.parametrize("bc", ["periodic", "zero_gradient", "cavity"])
@pytest.mark.parametrize("compute,storage", [("f64", "f64"), ("f32", "f32"), ("f32", "f16"), ("f32", "bf16")])
@pytest.mark.parametrize("steps", [0, 3])
@pytest.mark.parametrize("large", [False, True])
def test_totals_and_moments_of_the_populations(bc, compute, storage, steps, large):
    """Totals and moments against the populations read from the same state, in exact sums; deviations
    above 2^-4 and 2^-7 (large) take the integer paths of FP16.  Tolerance: one rounding of each
    population (2^-53) and, for FP32 and BF16 totals, FP32 pairs (2^-46)."""
    dims = [(64, 33), (37, 70), (3, 3), (131, 5), (9, 129)] + ([(1, 1), (2, 3), (5, 1)] if bc != "cavity" else [])
    parts, rng = [], np.random.default_rng(4)
    for nx, ny in dims:
        f = wl.random_populations(9, ny, nx, eps=0.4 if large else 1e-3, rho_spread=0.5 if large else 1e-3,
                                  seed=nx)
        parts.append(f.ravel())
    f0 = np.concatenate(parts)
    nus = [0.05] * len(dims)
    with lbm.Lattice("d2q9", dims, nus, bc, u_lid=0.05, compute=compute, storage=storage,
                     collision="srt") as lat:
        lat.set_populations(f0)
        lat.step(steps)
        f, tot = lat.populations(), lat.conservation()
        rho, ux, uy = lat.moments(allow_unstable=True)
        each = [lat.moments_instance(i, allow_unstable=True) for i in range(len(dims))]
        psi = lat.stream_function(allow_unstable=True)
        psi_each = [lat.stream_function_instance(i, allow_unstable=True) for i in range(len(dims))]
    vx = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
    vy = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
    k = n0 = 0
    for i, (nx, ny) in enumerate(dims):
        n = nx * ny
        g = f[k:k + 9 * n].reshape(9, n)
        tol = 9 * n * 2.0 ** (-46 if storage in ("f32", "bf16") else -52) * np.abs(g).max()
        for c, v in enumerate((np.ones(9), vx, vy)):
            assert abs(tot[i, c] - math.fsum((v[:, None] * g).ravel())) <= tol, (i, c)
        r = g.sum(0)
        e = 40 * 2.0 ** -53
        s = slice(n0, n0 + n)
        assert np.abs(rho[s] - r).max() <= e * r.max()
        assert np.abs(ux[s] - (vx @ g) / r).max() <= e and np.abs(uy[s] - (vy @ g) / r).max() <= e
        for got, want in zip(each[i], (rho, ux, uy)):
            assert np.array_equal(got.ravel(), want[s])
        p = oracle.stream_function(uy[s].reshape(ny, nx))
        assert np.abs(psi[s].reshape(ny, nx) - p).max() <= 4 * nx * 2.0 ** -53 * max(np.abs(uy[s]).max() * nx, 1e-300)
        assert np.array_equal(psi_each[i].ravel(), psi[s])
        k, n0 = k + 9 * n, n0 + n


@pytest.mark.parametrize("storage", ["f64", "f32", "f16"])
@pytest.mark.parametrize("n", [1, 2, 9, 255, 2049])
@pytest.mark.parametrize("bc", ["periodic", "zero_gradient"])
def test_tube_totals(storage, n, bc):
    rng = np.random.default_rng(n)
    rho, u = 1.0 + 0.3 * rng.random(n), 0.1 * (rng.random(n) - 0.5)
    with lbm.Lattice("d1q3", [(n, 1)], 0.05, bc, compute="f64" if storage == "f64" else "f32",
                     storage=storage) as lat:
        lat.init(rho, u)
        lat.step(2)
        f, tot = lat.populations().reshape(3, n), lat.conservation()[0]
    assert abs(tot[0] - math.fsum(f.ravel())) <= 3 * n * 2.0 ** -45
    assert abs(tot[1] - (math.fsum(f[1]) - math.fsum(f[2]))) <= 3 * n * 2.0 ** -45
    assert tot[2] == 0.0


def test_large_instance_splits_alike_alone_and_in_a_batch():
    """An instance large enough for a cluster of CTAs per partial gives the same bits alone and beside a
    larger one (whose cluster is larger)."""
    rng = np.random.default_rng(2)
    a, b = (1100, 1300), (2100, 2100)
    rho = [1.0 + 1e-3 * rng.random(nx * ny) for nx, ny in (a, b)]
    with lbm.Lattice("d2q9", [a], 0.05, "periodic", compute="f32", storage="f32") as lat:
        lat.init(rho[0])
        lat.step(2)
        one = lat.conservation()[0]
    with lbm.Lattice("d2q9", [a, b], 0.05, "periodic", compute="f32", storage="f32") as lat:
        lat.init(np.concatenate(rho))
        lat.step(2)
        two = lat.conservation()
    assert np.array_equal(one, two[0])
    assert abs(two[1, 0] - math.fsum(rho[1])) <= 1e-6 * 2100 * 2100 * 2.0 ** -10


@pytest.mark.parametrize("storage", ["f32", "bf16"])
def test_moments_over_the_whole_exponent_range(storage):
    """Fixed-point sums of values of very different size, of vanishing ones and of none: rho, u against
    exact sums of the stored deviations.  Each sum is within 2^-53 of the largest value (fixed point
    keeps 2^-58 of it), and so is rho's rounding."""
    rng = np.random.default_rng(8)
    nx, ny = 64, 40
    d = np.ldexp(rng.uniform(-1, 1, (9, ny, nx)), rng.integers(-60, -4, (9, ny, nx)))
    d[:, :4] = 0.0
    d[:, 4:8] = np.ldexp(rng.uniform(-1, 1, (9, 4, nx)), -100)
    w = W9[:, None, None]
    with lbm.Lattice("d2q9", [(nx, ny)], 0.1, "periodic", compute="f32", storage=storage) as lat:
        # deviations survive the FP64 populations only down to 2^-53 W: read back what is stored
        lat.set_populations(w + d)
        g = lat.populations().reshape(9, ny, nx) - w
        rho, ux, uy = (v.reshape(ny, nx) for v in lat.moments(allow_unstable=True))
    vx = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
    vy = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
    m, jx, jy = (np.vectorize(lambda i, j: math.fsum(c * g[:, i, j]))(*np.mgrid[:ny, :nx])
                 for c in (np.ones(9), vx, vy))
    tol = 2.0 ** -52 * (1.0 + 9 * np.abs(g).max(0))
    assert np.all(np.abs(rho - (1.0 + m)) <= tol)
    assert np.all(np.abs(ux - jx / (1.0 + m)) <= 2 * tol) and np.all(np.abs(uy - jy / (1.0 + m)) <= 2 * tol)
