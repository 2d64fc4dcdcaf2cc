"""Rounding of the FP64 MinxEnt rules: one collision of raw deviations against extended precision."""
import numpy as np
import pytest

from paper_1801_03863_gb300 import lbm

pytestmark = pytest.mark.gpu

T = np.array([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
              [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1],
              [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
              [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]])
VX, VY = T[3], T[5]
LD = np.longdouble
W = np.array([LD(4) / 9] + [LD(1) / 9] * 4 + [LD(1) / 36] * 4)


def collide(d, rho0, omega, omega2, free):
    """f^post - W rho0 of deviations d = f - W rho0 in extended precision: the rule of Sec. IV.C-E,
    start point in deviations, Newton step by Gaussian elimination."""
    m = [sum(int(c) * x for c, x in zip(row, d) if c) for row in T]
    rho = rho0 + m[0]
    ux, uy = m[3] / rho, m[5] / rho
    s8, s9 = m[7] / rho - (ux * ux - uy * uy), m[8] / rho - ux * uy
    k = (1 - omega) / 4
    gx = gy = LD(0)
    if free == 2:
        gx, gy = ((omega2 - 1) * (-u * rho - q) / rho for u, q in ((ux, m[4]), (uy, m[6])))
    delta = []
    for a in range(9):
        vu = int(VX[a]) * ux + int(VY[a]) * uy
        delta.append(3 * vu + LD(4.5) * vu * vu - LD(1.5) * (ux * ux + uy * uy)
                     + k / W[a] * (int(T[7][a]) * s8 + int(T[8][a]) * s9)
                     + (int(T[4][a]) * gx + int(T[6][a]) * gy) / (12 * W[a]))
    rows = [1, 2, 4, 6][:free]
    A = [[sum(int(T[i][a] * T[j][a]) / (W[a] * (1 + delta[a])) for a in range(9) if T[i][a] * T[j][a])
          + 0 * rho for j in rows] for i in rows]
    b = [sum(int(T[i][a]) * np.log1p(delta[a]) for a in range(9) if T[i][a]) for i in rows]
    for p in range(free):
        for i in range(p + 1, free):
            c = A[i][p] / A[p][p]
            A[i] = [x - c * y for x, y in zip(A[i], A[p])]
            b[i] = b[i] - c * b[p]
    s = [None] * free
    for p in reversed(range(free)):
        s[p] = (b[p] - sum(A[p][j] * s[j] for j in range(p + 1, free))) / A[p][p]
    return [W[a] * (m[0] + rho * delta[a]) - rho * sum(int(T[i][a]) * x for i, x in zip(rows, s))
            for a in range(9)]


# the error of the plain FP64 evaluation (rows of T, IEEE divisions, log1p) on states drawn like these
PLAIN = {("minxent4", 0.1): 0.826, ("minxent4", 0.01): 0.833, ("minxent2", 0.1): 0.866,
         ("minxent2", 0.01): 0.874}


@pytest.mark.parametrize("rule,u", list(PLAIN))
def test_collision_rounds_no_more_than_the_plain_rule(rule, u):
    """Root mean square error over populations and nodes, in units of 2^-53 of a node's largest
    deviation: no more than the plain evaluation's, with 1.5 % for the sample."""
    count, n, rho0 = 8, 48, 2.7
    nu = np.array([1, 2, 4, 8, 12, 20, 30, 40]) / 256  # tau and both terms of tau2 are exact
    rng = np.random.default_rng(7)
    rho = rho0 * (1 + 0.05 * u * rng.uniform(-1, 1, (count, n * n)))
    ux, uy = u * rng.uniform(-1, 1, (2, count, n * n))
    w = W.astype(np.float64)
    d = np.empty((count, 9, n * n))
    for a in range(9):
        vu = VX[a] * ux + VY[a] * uy
        d[:, a] = w[a] * (rho * (1 + 3 * vu + 4.5 * vu * vu - 1.5 * (ux * ux + uy * uy)) - rho0
                          + rho0 * 0.1 * u * rng.uniform(-1, 1, rho.shape))
    with lbm.Lattice("d2q9", [(n, n)] * count, list(nu), "periodic", collision=rule, rho0=rho0) as lat:
        lat.init(np.full(count * n * n, rho0))
        state = lat.save_state()
        raw = state[128 + 16 * count:].view(np.float64)[:d.size]  # planes of n x n nodes, no padding
        raw[:] = d.ravel()
        lat.load_state(state)
        lat.step(1)
        out = lat.save_state()[128 + 16 * count:].view(np.float64)[:d.size].reshape(d.shape)
    total = 0.0
    for i in range(count):
        tau = 3 * nu[i] + 0.5
        omega, omega2 = 1 / tau, 1 / ((8 * tau - 1) / (2 * tau - 1))  # the rates as the library holds them
        exact = np.array(collide([x.astype(LD) for x in d[i]], LD(rho0), LD(omega), LD(omega2),
                                 4 if rule == "minxent4" else 2))
        err = (out[i] - exact) / np.abs(exact).max(axis=0) * LD(2) ** 53
        total += float((err ** 2).mean()) / count
    assert np.sqrt(total) <= 1.015 * PLAIN[rule, u]
