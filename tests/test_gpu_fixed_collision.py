"""The FP64 sweep's fixed-point collision at the edges of its range.

A node's collision runs in block fixed point when its deviations are below rho0/16 and
not all under 2^-895, and in FP64 otherwise.  Velocities after a few steps on a periodic
box are compared with a deviation-form numpy restatement, for scales on both sides of
each edge, from a uniform start, and with one node far above its neighbours.

Tolerance: both sides round each population a handful of times per step at half an ulp
of the node's largest deviation; over 3 steps and the sum over Q populations this stays
below 3 * Q * 8 * 2^-53 < 6e-14 of the largest velocity.
"""

import numpy as np
import pytest

from oracle import lattices as OL
from paper_1712_08288_gb300 import binding as B
from paper_1712_08288_gb300 import workloads as W
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu
TOL = 6e-14
STEPS = 3


def _reference(lat, shape, s, rho0, force, drho, u):
    """Deviations after STEPS periodic steps, dense M, float64."""
    c, w = lat.e.astype(float), lat.w
    M = lat.M.astype(float)
    K = np.linalg.inv(M) @ np.diag(s) @ M
    push = np.zeros(lat.Q)
    for a, k in enumerate([3, 5, 7][: lat.D]):
        push += np.linalg.inv(M)[:, k] * rho0 * force[a]

    def eq(dr, j):
        cj = c @ j
        return w[:, None] * (dr + 3 * cj + (4.5 * cj * cj - 1.5 * (j * j).sum(0)) / rho0)

    g = eq(drho, rho0 * u.T)
    for _ in range(STEPS):
        gp = g - K @ (g - eq(g.sum(0), c.T @ g)) + push[:, None]
        f = gp.reshape((lat.Q,) + shape[::-1])
        g = np.stack([np.roll(f[i], tuple(lat.e[i][::-1]), axis=(0, 1, 2)) for i in range(lat.Q)]).reshape(lat.Q, -1)
    return (c.T @ g).T / rho0 + 0.5 * np.asarray(force)


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("rho0", [1.0, 3e-3, 41.0])
@pytest.mark.parametrize("scale, force", [(1e-285, 0.0), (1e-250, 0.0), (1e-30, 1e-32), (1e-6, 1e-3), (0.05, 1e-5),
                                          (0.2, 0.0), (0.9, 1e-4), ("peak", 0.0)])
def test_fixed_point_collision_at_the_edges_of_its_range(lattice, rho0, scale, force):
    require_gpu()
    lat = OL.BY_NAME[lattice]
    shape = (37, 5, 1) if lattice == "D2Q9" else (33, 4, 3)
    N = int(np.prod(shape))
    rng = np.random.default_rng(7)
    u = np.zeros((N, 3))
    u[:, : lat.D] = rng.uniform(-1, 1, (N, lat.D)) * (0.02 if scale == "peak" else scale)
    if scale == "peak":
        u *= 1e-9
        u[N // 2] = [0.15, -0.1, 0.1 if lat.D == 3 else 0.0]
    drho = np.zeros(N)
    f = np.array([force, -0.7 * force, 0.3 * force if lat.D == 3 else 0.0])
    s = W.relaxation_rates(lattice, 1.31)
    sim = B.Lbm(lattice, shape, s, "f64", rho0)
    sim.set_force(f)
    sim.init_equilibrium(None, u)
    sim.step(STEPS)
    _, got = sim.moments()
    want = _reference(lat, shape, s, rho0, f, drho, u)[:, : lat.D]
    assert np.abs(got - want).max() <= TOL * np.abs(want).max()
    sim.close()


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
def test_rest_stays_exactly_at_rest(lattice):
    require_gpu()
    sim = B.Lbm(lattice, (33, 3, 1) if lattice == "D2Q9" else (33, 3, 2), W.relaxation_rates(lattice, 1.1), "f64", 1.0)
    sim.step(5)
    rho, u = sim.moments()
    assert (rho == 1.0).all() and (u == 0.0).all()
    sim.close()
