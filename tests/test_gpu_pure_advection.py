"""FP64 storage without relaxation (every rate zero): the populations only move, so on a
periodic box of 4 nodes a side every state returns bit for bit after 4 steps."""

import numpy as np
import pytest

from paper_1712_08288_gb300 import binding as B
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("batch", [False, True])
def test_advection_without_relaxation_is_exact(lattice, batch):
    require_gpu()
    shape = (4, 4, 1) if lattice == "D2Q9" else (4, 4, 4)
    Q, D = {"D2Q9": (9, 2), "D3Q15": (15, 3), "D3Q19": (19, 3)}[lattice]
    N = int(np.prod(shape))
    rng = np.random.default_rng(2)
    u = np.zeros((N, 3))
    u[:, :D] = 1e-9 * rng.standard_normal((N, D))          # far below the density's deviations
    sim = B.Lbm(lattice, shape, np.zeros(Q), "f64", 1.0)
    sim.init_equilibrium(1.0 + 0.02 * rng.standard_normal(N), u)
    rho0, u0 = sim.moments()
    many = B.Batch([sim]) if batch else None
    for _ in range(2):
        (many or sim).step(4)
        rho, got = sim.moments()
        assert np.array_equal(rho, rho0) and np.array_equal(got, u0)
    if many:
        many.close()
    sim.close()
