"""FP64 read-outs where a node's sums leave the range of FP64 or come close: densities that
overflow, and velocities and momenta next to it at densities that are powers of two.

Expected values follow from the populations: a sum past the largest double is not finite, and
finite sums of a few populations round by 1e-12 at most.
"""

import numpy as np
import pytest

from oracle import lattices as OL
from paper_1712_08288_gb300 import binding as B
from paper_1712_08288_gb300 import workloads as W
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _sim(lattice, rho0=1.0):
    shape = (5, 4, 1) if lattice == "D2Q9" else (5, 4, 3)
    return B.Lbm(lattice, shape, W.relaxation_rates(lattice, 1.0), "f64", rho0), int(np.prod(shape))


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("which", ["all", "three", "opposite"])
def test_overflowing_density_is_not_finite(lattice, which):
    torch = require_gpu()
    lat = OL.BY_NAME[lattice]
    sim, N = _sim(lattice)
    big = 1.5 * 2.0 ** 1023
    f = np.repeat(lat.w[:, None], N, axis=1)
    picked = {"all": slice(0, lat.Q), "three": slice(0, 3), "opposite": [0, 1, lat.opp[1]]}[which]
    f[picked, 7] = big
    sim.set_populations(f)
    rho, u = sim.moments()
    assert not np.isfinite(rho[7])
    assert (np.delete(rho, 7) == 1.0).all() and np.isfinite(np.delete(u, 7, axis=0)).all()
    out = torch.zeros(7, device="cuda", dtype=torch.float64)
    sim.error_norms_noalloc(0, out.data_ptr())
    assert out[6].item() == 1.0
    assert sim.error_norms(check=False)["status"] == -5
    sim.close()


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("exponent", [1018, 1000, 900])
def test_large_finite_sums(lattice, exponent):
    require_gpu()
    lat = OL.BY_NAME[lattice]
    sim, N = _sim(lattice)
    f = np.repeat(lat.w[:, None], N, axis=1)
    f[1, 3] = 2.0 ** exponent
    sim.set_populations(f)
    rho, u = sim.moments()
    assert rho[3] == 2.0 ** exponent and u[3, 0] == lat.e[1, 0] * 2.0 ** exponent
    n = sim.error_norms(check=False)
    assert n["mass"] == 2.0 ** exponent and n["mom"][0] == lat.e[1, 0] * 2.0 ** exponent
    sim.close()


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
def test_small_velocities_at_a_large_density(lattice):
    # rho0 = 2^99: j is a normal number, j / rho0 of the second component is not
    require_gpu()
    sim, N = _sim(lattice, 2.0 ** 99)
    u0 = np.zeros((N, 3))
    u0[:, 0], u0[:, 1] = 2.0 ** -980, 2.0 ** -1030
    sim.init_equilibrium(None, u0)
    _, u = sim.moments()
    assert np.abs(u - u0[:, : u.shape[1]]).max() <= 1e-12 * 2.0 ** -980
    sim.close()


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
def test_momentum_where_the_velocity_leaves_the_range(lattice):
    torch = require_gpu()
    lat = OL.BY_NAME[lattice]
    out = torch.zeros(7, device="cuda", dtype=torch.float64)
    # j = 2^970 at rho0 = 2^-100: the velocity is infinite, the momentum is not
    sim, N = _sim(lattice, 2.0 ** -100)
    f = np.repeat(lat.w[:, None], N, axis=1) * 2.0 ** -100
    f[1, 3] = 2.0 ** 970
    sim.set_populations(f)
    sim.error_norms_noalloc(0, out.data_ptr())
    want = lat.e[1, 0] * 2.0 ** 970
    assert sim.error_norms(check=False)["mom"][0] == want and out[3].item() == want
    sim.close()
    # velocities below the normal numbers at rho0 = 2^99: the momentum is a normal number
    sim, N = _sim(lattice, 2.0 ** 99)
    tiny = 3.3e-317
    sim.init_equilibrium(None, np.repeat([[tiny, 0.0, 0.0]], N, axis=0))
    sim.error_norms_noalloc(0, out.data_ptr())
    want = N * tiny * 2.0 ** 99
    assert abs(sim.error_norms(check=False)["mom"][0] - want) <= 1e-12 * want
    assert abs(out[3].item() - want) <= 1e-12 * want
    sim.close()
