"""The FP64 adjoint's fixed-point collision transpose at the edges of its ranges.

Tolerances: against the oracle's adjoint 1e-10 of the largest gradient entry of its kind, as for
the other oracle comparisons; for the linearity in the adjoint's magnitude 1e-12 (two
runs of the same arithmetic whose roundings differ only in the exponent's alignment).
"""

import numpy as np
import pytest

from oracle import adjoint as OA
from oracle import lattices as OL
from oracle import lbm as O
from paper_1712_08288_gb300 import workloads as W
from gpu_common import check_close, gpu_sim, require_gpu

pytestmark = pytest.mark.gpu


def _box(lattice):
    rng = np.random.default_rng(8)
    shape = (7, 6, 1) if lattice == "D2Q9" else (6, 5, 4)
    skew = (2, 0)
    solid = rng.uniform(size=int(np.prod(shape))) < 0.15
    node, d = W.cut_links(lattice, shape, skew, solid)
    uw = 0.02 * rng.standard_normal((len(node), 3))
    if lattice == "D2Q9":
        uw[:, 2] = 0.0
    return dict(lattice=lattice, shape=shape, skew=skew, solid=solid, rho0=1.0, force=(1e-4, -5e-5, 0.0),
                links=dict(node=node, d=d, q=rng.uniform(0.1, 1.0, len(node)), uw=uw), S=W.relaxation_rates(lattice, 1.7))


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("speed", [1e-9, 0.03, 0.25])     # the last: some nodes beyond rho0/16
def test_adjoint_inside_and_outside_the_state_range(lattice, speed):
    require_gpu()
    w = _box(lattice)
    lat = OL.BY_NAME[lattice]
    N = len(w["solid"])
    rng = np.random.default_rng(9)
    u = np.zeros((N, 3))
    u[:, : lat.D] = speed * rng.uniform(-1, 1, (N, lat.D))
    rho = 1.0 + 0.2 * speed * rng.standard_normal(N)
    mask, ut = rng.random(N) < 0.6, 0.05 * rng.standard_normal((N, lat.D))
    scheme = (0, 1, 0, 0.8)
    o = O.Simulation(lat, w["shape"], w["S"], 1.0, w["solid"], w["links"], scheme=scheme, force=w["force"], skew=w["skew"])
    o.init_equilibrium(rho, u)
    J0, gs0, gq0, gp0 = OA.adjoint(o, 5, mask, ut)
    g = gpu_sim(w, "f64", scheme=scheme)
    g.init_equilibrium(rho, u)
    J, gs, gq, gp = g.adjoint(5, mask, ut)
    assert abs(J - J0) <= 1e-12 * abs(J0)
    check_close(gs, gs0, 1e-10, None, "dJ/ds")
    check_close(gq, gq0, 1e-10, None, "dJ/dq")
    check_close(gp[:, : lat.D], gp0[:, : lat.D], 1e-10, None, "dJ/dphi")
    # the kept states serve a second backward pass and give the same gradients
    again = g.adjoint_backward()
    for a, b in zip(again, (gs, gq, gp)):
        assert np.array_equal(a, b)
    g.close()


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("scale", [1e-285, 1e-200, 1e-30, 1e100])
def test_adjoint_is_linear_in_its_magnitude(lattice, scale):
    # at rest without force or moving walls the state is exactly zero, so the adjoint is
    # the only thing that carries the target's scale
    require_gpu()
    w = dict(_box(lattice), force=(0.0, 0.0, 0.0))
    w["links"]["uw"][:] = 0.0
    lat = OL.BY_NAME[lattice]
    N = len(w["solid"])
    rng = np.random.default_rng(3)
    mask, ut = np.ones(N, bool), rng.standard_normal((N, lat.D))

    def phi_gradient(c):
        g = gpu_sim(w, "f64")
        g.init_equilibrium()
        out = g.adjoint(6, mask, c * ut)[3]
        g.close()
        return out

    check_close(phi_gradient(scale) / scale, phi_gradient(1.0), 1e-12, None, "dJ/dphi at %g" % scale)
