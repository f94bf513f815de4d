"""The sweep's link-parallel boundary against the oracle where its bookkeeping can go wrong:
dense and sparse tiles, links on the x-wrap, nodes cut on both sides of a direction, nodes with
every direction cut, rows that do and do not start on 16-byte boundaries, remainders.

Tolerances as for the other one-to-few-step parity runs: FP64 1e-12 of the largest
deviation per entry, FP32 1e-6.
"""

import numpy as np
import pytest

from paper_1712_08288_gb300 import workloads as W
from gpu_common import check_close, deviation, gpu_sim, oracle_sim, require_gpu
from oracle import lattices as OL

pytestmark = pytest.mark.gpu


def _problem(lattice, nx, porosity, skew):
    ny, nz = (9, 1) if lattice == "D2Q9" else (6, 5)
    shape = (nx, ny, nz)
    rng = np.random.default_rng(nx + int(100 * porosity))
    x, y, z = W._coords(shape)
    solid = rng.uniform(size=nx * ny * nz) < porosity
    if porosity < 0.2:                       # a channel: dense rows of links along its walls
        solid |= y == 0
        if lattice != "D2Q9":
            solid |= z == 0
    node, d = W.cut_links(lattice, shape, skew, solid)
    order = rng.permutation(len(node))       # the caller's link order is free
    links = dict(node=node[order], d=d[order], q=rng.uniform(0.05, 1.0, len(node)),
                 uw=0.02 * rng.standard_normal((len(node), 3)))
    if lattice == "D2Q9":
        links["uw"][:, 2] = 0.0
    return dict(lattice=lattice, shape=shape, skew=skew, solid=solid, links=links, force=(1e-5, -2e-5, 0.0),
                S=W.relaxation_rates(lattice, 1.2), rho0=1.0)


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("nx, porosity, skew", [(71, 0.0, (0, 0)), (72, 0.02, (0, 0)), (97, 0.35, (0, 0)), (40, 0.6, (2, 0)),
                                                (33, 0.1, (1, 0)), (1, 0.3, (0, 0)), (3, 0.3, (1, 0)), (130, 0.05, (0, 0))])
def test_link_parallel_boundary_matches_oracle(lattice, precision, nx, porosity, skew):
    require_gpu()
    w = _problem(lattice, nx, porosity, skew)
    scheme = (0.0, 1.0, 0.0, 0.7)
    N = len(w["solid"])
    rho, u = W.random_state(w["shape"], lattice, 1.0, 0.01, 3)
    ref = oracle_sim(w, scheme)
    ref.init_equilibrium(rho, u)
    sim = gpu_sim(w, precision, scheme)
    sim.init_equilibrium(rho, u)
    lat, fluid = OL.BY_NAME[lattice], ~w["solid"]
    for steps in (1, 1, 3):
        ref.step(steps)
        sim.step(steps)
        check_close(deviation(sim.get_populations(), lat)[:, fluid], deviation(ref.f, lat)[:, fluid],
                    1e-12 if precision == "f64" else 1e-6, label="%s nx %d" % (lattice, nx))
    assert N == w["shape"][0] * w["shape"][1] * w["shape"][2]
    sim.close()
