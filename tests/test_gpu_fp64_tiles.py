"""The FP64 sweep's choice between 64-node tiles and half tiles: a grid on the wide side of the
rule, with rows that do not start on 16-byte boundaries, a remainder tile and cut links,
steps bit for bit like the same problem through a batch's half tiles."""

import numpy as np
import pytest

from paper_1712_08288_gb300 import binding as B
from paper_1712_08288_gb300 import workloads as W
from gpu_common import gpu_sim, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["couette_1101", "couette_1024", "sphere_131x60x70"])
def test_wide_tiles_equal_half_tiles(kind):
    require_gpu()
    if kind.startswith("couette"):
        w = W.couette_config(int(kind.split("_")[1]))
        lattice = "D2Q9"
    else:
        lattice, shape = "D3Q15", (131, 60, 70)
        x, y, z = W._coords(shape)
        solid = (x - 60.3) ** 2 + (y - 30.2) ** 2 + (z - 35.4) ** 2 <= 15.0 ** 2
        node, d = W.cut_links(lattice, shape, (0, 0), solid)
        rng = np.random.default_rng(1)
        w = dict(lattice=lattice, shape=shape, skew=(0, 0), solid=solid, force=(1e-5, 0.0, 0.0), rho0=1.0,
                 links=dict(node=node, d=d, q=rng.uniform(0.1, 1.0, len(node)), uw=np.zeros((len(node), 3))),
                 S=W.relaxation_rates(lattice, 1.1))
    rho, u = W.random_state(w["shape"], lattice, 1.0, 0.01, 5)
    one, other = gpu_sim(w, "f64"), gpu_sim(w, "f64")
    for sim in (one, other):
        sim.init_equilibrium(rho, u)
    batch = B.Batch([other])
    batch.set_config(0, 0, 1, 32)
    one.step(3)
    batch.step(3)
    fluid = ~np.asarray(w["solid"], bool)
    assert np.array_equal(one.get_populations()[:, fluid], other.get_populations()[:, fluid])
    batch.close()
