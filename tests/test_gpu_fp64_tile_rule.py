"""The FP64 sweep's tile width on both sides of its rule: grids that the rule (restated here)
gives to 64-node tiles and to half tiles, with and without a skewed wrap, with rows that do
and do not start on 16-byte boundaries, step bit for bit like batches of either width."""

import numpy as np
import pytest

from paper_1712_08288_gb300 import binding as B
from paper_1712_08288_gb300 import workloads as W
from gpu_common import gpu_sim, require_gpu

pytestmark = pytest.mark.gpu


def _takes_wide_tiles(w):
    """wide_tiles_f64 (csrc/sweep.cuh) for the geometry."""
    nx, ny, nz = w["shape"]
    fluid = np.zeros((ny * nz, (nx + 63) // 64 * 64), bool)
    fluid[:, :nx] = ~np.asarray(w["solid"], bool).reshape(ny * nz, nx)
    halves = fluid.reshape(ny * nz, -1, 2, 32).any(-1)
    tiles = int(halves.any(-1).sum())
    return tiles >= 3 * 152 * 4 * 4 and 5 * int(halves.sum()) >= 8 * tiles


@pytest.mark.parametrize("lattice, shape, skew, wide", [
    ("D3Q19", (128, 64, 60), (5, 3), True), ("D3Q19", (131, 60, 44), (7, 2), True),
    ("D3Q15", (131, 60, 44), (0, 9), True), ("D3Q19", (128, 64, 60), (0, 0), True),
    ("D2Q9", (1101, 460, 1), (3, 0), True), ("D3Q19", (96, 64, 60), (5, 3), False),
    ("D3Q19", (127, 57, 56), (4, 1), False), ("D2Q9", (1100, 400, 1), (3, 0), False)])
def test_tile_width_does_not_change_the_step(lattice, shape, skew, wide):
    require_gpu()
    x, y, z = W._coords(shape)
    c = [0.47 * n for n in shape]
    solid = (x - c[0]) ** 2 + (y - c[1]) ** 2 + ((z - c[2]) ** 2 if shape[2] > 1 else 0) <= (0.2 * min(shape[:2])) ** 2
    node, d = W.cut_links(lattice, shape, skew, solid)
    rng = np.random.default_rng(1)
    uw = 0.01 * rng.standard_normal((len(node), 3))
    if lattice == "D2Q9":
        uw[:, 2] = 0.0
    w = dict(lattice=lattice, shape=shape, skew=skew, solid=solid, force=(1e-5, 0.0, 0.0), rho0=1.0,
             links=dict(node=node, d=d, q=rng.uniform(0.1, 1.0, len(node)), uw=uw), S=W.relaxation_rates(lattice, 1.1))
    assert _takes_wide_tiles(w) == wide
    rho, u = W.random_state(shape, lattice, 1.0, 0.01, 5)
    one = gpu_sim(w, "f64")
    one.init_equilibrium(rho, u)
    one.step(3)
    fluid = ~np.asarray(solid, bool)
    want = one.get_populations()[:, fluid]
    for width in (64, 32):
        other = gpu_sim(w, "f64")
        other.init_equilibrium(rho, u)
        batch = B.Batch([other])
        batch.set_config(0, 0, 1, width)
        batch.step(3)
        assert np.array_equal(want, other.get_populations()[:, fluid])
        batch.close()
        other.close()
    one.close()
