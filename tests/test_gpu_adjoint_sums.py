"""The link gradients' sums over a long run, with and without checkpoints.

16-bit storage recomputes a segment with the sweep itself, so the states and the adjoint of a
run are the same bit for bit for every checkpoint interval, and the gradients of two intervals
differ only in how the sums over the steps are rounded.

An interval of one step adds every term in FP64.

Tolerance: in a slowly decaying channel the terms of a link keep their sign and size, so n
sequential FP32 additions are off by at most n roundings of 2^-25 of a sum that is on
average half the result: n 2^-26, 3.7e-6 where 245 steps, sqrt(T), are added up in FP32 before FP64 takes them
(2e-7 where the roundings are random).  Over all 60000 steps the same bound is 9e-4.
"""

import numpy as np
import pytest

from paper_1712_08288_gb300 import workloads as W
from gpu_common import gpu_sim, require_gpu

pytestmark = pytest.mark.gpu


def _channel():
    """Plane channel, 60 wide, viscosity 0.004: decays over some 80000 steps."""
    shape = (4, 62, 1)
    x, y, z = W._coords(shape)
    solid = (y == 0) | (y == 61)
    node, d = W.cut_links("D2Q9", shape, (0, 0), solid)
    rng = np.random.default_rng(6)
    uw = np.zeros((len(node), 3))
    return dict(lattice="D2Q9", shape=shape, skew=(0, 0), solid=solid, rho0=1.0, force=(1e-8, 0.0, 0.0),
                S=W.relaxation_rates("D2Q9", 1.95), links=dict(node=node, d=d, q=rng.uniform(0.2, 1.0, len(node)), uw=uw)), y


@pytest.mark.parametrize("precision", ["f16", "bf16"])
def test_link_sums_of_a_long_run_keep_their_digits(precision):
    require_gpu()
    w, y = _channel()
    N, T = len(w["solid"]), 60000
    u = np.zeros((N, 3))
    u[:, 0] = 0.05 * np.sin(np.pi * y / 61.0)
    mask, ut = ~w["solid"], np.full((N, 2), -0.05)
    grads = {}
    for every in (0, 1):
        sim = gpu_sim(w, precision)
        sim.init_equilibrium(None, u)
        grads[every] = sim.adjoint(T, mask, ut, checkpoint_every=every)
        sim.close()
    assert np.array_equal(grads[0][1], grads[1][1])          # dJ/ds: the same states and adjoint
    for k, name in ((2, "dJ/dq"), (3, "dJ/dphi")):
        a, b = grads[0][k], grads[1][k]
        off = np.abs(a - b).max() / np.abs(b).max()
        print("%s %s: %.2e" % (precision, name, off))
        assert off <= 3.7e-6, (name, off)
