"""The FP64 D3Q19 adjoint where rows e and eps of the adjoint are as large as they get: a target
whose lambda' at one node has the signs of row e (faces against edges), at rates that
relax e and eps differently, on a state that moves.

Tolerance: 1e-10 of the largest gradient entry against the oracle's adjoint, as for
the other oracle comparisons.
"""

import numpy as np
import pytest

from oracle import adjoint as OA
from oracle import lattices as OL
from oracle import lbm as O
from paper_1712_08288_gb300 import workloads as W
from gpu_common import check_close, gpu_sim, require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s_e, s_eps", [(2.0, 0.0), (2.0, 0.3), (0.0, 2.0), (1.8, 1.2)])
def test_adjoint_of_an_energy_mode(s_e, s_eps):
    require_gpu()
    lat, shape = OL.D3Q19, (8, 7, 6)
    N = int(np.prod(shape))
    rng = np.random.default_rng(4)
    solid = np.zeros(N, bool)
    solid[0] = True
    node, d = W.cut_links("D3Q19", shape, (0, 0), solid)
    S = W.relaxation_rates("D3Q19", 1.2)
    S[1:3] = s_e, s_eps
    w = dict(lattice="D3Q19", shape=shape, skew=(0, 0), solid=solid, rho0=1.0, force=(0.0, 0.0, 0.0), S=S,
             links=dict(node=node, d=d, q=rng.uniform(0.2, 1.0, len(node)), uw=0.01 * rng.standard_normal((len(node), 3))))
    u = 0.05 * np.array([1.0, -0.6, 0.4]) + 0.01 * rng.standard_normal((N, 3))
    rho = 1.0 + 1e-3 * rng.standard_normal(N)
    # lambda_i(x + e_i) = 2 (u - u*).e_i: about -1.9 * 1024 on the faces of the centre, 1.9 * 1024 on the edges
    mask, ut = np.zeros(N, bool), np.zeros((N, 3))
    centre = np.array([4, 3, 3])
    for i in range(1, 19):
        e = lat.e[i]
        x, y, z = centre + e
        n = x + shape[0] * (y + shape[1] * z)
        mask[n] = True
        ut[n] = 0.5 * 1.9 * 1024 * e * (1.0 if np.abs(e).sum() == 1 else -0.5)
    o = O.Simulation(lat, shape, S, 1.0, solid, w["links"], force=w["force"])
    o.init_equilibrium(rho, u)
    J0, gs0, gq0, gp0 = OA.adjoint(o, 4, mask, ut)
    g = gpu_sim(w, "f64")
    g.init_equilibrium(rho, u)
    J, gs, gq, gp = g.adjoint(4, mask, ut)
    assert abs(J - J0) <= 1e-12 * abs(J0)
    check_close(gs, gs0, 1e-10, None, "dJ/ds")
    check_close(gq, gq0, 1e-10, None, "dJ/dq")
    check_close(gp, gp0, 1e-10, None, "dJ/dphi")
    g.close()
