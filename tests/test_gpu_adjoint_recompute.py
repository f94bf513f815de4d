"""The adjoint through checkpoints and recomputation: runs whose interval is given, so that every
segment but the last is recomputed whatever the memory allows (short runs keep every state
at the default interval).

Tolerances as in test_gpu_adjoint.py: 1e-10 of the largest gradient entry against the
oracle's adjoint, FP32 against FP64 1e-3, central differences 1e-4 of the quotient above
its rounding floor.
"""

import numpy as np
import pytest

from oracle import adjoint as OA
from oracle import lattices as OL
from oracle import lbm as O
from paper_1712_08288_gb300 import workloads as W
from gpu_common import check_close, check_fd, gpu_sim, require_gpu
from test_gpu_adjoint import _case, _inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind, steps, every", [("couette", 9, 3), ("sphere", 7, 3), ("pipe", 12, 4), ("pipe", 11, 3)])
@pytest.mark.parametrize("scheme", [(0, 1, 0, 1.0), (0, 1, 1, 0.7)])
def test_recomputed_segments_equal_the_oracle(kind, steps, every, scheme):
    require_gpu()
    w = _case(kind)
    rho, u, mask, ut = _inputs(w, 7)
    lat = OL.BY_NAME[w["lattice"]]
    o = O.Simulation(lat, w["shape"], w["S"], 1.0, w["solid"], w["links"], scheme=scheme, force=w["force"],
                     skew=w.get("skew", (0, 0)))
    o.init_equilibrium(rho, u)
    J0, gs0, gq0, gp0 = OA.adjoint(o, steps, mask, ut)
    g = gpu_sim(w, "f64", scheme=scheme)
    g.init_equilibrium(rho, u)
    J, gs, gq, gp = g.adjoint(steps, mask, ut, checkpoint_every=every)
    assert abs(J - J0) <= 1e-12 * abs(J0)
    check_close(gs, gs0, 1e-10, None, "dJ/ds")
    check_close(gq, gq0, 1e-10, None, "dJ/dq")
    check_close(gp[:, : lat.D], gp0[:, : lat.D], 1e-10, None, "dJ/dphi")
    g.close()


def test_fp32_recomputation_close_to_fp64():
    require_gpu()
    w = _case("pipe")
    rho, u, mask, ut = _inputs(w, 11)
    res = {}
    for prec in ("f64", "f32"):
        g = gpu_sim(w, prec)
        g.init_equilibrium(rho, u)
        res[prec] = g.adjoint(20, mask, ut, checkpoint_every=6)
        g.close()
    scale = max(np.abs(x).max() for x in res["f64"][1:])
    assert abs(res["f32"][0] - res["f64"][0]) <= 1e-3 * res["f64"][0]
    for a, b in zip(res["f32"][1:], res["f64"][1:]):
        assert np.abs(a - b).max() <= 1e-3 * scale


def test_recomputed_gradients_against_central_differences():
    """32^3 box with a sphere, 40 steps in segments of 7."""
    require_gpu()
    w = W.sphere_3d(32, 5.2, (16.37, 15.71, 16.13), s_nu=1.0, force=(1e-5, 0.0, 0.0))
    N, steps, h = 32 ** 3, 40, 1e-4
    x = np.arange(N) % 32
    mask = (x >= 22) & (x < 26)
    rng = np.random.default_rng(5)
    ut = 1e-4 * rng.standard_normal((N, 3))
    viscous = [9, 11, 13, 14, 15]
    q0 = w["links"]["q"].copy()

    def run(s=None, q=None):
        sim = gpu_sim(w, "f64")
        if s is not None:
            sim.set_relaxation(s)
        if q is not None:
            sim.set_link_values(q, None)
        sim.init_equilibrium()
        out = sim.adjoint(steps, mask, ut, checkpoint_every=7)
        sim.close()
        return out

    J, gs, gq, _ = run()
    floor = 1e-12 * abs(J) / h
    S = w["S"]
    up, down = S.copy(), S.copy()
    up[viscous] += h
    down[viscous] -= h
    check_fd((run(s=up)[0] - run(s=down)[0]) / (2 * h), gs[viscous].sum(), 1e-4, floor, "dJ/ds_nu")
    for k in rng.choice(len(q0), 3, replace=False):
        qp, qm = q0.copy(), q0.copy()
        qp[k], qm[k] = min(q0[k] + h, 1.0), q0[k] - h
        check_fd((run(q=qp)[0] - run(q=qm)[0]) / (qp[k] - qm[k]), gq[k], 1e-4, floor, "dJ/dq[%d]" % k)
