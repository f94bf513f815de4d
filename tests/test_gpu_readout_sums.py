"""Density and velocity read-outs against FP64 sums of the same populations.

The read-out kernels sum a node's populations in integers aligned to its largest one;
tiny, huge, mixed and non-finite populations and both time parities are compared with
numpy sums of the populations that lbm_get_populations returns for storage whose
values the host knows exactly (they are set, and rounded to the storage type, here).

Tolerance: FP64 storage Q * 2^-53 of the node's sum of |f_i - w_i rho0| on either side,
that is 2 * 19 * 1.2e-16 < 5e-15 of it; the narrower types' sums are exact in range.
"""

import numpy as np
import pytest

from oracle import lattices as OL
from paper_1712_08288_gb300 import binding as B
from paper_1712_08288_gb300 import workloads as W
from gpu_common import require_gpu

pytestmark = pytest.mark.gpu
TOL = 5e-15


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("precision", ["f64", "f32", "f16"])
@pytest.mark.parametrize("rho0", [1.0, 1.7])
def test_readout_sums_match_fp64(lattice, precision, rho0):
    torch = require_gpu()
    lat = OL.BY_NAME[lattice]
    shape = (35, 3, 1) if lattice == "D2Q9" else (35, 3, 3)
    N = int(np.prod(shape))
    rng = np.random.default_rng(11)
    g = rng.standard_normal((lat.Q, N)) * np.exp(3.0 * rng.standard_normal((lat.Q, N)))
    g[:, 0] = 0.0
    g[1:, 1] = 0.0
    scale = {"f64": 1e-3, "f32": 1e-3, "f16": 1.0}[precision]
    wr = lat.w[:, None] * rho0
    f = wr + scale * g
    # what the context stores: f - w rho0 in one rounding (a fused multiply-add), then the type's
    wide = np.longdouble
    held = (f.astype(wide) - lat.w[:, None].astype(wide) * wide(rho0)).astype(np.float64)
    t = {"f64": np.float64, "f32": np.float32, "f16": np.float16}[precision]
    with np.errstate(over="ignore"):
        held = held.astype(t).astype(np.float64)
    fine = np.isfinite(held).all(0)                   # a few values exceed the FP16 range
    sim = B.Lbm(lattice, shape, W.relaxation_rates(lattice, 1.0), precision, rho0)
    sim.set_force((1e-4, 0.0, 0.0))
    sim.set_populations(f)
    rho, u = sim.moments()
    assert not np.isfinite(rho[~fine]).any()
    with np.errstate(invalid="ignore"):
        size = np.abs(held).sum(0)
        off = np.abs(rho - (rho0 + held.sum(0)))
    assert (off[fine] <= TOL * (size + rho0)[fine]).all()
    held[:, ~fine] = 0.0
    want = (lat.e[:, : lat.D].T.astype(float) @ held).T / rho0 + np.array([5e-5, 0.0, 0.0])[: lat.D]
    assert (np.abs(u - want)[fine] <= TOL * (size / rho0 + 1e-4)[fine, None]).all()
    out = torch.zeros(7, device="cuda", dtype=torch.float64)
    sim.error_norms_noalloc(0, out.data_ptr())
    norms = sim.error_norms(check=False)
    assert out[6].item() == (~fine).sum() and norms["status"] == (0 if fine.all() else -5)
    if fine.all():
        assert abs(out[2].item() - rho.sum()) <= 1e-13 * np.abs(rho).sum()
        assert abs(norms["mass"] - rho.sum()) <= 1e-13 * np.abs(rho).sum()
    # a step later the populations sit in the neighbours' slots; mass and momentum stay
    sim.set_force((0.0, 0.0, 0.0))
    sim.init_equilibrium(None, 1e-2 * np.ones((N, 3)))
    sim.step(1)
    rho, u = sim.moments()
    eps = {"f64": 1e-14, "f32": 1e-6, "f16": 2e-3}[precision]
    assert np.abs(rho - rho0).max() <= eps * rho0 and np.abs(u - 1e-2).max() <= eps
    sim.close()


@pytest.mark.parametrize("precision", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("value", [1e-36, 3e38, float("inf"), float("nan")])
def test_readout_outside_the_integer_range(precision, value):
    require_gpu()
    lat = OL.BY_NAME["D2Q9"]
    sim = B.Lbm("D2Q9", (4, 4, 1), W.relaxation_rates("D2Q9", 1.0), precision, 1.0)
    f = np.repeat(lat.w[:, None], 16, axis=1)
    if value == 1e-36:
        sim.init_equilibrium(None, value * np.ones((16, 3)))
        _, u = sim.moments()
        assert np.abs(u / value - 1.0).max() <= (1e-14 if precision == "f64" else 1e-2)
        return
    f[3, 5] = value
    sim.set_populations(f)
    rho, u = sim.moments()
    want = f.sum(0)
    if np.isfinite(value):
        assert abs(rho[5] / want[5] - 1.0) <= 1e-2 and (np.delete(rho, 5) == 1.0).all()
    else:
        assert not np.isfinite(rho[5]) and not np.isfinite(u[5, 0]) and np.isfinite(np.delete(rho, 5)).all()
    sim.close()
