"""The fixed-point arithmetic of FP64 storage (csrc/fixed.cuh, csrc/fixed_adjoint.cuh), compiled
for the host with every signed addition and product checked for overflow, at the
extremes of its stated ranges: entries of the largest size the range admits with the
signs of the lattice's moment rows and of combinations of them, relaxation rates at the
corners of [0, 2], the largest force.

Reference: the same map in extended precision (numpy longdouble, 64 mantissa bits here).
Tolerance: a result rounds to half an ulp of itself and carries the cuts of the products,
each under one unit (1/4 ulp of the largest entry for the transpose, 1/16 for the
collision) times the at most 4 Q |M| terms that use it; results reach 16 times the largest entry.  64
half-ulps of the largest entry cover that; a sum that wraps is off by a whole entry
(2^53 half-ulps).

Accuracy: at the rates that the workloads use, the rms error of the fixed-point form is no
larger than that of the FP64 form of the same code (both without fused multiply-adds here).
"""

import itertools
import shutil
import subprocess

import numpy as np
import pytest

from oracle import lattices as OL
from paper_1712_08288_gb300 import _build
from paper_1712_08288_gb300 import workloads as W

LD = np.longdouble
TOP = 2.0 - 2.0 ** -52          # largest mantissa
TOL = 64.0


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    """run(op, lat, s, rho0, F, *node arrays): (covered, first, second output)."""
    if shutil.which("nvcc") is None:
        pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("fixed") / "fixed_host")
    flags = [f for f in _build.FLAGS if f not in ("-lineinfo", "-O3") and "fPIC" not in f]
    flags = [f for f in flags if f != "-Xcompiler"]
    cmd = [_build.nvcc(), *_build.ARCH, *flags, "-O2", "-Xcompiler",
           "-ffp-contract=off,-fsanitize=signed-integer-overflow,-fsanitize-undefined-trap-on-error",
           __file__.replace("test_fixed_point_host.py", "fixed_host.cu"), "-o", exe]
    built = subprocess.run(cmd, capture_output=True, text=True)
    assert built.returncode == 0, built.stderr

    def run(op, lat, s, rho0, F, *nodes):
        n = nodes[0].shape[1]
        head = np.concatenate([[n, rho0], F, s, np.zeros(19 - lat.Q)])
        data = np.concatenate([head, np.concatenate(nodes, 0).T.ravel()]).astype(np.float64)
        r = subprocess.run([exe, op, lat.name], input=data.tobytes(), stdout=subprocess.PIPE)
        assert r.returncode == 0, "a signed overflow (or bad input) stopped the program: %d" % r.returncode
        out = np.frombuffer(r.stdout).reshape(n, 2 * lat.Q + 1)
        return out[:, 0] == 1.0, out[:, 1:1 + lat.Q].T, out[:, 1 + lat.Q:].T

    run.exe = exe
    return run


def _maps(lat, s, rho0, g):
    """M, its row norms, the relaxed rates, g^eq and e.j of the deviations g, extended."""
    M, e = lat.M.astype(LD), lat.e.astype(LD)
    w = np.array([LD(round(x * 216)) / LD(216) for x in lat.w])
    sk = s.astype(LD)
    sk[[0] + list(lat.j_rows)] = 0
    j = e.T @ g.astype(LD)
    ej = e @ j
    geq = w[:, None] * (g.astype(LD).sum(0) + 3 * ej + (LD(9) / 2 * ej * ej - LD(3) / 2 * (j * j).sum(0)) / LD(rho0))
    return M, (M * M).sum(1), sk, e, w, j, ej, geq


def collision(lat, s, rho0, F, g):
    """g' of the deviations g."""
    M, norm, sk, _, _, _, _, geq = _maps(lat, s, rho0, g)
    r = (sk / norm)[:, None] * (M @ (g - geq))
    for a, k in enumerate(lat.j_rows):
        r[k] -= LD(F[a])
    return g - M.T @ r


def transpose(lat, s, rho0, g, lp):
    """Collision transpose of lambda' at the deviations g, and dJ/ds."""
    M, norm, sk, e, w, j, ej, geq = _maps(lat, s, rho0, g)
    lp = lp.astype(LD)
    mu = (M @ lp) / norm[:, None]
    back = M.T @ (sk[:, None] * mu)
    wk = w[:, None] * back
    t = lp - back + wk.sum(0)
    for a in range(lat.D):
        t = t + e[:, a:a + 1] * (wk * (3 * e[:, a:a + 1] + (9 * ej * e[:, a:a + 1] - 3 * j[a]) / LD(rho0))).sum(0)
    gs = mu * (M @ (geq - g))
    gs[[0] + list(lat.j_rows)] = 0
    return t, gs


def half_ulps(x, g):
    """x in half ulps of each node's largest |g|."""
    largest = np.abs(g).max(0)
    return np.abs(x.astype(LD)) / (2.0 ** np.floor(np.log2(largest)) * 2.0 ** -53)


def sign_patterns(lat, rng, n):
    """Columns of -1, 0, 1: constant on rest, faces, edges or corners; the signs of the
    moment rows; of combinations of rows e and eps; of n random combinations of rows."""
    kind = (lat.e != 0).sum(1)
    kinds = sorted(set(kind))
    cols = [[c[kinds.index(k)] for k in kind] for c in itertools.product((-1, 0, 1), repeat=len(kinds))]
    unit = lat.M / np.sqrt((lat.M ** 2).sum(1))[:, None]
    cols += list(np.sign(unit)) + [np.sign(np.cos(a) * unit[1] + np.sin(a) * unit[2]) for a in np.linspace(0, 6.3, 25)]
    for _ in range(n):
        cols.append(np.sign((rng.standard_normal(lat.Q) * (rng.random(lat.Q) < rng.uniform(0.1, 0.6))) @ unit))
    p = np.array(cols, dtype=float).T
    return p[:, np.abs(p).max(0) > 0]


def corner_rates(lat, rng):
    yield W.relaxation_rates(lat.name, 0.5)
    yield W.relaxation_rates(lat.name, 1.99)
    yield np.full(lat.Q, 2.0)
    for s_e, s_eps in ((2.0, 0.0), (0.0, 2.0), (2.0, 0.5), (1.8, 0.8)):
        s = W.relaxation_rates(lat.name, 1.0)
        s[1:3] = s_e, s_eps
        yield s
    for _ in range(12):
        yield 2.0 * (rng.random(lat.Q) < 0.5)


def largest_in_range(rho0):
    """Largest deviation that the fixed-point form takes: just below rho0 / 16."""
    return TOP * 2.0 ** (np.floor(np.log2(rho0)) - 5)


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("rho0", [1.0, 1.9375, 3e-3])
def test_transpose_at_the_extremes_of_its_range(host, lattice, rho0):
    lat = OL.BY_NAME[lattice]
    rng = np.random.default_rng(5)
    for s in corner_rates(lat, rng):
        lp = TOP * sign_patterns(lat, rng, 300)
        states = np.concatenate([sign_patterns(lat, rng, 100), np.sign(lat.e @ rng.integers(-2, 3, (3, 200)))], 1)
        g = largest_in_range(rho0) * states[:, rng.integers(0, states.shape[1], lp.shape[1])]
        ok, t, gs = host("adjoint", lat, s, rho0, np.zeros(3), g, lp)
        want, _ = transpose(lat, s, rho0, g, lp)
        assert ok.all()
        assert half_ulps(t - want, lp).max() <= TOL


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("rho0", [1.0, 1.9375, 3e-3])
def test_collision_at_the_extremes_of_its_range(host, lattice, rho0):
    lat = OL.BY_NAME[lattice]
    rng = np.random.default_rng(6)
    big = largest_in_range(rho0)
    for force in (0.0, big):
        F = force * np.array([1.0, -1.0, 1.0 if lat.D == 3 else 0.0])
        for s in corner_rates(lat, rng):
            states = np.concatenate([sign_patterns(lat, rng, 200), np.sign(lat.e @ rng.integers(-2, 3, (3, 200)))], 1)
            g = big * states[:, np.abs(states).max(0) > 0]
            ok, got, _ = host("collide", lat, s, rho0, F, g)
            if not (s[[k for k in range(1, lat.Q) if k not in lat.j_rows]] > 0).any():
                assert not ok[np.abs(g).max(0) > 0].any()          # no relaxed row: the FP64 form
                continue
            assert ok.all()
            assert half_ulps(got - collision(lat, s, rho0, F, g), g).max() <= TOL


# velocity, density deviation and non-equilibrium part of a node
STATES = [(0.05, 1e-3, 1e-3), (0.05, 0.0, 1e-5), (1e-3, 1e-6, 1e-5), (0.01, 0.01, 1e-3)]


def near_equilibrium(lat, rng, speed, drho, neq, n=4000):
    w, e = lat.w[:, None], lat.e[:, : lat.D]
    j = speed * rng.uniform(-1, 1, (lat.D, n))
    ej = e @ j
    geq = w * (drho * rng.standard_normal(n) + 3 * ej + 4.5 * ej * ej - 1.5 * (j * j).sum(0))
    return geq + neq * w * rng.standard_normal((lat.Q, n))


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("s_nu", [0.5, 1.0, 1.9])
def test_collision_error_is_below_that_of_fp64(host, lattice, s_nu):
    lat = OL.BY_NAME[lattice]
    rng = np.random.default_rng(7)
    s, F = W.relaxation_rates(lattice, s_nu), np.array([1e-6, -2e-6, 0.0])
    for state in STATES:
        g = near_equilibrium(lat, rng, *state)
        ok, fixed, plain = host("collide", lat, s, 1.0, F, g)
        want = collision(lat, s, 1.0, F, g)
        rms = [float(np.sqrt((half_ulps(x - want, g) ** 2).mean())) for x in (fixed, plain)]
        print("%s s_nu %g state %s: rms %.2f fixed point, %.2f FP64 (half ulps)" % (lattice, s_nu, state, *rms))
        assert ok.all() and rms[0] <= rms[1]


@pytest.mark.parametrize("lattice", ["D2Q9", "D3Q15", "D3Q19"])
@pytest.mark.parametrize("s_nu", [0.5, 1.0, 1.9])
@pytest.mark.parametrize("field", ["random", "smooth", "density"])
def test_transpose_error_is_below_that_of_fp64(host, lattice, s_nu, field):
    # smooth fields, whose moments other than rho and j are small, are what an adjoint
    # settles to; dJ/ds is made of just those small moments
    lat = OL.BY_NAME[lattice]
    rng = np.random.default_rng(8)
    s = W.relaxation_rates(lattice, s_nu)
    for state in STATES:
        g = near_equilibrium(lat, rng, *state)
        n = g.shape[1]
        lp = rng.standard_normal((lat.Q, n))
        if field == "smooth":
            lp = lat.e @ rng.standard_normal((3, n)) + 1e-3 * lp
        elif field == "density":
            lp = rng.standard_normal(n) + 0.1 * (lat.e @ rng.standard_normal((3, n))) + 1e-3 * lp
        want, want_s = transpose(lat, s, 1.0, g, lp)
        size = np.abs(want_s).max(0)
        rms = []
        for op in ("adjoint", "adjoint_fp64"):
            ok, t, gs = host(op, lat, s, 1.0, np.zeros(3), g, lp)
            assert ok.all()
            rms += [float(np.sqrt((half_ulps(t - want, lp) ** 2).mean())), float(np.sqrt((((gs - want_s) / size) ** 2).mean()))]
        print("%s s_nu %g %s, state %s: lambda %.2f fixed point, %.2f FP64 (half ulps); dJ/ds %.2e, %.2e"
              % (lattice, s_nu, field, state, rms[0], rms[2], rms[1], rms[3]))
        assert rms[0] <= rms[2] and rms[1] <= rms[3]


def test_widening_by_bits_is_the_conversion(host):
    rng = np.random.default_rng(3)
    edges = [0, 1, 2, 0x7fffff, 0x800000, 0x800001, 0x3f800000, 0x7f7fffff, 0x7f800000, 0x7f800001, 0x7fc00000, 0x7fffffff]
    bits = np.concatenate([np.array(edges, np.uint32), rng.integers(0, 1 << 31, 200000).astype(np.uint32),
                           rng.integers(0, 1 << 23, 20000).astype(np.uint32)])
    v = np.concatenate([bits, bits | np.uint32(1 << 31)]).view(np.float32)
    r = subprocess.run([host.exe, "widen", "any"], input=v.tobytes(), stdout=subprocess.PIPE)
    with np.errstate(invalid="ignore"):              # signalling NaN
        got, want = np.frombuffer(r.stdout), v.astype(np.float64)
    nan = np.isnan(want)
    assert r.returncode == 0 and np.isnan(got[nan]).all()
    assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))
