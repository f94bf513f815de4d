"""The work that a user of this library has it do, as cases that can be timed.

A case is a geometry, a lattice, a storage precision and a number of time steps; one
pass of a case is what a program calls between two looks at the flow: ``step(n)`` and
the read-out of density and velocity, a checkpointed adjoint, or a whole job from host
fields to host fields.  The geometries are those of the library's configurations:
circular Couette flow between cylinders (D2Q9), a tilted periodic pipe with a skewed
x-wrap, and a sphere in a periodic box with ragged extents (D3Q19, D3Q15).

Read-outs of 32-bit and 16-bit storage are kept in the storage's own type, as a program
that chose that storage keeps its snapshots (the density as its deviation from rho0,
which is what such a type can hold).

``exact`` runs the same steps in 64 bits with plain torch operations: a dense collision
matrix, a gather per direction and the boundary formula of the scheme link by link.
"""

import math
import random

import numpy as np
import torch

from paper_1712_08288_gb300 import binding as B

DEV = "cuda"
RHO0 = 1.0
Q_OF = {"D2Q9": 9, "D3Q19": 19, "D3Q15": 15}
BYTES_OF = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}
TYPE_OF = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


# ---------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------

def _case(name, kind, lattice, precision, nx, ny, nz, steps, c1=1.0, c2=0.0, b=1.0, s_nu=1.0, members=0):
    return dict(name=name, kind=kind, lattice=lattice, precision=precision, nx=nx, ny=ny, nz=nz,
                steps=steps, c1=c1, c2=c2, b=b, s_nu=s_nu, members=members)


def listed():
    return [
        # the 64^2 circular Couette configuration in FP64: a problem of a few thousand
        # nodes stepped thousands of times, where the cost of a step is its latency
        _case("couette_64_f64", "couette", "D2Q9", "f64", 64, 64, 1, 200),
        # one grid of a refinement study in FP64; an odd size, so no row is aligned
        _case("couette_511_f64", "couette", "D2Q9", "f64", 511, 511, 1, 60),
        # the refinement study's largest grid in FP32 storage
        _case("couette_2048_f32", "couette", "D2Q9", "f32", 2048, 2048, 1, 40),
        # the smallest pipe of the convergence study
        _case("pipe_64_f32", "pipe", "D3Q19", "f32", 64, 64, 64, 100),
        # the headline workload: the L = 256 tilted pipe in FP32 storage
        _case("pipe_256_f32", "pipe", "D3Q19", "f32", 256, 256, 256, 40),
        # the same flow in FP64, the reference of the accuracy study
        _case("pipe_128_f64", "pipe", "D3Q19", "f64", 128, 128, 128, 20),
        # 16-bit storage, for throughput at reduced accuracy
        _case("pipe_192_bf16", "pipe", "D3Q19", "bf16", 192, 192, 192, 40),
        # the paper's own 3D lattice, around an obstacle in a box with ragged extents
        _case("sphere_131_d3q15_f32", "sphere", "D3Q15", "f32", 131, 97, 113, 50, c1=1.5),
        # an ensemble of uneven Couette instances advanced together
        _case("ensemble_32_f32", "ensemble", "D2Q9", "f32", 48, 768, 1, 40, members=32),
        # the gradient of a velocity mismatch: forward with checkpoints, then backward
        _case("adjoint_sphere_64_f32", "adjoint", "D3Q19", "f32", 64, 64, 64, 144),
        # the same in FP64 on a small 2D flow, as in verification and parameter fits
        _case("adjoint_couette_96_f64", "adjoint", "D2Q9", "f64", 96, 96, 1, 100),
        # a whole job: fields from the host, steps with the error norms watched every
        # few steps, fields back to the host
        _case("job_pipe_128_f32", "job", "D3Q19", "f32", 128, 128, 128, 120),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    c1, c2, b = rng.choice([(1.0, 0.0, 1.0), (1.5, 0.0, 1.0), (1.0, 1.0, 1.0), (0.0, 1.0, 1.0), (1.0, 0.0, 0.6)])
    s_nu = round(rng.uniform(0.6, 1.8), 3)
    kind = rng.choice(["couette", "couette", "pipe", "pipe", "sphere", "sphere", "ensemble", "adjoint", "job"])
    opt = dict(c1=c1, c2=c2, b=b, s_nu=s_nu)
    if kind == "couette":
        n = _log_int(rng, 48, 2048)
        prec = rng.choice(["f64", "f32", "f32", "bf16", "f16"])
        c = _case("", kind, "D2Q9", prec, n, n, 1, rng.randint(20, 40) if n > 600 else rng.randint(40, 200), **opt)
    elif kind == "pipe":
        L = 16 * _log_int(rng, 3, 15)
        prec = rng.choice(["f64", "f32", "f32", "bf16", "f16"] if L <= 160 else ["f32", "f32", "bf16", "f16"])
        c = _case("", kind, rng.choice(["D3Q19", "D3Q19", "D3Q15"]), prec, L, L, L, rng.randint(10, 40), **opt)
    elif kind == "sphere":
        e = [_log_int(rng, 24, 180) for _ in range(3)]
        prec = rng.choice(["f64", "f32", "f32", "bf16", "f16"])
        c = _case("", kind, rng.choice(["D3Q19", "D3Q15"]), prec, *e, rng.randint(10, 40), **opt)
    elif kind == "ensemble":
        c = _case("", kind, "D2Q9", rng.choice(["f32", "f32", "f64", "bf16"]), rng.randint(33, 64),
                  rng.randint(200, 600), 1, rng.randint(10, 30), members=rng.randint(4, 28), **opt)
    elif kind == "adjoint":
        if rng.random() < 0.5:
            n = _log_int(rng, 40, 200)
            c = _case("", kind, "D2Q9", rng.choice(["f64", "f32"]), n, n, 1, rng.randint(40, 120), **opt)
        else:
            n = _log_int(rng, 20, 56)
            c = _case("", kind, rng.choice(["D3Q19", "D3Q15"]), rng.choice(["f64", "f32", "f32"]), n, n + rng.randint(0, 7),
                      n + rng.randint(0, 7), rng.randint(30, 100), **opt)
    else:
        L = 16 * _log_int(rng, 3, 8)
        c = _case("", kind, "D3Q19", rng.choice(["f64", "f32", "f32"]), L, L, L, 10 * rng.randint(3, 10), **opt)
    del c["name"]
    return c


# ---------------------------------------------------------------------------------
# inputs: solid nodes, cut links, fields (plain torch on the GPU)
# ---------------------------------------------------------------------------------

E_OF = {
    "D2Q9": [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)],
    "D3Q19": [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
              (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)],
    "D3Q15": [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 1), (-1, 1, 1), (1, -1, 1), (-1, -1, 1), (1, 1, -1), (-1, 1, -1), (1, -1, -1), (-1, -1, -1)],
}


def _weights(lattice):
    by = {"D2Q9": (4 / 9, 1 / 9, 1 / 36), "D3Q19": (1 / 3, 1 / 18, 1 / 36), "D3Q15": (2 / 9, 1 / 9, 1 / 72)}[lattice]
    return [by[min(sum(abs(v) for v in e), 2)] for e in E_OF[lattice]]


def _rates(lattice, s_nu):
    return {"D2Q9": [1, 1.8, 1.2, 1, 0.5, 1, 0.5, s_nu, s_nu],
            "D3Q19": [1, 1.8, 1.2, 1, 0.5, 1, 0.5, 1, 0.5, s_nu, 1.2, s_nu, 1.2, s_nu, s_nu, s_nu, 1.5, 1.5, 1.5],
            "D3Q15": [1, 1.8, 1.2, 1, 0.5, 1, 0.5, 1, 0.5, s_nu, s_nu, s_nu, s_nu, s_nu, 1.5]}[lattice]


class _Grid:
    """Node coordinates of a periodic box whose x-wrap is skewed by (sy, sz)."""

    def __init__(self, nx, ny, nz, skew):
        self.shape, self.skew = (nx, ny, nz), skew
        self.x = torch.arange(nx, device=DEV)
        self.y = torch.arange(ny, device=DEV)
        self.z = torch.arange(nz, device=DEV)

    def coords(self):
        z, y, x = torch.meshgrid(self.z, self.y, self.x, indexing="ij")
        return x.reshape(-1), y.reshape(-1), z.reshape(-1)

    def neighbour(self, e):
        """Index of the node at x + e, for every node."""
        nx, ny, nz = self.shape
        x = self.x + e[0]
        k = torch.div(x, nx, rounding_mode="floor")
        x = x - k * nx
        y = (self.y[:, None] + e[1] - k[None, :] * self.skew[0]) % ny
        z = (self.z[:, None] + e[2] - k[None, :] * self.skew[1]) % nz
        return (x[None, None, :] + nx * (y[None, :, :] + ny * z[:, None, :])).reshape(-1)


def _first_root(a, b, c):
    s = torch.sqrt(torch.clamp(b * b - 4 * a * c, min=0.0))
    t1, t2 = (-b - s) / (2 * a), (-b + s) / (2 * a)
    return torch.clamp(torch.where(t1 > 0, t1, t2), 1e-12, 1.0)


def _links(lattice, grid, solid, wall_quadratic):
    """Cut links in node order: node, direction and wall fraction.  wall_quadratic(node,
    e) gives the coefficients of the quadratic in q whose first root is on the wall."""
    nodes, dirs, qs = [], [], []
    for d, e in enumerate(E_OF[lattice]):
        if d == 0:
            continue
        at = torch.nonzero(~solid & solid[grid.neighbour(e)]).reshape(-1)
        nodes.append(at)
        dirs.append(torch.full_like(at, d))
        qs.append(_first_root(*wall_quadratic(at, e)))
    node, d, q = torch.cat(nodes), torch.cat(dirs), torch.cat(qs)
    order = torch.argsort(node * 32 + d)
    return node[order], d[order], q[order]


def _couette(lattice, n, centre, R1, R2, U1):
    grid = _Grid(n, n, 1, (0, 0))
    x, y, _ = grid.coords()
    px, py = x.double() - centre[0], y.double() - centre[1]
    r = torch.hypot(px, py)
    solid = ~((r > R1) & (r < R2))

    def wall(at, e):
        wx, wy = px[at], py[at]
        R = torch.where(torch.hypot(wx + e[0], wy + e[1]) <= R1, R1, R2)
        return (torch.full_like(wx, e[0] ** 2 + e[1] ** 2), 2 * (e[0] * wx + e[1] * wy), wx * wx + wy * wy - R * R)

    node, d, q = _links(lattice, grid, solid, wall)
    e = torch.tensor(E_OF[lattice], device=DEV, dtype=torch.float64)[d]
    xb, yb = px[node] + q * e[:, 0], py[node] + q * e[:, 1]
    turns = torch.hypot(xb, yb) < 0.5 * (R1 + R2)
    uw = torch.zeros(len(node), 3, device=DEV, dtype=torch.float64)
    uw[:, 0] = torch.where(turns, -U1 * yb / R1, 0.0)
    uw[:, 1] = torch.where(turns, U1 * xb / R1, 0.0)
    ut = U1 * R1 * (R2 * R2 / r.clamp(min=R1) - r) / (R2 * R2 - R1 * R1)
    u = torch.stack([-ut * py / r.clamp(min=1.0), ut * px / r.clamp(min=1.0)], 1)
    u[solid] = 0.0
    return dict(grid=grid, solid=solid, node=node, d=d, q=q, uw=uw, u=u, force=(0.0, 0.0, 0.0))


def _pipe(lattice, L, s_nu):
    skew = (L // 4, 3 * L // 16)
    grid = _Grid(L, L, L, skew)
    a = torch.tensor([16.0, 4.0, 3.0], device=DEV, dtype=torch.float64)
    a = a / a.norm()
    R = 0.4 * L
    x, y, z = grid.coords()
    p = torch.stack([x, y, z], 1).double() - torch.tensor([L / 2, L / 2 + 0.37, L / 2 + 0.21], device=DEV, dtype=torch.float64)
    best = near = None
    for my in (-1, 0, 1):
        for mz in (-1, 0, 1):
            v = p - torch.tensor([0.0, my * L, mz * L], device=DEV, dtype=torch.float64)
            v -= (v @ a)[:, None] * a
            d2 = (v * v).sum(1)
            if best is None:
                best, near = d2, v
            else:
                closer = d2 < best
                best = torch.where(closer, d2, best)
                near = torch.where(closer[:, None], v, near)
            del v, d2
    solid = ~(best < R * R)

    def wall(at, e):
        e = torch.tensor(e, device=DEV, dtype=torch.float64)
        e = e - (e @ a) * a
        w = near[at]
        return (e @ e).expand(len(at)), 2 * (w @ e), (w * w).sum(1) - R * R

    node, d, q = _links(lattice, grid, solid, wall)
    u_max = 0.347 / L
    g = 4 * (1.0 / s_nu - 0.5) / 3.0 * u_max / (R * R)
    u = (u_max * (1 - best / (R * R)))[:, None] * a
    u[solid] = 0.0
    return dict(grid=grid, solid=solid, node=node, d=d, q=q, uw=torch.zeros(len(node), 3, device=DEV, dtype=torch.float64),
                u=u, force=tuple((g * a).tolist()))


def _sphere(lattice, nx, ny, nz):
    grid = _Grid(nx, ny, nz, (0, 0))
    x, y, z = grid.coords()
    R = 0.16 * min(nx, ny, nz)
    p = torch.stack([x, y, z], 1).double() - torch.tensor([nx / 2 + 0.37, ny / 2 - 0.29, nz / 2 + 0.13], device=DEV, dtype=torch.float64)
    d2 = (p * p).sum(1)
    solid = d2 <= R * R

    def wall(at, e):
        e = torch.tensor(e, device=DEV, dtype=torch.float64)
        w = p[at]
        return (e @ e).expand(len(at)), 2 * (w @ e), (w * w).sum(1) - R * R

    node, d, q = _links(lattice, grid, solid, wall)
    u = torch.zeros(len(x), 3, device=DEV, dtype=torch.float64)
    u[:, 0] = 0.02 * (1 - R / d2.sqrt().clamp(min=R))
    return dict(grid=grid, solid=solid, node=node, d=d, q=q, uw=torch.zeros(len(node), 3, device=DEV, dtype=torch.float64),
                u=u, force=(1e-6, 0.0, 0.0))


def _stirred(geo, seed):
    """Initial density and velocity: the geometry's base flow with a few smooth modes
    of seeded amplitude, direction and phase on top; (rho, u) of every node."""
    r = random.Random(int(seed))
    g = geo["grid"]
    nx, ny, nz = g.shape
    u = geo["u"].clone()
    top = max(float(u.abs().max()), 1e-4)
    rho = torch.full((nx * ny * nz,), RHO0, device=DEV, dtype=torch.float64)
    for k in range(6):
        phase = r.uniform(0, 2 * math.pi)
        w = 2 * math.pi * torch.tensor([r.choice([1, 2, 3]) / nx, r.choice([1, 2, 3]) / ny, r.choice([0, 1, 2]) / nz], dtype=torch.float64)
        mode = torch.sin(w[0] * g.x[None, None, :].double() + w[1] * g.y[None, :, None].double() + w[2] * g.z[:, None, None].double() + phase).reshape(-1)
        if k < 3:
            for c in range(u.shape[1]):
                u[:, c] += 0.1 * top * r.uniform(-1, 1) * mode
        else:
            rho += 0.1 * top * r.uniform(-1, 1) * mode
    u[geo["solid"]] = 0.0
    return rho, u


def _geometry(case):
    lat, n = case["lattice"], case["nx"]
    if case["kind"] in ("pipe", "job"):
        return _pipe(lat, n, case["s_nu"])
    if case["kind"] == "couette" or (case["kind"] == "adjoint" and lat == "D2Q9"):
        s = n / 64.0
        return _couette(lat, n, (32.3 * s, 31.7 * s), 10.0 * s, 28.0 * s, 0.01 / s)
    return _sphere(lat, case["nx"], case["ny"], case["nz"])


def _members(case, seed):
    """The ensemble's geometries: sizes fixed by the case, flow parameters by the seed."""
    sizes = np.random.RandomState(case["members"] * 1000 + case["nx"])
    r = random.Random(int(seed))
    got = []
    for _ in range(case["members"]):
        n = int(sizes.randint(case["nx"], case["ny"] + 1))
        R1, R2 = float(sizes.uniform(0.1, 0.25)) * n, float(sizes.uniform(0.35, 0.45)) * n
        ox, oy = sizes.uniform(0, 1, 2)
        geo = _couette("D2Q9", n, (n / 2 + float(ox), n / 2 + float(oy)), R1, R2, r.uniform(0.005, 0.02))
        geo["s_nu"] = 1.0 / (3.0 * r.uniform(0.02, 0.2) + 0.5)
        got.append(geo)
    return got


def _simulation(case, geo, s_nu):
    g = geo["grid"]
    sim = B.Lbm(case["lattice"], g.shape, np.array(_rates(case["lattice"], s_nu), dtype=np.float64), case["precision"], RHO0)
    sim.set_stream(torch.cuda.current_stream().cuda_stream)
    if g.skew != (0, 0):
        sim.set_skew(*g.skew)
    sim.set_scheme(0.0, case["c1"], case["c2"], case["b"], allow_nonconvex=True)
    links = dict(node=geo["node"].cpu().numpy(), d=geo["d"].cpu().numpy().astype(np.int32), q=geo["q"].cpu().numpy(), uw=geo["uw"].cpu().numpy())
    sim.set_geometry(geo["solid"].cpu().numpy(), links)
    sim.set_force(geo["force"])
    return sim


def _target(case, geo, u):
    """The adjoint's probe slab and target velocity (a damped copy of the start)."""
    g = geo["grid"]
    x, y, _ = g.coords()
    slab = (x >= g.shape[0] // 2) & (x < g.shape[0] // 2 + max(2, g.shape[0] // 8))
    return slab.to(torch.uint8), 0.7 * u


# ---------------------------------------------------------------------------------
# prepare, run, work
# ---------------------------------------------------------------------------------

def prepare(case, seed):
    D = 2 if case["lattice"] == "D2Q9" else 3
    st = dict(case=case, D=D)
    geos = _members(case, seed) if case["kind"] == "ensemble" else [_geometry(case)]
    sims, start, nodes = [], [], 0
    for k, geo in enumerate(geos):
        rho, u = _stirred(geo, int(seed) + 7919 * k)
        sim = _simulation(case, geo, geo.get("s_nu", case["s_nu"]))
        host = rho.cpu().numpy(), u[:, :D].contiguous().cpu().numpy()
        sim.init_equilibrium(*host)
        sims.append(sim)
        start.append(nodes)
        nodes += sim.N
    st.update(sims=sims, start=start, nodes=nodes)
    if case["kind"] == "ensemble":
        st["batch"] = B.Batch(sims)
        st["batch"].set_stream(torch.cuda.current_stream().cuda_stream)
    if case["kind"] == "adjoint":
        mask, target = _target(case, geos[0], u[:, :D])
        st.update(mask=mask.cpu().numpy(), target=target.contiguous().cpu().numpy())
    elif case["kind"] == "job":
        st.update(host=host, reference=geos[0]["u"][:, :D].contiguous(),
                  norms=torch.zeros(case["steps"] // 10, 7, device=DEV, dtype=torch.float64))
    else:
        st.update(rho=torch.empty(nodes, device=DEV, dtype=torch.float64), u=torch.empty(nodes, D, device=DEV, dtype=torch.float64))
    torch.cuda.synchronize()
    return st


def _kept(st, rho, u):
    """A read-out in the type of the storage."""
    t = TYPE_OF[st["case"]["precision"]]
    if t == torch.float64:
        return {"rho": rho, "u": u}
    return {"drho": (rho - RHO0).to(t), "u": u.to(t)}


def run(st):
    case, sim = st["case"], st["sims"][0]
    n = case["steps"]
    if case["kind"] == "adjoint":
        J, gs, gq, gu = sim.adjoint(n, st["mask"], st["target"])
        t = np.float64 if case["precision"] == "f64" else np.float32
        return {"J": J, "dJ_ds": gs.astype(t), "dJ_dq": gq.astype(t), "dJ_duw": gu.astype(t)}
    if case["kind"] == "job":
        sim.init_equilibrium(*st["host"])
        for k in range(n // 10):
            sim.step(10)
            sim.error_norms_noalloc(st["reference"].data_ptr(), st["norms"][k].data_ptr())
        rho, u = sim.moments()
        t = np.float64 if case["precision"] == "f64" else np.float32
        return {"drho": (rho - RHO0).astype(t), "u": u.astype(t), "norms": st["norms"].to(torch.float64 if case["precision"] == "f64" else torch.float32)}
    if case["kind"] == "ensemble":
        st["batch"].step(n)
    else:
        sim.step(n)
    for one, at in zip(st["sims"], st["start"]):
        one.moments_device(st["rho"].data_ptr() + 8 * at, st["u"].data_ptr() + 8 * st["D"] * at)
    return _kept(st, st["rho"], st["u"])


def _nodes(case):
    """(all nodes, fluid nodes), the fluid from the areas and volumes of the geometry."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["kind"] == "ensemble":
        sizes = np.random.RandomState(case["members"] * 1000 + nx)
        N = nf = 0
        for _ in range(case["members"]):
            n = int(sizes.randint(nx, ny + 1))
            R1, R2 = float(sizes.uniform(0.1, 0.25)) * n, float(sizes.uniform(0.35, 0.45)) * n
            sizes.uniform(0, 1, 2)
            N, nf = N + n * n, nf + math.pi * (R2 * R2 - R1 * R1)
        return N, nf
    N = nx * ny * nz
    if case["kind"] in ("pipe", "job"):
        return N, math.pi * 0.4 ** 2 * nx * nx * nx * math.sqrt(281.0) / 16.0
    if case["lattice"] == "D2Q9":
        return N, math.pi * (28.0 ** 2 - 10.0 ** 2) / 64.0 ** 2 * N
    return N, N - 4.0 / 3.0 * math.pi * (0.16 * min(nx, ny, nz)) ** 3


def work(case):
    """A step reads and writes every population of a fluid node once; a read-out reads
    them once and writes its fields; the adjoint needs a forward step, the state and
    the adjoint state read and the adjoint state written, and one recomputed step."""
    Q, D = Q_OF[case["lattice"]], 2 if case["lattice"] == "D2Q9" else 3
    s = BYTES_OF[case["precision"]]
    N, nf = _nodes(case)
    n = case["steps"]
    per_step = 2 * Q * s * nf
    read_out = Q * s * nf + (1 + D) * 8 * N
    flops = {"D2Q9": 110.0, "D3Q19": 263.0, "D3Q15": 200.0}[case["lattice"]] * nf * n
    if case["kind"] == "adjoint":
        return {"bytes": n * (2 * per_step + 1.5 * per_step), "flops": 4 * flops}
    if case["kind"] == "job":
        return {"bytes": n * per_step + (n // 10) * (Q * s * nf + 8 * D * N) + 2 * read_out, "flops": flops}
    return {"bytes": n * per_step + read_out, "flops": flops}


# ---------------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------------

def _moment_matrix(lattice):
    rows = []
    for x, y, z in E_OF[lattice]:
        r2 = x * x + y * y + z * z
        if lattice == "D2Q9":
            rows.append([1, 3 * r2 - 4, (9 * r2 * r2 - 21 * r2 + 8) / 2, x, (3 * r2 - 5) * x, y, (3 * r2 - 5) * y, x * x - y * y, x * y])
        elif lattice == "D3Q19":
            p, w = 3 * x * x - r2, y * y - z * z
            rows.append([1, 19 * r2 - 30, (21 * r2 * r2 - 53 * r2 + 24) / 2, x, (5 * r2 - 9) * x, y, (5 * r2 - 9) * y, z, (5 * r2 - 9) * z,
                         p, (3 * r2 - 5) * p, w, (3 * r2 - 5) * w, x * y, y * z, x * z, w * x, (z * z - x * x) * y, (x * x - y * y) * z])
        else:
            rows.append([1, r2 - 2, (15 * r2 * r2 - 55 * r2 + 32) / 2, x, (5 * r2 - 13) * x / 2, y, (5 * r2 - 13) * y / 2, z, (5 * r2 - 13) * z / 2,
                         3 * x * x - r2, y * y - z * z, x * y, y * z, x * z, x * y * z])
    return torch.tensor(rows, device=DEV, dtype=torch.float64).T.contiguous()


class _Plain:
    """Time steps in deviations g = f - w rho0, two arrays, 64 bits."""

    def __init__(self, case, geo, s_nu):
        lat = case["lattice"]
        self.E = E_OF[lat]
        self.Q, self.D = len(self.E), 2 if lat == "D2Q9" else 3
        self.grid, self.solid = geo["grid"], geo["solid"]
        self.c = torch.tensor(self.E, device=DEV, dtype=torch.float64)
        self.w = torch.tensor(_weights(lat), device=DEV, dtype=torch.float64)
        self.M = _moment_matrix(lat)
        self.Minv = torch.linalg.inv(self.M)
        self.s = torch.tensor(_rates(lat, s_nu), device=DEV, dtype=torch.float64)
        self.q, self.uw = geo["q"], geo["uw"]
        self.family = (case["c1"], case["c2"], case["b"])
        F = torch.tensor(geo["force"], device=DEV, dtype=torch.float64)
        self.half_force = 0.5 * F
        rows = [3, 5, 7][: self.D]
        self.push = sum(self.Minv[:, k] * (RHO0 * F[a]) for a, k in enumerate(rows))
        self.opp = [self.E.index((-x, -y, -z)) for x, y, z in self.E]
        self.node, self.dir = geo["node"], geo["d"]
        self.of = [torch.nonzero(self.dir == d).reshape(-1) for d in range(self.Q)]

    def start(self, rho, u):
        u = torch.cat([u, torch.zeros(len(u), 3 - u.shape[1], device=DEV, dtype=torch.float64)], 1)
        g = self.equilibrium(rho - RHO0, RHO0 * u[:, 0], RHO0 * u[:, 1], RHO0 * u[:, 2])
        g[:, self.solid] = 0.0
        return g

    def equilibrium(self, drho, jx, jy, jz):
        j2 = (jx * jx + jy * jy + jz * jz) / RHO0
        out = []
        for i, (x, y, z) in enumerate(self.E):
            cj = x * jx + y * jy + z * jz
            out.append(self.w[i] * (drho + 3 * cj + 4.5 * cj * cj / RHO0 - 1.5 * j2))
        return torch.stack(out)

    def step(self, g, s, q, uw):
        drho = g.sum(0)
        j = self.c.T @ g
        K = self.Minv @ (s[:, None] * self.M)
        gp = g - K @ (g - self.equilibrium(drho, j[0], j[1], j[2])) + self.push[:, None]
        c1, c2, b = self.family
        new = []
        for i, e in enumerate(self.E):
            d = self.opp[i]
            row = gp[i] if i == 0 else gp[i][self.grid.neighbour((-e[0], -e[1], -e[2]))]
            at = self.of[d]
            if i and len(at):
                n, qq, l = self.node[at], q[at], c1 * q[at] + c2 * q[at] * q[at]
                wall = 2 / (1 + l) * self.w[i] * RHO0 * (uw[at] @ self.c[i]) * 3
                v = (1 - b) * g[i][n] + b * ((1 + l - 2 * qq) / (1 + l) * g[d][n] + l / (1 + l) * gp[i][n] + (2 * qq - l) / (1 + l) * gp[d][n] + wall)
                row = row.index_put((n,), v)
            new.append(row)
        return torch.where(self.solid, 0.0, torch.stack(new))

    def velocity(self, g):
        return ((self.c.T @ g) / RHO0 + self.half_force[:, None]).T[:, : self.D]

    def fields(self, g):
        rho, u = RHO0 + g.sum(0), self.velocity(g).clone()
        rho[self.solid] = float("nan")
        u[self.solid] = float("nan")
        return rho, u


def _exact_adjoint(case, geo, seed):
    p = _Plain(case, geo, case["s_nu"])
    rho, u = _stirred(geo, seed)
    mask, target = _target(case, geo, u[:, : p.D])
    s, q, uw = (v.clone().requires_grad_() for v in (p.s, p.q, p.uw))
    on = (mask != 0) & ~p.solid
    n, every = case["steps"], int(math.ceil(math.sqrt(case["steps"])))
    kept, g = [], p.start(rho, u)
    with torch.no_grad():
        for k in range(n):
            if k % every == 0:
                kept.append(g)
            g = p.step(g, p.s, p.q, p.uw)
    g = g.requires_grad_()
    J = ((p.velocity(g) - target)[on] ** 2).sum()
    lam = torch.autograd.grad(J, g)[0]
    total = [torch.zeros_like(v) for v in (s, q, uw)]
    for seg in reversed(range(len(kept))):
        states = [kept[seg]]
        with torch.no_grad():
            for _ in range(min(every, n - seg * every) - 1):
                states.append(p.step(states[-1], p.s, p.q, p.uw))
        for g in reversed(states):
            g = g.detach().requires_grad_()
            lam, *more = torch.autograd.grad(p.step(g, s, q, uw), (g, s, q, uw), lam)
            for t, m in zip(total, more):
                t += m
        del states
    return {"J": J.item(), "dJ_ds": total[0].cpu().numpy(), "dJ_dq": total[1].cpu().numpy(), "dJ_duw": total[2].cpu().numpy() if p.D == 3 else
            (total[2] * torch.tensor([1.0, 1.0, 0.0], device=DEV, dtype=torch.float64)).cpu().numpy()}


def exact(case, seed):
    torch.set_float32_matmul_precision("highest")
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, _geometry(case), seed)
    keep = "rho" if case["precision"] == "f64" and case["kind"] != "job" else "drho"
    geos = _members(case, seed) if case["kind"] == "ensemble" else [_geometry(case)]
    rhos, us, norms = [], [], []
    with torch.no_grad():
        for k, geo in enumerate(geos):
            p = _Plain(case, geo, geo.get("s_nu", case["s_nu"]))
            g = p.start(*_stirred(geo, int(seed) + 7919 * k))
            for t in range(case["steps"]):
                g = p.step(g, p.s, p.q, p.uw)
                if case["kind"] == "job" and (t + 1) % 10 == 0:
                    fluid = ~p.solid
                    ref, u = geo["u"][:, : p.D][fluid], p.velocity(g)[fluid]
                    j = (p.c.T @ g)[:, fluid].sum(1)
                    norms.append(torch.stack([(ref - u).norm() / ref.norm(), (ref - u).abs().max(), RHO0 * fluid.sum() + g[:, fluid].sum(), j[0], j[1], j[2], torch.zeros_like(j[0])]))
            rho, u = p.fields(g)
            rhos.append(rho - RHO0 if keep == "drho" else rho)
            us.append(u)
            del g, p
    out = {keep: torch.cat(rhos), "u": torch.cat(us)}
    if case["kind"] == "job":
        out = {k: v.cpu().numpy() for k, v in out.items()}
        out["norms"] = torch.stack(norms)
    return out
