"""The calls that users of this framework make, as measurable cases.

A case is a plain dict; its ``kind`` says which call it stands for:

* ``step``: ``steps`` coupled time steps (Simulation.step), then the particle
  state and the potential are read back -- the main loop of every run.
* ``fleet``: one lockstep time step of several resident runs of uneven size,
  as the batching server makes it: mapping and solve of each run on its own
  stream, one batched stream-collide, forces and rigid-body update.
* ``solve``: the potential from zero to the tolerance (mapping, solve, read
  back): what the first step of every run costs, and a calculation that only
  wants the double layers.
* ``flow``: ``steps`` stream-collide steps past spheres with prescribed
  velocities under a uniform body force, then force, torque and the velocity
  field (the Stokes-drag half of the validation runs).
* ``fields``: potential, density and velocity of a state, read back into
  device tensors (a snapshot).

Grids are (nx, ny, nz); ``walls`` names the axes that are bounded by walls
(the others are periodic); ``slip`` makes those walls free-slip.
"""
from __future__ import annotations

import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_1708_08741_gb300 as es
from paper_1708_08741_gb300 import serving
from paper_1708_08741_gb300 import workloads as W

_PRECISION = {"fp64": es.ES_FP64, "mixed32": es.ES_MIXED32, "mixed16": es.ES_MIXED16}
# the type that the populations, and what is summed from them, have in a form
_TYPE = {"fp64": torch.float64, "mixed32": torch.float32, "mixed16": torch.bfloat16}

# D3Q19 velocities and weights (Sec. 4.1), rest first
_C = [(0, 0, 0)] + [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)
                    if 1 <= abs(a) + abs(b) + abs(c) <= 2]
_W = [1.0 / 3.0] + [1.0 / 18.0 if sum(map(abs, c)) == 1 else 1.0 / 36.0 for c in _C[1:]]
_OPP = [_C.index((-a, -b, -c)) for a, b, c in _C]


def listed():
    base = dict(walls="", slip=False, kind_of="charge", zeta=1.0, debye=4.0, field=1e-3, tau=1.0, coarse_sweeps=8)
    return [
        # the smallest run: one sphere of fixed zeta in a 32^3 periodic box, plain FP64
        dict(base, name="step_sphere32_fp64", kind="step", nx=32, ny=32, nz=32, spheres=1, radius=4.0, kind_of="zeta",
             levels=3, res_rf=1e-10, coarse_sweeps=32, precision="fp64", steps=4),
        # a small ragged box between two x walls: no extent a multiple of the vector width
        dict(base, name="step_box42_mixed32", kind="step", nx=42, ny=24, nz=36, walls="x", spheres=4, radius=3.5,
             levels=2, res_rf=1e-10, coarse_sweeps=32, precision="mixed32", steps=4),
        # eight served runs of uneven size, stepped together
        dict(name="fleet_8_mixed32", kind="fleet", runs=8, mix=5, lo=32, hi=96, precision="mixed32"),
        # charged spheres in a channel between two z walls, in both arithmetic forms
        dict(base, name="step_channel128_fp64", kind="step", nx=128, ny=128, nz=128, walls="z", spheres=64, radius=6.0,
             debye=3.0, field=2e-3, levels=4, res_rf=1e-8, coarse_sweeps=32, precision="fp64", steps=2),
        dict(base, name="step_channel128_mixed32", kind="step", nx=128, ny=128, nz=128, walls="z", spheres=64,
             radius=6.0, debye=3.0, field=2e-3, levels=4, res_rf=1e-8, coarse_sweeps=32, precision="mixed32", steps=4),
        # the validation box: one sphere, free-slip walls all round, the paper's relaxation time
        dict(base, name="step_henry96_mixed32", kind="step", nx=96, ny=96, nz=96, walls="xyz", slip=True, spheres=1,
             radius=4.0, kind_of="zeta", debye=8.0, field=2.5e-3, tau=6.0, levels=4, res_rf=1e-8, coarse_sweeps=32,
             precision="mixed32", steps=4),
        # a suspension with 16-bit populations
        dict(base, name="step_suspension256_mixed16", kind="step", nx=256, ny=256, nz=256, spheres=360, radius=5.0,
             levels=5, res_rf=4e-6, precision="mixed16", steps=4),
        # one node's problem of the paper's scaling runs
        dict(base, name="step_node_mixed32", kind="step", nx=288, ny=576, nz=288, walls="xz", spheres=1024, radius=6.0,
             kind_of="zeta", debye=15.08, field=0.019, tau=6.0, levels=6, res_rf=4e-6, precision="mixed32", steps=2,
             placement="lattice"),
        # the benchmark's suspension
        dict(base, name="step_suspension512_mixed32", kind="step", nx=512, ny=512, nz=512, spheres=2880, radius=5.0,
             levels=6, res_rf=4e-6, precision="mixed32", steps=2),
        # the potential of a suspension from zero
        dict(base, name="solve_suspension192_mixed32", kind="solve", nx=192, ny=192, nz=192, spheres=152, radius=5.0,
             levels=5, res_rf=1e-8, precision="mixed32"),
        # flow past spheres, plain FP64
        dict(base, name="flow_160_fp64", kind="flow", nx=160, ny=136, nz=152, spheres=24, radius=5.0, levels=2,
             res_rf=1e-8, precision="fp64", steps=4),
        # a snapshot of a large state
        dict(base, name="fields_320_mixed32", kind="fields", nx=320, ny=320, nz=320, spheres=703, radius=5.0, levels=5,
             res_rf=4e-6, precision="mixed32"),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "solve", "flow", "fields", "fleet"])
    if kind == "fleet":
        lo = rng.choice([32, 40, 48])
        return dict(kind="fleet", runs=rng.randint(2, 12), mix=rng.randint(1, 10 ** 6), lo=lo,
                    hi=lo + rng.choice([16, 32, 64]), precision=rng.choice(["mixed32", "mixed32", "fp64"]))
    precision = rng.choice(["mixed32", "mixed32", "mixed32", "mixed16", "fp64"])
    top = {"fp64": 144, "mixed32": 288, "mixed16": 288}[precision]
    walls = rng.choice(["", "", "", "z", "z", "x", "xz", "xyz"])
    slip = walls != "" and rng.random() < 0.3
    levels = rng.choice([2, 3, 3, 4])
    dims = []
    for axis in "xyz":
        e = math.exp(rng.uniform(math.log(32), math.log(top)))
        # periodic extents stay even on the coarsest level; walled ones need not
        mult = (1 << (levels - 1)) * (1 if axis in walls else 2)
        dims.append(min(max(int(round(e / mult)), -(-32 // mult)), top // mult) * mult)
    radius = round(rng.uniform(3.0, 6.0), 2)
    cells = dims[0] * dims[1] * dims[2]
    most = max(1, int(0.04 * cells / (4.0 / 3.0 * math.pi * radius ** 3)))
    spheres = max(1, int(round(math.exp(rng.uniform(0.0, math.log(most))))))
    if walls == "xyz":
        spheres = 1  # (the field drives them towards a wall)
    return dict(kind=kind, nx=dims[0], ny=dims[1], nz=dims[2], walls=walls, slip=slip, spheres=spheres, radius=radius,
                kind_of="zeta" if spheres == 1 and walls != "xyz" else "charge",
                zeta=round(rng.uniform(0.5, 1.0), 3), debye=round(rng.uniform(2.0, 8.0), 2),
                field=round(rng.uniform(5e-4, 1e-3), 6), tau=rng.choice([1.0, 1.0, 6.0]), levels=levels,
                res_rf=rng.choice([1e-10, 1e-8, 4e-6]), coarse_sweeps=rng.choice([8, 32]), precision=precision,
                steps=rng.randint(1, 4))


# -- workloads --

def _workload(case, seed):
    dims = [case["nx"], case["ny"], case["nz"]]
    periodic = tuple(0 if a in case["walls"] else 1 for a in "xyz")
    n, R = case["spheres"], case["radius"]
    rng = W.PCG32(seed)
    if n == 1:
        x = np.array([[d / 2.0 + rng.uniform_range(-0.5, 0.5) for d in dims]])
    elif case.get("placement") == "lattice":
        x = W.paper_node().x + np.array([[rng.uniform_range(-0.5, 0.5) for _ in range(3)] for _ in range(n)])
    else:
        x = W.place_spheres(n, R, dims, periodic, rng)
    axis = periodic.index(1) if 1 in periodic else 0  # the field: along the first periodic axis
    E = [0.0, 0.0, 0.0]
    E[axis] = case["field"]
    flow = case["kind"] == "flow"
    zeta = np.full(n, 0.0 if flow else case["zeta"] if case["kind_of"] == "zeta" else 0.0)
    q = np.array([0.0 if flow or case["kind_of"] == "zeta" else rng.uniform_range(0.5, 1.5) for _ in range(n)])
    kind = np.full(n, W.KIND_ZETA if flow or case["kind_of"] == "zeta" else W.KIND_CHARGE, dtype=np.int32)
    v = np.zeros((n, 3))
    w = np.zeros((n, 3))
    accel = [0.0, 0.0, 0.0]
    if flow:
        v = np.array([[rng.uniform_range(-0.02, 0.02) for _ in range(3)] for _ in range(n)])
        w = np.array([[rng.uniform_range(-2e-3, 2e-3) for _ in range(3)] for _ in range(n)])
        accel[axis] = 1e-5
    return W.Workload(name="case", dims=dims, periodic=periodic, tau=case["tau"], kappa=1.0 / case["debye"], eps=1.0,
                      E_ext=tuple(E), accel=tuple(accel), levels=case["levels"], coarse_sweeps=case["coarse_sweeps"],
                      res_rf=case["res_rf"], max_cycles=200, wall_slip=(1 if case["slip"] else 0,) * 6,
                      x=x, v=v, w=w, R=np.full(n, R), kind=kind, zeta=zeta, q=q)


def _fleet_workloads(case, seed):
    """The runs' shapes belong to the case, the sphere positions to the seed."""
    out = []
    for rid in range(case["runs"]):
        wl = serving.request_workload(rid, seed=case["mix"], edge_range=(case["lo"], case["hi"]),
                                      field_range=(5e-4, 1e-3), zeta_range=(0.5, 1.0))
        wl.x = W.place_spheres(wl.n_particles, float(wl.R[0]), wl.dims, wl.periodic, W.PCG32(seed, stream=rid))
        out.append(wl)
    return out


def _populations(case, seed):
    """Seeded populations near equilibrium, (19, nz, ny, nx) in the order of _C: a smooth flow plus noise."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ph = torch.rand(6, generator=gen, device="cuda", dtype=torch.float64) * (2.0 * math.pi)
    z, y, x = (torch.arange(n, device="cuda", dtype=torch.float64) * (2.0 * math.pi / n) for n in (nz, ny, nx))
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    u = [0.02 * torch.sin(y + ph[0]) * torch.cos(z + ph[1]), 0.02 * torch.sin(z + ph[2]) * torch.cos(x + ph[3]),
         0.02 * torch.sin(x + ph[4]) * torch.cos(y + ph[5])]
    u = [t.expand(nz, ny, nx) for t in u]
    uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    f = torch.empty((19, nz, ny, nx), device="cuda", dtype=torch.float64)
    for q, (c, w) in enumerate(zip(_C, _W)):
        cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
        noise = torch.randn((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float32)
        f[q] = w * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu + 1e-3 * noise.double())
    return f


def _potential(case, seed):
    """A seeded smooth potential."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    ph = torch.rand(3, generator=gen, device="cuda", dtype=torch.float64) * (2.0 * math.pi)
    z, y, x = (torch.arange(n, device="cuda", dtype=torch.float64) * (2.0 * math.pi / 32.0) for n in (nz, ny, nx))
    return (0.5 * torch.sin(x + ph[0])[None, None, :] * torch.cos(y + ph[1])[None, :, None]
            * torch.sin(z + ph[2])[:, None, None]).contiguous()


# -- calls through the C ABI with device pointers --

def _ok(sim, rc, where):
    if rc != es.ES_OK:
        raise es.EsError(rc, where, sim.lib.es_last_error(sim.h).decode())


def _set_field(sim, which, t):
    _ok(sim, sim.lib.es_set_field(sim.h, which, t.data_ptr(), t.numel() * t.element_size(), 1), "es_set_field")


def _particles(sim, records):
    """Positions, velocities and spins from the C records (13 doubles each)."""
    _ok(sim, sim.lib.es_get_particles(sim.h, records, sim.np), "es_get_particles")
    a = np.frombuffer(records, dtype=np.float64).reshape(-1, 13)[: sim.np]
    return a[:, 0:3].copy(), a[:, 3:6].copy(), a[:, 6:9].copy()


def _in_type(case, a):
    """A host array in the type that the form computes it in (positions stay FP64)."""
    return torch.from_numpy(a).to(_TYPE[case["precision"]])


def _solved_type(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


# -- the interface --

def prepare(case, seed):
    if case["kind"] == "fleet":
        sims = [es.Simulation(wl, _PRECISION[case["precision"]], stream=torch.cuda.Stream())
                for wl in _fleet_workloads(case, seed)]
        for s in sims:
            s.step()
        torch.cuda.synchronize()
        return {"case": case, "sims": sims, "records": [(es.Particle * s.np)() for s in sims],
                "pool": ThreadPoolExecutor(max_workers=len(sims))}
    sim = es.Simulation(_workload(case, seed), _PRECISION[case["precision"]])
    state = {"case": case, "sim": sim, "records": (es.Particle * sim.np)()}
    shape = (case["nz"], case["ny"], case["nx"])
    if case["kind"] == "step":
        sim.step()  # the cold first solve is its own case
        state["psi"] = torch.empty(shape, dtype=torch.float64, device="cuda")
    elif case["kind"] == "solve":
        state["zero"] = torch.zeros(shape, dtype=torch.float64, device="cuda")
        state["psi"] = torch.empty(shape, dtype=torch.float64, device="cuda")
    else:
        c, _ = es.lattice()
        order = [_C.index(tuple(int(v) for v in row)) for row in c]
        _set_field(sim, es.FIELD_PDF, _populations(case, seed)[order])
        sim.map_particles()
        if case["kind"] == "fields":
            _set_field(sim, es.FIELD_PSI, _potential(case, seed))
            state["psi"] = torch.empty(shape, dtype=torch.float64, device="cuda")
            state["rho"] = torch.empty(shape, dtype=torch.float64, device="cuda")
        sim.solve(forced_cycles=0)
        state["u"] = torch.empty((3,) + shape, dtype=torch.float64, device="cuda")
    torch.cuda.empty_cache()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "fleet":
        sims = state["sims"]
        for s in sims:
            s.map_particles()
        for f in [state["pool"].submit(s.solve) for s in sims]:
            f.result()
        es.lbm_step_batch(sims)
        for s in sims:
            s.forces_device()
            s.advance()
        out = []
        for s, r in zip(sims, state["records"]):
            x, v, w = _particles(s, r)
            out.append({"x": x, "v": _in_type(case, v), "w": _in_type(case, w)})
        return out
    sim = state["sim"]
    if case["kind"] == "step":
        for _ in range(case["steps"]):
            sim.step()
        x, v, w = _particles(sim, state["records"])
        sim.field_device(es.FIELD_PSI, state["psi"])
        return {"x": x, "v": _in_type(case, v), "w": _in_type(case, w), "psi": state["psi"].to(_solved_type(case))}
    if case["kind"] == "solve":
        _set_field(sim, es.FIELD_PSI, state["zero"])
        sim.map_particles()
        sim.solve()
        sim.field_device(es.FIELD_PSI, state["psi"])
        return state["psi"].to(_solved_type(case))
    if case["kind"] == "flow":
        for _ in range(case["steps"]):
            sim.lbm_step()
        F, T = sim.forces()
        sim.field_device(es.FIELD_U, state["u"])
        return {"F": _in_type(case, F), "T": _in_type(case, T), "u": state["u"].to(_TYPE[case["precision"]])}
    sim.field_device(es.FIELD_PSI, state["psi"])
    sim.field_device(es.FIELD_RHO, state["rho"])
    sim.field_device(es.FIELD_U, state["u"])
    return {"psi": state["psi"], "rho": state["rho"], "u": state["u"]}


def work(case):
    """Bytes: populations in and out (19 streams each way), the potential in and out, a flag byte, what is read back."""
    pop = {"fp64": 8, "mixed32": 4, "mixed16": 2}[case["precision"]]
    kind = case["kind"]
    if kind == "fleet":
        cells = sum(wl.n_cells for wl in _fleet_workloads(case, 1))
        return {"bytes": cells * (38 * pop + 16 + 1), "flops": 342.0 * cells}
    cells = case["nx"] * case["ny"] * case["nz"]
    out = 4 if case["precision"] != "fp64" else 8
    if kind == "step":
        return {"bytes": cells * (case["steps"] * (38 * pop + 16 + 1) + 8 + out),
                "flops": 342.0 * cells * case["steps"]}
    if kind == "solve":
        return {"bytes": cells * (8 + 8 + 1 + out), "flops": 12.0 * cells}
    if kind == "flow":
        return {"bytes": cells * (case["steps"] * (38 * pop + 8 + 1) + 19 * pop + 24 + 3 * out),
                "flops": 342.0 * cells * case["steps"]}
    return {"bytes": cells * (8 + 19 * pop + 5 * 8), "flops": 60.0 * cells}


# -- the same results in plain torch, 64 bits --

class _Geometry:
    """Which sphere owns a cell, and what lies beyond each face of it."""

    def __init__(self, case, seed):
        self.wl = wl = _workload(case, seed)
        self.dims = nx, ny, nz = wl.dims
        self.per = wl.periodic
        owner = np.full((nz, ny, nx), -1, dtype=np.int64)
        for p in range(wl.n_particles):
            idx, d2 = [], 0.0
            for a in range(3):
                lo, hi = math.floor(wl.x[p][a] - wl.R[p]) - 1, math.ceil(wl.x[p][a] + wl.R[p]) + 1
                i = np.arange(lo, hi + 1)
                if not self.per[a]:
                    i = i[(i >= 0) & (i < self.dims[a])]
                idx.append(i % self.dims[a])
                d = (i + 0.5 - wl.x[p][a]) ** 2
                d2 = d2 + d.reshape([-1 if k == 2 - a else 1 for k in range(3)])
            inside = d2 <= wl.R[p] ** 2
            block = owner[np.ix_(idx[2], idx[1], idx[0])]
            owner[np.ix_(idx[2], idx[1], idx[0])] = np.where(inside, p, block)
        self.owner = torch.from_numpy(owner).cuda()
        self.solid = self.owner >= 0
        faces = torch.zeros(wl.n_particles, dtype=torch.float64, device="cuda")
        for c in _C[1:]:
            if sum(map(abs, c)) == 1:
                o = torch.where(self.outside(c) | self.solid, torch.full_like(self.owner, -1), self.at(self.owner, c))
                faces += torch.bincount(o[o >= 0], minlength=wl.n_particles).double()
        dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()  # noqa: E731
        self.zeta, self.sigma = dev(wl.zeta), dev(wl.q) / faces.clamp(min=1.0)
        self.dirichlet = torch.from_numpy(wl.kind == W.KIND_ZETA).cuda()
        self.x, self.v, self.w = dev(wl.x), dev(wl.v), dev(wl.w)

    def at(self, t, c):
        """t at each cell's neighbour in direction c (axes wrapped)."""
        return torch.roll(t, shifts=(-c[2], -c[1], -c[0]), dims=(-3, -2, -1))

    def outside(self, c):
        """Cells whose neighbour in direction c lies beyond a wall."""
        out = torch.zeros(self.dims[::-1], dtype=torch.bool, device="cuda")
        for a in range(3):
            if c[a] and not self.per[a]:
                out.select(2 - a, self.dims[a] - 1 if c[a] > 0 else 0).fill_(True)
        return out

    def arm(self, cells, p, c):
        """x_s - X for the surface cells one step c from the cells (k, j, i), minimum image."""
        r = []
        for a in range(3):
            d = cells[2 - a].double() + c[a] + 0.5 - self.x[p, a]
            if self.per[a]:
                n = float(self.dims[a])
                d = d - n * torch.round(d / n)
            r.append(d)
        return r

    def wall_speed(self, cells, p, c):
        """c . u_s at those surface cells."""
        r = self.arm(cells, p, c)
        w, v = self.w[p], self.v[p]
        u = [v[:, 0] + w[:, 1] * r[2] - w[:, 2] * r[1], v[:, 1] + w[:, 2] * r[0] - w[:, 0] * r[2],
             v[:, 2] + w[:, 0] * r[1] - w[:, 1] * r[0]]
        return r, c[0] * u[0] + c[1] * u[1] + c[2] * u[2]


def _exact_solve(case, seed):
    g = _Geometry(case, seed)
    fluid = ~g.solid
    diag = torch.full(g.solid.shape, 6.0 + g.wl.kappa ** 2, dtype=torch.float64, device="cuda")
    b = torch.zeros_like(diag)
    open_ = []
    for c in _C[1:]:
        if sum(map(abs, c)) != 1:
            continue
        out, o = g.outside(c), g.at(g.owner, c)
        diag -= out.double()  # zero-flux wall
        hit = ~out & (o >= 0)
        p = o[hit]
        dirichlet = g.dirichlet[p]
        diag[hit] += torch.where(dirichlet, 1.0, -1.0).double()
        b[hit] += torch.where(dirichlet, 2.0 * g.zeta[p], g.sigma[p])
        open_.append((c, (~out & (o < 0)).double()))
    m = fluid.double()
    b = b * m

    def apply(v):
        r = diag * v
        for c, k in open_:
            r = r - k * g.at(v, c)
        return r * m

    x = torch.zeros_like(b)
    r = b.clone()
    z = r / diag
    p = z.clone()
    rz = (r * z).sum()
    stop = 1e-13 * float(r.norm())
    for it in range(4000):
        ap = apply(p)
        a = rz / (p * ap).sum()
        x += a * p
        r -= a * ap
        if it % 20 == 0 and float(r.norm()) <= stop:
            break
        z = r / diag
        rz, old = (r * z).sum(), rz
        p = z + (rz / old) * p
    o = g.owner.clamp(min=0)
    return torch.where(g.solid, torch.where(g.dirichlet[o], g.zeta[o], torch.zeros_like(x)), x)


def _exact_flow(case, seed):
    g = _Geometry(case, seed)
    wl = g.wl
    lam_e = -1.0 / wl.tau
    lam_o = -8.0 * (2.0 - 1.0 / wl.tau) / (8.0 - 1.0 / wl.tau)
    fx = list(wl.accel)
    bufs = [_populations(case, seed), torch.empty(0)]
    bufs[1] = torch.tensor(_W, dtype=torch.float64, device="cuda").reshape(19, 1, 1, 1).expand_as(bufs[0]).clone()
    walls = {q: g.outside(tuple(-v for v in c)) for q, c in enumerate(_C)}
    hits = {}
    for q, c in enumerate(_C[1:], start=1):
        back = tuple(-v for v in c)
        o = g.at(g.owner, back)
        cells = (~g.solid & ~walls[q] & (o >= 0)).nonzero(as_tuple=True)
        p = o[cells]
        hits[q] = (cells, p) + g.wall_speed(cells, p, back)
    cur = 0
    for _ in range(case["steps"]):
        src = bufs[cur]
        f = torch.empty_like(src)
        for q, c in enumerate(_C):
            back = tuple(-v for v in c)
            f[q] = g.at(src[q], back)
            if q == 0:
                continue
            if not case["slip"]:
                f[q] = torch.where(walls[q], src[_OPP[q]], f[q])
            else:
                f[q] = _mirrored(g, src, f[q], q, c)
            cells, _p, _r, speed = hits[q]
            # u_s . c_q: wall_speed's direction is -c_q
            f[q][cells] = src[_OPP[q]][cells] + 6.0 * _W[q] * -speed
        rho = f.sum(0)
        u = [sum(c[a] * f[q] for q, c in enumerate(_C) if c[a]) + 0.5 * fx[a] for a in range(3)]
        uu = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
        uf = u[0] * fx[0] + u[1] * fx[1] + u[2] * fx[2]
        new = bufs[1 - cur]
        for q, c in enumerate(_C):
            o, w = _OPP[q], _W[q]
            cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
            cf = c[0] * fx[0] + c[1] * fx[1] + c[2] * fx[2]
            even, odd = 0.5 * (f[q] + f[o]), 0.5 * (f[q] - f[o])
            post = (f[q] + lam_e * (even - w * (rho + 4.5 * cu * cu - 1.5 * uu)) + lam_o * (odd - 3.0 * w * cu)
                    + (1.0 + 0.5 * lam_e) * w * (9.0 * cu * cf - 3.0 * uf) + (1.0 + 0.5 * lam_o) * 3.0 * w * cf)
            new[q] = torch.where(g.solid, new[q], post)
        del f, rho, u, uu, uf
        cur = 1 - cur
    n = wl.n_particles
    F = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    T = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    src = bufs[1 - cur]
    for q, c in enumerate(_C[1:], start=1):
        o = _OPP[q]  # a link from the cell along c ends where the pull of the opposite direction starts
        cells, p, r, speed = hits[o]
        m = 2.0 * src[q][cells] - 6.0 * _W[q] * speed
        d = [m * c[0], m * c[1], m * c[2]]
        F.index_add_(0, p, torch.stack(d, 1))
        T.index_add_(0, p, torch.stack([r[1] * d[2] - r[2] * d[1], r[2] * d[0] - r[0] * d[2],
                                        r[0] * d[1] - r[1] * d[0]], 1))
    f = bufs[cur]
    u = torch.stack([sum(c[a] * f[q] for q, c in enumerate(_C) if c[a]) - 0.5 * fx[a] for a in range(3)])
    return {"F": F, "T": T, "u": u}


def _mirrored(g, src, f, q, c):
    """Free-slip walls: a population from beyond the crossed faces is the mirrored one of the fluid cell that lies
    along the uncrossed components (bounced back where that cell is an obstacle)."""
    crossed = [torch.zeros_like(g.solid) for _ in range(3)]
    for a in range(3):
        if c[a] and not g.per[a]:
            one = [0, 0, 0]
            one[a] = -c[a]
            crossed[a] = g.outside(tuple(one))
    f = f.clone()
    for m in range(1, 8):
        axes = [bool(m >> a & 1) for a in range(3)]
        if any(axes[a] and (not c[a] or g.per[a]) for a in range(3)):
            continue
        here = torch.ones_like(g.solid)
        for a in range(3):
            here &= crossed[a] if axes[a] else ~crossed[a]
        step = tuple(0 if axes[a] else -c[a] for a in range(3))
        mirror = _C.index(tuple(-c[a] if axes[a] else c[a] for a in range(3)))
        value = torch.where(g.at(g.solid, step), src[_OPP[q]], g.at(src[mirror], step))
        f = torch.where(here, value, f)
    return f


def _exact_fields(case, seed):
    g = _Geometry(case, seed)
    wl = g.wl
    f, psi = _populations(case, seed), _potential(case, seed)
    near = torch.zeros_like(g.solid)
    for c in _C[1:]:
        near |= g.outside(c) | g.at(g.solid, c)
    grad = []
    for a in range(3):
        e = [0, 0, 0]
        e[a] = 1
        iso = sum((3.0 * _W[q] * c[a]) * g.at(psi, c) for q, c in enumerate(_C) if c[a])
        side = []
        for s in (1, -1):
            c = tuple(s * v for v in e)
            o = g.at(g.owner, c).clamp(min=0)
            ghost = torch.where(g.dirichlet[o], 2.0 * g.zeta[o] - psi, psi + g.sigma[o] / wl.eps)
            value = torch.where(g.at(g.solid, c), ghost, g.at(psi, c))
            side.append(torch.where(g.outside(c), psi, value))
        grad.append(torch.where(near, 0.5 * (side[0] - side[1]), iso))
    rho_e = -wl.kappa ** 2 * wl.eps * psi
    fb = [torch.where(g.solid, torch.zeros_like(psi), rho_e * (wl.E_ext[a] - grad[a])) for a in range(3)]
    u = torch.stack([sum(c[a] * f[q] for q, c in enumerate(_C) if c[a]) - 0.5 * fb[a] for a in range(3)])
    return {"psi": psi, "rho": f.sum(0), "u": u}


def exact(case, seed):
    """The single parts in 64 bits; a whole coupled step (cells flip, the solve stops at its tolerance) has none."""
    kind = case["kind"]
    if kind == "solve":
        return _exact_solve(case, seed)
    if kind == "flow":
        return _exact_flow(case, seed)
    if kind == "fields":
        return _exact_fields(case, seed)
    return None
