"""The measured cases: what a user of this library has it do, each through the
public calls of ``binding.Solver``, ``binding.cfl_dt_noalloc`` and
``serve.SolveServer``.

A pass of a stepping case is what a driver program does between two looks at the
flow: hand over a state, advance it, and read it back (device pointers, as a
program whose fields live on the GPU has them). The states are what the solver
meets in earnest: a vortex on a periodic mesh, and a Mach-3 channel flow whose
free stream ahead of the bow shock is uniform to the bit, with a shock, smooth
structure behind it and a band that differs from the free stream by a few ulps
only ("shocked"), or with smooth structure everywhere ("perturbed").

``exact`` is the method itself (Algorithm 1 of arXiv:2106.02159 with its
boundary post-processing, SSPRK(3,3) and the parabolic sub-step of Sec. 5)
written with plain tensor operations in 64 bits; only the meshes' coefficient
arrays, which are inputs, come from the package.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2106_02159_gb300 import binding, meshes, serve

DEV = "cuda"
F64 = torch.float64
INFLOW = (1.4, 3.0, 1.0)  # rho, u, p of the Mach-3 channel


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def _case(kind, size, steps=1, mixed=False, relax=False, gamma=1.4, state="shocked", layers=0, cfl=0.5, passes=2):
    return dict(kind=kind, size=size, steps=steps, mixed=mixed, relax=relax, gamma=gamma, state=state, layers=layers,
                cfl=cfl, passes=passes)


def listed():
    c = [
        # the isentropic vortex on the 64 x 64 periodic P1 mesh, relaxed bounds (second order): the smallest
        # solve in use, a few thousand rows, where latency and launches count
        ("vortex_p1_4k", _case("vortex", 64, steps=10, relax=True)),
        # the vortex leaving an 80 x 80 Q1 box through non-reflecting sides, CFL 0.75
        ("nrbc_q1_6k", _case("nrbc", 80, steps=10, cfl=0.75)),
        # a parameter sweep: 256 small Q1 cylinder instances (32x8 to 64x16 cells) stepped together
        ("sweep_256x_q1", _case("sweep", 256, steps=2)),
        # a coarse Mach-3 cylinder, strict bounds: an ordinary 2D run
        ("cylinder_q1_62k", _case("cylinder", 112, steps=4)),
        # the same flow at 0.25M vertices, monatomic gas exponent off the 7/5 fast path
        ("cylinder_q1_246k_g13", _case("cylinder", 225, steps=1, gamma=1.3)),
        # a developed flow with structure in every cell, 1M vertices, FP64
        ("cylinder_q1_1m_full", _case("cylinder", 453, steps=1, state="perturbed")),
        # the same in mixed precision
        ("cylinder_q1_1m_mixed", _case("cylinder", 453, steps=1, state="perturbed", mixed=True)),
        # the benchmark's mesh: 4.0M vertices, bow shock and uniform free stream
        ("cylinder_q1_4m", _case("cylinder", 908, steps=1)),
        # 3D: the cylinder extruded over 24 layers of hexahedra (27-entry rows)
        ("cylinder3d_q1_375k", _case("cylinder3d", 56, steps=1, state="perturbed", layers=24)),
        # one Strang-split Navier-Stokes step on the cylinder with no-slip walls
        ("ns_q1_246k", _case("ns", 225, steps=1, state="perturbed")),
        # the CFL step from the caller's own device arrays, for callers that may not allocate
        ("cfl_noalloc_1m", _case("cfl", 453, state="perturbed")),
        # a stream of eight small requests (P1 and Q1 cylinders) served to a common final time
        ("serve_8", _case("serve", 8, steps=16, state="inflow")),
    ]
    return [dict(x, name=n) for n, x in c]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["vortex", "nrbc", "sweep", "cylinder", "cylinder", "cylinder", "cylinder3d", "cylinder3d", "ns",
                       "cfl", "serve"])
    gamma = rng.choice([1.4, 1.4, 1.4, 1.3, 5.0 / 3.0])
    mixed = rng.random() < 0.35
    relax = rng.random() < 0.4
    state = rng.choice(["shocked", "perturbed"])
    if kind == "vortex":
        return _case(kind, log_int(24, 300), steps=rng.randint(1, 10), mixed=mixed, relax=relax)
    if kind == "nrbc":
        return _case(kind, log_int(30, 240), steps=rng.randint(1, 10), mixed=mixed, relax=relax,
                     cfl=rng.choice([0.5, 0.75]))
    if kind == "sweep":
        return _case(kind, log_int(8, 300), steps=rng.randint(1, 4), mixed=mixed, relax=relax)
    if kind == "cylinder":
        m = log_int(20, 640)
        return _case(kind, m, steps=rng.randint(1, 4) if m < 300 else 1, mixed=mixed, relax=relax, gamma=gamma,
                     state=state, passes=rng.choice([1, 2, 2, 2, 3]))
    if kind == "cylinder3d":
        return _case(kind, log_int(9, 56), steps=1, mixed=mixed, relax=relax, gamma=gamma, state=state,
                     layers=rng.randint(3, 24))
    if kind == "ns":
        return _case(kind, log_int(24, 320), steps=1, relax=relax, state=state)
    if kind == "cfl":
        return _case(kind, log_int(24, 900), gamma=gamma, state=state, layers=0)
    return _case("serve", rng.randint(2, 12), steps=rng.randint(8, 24), mixed=mixed, state="inflow")


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

@functools.lru_cache(maxsize=6)
def _cylinder(m):
    return meshes.cylinder_channel_q1(m)


@functools.lru_cache(maxsize=3)
def _cylinder_p1(m):
    return meshes.cylinder_channel_p1(m)


@functools.lru_cache(maxsize=2)
def _cylinder3d(m, layers):
    return meshes.extruded_q1(meshes.cylinder_channel_q1(m), layers)


@functools.lru_cache(maxsize=2)
def _vortex_mesh(nv):
    return meshes.periodic_p1_square(nv)


@functools.lru_cache(maxsize=2)
def _nrbc_mesh(cells):
    return meshes.structured_q1(cells, cells, -1.0, 1.0, -1.0, 1.0, kinds=(meshes.BC_CHARACTERISTIC,) * 4)


@functools.lru_cache(maxsize=2)
def _parabolic(m):
    return meshes.parabolic_data(_cylinder(m))


@functools.lru_cache(maxsize=2)
def _sweep_mesh(count):
    sizes = np.exp(np.random.RandomState(4).uniform(math.log(8), math.log(16), count)).round().astype(int)
    parts = [_sweep_part(int(m)) for m in sizes]
    mesh, off, _ = meshes.concatenate(parts)
    return mesh, off


@functools.lru_cache(maxsize=16)
def _sweep_part(m):
    return meshes.cylinder_channel_q1(m)


def _mesh(case):
    kind, size = case["kind"], case["size"]
    if kind == "vortex":
        return _vortex_mesh(size)
    if kind == "nrbc":
        return _nrbc_mesh(size)
    if kind == "sweep":
        return _sweep_mesh(size)[0]
    if kind == "cylinder3d":
        return _cylinder3d(size, case["layers"])
    return _cylinder(size)


def _conserved(rho, vel, p, gamma):
    ke = sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [p / (gamma - 1.0) + 0.5 * rho * ke]).contiguous()


def _inflow(shape, dim, gamma, mach=None):
    one = torch.ones(shape, dtype=F64, device=DEV)
    u = INFLOW[1] if mach is None else mach
    return _conserved(INFLOW[0] * one, [u * one] + [0.0 * one] * (dim - 1), INFLOW[2] * one, gamma)


def _channel_state(mesh, kind, gamma, seed):
    """A state of the Mach-3 channel from the seed: "perturbed" (smooth bumps of
    density, pressure and velocity everywhere) or "shocked" (uniform ahead of a
    bow-shaped shock front, post-shock values and bumps of compact support
    behind it, and a band of the free stream that differs by a few ulps)."""
    rng = np.random.RandomState(seed % (1 << 31))
    x = torch.from_numpy(mesh.coords).to(DEV)
    rho0, u0, p0 = INFLOW
    dim = mesh.dim
    rho = torch.full((mesh.n,), rho0, dtype=F64, device=DEV)
    p = torch.full((mesh.n,), p0, dtype=F64, device=DEV)
    vel = [torch.full((mesh.n,), u0 if d == 0 else 0.0, dtype=F64, device=DEV) for d in range(dim)]
    lo, hi = mesh.coords.min(0), mesh.coords.max(0)
    if kind == "shocked":
        # normal shock relations at Mach 3 behind a parabolic front through x = 0.3
        m2, g = 9.0, gamma
        rr = (g + 1.0) * m2 / ((g - 1.0) * m2 + 2.0)
        pr = 1.0 + 2.0 * g / (g + 1.0) * (m2 - 1.0)
        front = rng.uniform(0.28, 0.32) + rng.uniform(1.5, 2.5) * (x[:, 1] - 0.5) ** 2
        behind = (x[:, 0] > front) & (x[:, 0] < front + rng.uniform(0.5, 0.9))
        rho = torch.where(behind, rho * rr, rho)
        p = torch.where(behind, p * pr, p)
        vel[0] = torch.where(behind, vel[0] / rr, vel[0])
    for _ in range(12):
        if kind == "shocked":
            c = [rng.uniform(0.5, 2.6)] + [rng.uniform(lo[d], hi[d]) for d in range(1, dim)]
            r = rng.uniform(0.15, 0.4)
        else:
            c = [rng.uniform(lo[d], hi[d]) for d in range(dim)]
            r = rng.uniform(0.12, 0.6)
        r2 = sum((x[:, d] - c[d]) ** 2 for d in range(dim)) / (r * r)
        g_ = torch.clamp(1.0 - r2, min=0.0) ** 3 if kind == "shocked" else torch.exp(-r2)
        rho = rho * (1.0 + 0.3 * rng.uniform(-0.9, 1.0) * g_)
        p = p * (1.0 + 0.3 * rng.uniform(-0.9, 2.0) * g_)
        for d in range(dim):
            vel[d] = vel[d] + 0.3 * rng.uniform(-2.0, 2.0) * g_
    if kind == "shocked":
        band = (x[:, 0] > 3.0) & (x[:, 0] < 3.4)
        k = torch.from_numpy(rng.randint(-3, 4, mesh.n).astype(np.float64)).to(DEV)
        rho = torch.where(band, rho * (1.0 + k * 2.0 ** -52), rho)
    return _conserved(rho, vel, p, gamma)


def _inputs(case, seed):
    """(mesh, U0 on the GPU, boundary states or None, row offsets or None)."""
    kind, gamma = case["kind"], case["gamma"]
    mesh = _mesh(case)
    rng = np.random.RandomState(seed % (1 << 31))
    x = torch.from_numpy(mesh.coords).to(DEV)
    off = None
    if kind == "vortex":
        # Yee's vortex of seeded strength at a seeded place of the periodic box
        beta, cx, cy = rng.uniform(4.0, 6.0), rng.uniform(-1.0, 1.0), rng.uniform(-1.0, 1.0)
        dx = torch.remainder(x[:, 0] - cx + 5.0, 10.0) - 5.0
        dy = torch.remainder(x[:, 1] - cy + 5.0, 10.0) - 5.0
        r2 = dx * dx + dy * dy
        du = beta / (2.0 * math.pi) * torch.exp(0.5 * (1.0 - r2))
        T = 1.0 - (gamma - 1.0) * beta * beta / (8.0 * gamma * math.pi ** 2) * torch.exp(1.0 - r2)
        rho = T ** (1.0 / (gamma - 1.0))
        return mesh, _conserved(rho, [1.0 - du * dy, 1.0 + du * dx], rho * T, gamma), None, None
    if kind == "nrbc":
        mach, vbar, r0 = 0.5, rng.uniform(0.25, 0.75), 0.1
        dx, dy = x[:, 0] - rng.uniform(0.6, 0.9), x[:, 1] - rng.uniform(-0.2, 0.2)
        psi = torch.exp(0.5 * (1.0 - (dx * dx + dy * dy) / (r0 * r0)))
        p_inf = (1.0 / mach) ** 2 / gamma
        one = torch.ones_like(dx)
        U = _conserved(one, [1.0 - vbar / r0 * psi * dy, vbar / r0 * psi * dx], p_inf - 0.5 * (vbar * psi) ** 2, gamma)
        ob = torch.ones(mesh.n_bnd, dtype=F64, device=DEV)
        return mesh, U, _conserved(ob, [ob, 0.0 * ob], p_inf * ob, gamma), None
    if kind == "sweep":
        mesh, off = _sweep_mesh(case["size"])
        mach = torch.from_numpy(np.repeat(rng.uniform(1.5, 4.0, off.size - 1), np.diff(off))).to(DEV)
        U = _inflow(mesh.n, 2, gamma, mach)
        bs = U[:, torch.from_numpy(mesh.bnd_node).long().to(DEV)].contiguous()
        g_ = torch.exp(-((x[:, 0] - rng.uniform(1.0, 3.0)) ** 2 + (x[:, 1] - 0.5) ** 2) / 0.2)
        U = U * (1.0 + 0.2 * g_)
    else:
        U = _channel_state(mesh, case["state"], gamma, seed)
        bs = _inflow(mesh.n_bnd, mesh.dim, gamma)
        if kind == "ns":
            wall = torch.from_numpy(mesh.bnd_node[mesh.bnd_kind == meshes.BC_SLIP]).long().to(DEV)
            ke = 0.5 * (U[1, wall] ** 2 + U[2, wall] ** 2) / U[0, wall]
            U[3, wall] -= ke
            U[1:3, wall] = 0.0
    return mesh, _Boundary(mesh, bs, gamma).apply(U).contiguous(), bs, off


def _wall(mesh):
    return mesh.bnd_node[mesh.bnd_kind == meshes.BC_SLIP]


NS_MU, NS_KC = 1e-4, 1.4e-4


def _requests(case, seed):
    """Serve requests: P1 and Q1 cylinders of 1e4 to 6e4 vertices, uniform
    inflow at a seeded Mach number, all to one final time."""
    rng = np.random.RandomState(seed % (1 << 31))
    reqs = []
    for k in range(case["size"]):
        p1 = k % 2 == 1
        m = (45, 64, 90, 110)[(k // 2) % 4]
        mesh = _cylinder_p1(m) if p1 else _cylinder(m)
        U = _inflow(mesh.n, 2, case["gamma"], rng.uniform(1.5, 4.0)).cpu().numpy()
        reqs.append(serve.Request(mesh, U, np.ascontiguousarray(U[:, mesh.bnd_node]), case["steps"] * 2.5e-4, 0.0, f"r{k}"))
    return reqs


def prepare(case, seed):
    kind = case["kind"]
    precision = binding.EH_PRECISION_MIXED if case["mixed"] else binding.EH_PRECISION_FP64
    if kind == "serve":
        # the requests are host data by nature: they arrive from outside and are admitted one by one
        server = serve.SolveServer(8 << 30, precision=precision)
        return dict(kind=kind, server=server, requests=_requests(case, seed))
    mesh, U, bs, off = _inputs(case, seed)
    if kind == "cfl":
        row_ptr = torch.from_numpy(mesh.row_ptr).to(DEV)
        isb = torch.zeros(mesh.n, dtype=torch.uint8, device=DEV)
        isb[torch.from_numpy(mesh.bnd_node).long().to(DEV)] = 1
        return dict(kind=kind, args=(mesh.dim, case["gamma"], case["cfl"], row_ptr, torch.from_numpy(mesh.col).to(DEV),
                                     torch.from_numpy(mesh.cij).to(DEV), torch.from_numpy(mesh.mi).to(DEV), isb, U),
                    dt=torch.zeros(1, dtype=F64, device=DEV))
    s = binding.Solver(dim=mesh.dim, gamma=case["gamma"], cfl=case["cfl"], limiter_passes=case["passes"],
                       bound_relaxation=case["relax"], precision=precision)
    s.upload_mesh(mesh, None if bs is None else bs.cpu().numpy())
    if off is not None:
        s.set_instances(off)
    if kind == "ns":
        s.set_viscosity(_parabolic(case["size"]), NS_MU, 0.0, NS_KC, wall=_wall(mesh))
    return dict(kind=kind, solver=s, U0=U, out=torch.empty_like(U), steps=case["steps"])


def run(state):
    kind = state["kind"]
    if kind == "serve":
        done = {r.name: r for r in state["server"].run(state["requests"])}
        return {k: {"U": done[k].U, "t": done[k].t, "steps": done[k].steps} for k in sorted(done)}
    if kind == "cfl":
        binding.cfl_dt_noalloc(*state["args"], state["dt"], stream=torch.cuda.current_stream())
        return state["dt"]
    s = state["solver"]
    s.set_state(state["U0"])
    if kind == "ns":
        tau, _ = s.step_ns()
        return {"U": s.get_state(state["out"]), "tau": tau}
    s.run(state["steps"])
    return s.get_state(state["out"])


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _stage_work(n, nnz, dim):
    """Bytes and operations of one forward-Euler stage: the static edge data
    read once (c_ij, m_ij and the column per entry, m_i per node), the state
    read and written once; operations counted once from the method's formulas
    (+, -, x, /, sqrt and each elementary function = 1)."""
    d, S = dim, dim + 2
    e = nnz - n
    check = S + 2 * d + 6
    node = (d * d + 9 * d + 25) + 1 + 3 + (2 * S + 2) + 2 + 3 * S
    entry = ((7 * d + 20) / 2.0 + S * (3 * d - 1) + (3 * d - 1) + (2 * S - 1) + 4 + (7 * S + 1) + (4 * S + 3) + 1
             + (6 * S + 3) + check + 3 * S + (S + 1) + check + 3 * S)
    return (8 * d + 8 + 4) * nnz + (2 * 8 * S + 8 + 4) * n, entry * e + node * n


def work(case):
    kind = case["kind"]
    if kind == "serve":
        b = f = 0.0
        for k in range(case["size"]):
            m = (45, 64, 90, 110)[(k // 2) % 4]
            mesh = _cylinder_p1(m) if k % 2 else _cylinder(m)
            sb, sf = _stage_work(mesh.n, mesh.nnz, 2)
            b += 3 * case["steps"] * sb
            f += 3 * case["steps"] * sf
        return {"bytes": b, "flops": f}
    mesh = _mesh(case)
    n, nnz, d = mesh.n, mesh.nnz, mesh.dim
    if kind == "cfl":
        # c_ij and the column per entry, the state and m_i per node; the wave-speed bound once per edge
        return {"bytes": (8 * d + 4) * nnz + (8 * (d + 2) + 8 + 8 + 1) * n,
                "flops": (nnz - n) / 2.0 * (7 * d + 20) + n * (3 * d + 12)}
    sb, sf = _stage_work(n, nnz, d)
    b, f = 3.0 * case["steps"] * sb, 3.0 * case["steps"] * sf
    if kind == "ns":
        # two hyperbolic steps, and of the parabolic one the operators (L; the 2 x 2 velocity blocks) and the
        # cells' quadrature read once
        nc = mesh.cells.shape[0]
        b, f = 2 * b + 44 * nnz + 8 * 4 * (1 + 4 + 8) * nc + 2 * 32 * n, 2 * f + 10 * nnz + 4 * 60 * nc
    return {"bytes": b, "flops": f}


# --------------------------------------------------------------------------
# the method in plain tensor operations, 64 bits
# --------------------------------------------------------------------------

class _Boundary:
    def __init__(self, mesh, bs, gamma):
        self.node = torch.from_numpy(mesh.bnd_node).long().to(DEV)
        self.kind = torch.from_numpy(mesh.bnd_kind).long().to(DEV)
        self.normal = torch.from_numpy(mesh.bnd_normal).to(DEV)
        self.bs, self.gamma, self.dim = bs, gamma, mesh.dim

    def apply(self, U):
        if self.node.numel() == 0:
            return U
        U, d, g = U.clone(), self.dim, self.gamma
        for kind in torch.unique(self.kind).tolist():
            sel = self.kind == kind
            i, nv = self.node[sel], self.normal[:, sel]
            if kind == meshes.BC_SLIP:
                U[1:1 + d, i] -= (U[1:1 + d, i] * nv).sum(0) * nv
            elif kind == meshes.BC_DIRICHLET:
                U[:, i] = self.bs[:, sel]
            elif kind == meshes.BC_CHARACTERISTIC:
                U[:, i] = self._characteristic(U[:, i], nv, self.bs[:, sel], d, g)
        return U

    @staticmethod
    def _normal(u, nv, d, g):
        v = u[1:1 + d] / u[0]
        un = (v * nv).sum(0)
        p = (g - 1.0) * (u[1 + d] - 0.5 * u[0] * (v * v).sum(0))
        return u[0], un, v - un * nv, p, torch.sqrt(g * p / u[0])

    def _characteristic(self, u, nv, ud, d, g):
        rho, un, ut, p, a = self._normal(u, nv, d, g)
        rf, unf, utf, pf, af = self._normal(ud, nv, d, g)
        inflow = un < 0.0
        c3, c1 = un + 2.0 * a / (g - 1.0), unf - 2.0 * af / (g - 1.0)
        ent = torch.where(inflow, pf * rf ** -g, p * rho ** -g)
        t = torch.where(inflow, utf, ut)
        ap, vn = 0.25 * (g - 1.0) * (c3 - c1), 0.5 * (c1 + c3)
        rp = (ap * ap / (g * ent)) ** (1.0 / (g - 1.0))
        v = t + vn * nv
        w = torch.cat([rp[None], rp * v, (ent * rp ** g / (g - 1.0) + 0.5 * rp * (v * v).sum(0))[None]])
        w = torch.where(inflow & (-un > a), ud, w)
        return torch.where(~inflow & (un >= a), u, w)


class _Reference:
    """One mesh with its off-diagonal entries (i, j) in row order. State
    vectors are [S, n], entry arrays [.., E]."""

    def __init__(self, mesh, bs, case, off=None):
        self.d, self.S, self.n = mesh.dim, mesh.dim + 2, mesh.n
        self.g, self.cfl, self.passes = case["gamma"], case["cfl"], case["passes"]
        rows = np.repeat(np.arange(mesh.n, dtype=np.int64), np.diff(mesh.row_ptr))
        keep = rows != mesh.col
        self.row = torch.from_numpy(rows[keep]).to(DEV)
        self.col = torch.from_numpy(mesh.col[keep].astype(np.int64)).to(DEV)
        self.tr = torch.searchsorted(self.row * mesh.n + self.col, self.col * mesh.n + self.row)
        self.c = torch.from_numpy(np.ascontiguousarray(mesh.cij[:, keep])).to(DEV)
        self.mij = torch.from_numpy(mesh.mij[keep]).to(DEV)
        self.mi = torch.from_numpy(mesh.mi).to(DEV)
        self.len = torch.from_numpy(np.diff(mesh.row_ptr) - 1).to(DEV)
        isb = torch.zeros(mesh.n, dtype=torch.bool, device=DEV)
        isb[torch.from_numpy(mesh.bnd_node).long().to(DEV)] = True
        self.both = isb[self.row] & isb[self.col]
        self.bnd = _Boundary(mesh, bs, self.g)
        k = 1 if off is None else off.size - 1
        self.inst = (torch.zeros(mesh.n, dtype=torch.long, device=DEV) if off is None else
                     torch.from_numpy(np.repeat(np.arange(k), np.diff(off))).to(DEV))
        self.ninst = k
        area = torch.zeros(k, dtype=F64, device=DEV).index_add_(0, self.inst, self.mi)
        self.relax = (self.mi / area[self.inst]) ** (1.5 / self.d) if case["relax"] else torch.zeros_like(self.mi)

    def rows(self, e, how="sum"):
        """Reduction of an entry array over every row."""
        if e.dim() == 2:
            return torch.stack([self.rows(x, how) for x in e])
        return torch.segment_reduce(e, how, lengths=self.len, axis=0, unsafe=True)

    def pressure(self, U):
        return (self.g - 1.0) * (U[self.d + 1] - 0.5 * (U[1:1 + self.d] ** 2).sum(0) / U[0])

    def wave_speed(self, ul, pl, al, ur, pr, ar):
        g = self.g
        z = (g - 1.0) / (2.0 * g)
        num = torch.clamp(al + ar - 0.5 * (g - 1.0) * (ur - ul), min=0.0)
        ptr = (num / (al * pl ** -z + ar * pr ** -z)) ** (1.0 / z)
        k = (g + 1.0) / (2.0 * g)
        l1 = ul - al * torch.sqrt(1.0 + k * torch.clamp(ptr - pl, min=0.0) / pl)
        l3 = ur + ar * torch.sqrt(1.0 + k * torch.clamp(ptr - pr, min=0.0) / pr)
        return torch.maximum(torch.clamp(-l1, min=0.0), torch.clamp(l3, min=0.0))

    def viscosity(self, U):
        """d_ij per entry and the CFL step per instance."""
        i, j = self.row, self.col
        v, p = U[1:1 + self.d] / U[0], self.pressure(U)
        a = torch.sqrt(self.g * p / U[0])
        cn = (self.c ** 2).sum(0).sqrt()
        nv = self.c / cn
        d = self.wave_speed((v[:, i] * nv).sum(0), p[i], a[i], (v[:, j] * nv).sum(0), p[j], a[j]) * cn
        dt = d[self.tr]
        d = torch.where(self.both, torch.maximum(d, dt), torch.where(i < j, d, dt))
        bound = self.cfl * self.mi / (2.0 * self.rows(d))
        tau = torch.full((self.ninst,), math.inf, dtype=F64, device=DEV)
        return d, tau.scatter_reduce(0, self.inst, bound, "amin")

    def psi(self, u, P, l, phi):
        w = u + l * P
        return w[-1] - 0.5 * (w[1:-1] ** 2).sum(0) / w[0] - phi * w[0] ** self.g

    def line_search(self, U, P, b):
        """The largest l in [0, 1] that keeps the row's bounds, per entry."""
        lim = torch.ones_like(P[0])
        at = torch.nonzero((P != 0.0).any(0))[:, 0]
        i, P = self.row[at], P[:, at]
        u, rmin, rmax, phi = U[:, i], b[0][i], b[1][i], b[2][i]
        room = torch.where(P[0] > 0.0, rmax - u[0], rmin - u[0])
        l = torch.where(P[0] != 0.0, torch.clamp(room / torch.where(P[0] != 0.0, P[0], 1.0), 0.0, 1.0), 1.0)
        pr = self.psi(u, P, l, phi)
        pl = self.psi(u, P, torch.zeros_like(l), phi)
        l = torch.where((pr < 0.0) & (pl <= 0.0), 0.0, l)
        it = torch.nonzero((pr < 0.0) & (pl > 0.0))[:, 0]
        if it.numel():
            u, P, phi, lR, pl, pr = u[:, it], P[:, it], phi[it], l[it], pl[it], pr[it]
            lL = torch.zeros_like(lR)
            for _ in range(6):
                ls = lL + pl * (lR - lL) / (pl - pr)
                w = u + lR * P
                v = w[1:-1] / w[0]
                dr = (P[-1] - (v * P[1:-1]).sum(0) + 0.5 * (v * v).sum(0) * P[0]
                      - phi * self.g * w[0] ** (self.g - 1.0) * P[0])
                ln = torch.where(dr < 0.0, lR - pr / torch.where(dr < 0.0, dr, -1.0), lR)
                ln = torch.maximum(ln, ls)
                ps, pn = self.psi(u, P, ls, phi), self.psi(u, P, ln, phi)
                lL, pl = torch.where(ps >= 0.0, ls, lL), torch.where(ps >= 0.0, ps, pl)
                lR, pr, lL, pl = (torch.where(pn < 0.0, ln, lR), torch.where(pn < 0.0, pn, pr),
                                  torch.where(pn < 0.0, lL, ln), torch.where(pn < 0.0, pl, pn))
            l = l.clone()
            l[it] = lL
        lim[at] = l
        return lim

    def euler(self, U, tau):
        """One forward-Euler stage (Algorithm 1); tau: per instance, or None for the CFL step."""
        i, j, g, d = self.row, self.col, self.g, self.d
        dij, bound = self.viscosity(U)
        tau = bound if tau is None else tau
        tn = tau[self.inst]
        v, p = U[1:1 + d] / U[0], self.pressure(U)
        eps = p / (g - 1.0)
        phi = eps * U[0] ** -g
        s = torch.log(phi) / (g - 1.0)
        eta = -U[0] * s
        dU = U[:, j] - U[:, i]
        vjc, vic = (v[:, j] * self.c).sum(0), (v[:, i] * self.c).sum(0)
        dv = vjc - vic
        w = torch.stack([(dU[1:1 + d] * self.c).sum(0)]
                        + [dU[1 + q] * vjc + U[1 + q][i] * dv + (p[j] - p[i]) * self.c[q] for q in range(d)]
                        + [(dU[d + 1] + p[j] - p[i]) * vjc + (U[d + 1] + p)[i] * dv])
        a = (eta[j] - eta[i]) * vjc + eta[i] * dv
        g1 = U[0] / ((g - 1.0) * eps)
        deta = torch.cat([(-s - U[0] / (g - 1.0) * ((v * v).sum(0) / (2.0 * eps) - g / U[0]))[None], g1 * v, -g1[None]])
        b = (deta[:, i] * w).sum(0)
        N, D = self.rows(a - b).abs(), self.rows(a.abs() + b.abs())
        alpha = torch.where(D > 0.0, N / torch.where(D > 0.0, D, 1.0), 0.0)
        dH = 0.5 * (alpha[i] + alpha[j]) * dij
        UL = U + tn / self.mi * self.rows(dij * dU - w)
        G = self.rows(dH * dU - w) / self.mi
        rbar = 0.5 * (U[0][i] + U[0][j]) - w[0] / (2.0 * dij)
        bounds = torch.stack([(1.0 - self.relax) * torch.minimum(U[0], self.rows(rbar, "min")),
                              (1.0 + self.relax) * torch.maximum(U[0], self.rows(rbar, "max")),
                              (1.0 - self.relax) * torch.minimum(phi, self.rows(phi[j], "min"))])
        count = self.len[i].to(F64)
        P = tn[i] * count / self.mi[i] * (self.mij * (G[:, i] - G[:, j]) + (dH - dij) * dU)
        W, l = UL, self.line_search(UL, P, bounds)
        for k in range(self.passes):
            l = torch.minimum(l, l[self.tr])
            W = W + self.rows(l * P / count)
            if k + 1 < self.passes:
                P = (1.0 - l) * P
                l = self.line_search(W, P, bounds)
        return W, tau

    def step(self, U, left=None, tau=None):
        """One SSPRK(3,3) step; left: the time to the end, which shortens the step."""
        if tau is None:
            tau = self.viscosity(U)[1]
        if left is not None:
            tau = torch.clamp(tau, max=left)
        w = self.bnd.apply(self.euler(U, tau)[0])
        w = U + 0.25 * (self.bnd.apply(self.euler(w, tau)[0]) - U)
        return U + 2.0 / 3.0 * (self.bnd.apply(self.euler(w, tau)[0]) - U), tau

    # the parabolic sub-step (2D): Crank-Nicolson velocity and internal energy
    def parabolic(self, U, dt, data, wall, mu, kc):
        t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
        rows, col = self._all
        L, G = t(data["L"]), t(data["G"])
        lm = -2.0 * mu / 3.0
        isw = torch.zeros(self.n, dtype=torch.bool, device=DEV)
        isw[t(wall).long()] = True
        A = [[(mu * L if a == b else 0.0) + mu * G[b, a] + lm * G[a, b] for b in range(2)] for a in range(2)]
        A = [[torch.where(isw[col], 0.0, x) for x in r] for r in A]
        D = U[0] * self.mi
        V = U[1:3] / U[0]
        diag = rows == col
        at = rows[diag]

        def total(e):
            return torch.segment_reduce(e, "sum", lengths=self.len + 1, axis=0, unsafe=True)

        def velocity(x):
            y = torch.stack([D * x[a] + 0.5 * dt * total(A[a][0] * x[0][col] + A[a][1] * x[1][col]) for a in range(2)])
            return torch.where(isw, x, y)

        pd = torch.stack([torch.where(isw, 1.0, D + 0.5 * dt * torch.zeros_like(D).index_copy(0, at, A[a][a][diag]))
                          for a in range(2)])
        Vh = self._pcg(velocity, torch.where(isw, 0.0, D * V), torch.where(isw, 0.0, V), pd)
        cells, qw, qphi, qgrad = t(data["cells"]).long(), t(data["qw"]), t(data["qphi"]), t(data["qgrad"])
        vc = Vh[:, cells]                                       # [2, nc, nv]
        Dv = torch.einsum("kca,cqma->cqkm", vc, qgrad)
        E = 0.5 * (Dv + Dv.transpose(-1, -2))
        div = Dv[..., 0, 0] + Dv[..., 1, 1]
        se = 2.0 * mu * (E * E).sum((-1, -2)) + lm * div * div
        share = torch.einsum("cq,cqa,cq->ca", qw, qphi, se)
        mK = torch.zeros_like(D).index_add_(0, cells.reshape(-1), share.reshape(-1))
        en = U[3] / U[0] - 0.5 * (V * V).sum(0)
        Ld = torch.zeros_like(D).index_copy(0, at, L[diag])
        c = 0.5 * dt * kc
        eh = self._pcg(lambda x: D * x + c * total(L * x[col]), D * en + 0.5 * dt * mK, en.clone(), D + c * Ld)
        eH, Vn = 2.0 * eh - en, 2.0 * Vh - V
        if bool((eH <= 0.0).any()):
            return None  # the limited branch
        return torch.stack([U[0], U[0] * Vn[0], U[0] * Vn[1], U[0] * eH + 0.5 * U[0] * (Vn * Vn).sum(0)])

    @staticmethod
    def _pcg(apply, b, x, pd):
        r = b - apply(x)
        z = r / pd
        p, rz, stop = z, (r * z).sum(), 1e-15 * b.norm()
        for _ in range(60):
            if float(r.norm()) <= float(stop) or float(rz) == 0.0:
                break
            q = apply(p)
            al = rz / (p * q).sum()
            x, r = x + al * p, r - al * q
            z = r / pd
            new = (r * z).sum()
            p, rz = z + new / rz * p, new
        return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        out = {}
        for q in _requests(case, seed):
            bs = torch.from_numpy(q.bnd_state).to(DEV)
            ref = _Reference(q.mesh, bs, case)
            U, t = ref.bnd.apply(torch.from_numpy(q.U0).to(DEV)), 0.0
            while t < q.t_final:
                U, tau = ref.step(U, left=q.t_final - t)
                t += float(tau[0])
            out[q.name] = {"U": U, "t": t, "steps": None}
        return {k: out[k] for k in sorted(out)}
    mesh, U, bs, off = _inputs(case, seed)
    ref = _Reference(mesh, bs, case, off)
    if kind == "cfl":
        return ref.viscosity(U)[1]
    if kind == "ns":
        rows = np.repeat(np.arange(mesh.n, dtype=np.int64), np.diff(mesh.row_ptr))
        ref._all = (torch.from_numpy(rows).to(DEV), torch.from_numpy(mesh.col.astype(np.int64)).to(DEV))
        U, tau = ref.step(U)
        U = ref.parabolic(U, 2.0 * float(tau[0]), _parabolic(case["size"]), _wall(mesh), NS_MU, NS_KC)
        if U is None:
            return None
        return {"U": ref.step(U, tau=tau)[0], "tau": float(tau[0])}
    for _ in range(case["steps"]):
        U = ref.step(U)[0]
    return U
