"""Performance cases: what programs have this solver do, through its public
entry points (Mesh.set_rhs / set_initial / solve / vcycle / fmg_solve /
get_solution and autograd.stokes_solve), on device-resident data.

A case is a dict of plain values:
  kind      "solve" (set_rhs + solve to 1e-8 from zero), "fmg" (full
            multigrid), "vcycle" (cycles on a given iterate) or "adjoint"
            (differentiable solve and its backward pass)
  nx ny nz  unit cubes of the macro mesh, 6 tetrahedra each
  level     regular refinements: nodes per axis = cells * 2**level + 1
  fp32      FP32 V-cycles inside FP64 refinement, else plain FP64
  d_form    symmetric-gradient operator instead of the Laplace form
  outflow   inflow on x = 0 and do-nothing outflow on x = nx (a channel),
            else Dirichlet data on every face
  obstacles number of seeded interior cubes left out (0: none)
  slip      the obstacles' faces are free-slip faces
  sheared   the lattice axes are not orthogonal

Several right-hand sides are solved on one hierarchy, as a time loop, an
optimisation or a parameter study does: prepare() makes the inputs and output
buffers and keeps the most recently used Mesh.  Nothing else outlives a call.

exact() computes the discrete solution itself: a matrix-free element-by-element
operator on the tetrahedra and conjugate gradients on the pressure Schur
complement, in 64 bits with plain torch.
"""
import itertools
import math
import random

import numpy as np
import torch

import paper_1511_02134_gb300 as hhg
import workloads as W
from paper_1511_02134_gb300.autograd import stokes_solve

SHEAR = W.SHEAR


def _case(name, kind, cells, level, fp32, **more):
    c = {"name": name, "kind": kind, "nx": cells[0], "ny": cells[1], "nz": cells[2], "level": level, "fp32": fp32,
         "d_form": False, "outflow": False, "obstacles": 0, "slip": False, "sheared": False}
    c.update(more)
    return c


def listed():
    one, channel = (1, 1, 1), (16, 4, 4)
    return [
        # a small problem solved many times: latency of launches and of the coarse solve
        _case("cube4_fp64", "solve", one, 4, False),
        # a mid-size solve of an interactive or outer-loop use
        _case("cube6_ir", "solve", one, 6, True),
        # the paper's serial problem (8.3e6 unknowns) in both precision modes
        _case("cube7_ir", "solve", one, 7, True),
        _case("cube7_fp64", "solve", one, 7, False),
        # the largest cube: 5.4e8 unknowns, the headline solve
        _case("cube9_ir", "solve", one, 9, True),
        # flow past obstacles, the application run: 2.6e8 unknowns
        _case("channel6_ir", "solve", channel, 6, True, outflow=True, obstacles=6),
        # the same with free-slip obstacles, a quick parameter-study size
        _case("slip_channel4_ir", "solve", channel, 4, True, outflow=True, obstacles=6, slip=True),
        # gradient of an outflow functional with respect to the body force
        _case("channel4_adjoint", "adjoint", channel, 4, False, outflow=True, obstacles=6),
        # full multigrid, two cycles per level: the discretisation error in one pass
        _case("cube8_fmg_ir", "fmg", one, 8, True),
        # symmetric-gradient operator (variable-viscosity and traction problems start from it)
        _case("cube6_dform_ir", "solve", one, 6, True, d_form=True),
        # a lattice that is not axis-aligned: every node takes its stencil-class rows
        _case("sheared6_ir", "solve", (1, 1, 1), 6, True, sheared=True),
        # cycles as a smoother or preconditioner on an iterate of the caller's, ragged box with an obstacle
        _case("box4_vcycle", "vcycle", (5, 3, 3), 4, False, obstacles=1),
    ]


def _nodes(c):
    return math.prod(c[a] * 2 ** c["level"] + 1 for a in ("nx", "ny", "nz"))


def draw(rng):
    while True:
        kind = rng.choice(["solve"] * 6 + ["fmg", "vcycle", "vcycle", "adjoint"])
        fp32 = kind in ("solve", "fmg") and rng.random() < 0.65
        c = _case("", kind, (1, 1, 1), 0, fp32)
        del c["name"]
        if kind == "adjoint" or (kind == "solve" and rng.random() < 0.3):
            big = kind == "solve"
            c.update(nx=rng.randint(3, 16 if big else 8), ny=rng.randint(3, 5 if big else 4), nz=rng.randint(3, 5 if big else 4),
                     outflow=True)
            c["obstacles"] = rng.randint(0, 5)
            c["slip"] = big and c["obstacles"] > 0 and rng.random() < 0.4
        else:
            c.update(nx=rng.randint(1, 5), ny=rng.randint(1, 4), nz=rng.randint(1, 3))
            if min(c["nx"], c["ny"], c["nz"]) == 3 and rng.random() < 0.5:
                c["obstacles"] = 1
            r = rng.random()
            c["sheared"] = kind == "solve" and not c["obstacles"] and r < 0.15
            c["d_form"] = kind == "solve" and not c["sheared"] and r > 0.85
        # nodes, spread over the logarithm
        most = 3e5 if kind == "adjoint" else 2e6 if c["d_form"] or c["sheared"] or not fp32 else 1.7e7
        target = math.exp(rng.uniform(math.log(3e3), math.log(most)))
        c["level"] = 3
        while _nodes(dict(c, level=c["level"] + 1)) <= target:
            c["level"] += 1
        if _nodes(c) <= most:
            return c


# ---- geometry ------------------------------------------------------------------

def _removed(c):
    interior = list(itertools.product(range(1, c["nx"] - 1), range(1, c["ny"] - 1), range(1, c["nz"] - 1)))
    if not c["obstacles"] or not interior:
        return ()
    order = np.random.default_rng(0).permutation(len(interior))
    return tuple(sorted(interior[m] for m in order[:c["obstacles"]]))


def _macro(c):
    m = W.box_of_cubes(c["nx"], c["ny"], c["nz"], removed=_removed(c), outflow_x_max=c["outflow"],
                       slip_obstacles=c["slip"])
    if c["sheared"]:
        m.vertices = m.vertices @ SHEAR.T
        m.basis = SHEAR.copy()
    return m


def _dims(c):
    return tuple(c[a] * 2 ** c["level"] + 1 for a in ("nx", "ny", "nz"))


_kept = {}


def _mesh(c):
    """The hierarchy of the case's mesh; the last one made is kept."""
    key = tuple(sorted((k, v) for k, v in c.items() if k not in ("name", "kind", "fp32")))
    if key not in _kept:
        _kept.clear()
        m = _macro(c)
        opts = {}
        if c["nx"] * c["ny"] * c["nz"] > 1:
            opts = {"coarsest_level": 1, "coarse_minres_max": 300}
        _kept[key] = hhg.Mesh(m.vertices, m.tets, m.bc_flags, c["level"], operator_form=int(c["d_form"]), **opts)
    return _kept[key]


def _coords(c, dev):
    """Physical coordinates as arrays that broadcast to (nz, ny, nx)."""
    h = 1.0 / 2 ** c["level"]
    nx, ny, nz = _dims(c)
    x = h * torch.arange(nx, dtype=torch.float64, device=dev).view(1, 1, nx)
    y = h * torch.arange(ny, dtype=torch.float64, device=dev).view(1, ny, 1)
    z = h * torch.arange(nz, dtype=torch.float64, device=dev).view(nz, 1, 1)
    return (x + y, y, z) if c["sheared"] else (x, y, z)


def _inputs(c, seed, dev):
    """Nodal body force and Dirichlet data, both (n, 3): a smooth trigonometric
    flow with its forcing (amplitudes and phases from the seed), or the inflow
    profile of a channel with a smooth force; for gradients N(0,1) forces."""
    r = random.Random(seed)
    nx, ny, nz = _dims(c)
    x, y, z = _coords(c, dev)
    f = torch.empty((nz, ny, nx, 3), dtype=torch.float64, device=dev)
    ud = torch.zeros((nz, ny, nx, 3), dtype=torch.float64, device=dev)
    amp = [r.uniform(0.6, 1.4) for _ in range(4)]
    ph = [r.uniform(-1.0, 1.0) for _ in range(6)]
    wave = (-4.0 * amp[0] * torch.cos(4.0 * z + ph[0]), 8.0 * amp[1] * torch.cos(8.0 * x + ph[1]),
            -2.0 * amp[2] * torch.cos(2.0 * y + ph[2]))
    if c["kind"] == "adjoint":
        g = torch.Generator(device=dev).manual_seed(seed)
        f.normal_(generator=g)
    else:
        sx, cx = torch.sin(4.0 * x + ph[3]), torch.cos(4.0 * x + ph[3])
        sy, cy = torch.sin(8.0 * y + ph[4]), torch.cos(8.0 * y + ph[4])
        sz, cz = torch.sin(2.0 * z + ph[5]), torch.cos(2.0 * z + ph[5])
        f[..., 0] = 16.0 * wave[0] + amp[3] * 4.0 * cx * sy * sz
        f[..., 1] = 64.0 * wave[1] + amp[3] * 8.0 * sx * cy * sz
        f[..., 2] = 4.0 * wave[2] + amp[3] * 2.0 * sx * sy * cz
    if c["outflow"]:
        if c["kind"] != "adjoint":
            f *= 0.01
        by, bz = float(c["ny"]), float(c["nz"])
        prof = (y * (by - y)) * (z * (bz - z)) * (16.0 / (by * by * bz * bz))
        ud[:, :, 0, 0] = amp[0] * prof[:, :, 0]
    else:
        for d in range(3):
            ud[..., d] = wave[d]
        for (i, j, k) in _removed(c):  # obstacles at rest
            N = 2 ** c["level"]
            ud[k * N:(k + 1) * N + 1, j * N:(j + 1) * N + 1, i * N:(i + 1) * N + 1] = 0.0
    return f.view(-1, 3), ud.view(-1, 3)


def _functional(c, seed, dev):
    """Weights of a linear functional of the outflow velocity, (n, 3)."""
    r = random.Random(seed + 77)
    nx, ny, nz = _dims(c)
    _, y, z = _coords(c, dev)
    h = 1.0 / 2 ** c["level"]
    ju = torch.zeros((nz, ny, nx, 3), dtype=torch.float64, device=dev)
    psi = (r.uniform(0.5, 1.5) + torch.sin(y + r.uniform(0, 3))) * (r.uniform(0.5, 1.5) + torch.cos(z + r.uniform(0, 3)))
    ju[:, :, -1, 0] = h * h * psi[:, :, 0]
    ju[:, :, -1, 1] = 0.3 * h * h * psi[:, :, 0]
    return ju.view(-1, 3)


def prepare(case, seed):
    dev = torch.device("cuda")
    mesh = _mesh(case)
    f, ud = _inputs(case, seed, dev)
    n = f.shape[0]
    s = {"case": case, "mesh": mesh, "f": f, "ud": ud, "mode": hhg.MODE_FP32_IR if case["fp32"] else hhg.MODE_FP64}
    if case["kind"] == "adjoint":
        s["f"].requires_grad_(True)
        s["ju"] = _functional(case, seed, dev)
        s["jp"] = torch.zeros(n, dtype=torch.float64, device=dev)
    else:
        s["u"] = torch.empty((n, 3), dtype=torch.float64, device=dev)
        s["p"] = torch.empty((n,), dtype=torch.float64, device=dev)
    if case["kind"] == "vcycle":
        # the paper's start: u_0 ~ U[0, 1], p_0 ~ U[0, 1/h]
        g = torch.Generator(device=dev).manual_seed(seed + 1)
        s["u0"] = torch.rand((n, 3), dtype=torch.float64, device=dev, generator=g)
        s["p0"] = torch.rand((n,), dtype=torch.float64, device=dev, generator=g) * 2.0 ** case["level"]
    return s


def run(s):
    mesh, kind = s["mesh"], s["case"]["kind"]
    if kind == "adjoint":
        u, p = stokes_solve(s["f"], mesh, s["ud"], tol=1e-8, max_cycles=60, mode=s["mode"])
        (grad,) = torch.autograd.grad([u, p], [s["f"]], [s["ju"], s["jp"]])
        return {"u": u.detach(), "p": p.detach(), "grad": grad}
    if kind == "fmg":
        mesh.fmg_solve(s["f"], s["ud"], cycles=2, nu=2, mode=s["mode"], u_out=s["u"], p_out=s["p"])
    elif kind == "vcycle":
        mesh.set_rhs(s["f"], s["ud"])
        mesh.set_initial(s["u0"], s["p0"])
        mesh.vcycle(2)
        mesh.get_solution(s["u"], s["p"])
    else:
        mesh.set_rhs(s["f"], s["ud"])
        mesh.solve(tol=1e-8, max_cycles=60, mode=s["mode"], u_out=s["u"], p_out=s["p"])
    return {"u": s["u"], "p": s["p"]}


def work(case):
    """Bytes: the nodal inputs read and outputs written once.  Operations: those
    of the multigrid cycles of one pass, counted per lattice node of the finest
    level (a smoothing step applies A twice, B, B^T and C once; the coarser
    levels of V_var add a quarter)."""
    n = _nodes(case)
    step = (2 * 3 * 14 if not case["d_form"] else 2 * 9 * 30) + 84 + 84 + 14
    cycle = 1.26 * (6 * step + step + 60)
    if case["kind"] == "adjoint":
        return {"bytes": 8.0 * n * (3 + 3 + 4 + 4 + 3), "flops": 2 * 9 * cycle * n}
    if case["kind"] == "fmg":
        return {"bytes": 8.0 * n * 10, "flops": 2 * 0.7 * cycle * n * 8 / 7}
    if case["kind"] == "vcycle":
        return {"bytes": 8.0 * n * 14, "flops": 2 * cycle * n}
    return {"bytes": 8.0 * n * 10, "flops": 9 * cycle * n}


# ---- the discrete solution in 64 bits --------------------------------------------

class _Discrete:
    """The stabilised P1-P1 Stokes system on the Kuhn tetrahedra of a box of
    cubes (delta = 1/12, nu = 1), applied element by element."""

    def __init__(self, c, dev):
        self.c = c
        nx, ny, nz = _dims(c)
        N = 2 ** c["level"]
        self.h = h = 1.0 / N
        self.shape = (nz, ny, nx)
        B = SHEAR if c["sheared"] else np.eye(3)
        self.binv = np.linalg.inv(B)
        self.vol = abs(np.linalg.det(B)) * h ** 3 / 6.0
        self.dh2 = (1.0 / 12.0) * self.vol ** (2.0 / 3.0)
        cell = torch.ones((nz - 1, ny - 1, nx - 1), dtype=torch.float64, device=dev)
        wall = torch.zeros(self.shape, dtype=torch.bool, device=dev)
        wall[0], wall[-1], wall[:, 0], wall[:, -1], wall[:, :, 0] = True, True, True, True, True
        if not c["outflow"]:
            wall[:, :, -1] = True
        for (i, j, k) in _removed(c):
            cell[k * N:(k + 1) * N, j * N:(j + 1) * N, i * N:(i + 1) * N] = 0.0
            wall[k * N:(k + 1) * N + 1, j * N:(j + 1) * N + 1, i * N:(i + 1) * N + 1] = True
        self.cell = cell if _removed(c) else None
        act = torch.zeros(self.shape, dtype=torch.float64, device=dev)
        for o in itertools.product((0, 1), repeat=3):
            self._at(act, o).add_(cell)
        self.act = (act > 0).to(torch.float64)
        self.free = ((act > 0) & ~wall).to(torch.float64)
        self.paths = []
        for perm in itertools.permutations(range(3)):
            o, corners = [0, 0, 0], [(0, 0, 0)]
            for a in perm:
                o[a] += 1
                corners.append(tuple(o))
            self.paths.append((perm, corners))
        self.lump = torch.zeros(self.shape, dtype=torch.float64, device=dev)
        for _, corners in self.paths:
            for o in corners:
                self._at(self.lump, o).add_(cell, alpha=self.vol / 4.0)
        # the box's seven-point Laplacian, diagonalised axis by axis
        self.V, lam = [], []
        for a, n in enumerate((nx, ny, nz)):
            K = 2.0 * torch.eye(n, dtype=torch.float64) - torch.diag(torch.ones(n - 1, dtype=torch.float64), 1)
            K = K - torch.diag(torch.ones(n - 1, dtype=torch.float64), -1)
            D = torch.ones(n, dtype=torch.float64)
            hi = n - 1
            if a == 0 and c["outflow"]:
                K[-1, -1], D[-1], hi = 1.0, 0.5, n
            K, D = K[1:hi, 1:hi], D[1:hi].sqrt()
            w, Q = torch.linalg.eigh(K / D[:, None] / D[None, :])
            V = torch.zeros((n, hi - 1), dtype=torch.float64)
            V[1:hi] = Q / D[:, None]
            self.V.append(V.to(dev))
            lam.append(w.to(dev))
        self.lam = h * (lam[0].view(1, 1, -1) + lam[1].view(1, -1, 1) + lam[2].view(-1, 1, 1))

    def _at(self, x, o):
        nz, ny, nx = self.shape
        return x[..., o[2]:o[2] + nz - 1, o[1]:o[1] + ny - 1, o[0]:o[0] + nx - 1]

    def _grad(self, x, path):
        """Physical gradient per tetrahedron: (3, ..., cells)."""
        perm, cor = path
        g = [None] * 3
        for m, a in enumerate(perm):
            g[a] = (self._at(x, cor[m + 1]) - self._at(x, cor[m])) / self.h
        bi = self.binv
        if not self.c["sheared"]:
            return torch.stack(g)
        return torch.stack([sum(float(bi[a, d]) * g[a] for a in range(3)) for d in range(3)])

    def _div_add(self, y, s, path):
        """y_i += vol s . grad phi_i, s (3, ..., cells)."""
        perm, cor = path
        bi = self.binv
        for m, a in enumerate(perm):
            t = s[a] if not self.c["sheared"] else sum(float(bi[a, d]) * s[d] for d in range(3))
            t = t * (self.vol / self.h)
            if self.cell is not None:
                t = t * self.cell
            self._at(y, cor[m + 1]).add_(t)
            self._at(y, cor[m]).sub_(t)

    def _mean(self, x, path):
        return 0.25 * sum(self._at(x, o) for o in path[1])

    def A(self, u):
        """Velocity block on all rows; u (3, nz, ny, nx)."""
        y = torch.zeros_like(u)
        for path in self.paths:
            g = self._grad(u, path)  # (d, component, cells)
            self._div_add(y, g + g.transpose(0, 1) if self.c["d_form"] else g, path)
        return y

    def B(self, u):
        y = torch.zeros(self.shape, dtype=u.dtype, device=u.device)
        for path in self.paths:
            g = self._grad(u, path)
            q = (g[0, 0] + g[1, 1] + g[2, 2]) * (-0.25 * self.vol)
            if self.cell is not None:
                q = q * self.cell
            for o in path[1]:
                self._at(y, o).add_(q)
        return y

    def BT(self, p):
        y = torch.zeros((3,) + self.shape, dtype=p.dtype, device=p.device)
        for path in self.paths:
            m = -self._mean(p, path)
            for a in range(3):
                s = torch.zeros((3,) + m.shape, dtype=p.dtype, device=p.device)
                s[a] = m
                self._div_add(y[a], s, path)
        return y

    def C(self, p):
        y = torch.zeros_like(p)
        for path in self.paths:
            self._div_add(y, self._grad(p, path), path)
        return y * self.dh2

    def M(self, f):
        y = torch.zeros_like(f)
        for path in self.paths:
            s = sum(self._at(f, o) for o in path[1])
            for o in path[1]:
                t = (s + self._at(f, o)) * (self.vol / 20.0)
                self._at(y, o).add_(t if self.cell is None else t * self.cell)
        return y

    def G(self, f):
        """g(q) = -delta h_T^2 <f, grad q>, f (3, nz, ny, nx)."""
        y = torch.zeros(self.shape, dtype=f.dtype, device=f.device)
        for path in self.paths:
            self._div_add(y, torch.stack([self._mean(f[d], path) for d in range(3)]), path)
        return y * -self.dh2

    def GT(self, q):
        """Transpose of G on one pressure field: (3, nz, ny, nx)."""
        y = torch.zeros((3,) + self.shape, dtype=q.dtype, device=q.device)
        for path in self.paths:
            g = self._grad(q, path) * (0.25 * self.vol)
            if self.cell is not None:
                g = g * self.cell
            for o in path[1]:
                self._at(y, o).add_(g)
        return y * -self.dh2

    def _box(self, r):
        Vx, Vy, Vz = self.V
        t = torch.einsum("...x,xa->...a", r, Vx)
        t = torch.einsum("...ya,yb->...ba", t, Vy)
        t = torch.einsum("...zba,zc->...cba", t, Vz) / self.lam
        t = torch.einsum("...cba,zc->...zba", t, Vz)
        t = torch.einsum("...ba,yb->...ya", t, Vy)
        return torch.einsum("...a,xa->...x", t, Vx)

    def _pcg(self, op, prec, b, rtol, most):
        x, r = torch.zeros_like(b), b.clone()
        z = prec(r)
        d, rz, stop = z.clone(), (r * z).sum(), float((b * b).sum().sqrt()) * rtol
        for _ in range(most):
            if float((r * r).sum().sqrt()) <= stop:
                break
            q = op(d)
            a = rz / (d * q).sum()
            x += a * d
            r -= a * q
            z = prec(r)
            rn = (r * z).sum()
            d = z + (rn / rz) * d
            rz = rn
        return x

    def Ainv(self, b):
        return self._pcg(lambda v: self.A(v) * self.free, lambda v: self._box(v) * self.free, b * self.free, 1e-14, 400)

    def solve(self, fu, gp):
        """(u, p) of A u + B^T p = fu on free nodes, B u - C p = gp."""
        act, n = self.act, float(self.act.sum())

        def centre(v):
            return v if self.c["outflow"] else (v - (v.sum() / n)) * act
        gp = centre(gp * act)
        u1 = self.Ainv(fu)
        op = lambda p: centre((self.B(self.Ainv(self.BT(p) * self.free)) + self.C(p)) * act)  # noqa: E731
        inv = act / self.lump.clamp_min(1e-300)
        p = self._pcg(op, lambda r: r * inv, centre((self.B(u1) - gp) * act), 1e-13, 300)
        if not self.c["outflow"]:
            p = (p - (self.lump * p).sum() / self.lump.sum()) * act
        return self.Ainv(fu - self.BT(p) * self.free), p


def exact(case, seed):
    plain = not (case["obstacles"] or case["sheared"])
    if case["slip"] or case["kind"] == "vcycle" or _nodes(case) > (2.5e6 if plain and not case["outflow"] else 1e5):
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    S = _Discrete(case, dev)
    f, ud = (t.view(S.shape + (3,)).movedim(-1, 0) for t in _inputs(case, seed, dev))
    f, ud = f * S.act, ud * (S.act - S.free)
    u, p = S.solve((S.M(f) - S.A(ud)) * S.free, S.G(f) - S.B(ud))
    flat = lambda v: v.movedim(0, -1).reshape(-1, 3)  # noqa: E731
    out = {"u": flat(u + ud), "p": p.reshape(-1)}
    if case["kind"] == "adjoint":
        ju = _functional(case, seed, dev).view(S.shape + (3,)).movedim(-1, 0) * S.free
        lu, lp = S.solve(ju, torch.zeros_like(p))
        out["grad"] = flat((S.M(lu) + S.GT(lp)) * S.act)
    return out
