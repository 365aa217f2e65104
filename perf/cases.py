"""Performance cases: the calls a program on this library spends its time in, over the range of
sizes, precisions and meshes it makes them with.

A case names an entry point group ("kind"), a synthetic mesh and a precision. The meshes are the
ones of the benchmark and the tests: the Rayleigh-Taylor box ("rt"), the rising drop ("drop"),
uniform octrees and random balanced octrees. Inputs are seeded: the interface is displaced, and
velocities, potentials, pressures and Krylov vectors are drawn, from the seed.

exact() restates the finite-element forms in plain torch FP64 (dense per-element sums over the
2x2x2 Gauss points, its own node numbering and hanging constraints); it uses nothing of the
library.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

MAXD = 20
DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64


# ------------------------------------------------------------------ the cases
def listed():
    rt10 = dict(mesh="rt", lmin=6, lmax=10, cn=0.005, mseed=0)
    rt9 = dict(mesh="rt", lmin=6, lmax=9, cn=0.005, mseed=0)
    rt8 = dict(mesh="rt", lmin=5, lmax=8, cn=0.005, mseed=0)
    drop8 = dict(mesh="drop", lmin=5, lmax=8, cn=0.01, mseed=0)
    return [
        # one CG or smoother application of the pressure operator on the headline mesh (6.9e6
        # leaves): the call the pressure solve consists of
        dict(name="poisson_fp32_rt10", kind="apply", ops="poisson", prec="fp32", **rt10),
        # the velocity-update operator on the rising drop with bfloat16 coefficients
        dict(name="mass_bf16_drop8", kind="apply", ops="mass", prec="bf16", **drop8),
        # the Cahn-Hilliard Newton Jacobian inside GMRES, 1.4e6 leaves
        dict(name="ch_fp32_rt9", kind="apply", ops="ch", prec="fp32", **rt9),
        # the velocity-prediction operator, coefficients evaluated on the fly, 3e5 leaves
        dict(name="momentum_fp32_drop8", kind="apply", ops="momentum", prec="fp32", **drop8),
        # all four operators in FP64, as residuals and the all-FP64 path apply them
        dict(name="applies_fp64_rt8", kind="apply", ops="poisson,mass,ch,momentum", prec="fp64",
             **rt8),
        # the smallest calls: an octree of a few thousand leaves with many hanging nodes, where
        # launch and latency are all there is
        dict(name="applies_tiny", kind="apply", ops="poisson,mass,ch,momentum", prec="fp32",
             mesh="random", lmin=2, lmax=5, cn=0.05, mseed=1),
        # what a block of a time step assembles before and between its solves: the CH residual,
        # the three right-hand sides and the phase integral
        dict(name="rhs_fp64_drop8", kind="rhs", prec="fp64", **drop8),
        # the headline pressure solve: flexible CG with the multigrid V-cycle, FP32 iterations
        # refined in double-float
        dict(name="solve_pressure_mg_rt10", kind="solve", ops="poisson", pc="mg", inner="fp32",
             rtol=1e-10, **rt10),
        # one Newton correction of the Cahn-Hilliard pair: flexible GMRES with the Schur
        # preconditioner whose inner solves are V-cycles
        dict(name="solve_ch_schur_rt9", kind="solve", ops="ch", pc="schur_mg", inner="fp32",
             rtol=1e-11, **rt9),
        # a whole time step on a small mesh, mixed precision with the one-level preconditioners:
        # some thousand short launches, GMRES and CG on every operator
        dict(name="step_fp32_drop6", kind="step", inner="fp32", rtol=1e-11, mesh="drop", lmin=4,
             lmax=6, cn=0.03, mseed=0),
        # adaptive remeshing between steps: band flags, the new mesh, every field transferred
        dict(name="remesh_drop7", kind="remesh", mesh="drop", lmin=4, lmax=7, cn=0.02, mseed=0),
        # one training pass of the learned correction's network on the grid of the benchmark
        dict(name="learned_train_64", kind="learned", grid=64),
    ]


def draw(rng):
    """One more case: any kind, on a mesh of random type, depth, interface width and placement,
    from some hundred to about 1.5e6 leaves."""
    kind = rng.choice(["apply"] * 5 + ["rhs"] * 2 + ["solve"] * 3 + ["step", "remesh", "learned"])
    if kind == "learned":
        return dict(kind=kind, grid=rng.choice([8, 16, 32, 64]), mseed=rng.randrange(1, 10 ** 6))
    c = dict(kind=kind)
    small = kind in ("step", "remesh")
    mesh = rng.choice(["rt", "drop", "drop"] if kind != "apply" else
                      ["rt", "drop", "drop", "random", "uniform"])
    c["mesh"] = mesh
    c["mseed"] = rng.randrange(1, 10 ** 6)
    if mesh == "uniform":
        c.update(lmin=(l := rng.randint(2, 6)), lmax=l, cn=0.1)
    elif mesh == "random":
        c.update(lmin=rng.randint(1, 3), lmax=rng.randint(4, 6), cn=0.05)
    else:
        lmax = rng.randint(5, 6 if small else 8)
        if mesh == "rt" and not small and rng.random() < 0.4:
            lmax = 9
        lmin = rng.randint(max(3, lmax - 3), min(6, lmax - 1))
        # the interface spans one to four of the finest cells
        c.update(lmin=lmin, lmax=lmax, cn=round(rng.uniform(1.2, 3.0) * 2.0 ** -lmax, 6))
    if kind == "apply":
        ops = ["poisson", "mass", "ch", "momentum"]
        c["prec"] = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp64"])
        c["ops"] = rng.choice(ops) if rng.random() < 0.75 else ",".join(rng.sample(ops, 2))
    elif kind == "rhs":
        c["prec"] = "fp64"
    elif kind == "solve":
        op, pc = rng.choice([("poisson", "mg"), ("poisson", "jacobi"), ("poisson", "chebyshev"),
                             ("mass", "jacobi"), ("momentum", "jacobi"), ("ch", "schur_mg")])
        c.update(ops=op, pc=pc, inner=rng.choice(["fp32", "fp32", "bf16", "fp64"]),
                 rtol=1e-11 if op == "ch" else 1e-10)
        if pc in ("jacobi", "chebyshev") or c["inner"] == "fp64":
            c["lmax"] = min(c["lmax"], 7)
            c["lmin"] = min(c["lmin"], c["lmax"] - 1)
            c["cn"] = max(c["cn"], round(1.2 * 2.0 ** -c["lmax"], 6))
    elif kind == "step":
        c.update(inner=rng.choice(["fp32", "fp64"]), rtol=1e-11, mesh="drop")
    return c


# ------------------------------------------------------------------ synthetic octrees (torch)
def _spread(v):
    """Bit i of a 21-bit integer to bit 3 i."""
    v = v & 0x1FFFFF
    for s, m in ((32, 0x1F00000000FFFF), (16, 0x1F0000FF0000FF), (8, 0x100F00F00F00F00F),
                 (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        v = (v | (v << s)) & m
    return v


def _morton(x):
    """Morton keys (x lowest) of integer points (..., 3) with coordinates up to 2^20."""
    return _spread(x[..., 0]) | (_spread(x[..., 1]) << 1) | (_spread(x[..., 2]) << 2)


def _compact(k):
    """Inverse of _spread."""
    k = k & 0x1249249249249249
    for s, m in ((2, 0x10C30C30C30C30C3), (4, 0x100F00F00F00F00F), (8, 0x1F0000FF0000FF),
                 (16, 0x1F00000000FFFF), (32, 0x1FFFFF)):
        k = (k | (k >> s)) & m
    return k


_BITS = torch.tensor([[a & 1, a >> 1 & 1, a >> 2 & 1] for a in range(8)], device=DEV)


def _points(key):
    return torch.stack([_compact(key >> d) for d in range(3)], dim=-1)


def _children(key):
    """Keys, one level deeper, of the 8 children of octants given by the keys of their own level."""
    return (key[:, None] * 8 + torch.arange(8, device=DEV)[None, :]).reshape(-1)


def _complete(split, lmax):
    """Leaves of the coarsest full 2:1 balanced octree in which the octants split[l] (keys of
    level l) have children: an octant with children needs the parents of its 26 neighbours to
    have children too."""
    off = torch.tensor([[dx, dy, dz] for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)],
                       device=DEV)
    split = [s.unique() for s in split]
    for l in range(lmax - 1, 0, -1):
        if split[l].numel() == 0:
            continue
        nb = (_points(split[l])[:, None, :] + off[None]).reshape(-1, 3)
        nb = nb[((nb >= 0) & (nb < (1 << l))).all(dim=1)]
        split[l - 1] = torch.cat([split[l - 1], _morton(nb >> 1)]).unique()
    keys, levels = [], []
    for l in range(lmax):
        if split[l].numel() == 0:
            continue
        kids = _children(split[l])
        if l + 1 < lmax:
            kids = kids[~torch.isin(kids, split[l + 1])]
        keys.append(kids << (3 * (MAXD - l - 1)))
        levels.append(torch.full_like(kids, l + 1))
    key, level = torch.cat(keys), torch.cat(levels)
    order = key.argsort()
    return key[order], level[order]


def _phase(c, x, seed):
    """Signed distance to the interface over sqrt(2) Cn, at points x of the box, with the
    interface displaced by the seed."""
    r = np.random.default_rng([seed or 0, 11])
    if c["mesh"] == "rt":
        m = np.random.default_rng([c["mseed"], 5])
        y0 = 2.0 if c["mseed"] == 0 else 2.0 + m.uniform(-0.4, 0.4)
        amp = 0.05 * (1.0 if seed is None else r.uniform(0.9, 1.1))
        sx, sz = (0.0, 0.0) if seed is None else r.uniform(-0.02, 0.02, 2)
        t = 2.0 * math.pi
        d = x[:, 1] - y0 - amp * torch.cos(t * (x[:, 0] - sx)) * torch.cos(t * (x[:, 2] - sz))
    else:
        m = np.random.default_rng([c["mseed"], 5])
        ctr, rad = np.array([0.5, 0.5, 0.3]), 0.15
        if c["mseed"]:
            rad = m.uniform(0.08, 0.22)
            ctr = m.uniform(rad + 0.03, 0.97 - rad, 3)
        if seed is not None:
            ctr = ctr + r.uniform(-0.5, 0.5, 3) * c["cn"]
        d = (x - torch.tensor(ctr, device=DEV)[None]).norm(dim=1) - rad
    return d / (math.sqrt(2.0) * c["cn"])


def _extent(c):
    return (1.0, 4.0, 1.0) if c["mesh"] == "rt" else (1.0, 1.0, 1.0)


def _leaves(c):
    """Morton keys of the anchors and levels of the case's leaves."""
    lmin, lmax = c["lmin"], c["lmax"]
    ext = torch.tensor(_extent(c), device=DEV, dtype=F64)
    split = [torch.zeros(0, dtype=torch.int64, device=DEV) for _ in range(lmax)]
    cur = torch.zeros(1, dtype=torch.int64, device=DEV)
    g = torch.Generator(device="cpu").manual_seed(c["mseed"])
    for l in range(lmax):
        if l < lmin:
            sel = torch.ones(len(cur), dtype=torch.bool, device=DEV)
        elif c["mesh"] == "random":
            sel = (torch.rand(len(cur), generator=g) < 0.3).to(DEV)
        elif c["mesh"] == "uniform":
            sel = torch.zeros(len(cur), dtype=torch.bool, device=DEV)
        else:  # the smallest |phi| over the corners and the centre is below 0.9
            sel = torch.zeros(len(cur), dtype=torch.bool, device=DEV)
            a = _points(cur).to(F64)
            low = torch.full((len(cur),), math.inf, device=DEV, dtype=F64)
            for b in [*_BITS.to(F64), torch.full((3,), 0.5, device=DEV, dtype=F64)]:
                low = torch.minimum(low, _phase(c, (a + b) / (1 << l) * ext, None).abs())
            sel = low < math.atanh(0.9)
        split[l] = cur[sel]
        cur = _children(split[l])
    return _complete(split, lmax)


# ------------------------------------------------------------------ nodes and FE sums (FP64)
class _Nodes:
    """Nodes of a leaf list: the distinct corners that are not hanging, in Morton order; hanging
    corners are the midpoint of an edge or the centre of a face of some leaf."""

    def __init__(self, key, level, ext):
        self.key, self.level, self.ext = key, level, torch.tensor(ext, device=DEV, dtype=F64)
        anchor = _points(key)
        side = (1 << (MAXD - level))[:, None]
        pk = _morton(anchor[:, None, :] + side[:, None] * _BITS[None])          # (E, 8)
        pts, conn = pk.unique(return_inverse=True)
        par = torch.full((len(pts), 4), -1, dtype=torch.int64, device=DEV)

        def find(k):
            i = torch.searchsorted(pts, k).clamp_(max=len(pts) - 1)
            return i, pts[i] == k

        def mark(mid, ends):
            i, hit = find(_morton(mid))
            for s, e in enumerate(ends):
                j, ok = find(_morton(e[hit]))
                assert bool(ok.all())
                par[i[hit], s] = j

        e = torch.eye(3, dtype=torch.int64, device=DEV)
        for d in range(3):
            o1, o2 = [k for k in range(3) if k != d]
            for b1 in (0, 1):
                for b2 in (0, 1):
                    base = anchor + side * (b1 * e[o1] + b2 * e[o2])
                    mark(base + side // 2 * e[d], [base, base + side * e[d]])
            for b in (0, 1):
                base = anchor + side * b * e[d]
                mark(base + side // 2 * (e[o1] + e[o2]),
                     [base, base + side * e[o1], base + side * e[o2], base + side * (e[o1] + e[o2])])
        self.reg = (par[:, 0] < 0).nonzero().flatten()
        self.hang = (par[:, 0] >= 0).nonzero().flatten()
        p = par[self.hang]
        self.par = torch.where(p < 0, p[:, :1], p)
        self.wpar = torch.where(p[:, 2:3] >= 0, 0.25, 0.5).to(F64) * (p >= 0)
        self.conn, self.npts, self.n, self.n_elem = conn, len(pts), len(self.reg), len(key)
        self.n_hang = len(self.hang)
        self.node_int = _points(pts[self.reg])
        self.xyz = self.node_int.to(F64) / (1 << MAXD) * self.ext
        self.bnd = ((self.node_int == 0) | (self.node_int == 1 << MAXD)).any(dim=1)
        self.h = self.ext[None] / (1 << level)[:, None].to(F64)
        self.det = self.h.prod(dim=1) / 8

    def to_points(self, u):
        """Values at every distinct corner of nodal values u (n,)."""
        v = torch.zeros(self.npts, device=DEV, dtype=F64)
        v[self.reg] = u
        v[self.hang] = (v[self.par] * self.wpar).sum(dim=1)
        return v

    def from_points(self, v):
        """Transpose of to_points, with the contributions to a node added in a fixed order."""
        w = v[self.hang, None] * self.wpar
        v = v.clone().index_put_((self.par.reshape(-1),), w.reshape(-1), accumulate=True)
        return v[self.reg]

    def assemble(self, fields, fn, n_out):
        """P^T sum_e fn(e): fn gets the slice of elements and the corner values of the fields and
        gives n_out (e, 8) arrays."""
        pf = [self.to_points(f) for f in fields]
        out = [torch.zeros(self.npts, device=DEV, dtype=F64) for _ in range(n_out)]
        step = 1 << 19
        for a in range(0, self.n_elem, step):
            s = slice(a, min(a + step, self.n_elem))
            r = fn(_El(self.h[s], self.det[s]), [f[self.conn[s]] for f in pf])
            for o, x in zip(out, r):
                o.index_put_((self.conn[s].reshape(-1),), x.reshape(-1), accumulate=True)
        return [self.from_points(o) for o in out]


def _basis():
    b = _BITS.to(F64).cpu().numpy() * 2 - 1
    f = 0.5 * (1 + b[None] * b[:, None] / math.sqrt(3))          # (q, a, d)
    d = 0.5 * b
    N = f.prod(2)
    D = np.stack([d[None, :, k] * f.prod(2) / f[:, :, k] for k in range(3)], -1)
    H = {(i, j): d[None, :, i] * d[None, :, j] * f[:, :, 3 - i - j] for i in range(3) for j in range(i)}
    t = lambda a: torch.tensor(a, device=DEV, dtype=F64)  # noqa: E731
    return t(N), t(D), {k: t(v) for k, v in H.items()}


_N, _D, _H = _basis()


class _El:
    """Values, gradients and test-function sums of a chunk of elements at the 8 Gauss points."""

    def __init__(self, h, det):
        self.s, self.det = 2.0 / h, det

    def val(self, u):
        return u @ _N.T

    def grad(self, u):
        return torch.einsum("qad,ea->eqd", _D, u) * self.s[:, None]

    def mixed(self, u):
        """The mixed second derivatives (the pure ones vanish), {(i, j)}."""
        return {k: (u @ v.T) * (self.s[:, k[0]] * self.s[:, k[1]])[:, None] for k, v in _H.items()}

    def test(self, s=None, V=None):
        """detJ sum_q (s N_a + V . grad N_a)"""
        r = 0.0 if s is None else s @ _N
        if V is not None:
            r = r + torch.einsum("qad,eqd->ea", _D, V * self.s[:, None])
        return r * self.det[:, None]


class _Phys:
    def __init__(self, p):
        self.__dict__.update(p)
        self.alpha, self.beta = (1 - 1 / self.rho_ratio) / 2, (1 + 1 / self.rho_ratio) / 2
        self.gamma, self.xi = (1 - 1 / self.eta_ratio) / 2, (1 + 1 / self.eta_ratio) / 2

    def rho(self, v):
        return self.alpha * v.clamp(-1, 1) + self.beta


class _Vms:
    """Coefficients of the residual-based variational multiscale closure at the Gauss points."""

    def __init__(self, el, k, phi, u, mu):
        pv, self.gp = el.val(phi), el.grad(phi)
        self.rho, self.eta = k.rho(pv), k.gamma * pv.clamp(-1, 1) + k.xi
        self.ge = k.gamma * self.gp * (pv.abs() < 1)[..., None]
        self.u = torch.stack([el.val(c) for c in u], -1)
        self.J = -(k.alpha / k.Cn) * el.grad(mu)
        G = el.s[:, None] ** 2
        t = (4 / k.dt ** 2 + (self.u * G * self.u).sum(-1)
             + (self.u * G * self.J).sum(-1) / (self.rho * k.Pe)
             + k.C_I * (self.eta / (self.rho * k.Re)) ** 2 * (G * G).sum(-1))
        self.tau = t.clamp(min=4 / k.dt ** 2) ** -0.5
        self.b = 0.5 * self.rho[..., None] * self.u + 0.5 / k.Pe * self.J
        self.bp = self.b - 0.5 / k.Re * self.ge
        self.t = self.tau[..., None] * (0.5 * self.u + 0.5 / k.Pe * self.J / self.rho[..., None])
        m, g = el.mixed(phi), self.gp
        self.force = torch.stack([m[1, 0] * g[..., 1] + m[2, 0] * g[..., 2],
                                  m[1, 0] * g[..., 0] + m[2, 1] * g[..., 2],
                                  m[2, 0] * g[..., 0] + m[2, 1] * g[..., 1]], -1)

    def residual(self, el, k, i, v, uk, pk):
        """R_m,i for the velocity v (u_k, p_k of the last step)."""
        gt = 0.5 * (el.grad(v) + el.grad(uk))
        return (self.rho * (el.val(v) - el.val(uk)) / k.dt
                + ((self.rho[..., None] * self.u + self.J / k.Pe - self.ge / k.Re) * gt).sum(-1)
                + k.Cn / k.We * self.force[..., i] + el.grad(pk)[..., i]
                + (self.rho / k.Fr if i == 1 else 0.0))


def _operator(nodes, op, prm, phi, u, mu, x):
    """A x of one operator in FP64, components one after another."""
    k, n = _Phys(prm), nodes.n
    xs = list(x.reshape(-1, n))
    if op in ("mass", "momentum"):
        xs = [torch.where(nodes.bnd, 0.0, v) for v in xs]

    def poisson(el, f):
        return [el.test(V=el.grad(f[1]) / k.rho(el.val(f[0]))[..., None])]

    def mass(el, f):
        rho = k.rho(el.val(f[0]))
        return [el.test(rho * el.val(v)) for v in f[1:]]

    def ch(el, f):
        pv, fv = el.val(f[0]), el.val(f[4])
        uv = torch.stack([el.val(c) for c in f[1:4]], -1)
        return [el.test(fv / k.dt, 0.5 / (k.Pe * k.Cn) * el.grad(f[5]) - 0.5 * uv * fv[..., None]),
                el.test(0.5 * ((3 * pv ** 2 - 1) * fv - el.val(f[5])), 0.5 * k.Cn ** 2 * el.grad(f[4]))]

    def momentum(el, f):
        c, out = _Vms(el, k, f[0], f[1:4], f[4]), []
        for v in f[5:]:
            w, g = el.val(v), el.grad(v)
            s = c.rho / k.dt * w + (c.b * g).sum(-1)
            R = c.rho / k.dt * w + (c.bp * g).sum(-1)
            out.append(el.test(s, (0.5 / k.Re * c.eta)[..., None] * g + R[..., None] * c.t))
        return out

    fn, co = {"poisson": (poisson, [phi]), "mass": (mass, [phi]), "ch": (ch, [phi, *u]),
              "momentum": (momentum, [phi, *u, mu])}[op]
    y = torch.cat(nodes.assemble([*co, *xs], fn, len(xs))).reshape(len(xs), n)
    if op in ("mass", "momentum"):
        y = torch.where(nodes.bnd[None], x.reshape(len(xs), n), y)
    return y.reshape(-1)


def _right_hand_sides(nodes, prm, f):
    """CH residual, velocity prediction, pressure and velocity update right-hand sides, phase
    integral."""
    k = _Phys(prm)

    def residual(el, e):
        phi, mu, phik, muk = e[:4]
        pt, mt = 0.5 * (phi + phik), 0.5 * (mu + muk)
        pv = el.val(pt)
        uv = torch.stack([el.val(c) for c in e[4:7]], -1)
        return [el.test(el.val(phi - phik) / k.dt, el.grad(mt) / (k.Pe * k.Cn) - uv * pv[..., None]),
                el.test(pv ** 3 - pv - el.val(mt), k.Cn ** 2 * el.grad(pt))]

    def prediction(el, e):
        c, pk, out = _Vms(el, k, e[0], e[1:4], e[4]), el.grad(e[8]), []
        for i, ui in enumerate(e[5:8]):
            a, g = c.rho / k.dt * el.val(ui), el.grad(ui)
            grav = -c.rho / k.Fr if i == 1 else 0.0
            R = (c.bp * g).sum(-1) - a + k.Cn / k.We * c.force[..., i] + pk[..., i] - grav
            s = a - (c.b * g).sum(-1) - pk[..., i] + grav
            V = (k.Cn / k.We * c.gp[..., i:i + 1] * c.gp - (0.5 / k.Re * c.eta)[..., None] * g
                 - c.t * R[..., None])
            out.append(el.test(s, V))
        return out

    def pressure(el, e):
        c = _Vms(el, k, e[0], e[1:4], e[4])
        R = torch.stack([c.residual(el, k, i, e[5 + i], e[8 + i], e[11]) for i in range(3)], -1)
        div = sum(el.grad(e[5 + i])[..., i] for i in range(3))
        V = (el.grad(e[11]) - 2 / k.dt * c.tau[..., None] * R) / c.rho[..., None]
        return [el.test(-2 / k.dt * div, V)]

    def update(el, e):
        c, gd = _Vms(el, k, e[0], e[1:4], e[4]), el.grad(e[12] - e[11])
        return [el.test(c.rho * el.val(e[5 + i]) - 0.5 * k.dt * gd[..., i]
                        - c.tau * c.residual(el, k, i, e[5 + i], e[8 + i], e[11]))
                for i in range(3)]

    co = [f["phi"], *f["u"], f["mu"]]
    r = nodes.assemble([f["phi"], f["mu"], f["phik"], f["muk"], *f["u"]], residual, 2)
    vp = nodes.assemble([*co, *f["uk"], f["pk"]], prediction, 3)
    vp = [torch.where(nodes.bnd, 0.0, b) for b in vp]
    pp = nodes.assemble([*co, *f["v"], *f["uk"], f["pk"]], pressure, 1)[0]
    vu = nodes.assemble([*co, *f["v"], *f["uk"], f["pk"], f["pn"]], update, 3)
    vu = [torch.where(nodes.bnd, 0.0, b) for b in vu]
    mass = (nodes.to_points(f["phi"])[nodes.conn].sum(1) * nodes.det).sum()
    return [torch.cat(r), torch.cat(vp), pp, torch.cat(vu), float(mass)]


# ------------------------------------------------------------------ inputs
def _params(c):
    p = dict(Fr=1.0, C_I=6.0, Cn=c["cn"], Pe=1.0 / (3 * c["cn"] ** 2))
    if c["mesh"] == "rt":
        p.update(Re=1000.0, We=1000.0, rho_ratio=3.0, eta_ratio=1.0, dt=2.5e-4)
    elif c["mesh"] == "drop":
        p.update(Re=35.0, We=1.0, rho_ratio=1000.0, eta_ratio=100.0, dt=5e-4)
    elif c["mesh"] == "uniform":
        p.update(Re=100.0, We=10.0, Pe=100.0, rho_ratio=10.0, eta_ratio=10.0, dt=1e-3)
    else:
        p.update(Re=35.0, We=2.0, Pe=50.0, rho_ratio=20.0, eta_ratio=5.0, dt=1e-3)
    return p


class _Fields:
    """Seeded nodal fields at the nodes x (n, 3) of a box."""

    def __init__(self, c, xyz, seed):
        self.c, self.x, self.seed = c, xyz, seed
        self.z = xyz / torch.tensor(_extent(c), device=DEV, dtype=F64)
        self.r = np.random.default_rng([seed, 3])
        self.g = torch.Generator(device=DEV).manual_seed(seed)
        self.wall = ((self.z == 0) | (self.z == 1)).any(dim=1)

    def smooth(self, amp, wall=False):
        """Four random modes; wall: they vanish on the boundary (velocities at rest there)."""
        v = torch.zeros(len(self.x), device=DEV, dtype=F64)
        for _ in range(4):
            k, a, s = self.r.integers(1, 4, 3), self.r.standard_normal(), self.r.uniform(0, 6.3, 3)
            w = [torch.sin(math.pi * float(k[d]) * self.z[:, d]) if wall else
                 torch.cos(math.pi * float(k[d]) * self.z[:, d] + float(s[d])) for d in range(3)]
            v += amp * a * w[0] * w[1] * w[2]
        return v

    def noise(self, n=None):
        return torch.randn(n or len(self.x), device=DEV, dtype=F64, generator=self.g)

    def phase(self):
        if self.c["mesh"] in ("uniform", "random"):
            return self.smooth(0.7) + 0.02 * self.noise()
        return torch.tanh(_phase(self.c, self.x, self.seed)) + 0.005 * self.noise()

    def velocity(self, amp=0.1):
        return [self.smooth(amp, wall=True) for _ in range(3)]


_COMP = {"poisson": 1, "mass": 3, "ch": 2, "momentum": 3}


def _apply_inputs(c, xyz, seed):
    """phi~ (as stored: 1 + phi~ in bfloat16), u, mu and one vector per operator, in the storage
    types of the precision."""
    f = _Fields(c, xyz, seed)
    ct = dict(fp32=torch.float32, fp64=F64, bf16=torch.bfloat16)[c["prec"]]
    vt = F64 if c["prec"] == "fp64" else torch.float32
    phi = f.phase() + (1.0 if c["prec"] == "bf16" else 0.0)
    u, mu = f.velocity(), f.smooth(0.02)
    xs = []
    for op in c["ops"].split(","):  # velocities are corrected with zero boundary values
        x = f.noise(_COMP[op] * len(xyz)).reshape(-1, len(xyz))
        x = torch.where(f.wall[None], 0.0, x) if op in ("mass", "momentum") else x
        xs.append(x.reshape(-1))
    return phi.to(ct), [a.to(ct) for a in u], mu.to(ct), [x.to(vt) for x in xs]


def _solve_inputs(c, nodes, seed):
    """Coefficients, the solution the right-hand side is made from, and that right-hand side."""
    f = _Fields(c, nodes.xyz, seed)
    phi, u, mu, op = f.phase(), f.velocity(), f.smooth(0.02), c["ops"]
    x = torch.stack([f.smooth(1.0, wall=op in ("mass", "momentum")) + 0.1 * f.noise()
                     for _ in range(_COMP[op])])
    if op == "poisson":
        x -= x.mean()
    if op in ("mass", "momentum"):
        x = torch.where(nodes.bnd[None], 0.0, x)
    x = x.reshape(-1)
    return phi, u, mu, x, _operator(nodes, op, _params(c), phi, u, mu, x)


def _rhs_inputs(c, xyz, seed):
    f = _Fields(c, xyz, seed)
    phi, mu = f.phase(), f.smooth(0.02)
    u, uk = f.velocity(), f.velocity()
    return dict(phi=phi, mu=mu, phik=phi + f.smooth(0.01), muk=mu + f.smooth(0.002), u=u, uk=uk,
                v=[a + b for a, b in zip(uk, f.velocity(0.01))], pk=f.smooth(0.5), pn=f.smooth(0.5))


def _state_inputs(c, xyz, seed):
    f = _Fields(c, xyz, seed)
    u = f.velocity(0.02)
    # a remesh takes its new leaves from phi: the phase of the mesh itself, displaced
    phi = f.phase() if c["kind"] == "step" else _Fields(c, xyz, c["mseed"] + 1).phase()
    return dict(phi=phi, mu=f.smooth(0.005), u=torch.stack(u), u_old=0.99 * torch.stack(u),
                p=f.smooth(0.05))


def _learned_inputs(c, seed):
    """Parameters of the 16-channel network, an input of two channels and an output gradient."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    D = c["grid"]
    par = []
    for cin in (2, 16, 16, 16, 16, 16, 16):
        par.append(torch.randn(27 * 16 * cin, device=DEV, generator=g) * math.sqrt(2 / (27 * cin)))
        par.append(0.05 * torch.randn(16, device=DEV, generator=g))
    par += [0.25 * torch.randn(16, device=DEV, generator=g), torch.zeros(1, device=DEV)]
    x = torch.randn(2 * D ** 3, device=DEV, generator=g)
    return torch.cat(par), x, torch.randn(D ** 3, device=DEV, generator=g)


# ------------------------------------------------------------------ handles a program keeps
def _spec(c):
    return tuple((k, c[k]) for k in ("mesh", "lmin", "lmax", "cn", "mseed"))


@functools.lru_cache(maxsize=4)
def _nodes_of(spec):
    c = dict(spec)
    return _Nodes(*_leaves(c), _extent(c))


class _Handle:
    """A mesh and, when asked for, its multigrid hierarchy."""

    def __init__(self, spec):
        from paper_2107_05123_gb300.session import Mesh
        c = dict(spec)
        key, level = _leaves(c)
        self.mesh = Mesh(_points(key).cpu().numpy().astype(np.uint32),
                         level.cpu().numpy().astype(np.uint8), _extent(c))
        self.xyz = torch.as_tensor(self.mesh.node_int.astype(np.int64), device=DEV).to(F64)
        self.xyz = self.xyz / (1 << MAXD) * torch.tensor(_extent(c), device=DEV, dtype=F64)
        self._mg = None

    @property
    def mg(self):
        from paper_2107_05123_gb300 import capi
        if self._mg is None:
            self._mg = capi.chns_mg_create(self.mesh.handle, degree=2)
        return self._mg

    def __del__(self):
        if getattr(self, "_mg", None) is not None:
            from paper_2107_05123_gb300 import capi
            capi.chns_mg_destroy(self._mg)
            self._mg = None


@functools.lru_cache(maxsize=3)
def _handle(spec):
    return _Handle(spec)


class _Net:
    def __init__(self, grid, par):
        from paper_2107_05123_gb300 import capi
        self.handle = capi.chns_learned_create(grid, 0, 1)
        capi.chns_learned_set_params(self.handle, par.cpu().numpy())

    def __del__(self):
        from paper_2107_05123_gb300 import capi
        capi.chns_learned_destroy(self.handle)


def _solver(c, capi, h):
    inner = dict(fp32=capi.FP32, bf16=capi.FP32_BF16COEF, fp64=capi.FP64)[c["inner"]]
    df = capi.FP64 if c["inner"] == "fp64" else capi.FP64_DF
    if c["pc"] == "mg":
        return capi.make_solver(capi.KSP_FCG, capi.PC_MULTIGRID, c["rtol"], 2000, 30, inner, 1e-6, 40,
                                check_every=2, mg=h.mg, fp64_apply=df)
    if c["pc"] == "schur_mg":
        return capi.make_solver(capi.KSP_GMRES, capi.PC_SCHUR, c["rtol"], 400, 30, inner, 1e-4,
                                inner_its=20, mg=h.mg)
    if c["ops"] == "momentum":
        return capi.make_solver(capi.KSP_GMRES, capi.PC_JACOBI, c["rtol"], 4000, 30, inner, 1e-4)
    pc, restart = (capi.PC_CHEBYSHEV, 3) if c["pc"] == "chebyshev" else (capi.PC_JACOBI, 30)
    return capi.make_solver(capi.KSP_CG, pc, c["rtol"], 20000, restart, inner, 1e-6, check_every=8,
                            fp64_apply=df)


def prepare(case, seed):
    from paper_2107_05123_gb300 import capi
    from paper_2107_05123_gb300.session import DeviceState, default_step_params
    c, kind = case, case["kind"]
    if kind == "learned":
        par, x, gout = _learned_inputs(c, seed)
        return dict(kind=kind, net=_Net(c["grid"], par), x=x, gout=gout, out=torch.empty_like(gout),
                    grad=torch.empty(par.numel(), device=DEV))
    h = _handle(_spec(c))
    n, prm = h.mesh.n_nodes, capi.make_params(_params(c))
    st = dict(kind=kind, h=h, mesh=h.mesh.handle, prm=prm)
    if kind == "apply":
        phi, u, mu, xs = _apply_inputs(c, h.xyz, seed)
        prec = dict(fp32=capi.FP32, fp64=capi.FP64, bf16=capi.FP32_BF16COEF)[c["prec"]]
        fn = [getattr(capi, "chns_apply_" + op) for op in c["ops"].split(",")]
        st.update(coef=capi.make_coef(phi, u, mu), prec=prec,
                  calls=[(f, x, torch.empty_like(x)) for f, x in zip(fn, xs)])
    elif kind == "rhs":
        f = _rhs_inputs(c, h.xyz, seed)
        new = lambda m: torch.empty(m * n, device=DEV, dtype=F64)  # noqa: E731
        st.update(f=f, coef=capi.make_coef(f["phi"], f["u"], f["mu"]),
                  out=[new(2), new(3), new(1), new(3)])
    elif kind == "solve":
        phi, u, mu, _, b = _solve_inputs(c, _nodes_of(_spec(c)), seed)
        op = dict(poisson=capi.OP_POISSON, mass=capi.OP_MASS, ch=capi.OP_CH,
                  momentum=capi.OP_MOMENTUM)[c["ops"]]
        st.update(op=op, coef=capi.make_coef(phi, u, mu), b=b, x=torch.zeros_like(b),
                  solver=_solver(c, capi, h))
    elif kind == "step":
        f = {k: v.cpu().numpy() for k, v in _state_inputs(c, h.xyz, seed).items()}
        sp = default_step_params(rtol=c["rtol"], newton_rtol=1e-12,
                                 inner=capi.FP32 if c["inner"] == "fp32" else capi.FP64)
        st.update(start=DeviceState(f), now=DeviceState(f), sp=sp)
    elif kind == "remesh":
        f = {k: v.cpu().numpy() for k, v in _state_inputs(c, h.xyz, seed).items()}
        st.update(ds=DeviceState(f), lmin=c["lmin"], lmax=c["lmax"])
    return st


def _copy_state(src, dst):
    for a, b in zip((src.phi, src.mu, *src.u, *src.u_old, src.p),
                    (dst.phi, dst.mu, *dst.u, *dst.u_old, dst.p)):
        b.copy_(a)


def run(state):
    from paper_2107_05123_gb300 import capi, session
    s, kind = state, state["kind"]
    if kind == "apply":
        for fn, x, y in s["calls"]:
            fn(s["mesh"], s["prm"], s["coef"], x, y, s["prec"])
        return [y for _, _, y in s["calls"]]
    if kind == "rhs":
        f, (r, vp, pp, vu) = s["f"], s["out"]
        capi.chns_residual_ch(s["mesh"], s["prm"], f["phi"], f["mu"], f["phik"], f["muk"], f["u"], r)
        capi.chns_rhs_momentum(s["mesh"], s["prm"], s["coef"], f["uk"], f["pk"], vp)
        capi.chns_rhs_poisson(s["mesh"], s["prm"], s["coef"], f["v"], f["uk"], f["pk"], pp)
        capi.chns_rhs_velocity_update(s["mesh"], s["prm"], s["coef"], f["v"], f["uk"], f["pk"],
                                      f["pn"], vu)
        return [r, vp, pp, vu, capi.chns_phi_mass(s["mesh"], f["phi"])]
    if kind == "solve":
        s["x"].zero_()
        capi.chns_krylov_solve(s["mesh"], s["op"], s["prm"], s["coef"], s["b"], s["x"], s["solver"])
        return s["x"]
    if kind == "step":  # each pass advances the same initial state by one step
        _copy_state(s["start"], s["now"])
        capi.chns_step(s["mesh"], s["now"].c, s["prm"], s["sp"])
        d = s["now"]
        return [d.phi, d.mu, *d.u, *d.u_old, d.p]
    if kind == "remesh":
        mesh, d = session.remesh(s["h"].mesh, s["ds"], 0.95, s["lmin"], s["lmax"])
        return [mesh.n_elem, mesh.n_hanging, d.phi, d.mu, *d.u, *d.u_old, d.p]
    net = s["net"].handle
    capi.chns_learned_forward(net, s["x"], s["out"])
    capi.chns_learned_backward(net, s["gout"], s["grad"])
    return [s["out"], s["grad"]]


# ------------------------------------------------------------------ work and exact values
def work(case):
    """Each nodal vector, coefficient field and element or hanging-node table entry moved once.
    A solve is counted as one application of its operator: its iterations are the method's."""
    c, kind = case, case["kind"]
    if kind == "learned":
        v, macs = c["grid"] ** 3, 27 * 16
        cells = [v, v // 8, v // 64, v // 512, v // 64, v // 8, v]
        fwd = sum(2 * macs * (2 if i == 0 else 16) * k for i, k in enumerate(cells)) + 32 * v
        # 42,465 parameters: read, and their gradients written
        return dict(bytes=4.0 * (2 * v + 2 * v + 2 * 42465), flops=3.0 * fwd)
    m = _nodes_of(_spec(c))
    tables = 33 * m.n_elem + 16 * m.n_hang
    arrays = dict(poisson=3, mass=7, ch=8, momentum=11)     # x, y and coefficients per node
    flops = dict(poisson=290, mass=420, ch=760, momentum=1500)
    if kind == "apply":
        vb, cb = dict(fp32=(4, 4), fp64=(8, 8), bf16=(4, 2))[c["prec"]]
        ops = c["ops"].split(",")
        nb = sum(2 * _COMP[o] * vb + (arrays[o] - 2 * _COMP[o]) * cb for o in ops)
        return dict(bytes=float(nb * m.n + tables * len(ops)),
                    flops=float(sum(flops[o] for o in ops) * m.n_elem))
    if kind == "rhs":
        return dict(bytes=float(8 * (9 + 12 + 13 + 16 + 1) * m.n + 5 * tables),
                    flops=float(7000 * m.n_elem))
    if kind == "solve":
        o = c["ops"]
        return dict(bytes=float(8 * arrays[o] * m.n + tables), flops=float(flops[o] * m.n_elem))
    if kind == "step":
        return dict(bytes=float(8 * 18 * m.n + tables), flops=float(14000 * m.n_elem))
    return dict(bytes=float(8 * 2 * 9 * m.n + 2 * tables), flops=float(9 * 30 * m.n))


def _remeshed(c, nodes, f):
    """The leaves after one remesh and every field at their nodes."""
    v = nodes.to_points(f["phi"])[nodes.conn]
    low = torch.minimum(v.abs().amin(1), v.mean(1).abs())
    band, lev, lmin, lmax = low <= 0.95, nodes.level, c["lmin"], c["lmax"]
    split = [torch.zeros(0, dtype=torch.int64, device=DEV) for _ in range(lmax)]
    own = nodes.key >> (3 * (MAXD - lev))              # keys of the leaves' own levels
    for l in range(lmax):
        # octants with children now: ancestors of every leaf, and the leaves that split; parents
        # whose 8 children are all leaves outside the band merge
        keep = [own[(lev == l) & band]]
        for k in range(l + 1, lmax + 1):
            sel = lev == k
            anc = own[sel] >> (3 * (k - l))
            if k == l + 1:
                par, cnt = (anc[~band[sel] & (lev[sel] > lmin)]).unique(return_counts=True)
                anc = anc[~torch.isin(anc, par[cnt == 8])]
            keep.append(anc)
        split[l] = torch.cat(keep)
    new = _Nodes(*_complete(split, lmax), _extent(c))
    k = _morton(new.node_int.clamp(max=(1 << MAXD) - 1))
    e = torch.searchsorted(nodes.key, k, right=True) - 1
    side = (1 << (MAXD - nodes.level[e]))[:, None].to(F64)
    xi = (new.node_int - _points(nodes.key[e])).to(F64) / side
    w = torch.where(_BITS[None] == 1, xi[:, None], 1 - xi[:, None]).prod(2)
    at = lambda a: (nodes.to_points(a)[nodes.conn[e]] * w).sum(1)  # noqa: E731
    return [new.n_elem, new.n_hang, at(f["phi"]), at(f["mu"]), *[at(a) for a in f["u"]],
            *[at(a) for a in f["u_old"]], at(f["p"])]


def _network(par, x, D):
    """Output of the network in FP64. Its gradient has no such value: bfloat16 activations take
    other sides of the rectifiers, and the gradient of the FP64 network is that of another one."""
    import torch.nn.functional as F
    par = par.double()
    at, lay = 0, []
    for cin in (2, 16, 16, 16, 16, 16, 16):
        w = par[at:at + 432 * cin].reshape(3, 3, 3, 16, cin).permute(3, 4, 0, 1, 2)
        lay.append((w, par[at + 432 * cin:at + 432 * cin + 16]))
        at += 432 * cin + 16
    conv = lambda a, i: torch.relu(F.conv3d(a, lay[i][0], lay[i][1], padding=1))  # noqa: E731
    up = lambda a: F.interpolate(a, scale_factor=2, mode="nearest")  # noqa: E731
    e = [conv(x.double().reshape(1, 2, D, D, D), 0)]
    for i in range(1, 4):
        e.append(conv(F.avg_pool3d(e[-1], 2), i))
    d = e[3]
    for i, l in ((4, 2), (5, 1), (6, 0)):
        d = conv(up(d) + e[l], i)
    out = (d[0] * par[at:at + 16, None, None, None]).sum(0) + par[at + 16]
    return [out.detach().reshape(-1), None]


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "step":
        return None  # a nonlinear step: four coupled systems, solved twice
    if kind == "learned":
        return _network(*_learned_inputs(c, seed)[:2], c["grid"])
    nodes = _nodes_of(_spec(c))
    if kind == "solve":
        return _solve_inputs(c, nodes, seed)[3]
    if kind == "apply":
        phi, u, mu, xs = _apply_inputs(c, nodes.xyz, seed)
        phi = phi.double() - (1.0 if c["prec"] == "bf16" else 0.0)
        u, mu = [a.double() for a in u], mu.double()
        return [_operator(nodes, op, _params(c), phi, u, mu, x.double())
                for op, x in zip(c["ops"].split(","), xs)]
    if kind == "rhs":
        return _right_hand_sides(nodes, _params(c), _rhs_inputs(c, nodes.xyz, seed))
    f = {k: v for k, v in _state_inputs(c, nodes.xyz, seed).items()}
    return _remeshed(c, nodes, f)
