"""The work that users of this framework have it do, as cases that can be timed and compared.

Families ("what" of a case), each through the public entry points of paper_2603_29621_gb300.api:
  apply   one operator application (Problem.vmult): the inner loop of every solver, and what a
          program with its own Krylov method calls; FP64 is the outer residual, FP32 the multigrid's
  smooth  one smoothing step from zero on the finest level (Problem.smooth)
  vcycle  one multigrid V-cycle (Problem.vcycle): the preconditioner
  solve   a whole preconditioned FGMRES solve (Problem.solve)

Kinds: "ns" (linearised stabilised Navier--Stokes, Q_k Q_k, frozen Taylor--Green state), "stokes"
(Taylor--Hood Q_k/Q_{k-1}) and "a" (its velocity block).  Meshes are the unit square / cube with n cells
per direction, "ball" > 0 refined that many times inside the ball of radius 0.25 around the centre
(hanging nodes).  Vectors are uniform(-1, 1) with zero constrained entries, as the increments and residuals
of a solve have them.  A problem (mesh tables, hierarchy, workspaces) is laid out once and kept, as a program
that solves again and again keeps it; new inputs are new vectors.
"""
import collections
import math

import numpy as np
import torch

from paper_2603_29621_gb300 import _lib as L
from paper_2603_29621_gb300 import api

KIND = {"ns": L.STAB_NS, "stokes": L.STOKES, "a": L.STOKES_A}


def _case(name, what, kind, dim, k, n, prec, ball=0, nu=1e-2, lam=0.0):
    """prec: "f32" / "f64" of the vectors, of the multigrid inside a solve; lam: smoother bound on every
    level (0: the library's own estimate)."""
    c = dict(what=what, kind=kind, dim=dim, k=k, n=n, prec=prec, ball=ball, nu=nu, lam=lam)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one product of the 64^3 Q2Q2 stabilised operator in FP32: the benchmark's headline workload
        _case("ns_apply_q2_n64_f32", "apply", "ns", 3, 2, 64, "f32"),
        # the same operator in FP64 at 48^3: the residual of every outer iteration of a mixed-precision solve
        _case("ns_apply_q2_n48_f64", "apply", "ns", 3, 2, 48, "f64"),
        # cubic elements on an odd mesh, as requests of the serving stream bring them
        _case("ns_apply_q3_n31_f32", "apply", "ns", 3, 3, 31, "f32"),
        # five relaxation sweeps on linear elements, odd mesh: the degree of the coarse part of every hierarchy
        _case("ns_smooth_q1_n45_f32", "smooth", "ns", 3, 1, 45, "f32", lam=3.0),
        # the FP32 preconditioner of the 48^3 problem: seven levels
        _case("ns_vcycle_q2_n48_f32", "vcycle", "ns", 3, 2, 48, "f32", lam=3.0),
        # the same on the smallest mesh that the serving stream has: launches and latency
        _case("ns_vcycle_q2_n8_f32", "vcycle", "ns", 3, 2, 8, "f32", lam=3.0),
        # FP64 multigrid (the default precision) on an odd mesh with non-nested levels
        _case("ns_vcycle_q2_n21_f64", "vcycle", "ns", 3, 2, 21, "f64", lam=3.0),
        # a whole solve of the serving stream: FP32 multigrid inside FP64 FGMRES
        _case("ns_solve_q2_n20_f32", "solve", "ns", 3, 2, 20, "f32"),
        # the smallest call: 2D Stokes on 16 x 16 cells in FP64
        _case("stokes_apply_2d_q2_n16_f64", "apply", "stokes", 2, 2, 16, "f64", nu=1.0),
        # the outer product of a Taylor--Hood request of the serving stream
        _case("stokes_apply_q3_n24_f64", "apply", "stokes", 3, 3, 24, "f64", nu=1.0),
        # Stokes on a locally refined mesh with hanging nodes, the product inside its preconditioner
        _case("stokes_apply_q2_ball24_f32", "apply", "stokes", 3, 2, 24, "f32", ball=2, nu=1.0),
        # the velocity block's V-cycle (p-, then h-coarsening) on a locally refined mesh
        _case("a_vcycle_q2_ball16_f32", "vcycle", "a", 3, 2, 16, "f32", ball=2, nu=1.0),
    ]


def draw(rng):
    """One more case of the same families and ranges."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    nu = float("%.3g" % math.exp(rng.uniform(math.log(1e-3), 0.0)))
    f = rng.choice(["ns_apply", "ns_apply", "ns_smooth", "ns_vcycle", "ns_vcycle", "ns_solve", "stokes_apply", "ball"])
    k = rng.choice([1, 2, 2, 3])
    prec = rng.choice(["f32", "f32", "f64"])
    if f == "ns_apply":
        if rng.random() < 0.15:
            return _case("", "apply", "ns", 2, k, size(16, 192), prec, nu=nu)
        return _case("", "apply", "ns", 3, k, size(8, {1: 90, 2: 56, 3: 36}[k] if prec == "f32" else {1: 48, 2: 32, 3: 20}[k]),
                     prec, nu=nu)
    if f == "ns_smooth":
        return _case("", "smooth", "ns", 3, k, size(8, {1: 64, 2: 36, 3: 24}[k]), prec, nu=nu, lam=3.0)
    if f == "ns_vcycle":
        return _case("", "vcycle", "ns", 3, k, size(8, ({1: 48, 2: 40, 3: 20} if prec == "f32" else {1: 32, 2: 20, 3: 12})[k]),
                     prec, nu=nu, lam=3.0)
    if f == "ns_solve":
        return _case("", "solve", "ns", 3, rng.choice([1, 2]), size(8, 20), "f32", nu=rng.choice([1e-2, 2e-2, 5e-2]))
    if f == "stokes_apply":
        return _case("", "apply", "stokes", rng.choice([2, 3]), rng.choice([2, 3]), size(8, 28), prec, nu=nu)
    return _case("", "apply", rng.choice(["stokes", "a"]), 3, 2, size(8, 20), prec, ball=rng.choice([1, 2]), nu=nu)


# ------------------------------------------------------------------------------------ running
_plans = collections.OrderedDict()  # problems laid out by this program, the last few


def _plan(case):
    key = tuple(sorted((a, b) for a, b in case.items() if a != "name"))
    if key not in _plans:
        while len(_plans) >= 3:
            ctx, prob = _plans.popitem(last=False)[1]
            prob.close()
            ctx.close()
        ctx = api.Context(0)
        m = api.Mesh(ctx, case["dim"], case["n"])
        if case["ball"]:
            m.refine_ball((0.5, 0.5, 0.5), 0.25, case["ball"])
        _plans[key] = ctx, api.Problem(
            ctx, m, kind=KIND[case["kind"]], degree=case["k"], nu=case["nu"],
            dt=1e-2 if case["kind"] == "ns" else 0.0, lambda_max=case["lam"], tol=1e-13, maxit=200,
            mg_precision=L.FP32 if case["prec"] == "f32" else L.FP64)
    _plans.move_to_end(key)
    return _plans[key][1]


def _dtype(case):
    return torch.float32 if case["prec"] == "f32" and case["what"] != "solve" else torch.float64


def _random(case, seed, n):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (2.0 * torch.rand(n, generator=g, device="cuda", dtype=torch.float64) - 1.0).to(_dtype(case))


def prepare(case, seed):
    prob = _plan(case)
    cycle = case["what"] in ("vcycle", "smooth")
    x = _random(case, seed, prob.info.cycle_dofs if cycle else prob.info.n_dofs)
    x[torch.as_tensor(prob.constrained(0 if cycle else L.OP_SYSTEM), device="cuda")] = 0
    if case["what"] == "solve":  # a right-hand side whose solution is known
        b = torch.empty_like(x)
        prob.vmult(x, b)
        x = b
    return dict(what=case["what"], prob=prob, src=x, dst=torch.zeros_like(x))


def run(s):
    p = s["prob"]
    if s["what"] == "apply":
        return p.vmult(s["src"], s["dst"])
    if s["what"] == "smooth":
        return p.smooth(0, s["src"], s["dst"], x_is_zero=True)
    if s["what"] == "vcycle":
        return p.vcycle(s["src"], s["dst"])
    p.solve(s["src"], s["dst"])
    return s["dst"]


# ------------------------------------------------------------------------------- what it cannot do without
def _cells(case):
    """Cells and nodes of the finest mesh (refined meshes: the ball's cells are replaced by 2^dim each)."""
    n, dim = case["n"], case["dim"]
    cells = float(n ** dim)
    ball = 4.0 / 3.0 * math.pi * 0.25 ** 3 if dim == 3 else math.pi * 0.25 ** 2
    for level in range(case["ball"]):
        cells += ball * (n * 2 ** level) ** dim * (2 ** dim - 1)
    return cells


def _product(kind, dim, k, cells, es):
    """Bytes (vectors in and out, the frozen state's nodal fields) and operations (sum factorisation, every
    lane of the tensor product used once) of one product."""
    q, nodes = k + 1, cells * k ** dim
    fields = {"ns": dim + 1, "stokes": dim, "a": dim}[kind]
    dofs = nodes * fields + (cells * (k - 1) ** dim if kind == "stokes" else 0)
    sweep = 2.0 * dim * q ** (dim + 1)
    ops = cells * fields * 4 * sweep
    if kind == "ns":  # + second derivatives and the pointwise terms
        ops += cells * (dim * sweep + 180.0 * q ** dim * dim / 3)
    elif kind == "stokes":
        ops += cells * (2 * sweep + 40.0 * q ** dim)
    return es * (2 * dofs + (nodes * fields if kind == "ns" else 0)), ops


def work(case):
    kind, dim, k, cells = case["kind"], case["dim"], case["k"], _cells(case)
    es = 4 if _dtype(case) == torch.float32 else 8
    b, f = _product(kind, dim, k, cells, es)
    if case["what"] == "smooth":
        return {"bytes": b, "flops": 4 * f}
    if case["what"] in ("vcycle", "solve"):
        # ten products (5 + 5 sweeps from zero, one residual) on a hierarchy of geometrically smaller levels
        flops = 10 * f * (8 / 7 if dim == 3 else 4 / 3) if kind == "ns" else 10 * (f + _product(kind, dim, 1, cells, es)[1])
        if case["what"] == "solve":
            flops = 8 * (flops + f)
        return {"bytes": b, "flops": flops}
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------------------- plain 64-bit values
def _gll(k):
    return {1: [0.0, 1.0], 2: [0.0, 0.5, 1.0], 3: [0.0, 0.5 - 0.5 / math.sqrt(5), 0.5 + 0.5 / math.sqrt(5), 1.0]}[k]


def _basis(k, pts):
    """Values, first and second derivatives of the 1D Lagrange basis on the GLL nodes at pts."""
    x = np.array(_gll(k))
    out = np.zeros((3, len(pts), k + 1))
    for a in range(k + 1):
        p = np.poly1d([1.0])
        for m in range(k + 1):
            if m != a:
                p = p * np.poly1d([1.0, -x[m]]) / (x[a] - x[m])
        for d in range(3):
            out[d, :, a] = (p.deriv(d) if d else p)(np.array(pts))
    return out


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), device="cuda")


class _Space:
    """Q_k nodes of a mesh given by its cells (level, x, y, z): node ids per cell, positions, boundary flags
    and, on refined meshes (k <= 2), the interpolation of hanging nodes, coarse cells first."""

    def __init__(self, dim, n, k, cells):
        self.dim, self.n, self.k = dim, n, k
        lev, crd = cells[:, 0], cells[:, 1:1 + dim]
        top = int(lev.max())
        loc = np.stack(np.meshgrid(*[np.arange(k + 1)] * dim, indexing="ij"), -1).reshape(-1, dim)[:, ::-1]  # x fastest
        ext = n * 2 ** top * k + 1
        scale = (2 ** (top - lev))[:, None, None]
        pos = (crd[:, None, :] * k + loc[None]) * scale
        stride = np.array([ext ** d for d in range(dim)])
        self.keys, ids = np.unique((pos * stride).sum(-1), return_inverse=True)
        self.ids = ids.reshape(len(cells), -1)
        self.ext, self.stride, self.h = ext, stride, 1.0 / (n * 2.0 ** lev)
        q = self.keys[:, None] // stride % ext
        self.boundary = ((q == 0) | (q == ext - 1)).any(1)
        x = np.zeros((len(self.keys), dim))
        x[self.ids] = (crd[:, None, :] + np.array(_gll(k))[loc][None]) * self.h[:, None, None]
        self.x = x
        self.hang = []
        done = np.zeros(len(self.keys), bool)
        half = np.stack(np.meshgrid(*[np.arange(2 * k + 1)] * dim, indexing="ij"), -1).reshape(-1, dim)[:, ::-1]
        half = half[(half % 2).any(1)]
        if top:
            w = np.ones((len(half), len(loc)))
            for d in range(dim):
                w = w * _basis(k, np.arange(2 * k + 1) / (2.0 * k))[0][half[:, d]][:, loc[:, d]]
        for level in range(top):
            sel = np.nonzero(lev == level)[0]
            key = ((crd[sel][:, None, :] * 2 * k + half[None]) * 2 ** (top - level - 1) * stride).sum(-1)
            at = np.minimum(np.searchsorted(self.keys, key), len(self.keys) - 1)
            c, s = np.nonzero(self.keys[at] == key)
            nodes, first = np.unique(at[c, s], return_index=True)
            new = ~done[nodes]
            nodes, first = nodes[new], first[new]
            done[nodes] = True
            self.hang.append((_t(nodes), _t(self.ids[sel[c[first]]]), _t(w[s[first]])))
        self.hanging = done

    def find(self, xyz):
        """Node ids of positions (refined meshes: equispaced nodes)."""
        q = np.rint(xyz * (self.ext - 1)).astype(np.int64)
        return np.searchsorted(self.keys, (q * self.stride).sum(-1))

    def distribute(self, u):
        for nodes, masters, w in self.hang:
            u[nodes] = torch.einsum("hm,hmf->hf", w, u[masters])
        return u

    def condense(self, y):
        for nodes, masters, w in reversed(self.hang):
            y.index_add_(0, masters.reshape(-1), (w[:, :, None] * y[nodes][:, None, :]).reshape(-1, y.shape[1]))
            y[nodes] = 0
        return y


def _uniform_cells(dim, n):
    g = np.stack(np.meshgrid(*[np.arange(n)] * dim, indexing="ij"), -1).reshape(-1, dim)[:, ::-1]
    return np.concatenate([np.zeros((len(g), 1), np.int64), g], 1)


class _Plain:
    """The operators by direct quadrature with full tensor-product tables, cell by cell."""

    def __init__(self, kind, dim, n, k, nu, cells=None):
        self.kind, self.dim, self.k, self.n, self.nu = kind, dim, k, n, nu
        cells = _uniform_cells(dim, n) if cells is None else cells
        self.v = _Space(dim, n, k, cells)
        self.p = _Space(dim, n, k - 1, cells) if kind == "stokes" else None
        self.nf = dim + 1 if kind == "ns" else dim
        xg, wg = np.polynomial.legendre.leggauss(k + 1)
        self.phi, self.dphi, self.lap = self.tables(k, 0.5 * (xg + 1))
        if kind == "stokes":
            self.phip = self.tables(k - 1, 0.5 * (xg + 1))[0]
        w = np.array([1.0])
        for _ in range(dim):
            w = np.outer(w, 0.5 * wg).reshape(-1)
        self.w, self.h, self.ids = _t(w), _t(self.v.h), _t(self.v.ids)
        self.bnd = _t(self.v.boundary)
        if kind == "ns":
            x, tp = self.v.x, 2 * math.pi
            s, c = np.sin(tp * x), np.cos(tp * x)
            c2 = np.cos(2 * tp * x)
            if dim == 3:
                f = [s[:, 0] * c[:, 1] * c[:, 2], -c[:, 0] * s[:, 1] * c[:, 2], 0 * s[:, 0],
                     (c2[:, 0] + c2[:, 1]) * (c2[:, 2] + 2) / 16]
            else:
                f = [s[:, 0] * c[:, 1], -c[:, 0] * s[:, 1], (c2[:, 0] + c2[:, 1]) / 16]
            self.state = _t(np.stack(f, 1))

    def tables(self, k, pts):
        b, dim = _basis(k, pts), self.dim

        def kron(orders):  # x fastest
            m = np.ones((1, 1))
            for d in range(dim):
                m = np.kron(b[orders[d]], m)
            return m
        val = kron([0] * dim)
        grad = np.stack([kron([int(d == e) for e in range(dim)]) for d in range(dim)], -1)
        lap = sum(kron([2 * int(d == e) for e in range(dim)]) for d in range(dim))
        return _t(val), _t(grad), _t(lap)

    def fields(self, u, h):
        return (torch.einsum("qa,caf->cqf", self.phi, u), torch.einsum("qad,caf->cqfd", self.dphi, u) / h[:, None, None, None],
                torch.einsum("qa,caf->cqf", self.lap, u) / h[:, None, None] ** 2)

    def local(self, u, p, sel):
        """Cell contributions [c, a, f] (and the pressure block's) of nodal cell values u (and p)."""
        dim, h, nu = self.dim, self.h[sel], self.nu
        jxw = self.w[None] * h[:, None] ** dim
        hg = h[:, None, None, None]
        if self.kind != "ns":
            g = torch.einsum("qad,caf->cqfd", self.dphi, u) / hg
            t = nu * g
            if p is None:
                return torch.einsum("qad,cqfd->caf", self.dphi, t * (jxw / h[:, None])[:, :, None, None]), None
            pq = torch.einsum("qa,ca->cq", self.phip, p)
            t = t - pq[:, :, None, None] * torch.eye(dim, device="cuda", dtype=torch.float64)
            div = torch.einsum("cqdd->cq", g)
            return (torch.einsum("qad,cqfd->caf", self.dphi, t * (jxw / h[:, None])[:, :, None, None]),
                    torch.einsum("qa,cq->ca", self.phip, -div * jxw))
        dt = 1e-2
        sv, sg, sl = self.fields(self.state[self.ids[sel]], h)
        ub, gb = sv[..., :dim], sg[..., :dim, :]
        rb = torch.einsum("cqj,cqij->cqi", ub, gb) + sg[..., dim, :] - nu * sl[..., :dim]
        tau = 1.0 / torch.sqrt((2 / dt) ** 2 + 4 * (ub * ub).sum(-1) / h[:, None] ** 2 + (12 * nu / h[:, None] ** 2) ** 2)
        v, g, lap = self.fields(u, h)
        du, dg, q, gq = v[..., :dim], g[..., :dim, :], v[..., dim], g[..., dim, :]
        conv = 1.5 / dt * du + torch.einsum("cqd,cqid->cqi", ub, dg) + torch.einsum("cqd,cqid->cqi", du, gb)
        rl = conv + gq - nu * lap[..., :dim]
        ten = nu * dg - q[..., None, None] * torch.eye(dim, device="cuda", dtype=torch.float64)
        ten = ten + tau[..., None, None] * (rl[..., :, None] * ub[..., None, :] + rb[..., :, None] * du[..., None, :])
        c0 = torch.cat([conv, torch.einsum("cqdd->cq", dg)[..., None]], -1) * jxw[..., None]
        cg = torch.cat([ten, (tau[..., None] * rl)[..., None, :]], -2) * (jxw / h[:, None])[..., None, None]
        return torch.einsum("qa,cqf->caf", self.phi, c0) + torch.einsum("qad,cqfd->caf", self.dphi, cg), None

    def free(self, u):
        """Velocity zero on the boundary (nodal array [nodes, fields])."""
        u = u.clone()
        u[:, :self.dim] = torch.where(self.bnd[:, None], 0.0, u[:, :self.dim])
        return u

    def apply(self, u, p=None):
        """Nodal [nodes, nf] (and pressure [nodes, 1]) -> the same, constrained rows identity rows."""
        a = self.v.distribute(self.free(u))
        b = self.p.distribute(p.clone()) if p is not None else None
        y, z = torch.zeros_like(u), None if p is None else torch.zeros_like(p)
        pid = None if p is None else _t(self.p.ids)
        step = 8192 if self.k > 2 else 32768
        for i in range(0, len(self.ids), step):
            s = slice(i, i + step)
            r, rp = self.local(a[self.ids[s]], None if p is None else b[pid[s], 0], s)
            y.index_add_(0, self.ids[s].reshape(-1), r.reshape(-1, self.nf))
            if p is not None:
                z.index_add_(0, pid[s].reshape(-1), rp.reshape(-1, 1))
        y = self.v.condense(y)
        hang = _t(self.v.hanging)
        y[:, :self.dim] = torch.where((self.bnd | hang)[:, None], u[:, :self.dim], y[:, :self.dim])
        y = torch.where(hang[:, None], u, y)
        if p is not None:
            z = torch.where(_t(self.p.hanging)[:, None], p, self.p.condense(z))
        return y, z

    def diagonal(self):
        """diag of the uniform operator by local unit vectors, 1 on the boundary's velocity rows."""
        nb, d = self.ids.shape[1], torch.zeros(len(self.bnd), self.nf, device="cuda", dtype=torch.float64)
        for i in range(0, len(self.ids), 8192):
            s = slice(i, i + 8192)
            u = torch.zeros(len(self.ids[s]), nb, self.nf, device="cuda", dtype=torch.float64)
            for a in range(nb):
                for f in range(self.nf):
                    u[:, a, f] = 1
                    d[:, f].index_add_(0, self.ids[s][:, a], self.local(u, None, s)[0][:, a, f])
                    u[:, a, f] = 0
        d[:, :self.dim] = torch.where(self.bnd[:, None], 1.0, d[:, :self.dim])
        return d


class _Cycle:
    """V-cycle of the stabilised operator on uniform meshes: h-, then p-coarsening, five relaxation sweeps
    around point Jacobi, dense coarse solve."""

    def __init__(self, case, levels=None):
        n, k, dim = case["n"], case["k"], case["dim"]
        seq = [(n, k)]
        while seq[-1][0] > 2:
            seq.append(((seq[-1][0] + 1) // 2, k))
        seq += [(seq[-1][0], d) for d in range(k - 1, 0, -1)]
        self.ops = [_Plain("ns", dim, m, d, case["nu"]) for m, d in seq[:levels]]
        self.omega = 2.0 / (case["lam"] / 20.0 + case["lam"])
        self.dinv = [1.0 / o.diagonal() for o in self.ops]
        if levels is None:
            c = self.ops[-1]
            size = c.bnd.numel() * c.nf
            eye = torch.eye(size, device="cuda", dtype=torch.float64)
            a = torch.stack([c.apply(e.reshape(-1, c.nf))[0].reshape(-1) for e in eye], 1)
            pres = torch.arange(dim, size, c.nf, device="cuda")
            a[pres[:, None], pres[None]] += 1.0 / len(pres)
            self.coarse = torch.linalg.inv(a)

    def smooth(self, l, b, x):
        for it in range(5):
            r = b if x is None else b - self.ops[l].apply(x)[0]
            x = self.omega * self.dinv[l] * r + (0 if x is None else x)
        return x

    def transfer(self, l):
        """1D interpolation from level l + 1 to level l."""
        f, c = self.ops[l], self.ops[l + 1]
        pos = np.array([(i // f.k + _gll(f.k)[i % f.k]) / f.n for i in range(f.k * f.n + 1)])
        m = np.zeros((len(pos), c.k * c.n + 1))
        cell = np.minimum(np.floor(pos * c.n + 1e-12).astype(int), c.n - 1)
        for i, e in enumerate(cell):
            m[i, c.k * e:c.k * e + c.k + 1] = _basis(c.k, [pos[i] * c.n - e])[0][0]
        return _t(m)

    def along(self, m, u, dim):
        shape = [round(u.shape[0] ** (1.0 / dim))] * dim
        u = u.reshape(*shape, -1)
        for d in range(dim):
            u = torch.movedim(torch.tensordot(m, u, dims=([1], [d])), 0, d)
        return u.reshape(-1, u.shape[-1])

    def cycle(self, l, b):
        o = self.ops[l]
        if l == len(self.ops) - 1:
            return (self.coarse @ b.reshape(-1)).reshape(b.shape)
        x = self.smooth(l, b, None)
        m = self.transfer(l)
        r = self.along(m.T, o.free(b - o.apply(x)[0]), o.dim)
        z = self.cycle(l + 1, self.ops[l + 1].free(r))
        x = x + o.free(self.along(m, self.ops[l + 1].free(z), o.dim))
        return self.smooth(l, b, x)


def exact(case, seed):
    kind, dim, k, n = case["kind"], case["dim"], case["k"], case["n"]
    if case["what"] == "solve":  # the right-hand side was made from its solution; the mean pressure is free
        nodes = (k * n + 1) ** dim
        x = _Plain(kind, dim, n, k, case["nu"]).free(_random(case, seed, nodes * (dim + 1)).reshape(nodes, -1))
        x[:, dim] -= x[:, dim].mean()
        return x.reshape(-1)
    if case["ball"] and case["what"] != "apply":
        return None  # a cycle on a refined mesh: the product's values stand for it
    if case["ball"]:  # the numbering of a refined mesh is the library's: taken from its support points
        prob = _plan(case)
        m = api.Mesh(prob.ctx, dim, n)
        m.refine_ball((0.5, 0.5, 0.5), 0.25, case["ball"])
        o = _Plain(kind, dim, n, k, case["nu"], m.cells().astype(np.int64))
        xyz, field = prob.support_points()
        x = _random(case, seed, len(field)).double()
        isv = field < dim
        vel = _t(o.v.find(xyz[isv]) * dim + field[isv])
        u = torch.zeros(len(o.bnd) * dim, device="cuda", dtype=torch.float64)
        isv = _t(isv)
        u[vel] = x[isv]
        p = None
        if kind == "stokes":
            at = _t(o.p.find(xyz[field == dim]))
            p = torch.zeros(len(o.p.keys), 1, device="cuda", dtype=torch.float64)
            p[at, 0] = x[~isv]
            p[_t(o.p.hanging)] = 0
        u = o.free(u.reshape(-1, dim))
        u[_t(o.v.hanging)] = 0
        y, z = o.apply(u, p)
        out = torch.empty_like(x)
        out[isv] = y.reshape(-1)[vel]
        if p is not None:
            out[~isv] = z[at, 0]
        return out
    nodes = (k * n + 1) ** dim
    nf = dim + 1 if kind == "ns" else dim
    size = nodes * nf + (((k - 1) * n + 1) ** dim if kind == "stokes" else 0)
    x = _random(case, seed, size).double()
    u = x[:nodes * nf].reshape(nodes, nf)
    o = _Plain(kind, dim, n, k, case["nu"])
    u = o.free(u)
    if case["what"] == "apply":
        y, z = o.apply(u, x[nodes * nf:, None] if kind == "stokes" else None)
        return torch.cat([y.reshape(-1)] + ([z.reshape(-1)] if z is not None else []))
    if case["what"] == "smooth":
        return _Cycle(case, 1).smooth(0, u, None).reshape(-1)
    return _Cycle(case).cycle(0, u).reshape(-1)
