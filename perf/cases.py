"""The work that users of this package have it do, as cases that can be timed.

A case is one call pattern on one synthetic problem: P1 / P2 Poisson and
Helmholtz systems and two-component elastic waves on uniform and uneven
grids of the unit square (the package's problem classes), solved through the
public entry points of ``paper_2105_07791_gb300.ndhss`` and
``paper_2105_07791_gb300.autograd``.  ``op`` says which call:

  apply         one preconditioner application P^{-1} x on a kept factor (a program with its own Krylov loop)
  apply_multi   the same for 32 right-hand sides at once
  solve         one preconditioned GMRES solve on a kept factor
  factor_solve  a new matrix on a known tree: factor it and solve (frequency sweeps, Newton and time steps)
  batched       a forest of independent problems: factor it and solve all right-hand sides in lockstep
  adjoint       misfit and gradient through the autograd function (forward solves, adjoint solves, block forms)

GMRES runs to the tolerance that the autograd model takes by default.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2105_07791_gb300 import autograd, ndhss

PREC = {"f64": ndhss.NDHSS_FP64, "f32": ndhss.NDHSS_FP32, "bf16": ndhss.NDHSS_FP32_BF16}
TOL = 1e-10
BASE = dict(op="solve", problem="helmholtz", p=1, nx=64, ny=64, k=20.0, prec="f32", hss=4, leaf=64, count=1, nrhs=1)


def _case(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # the smallest call: one application on a coarse grid, dense FP64 fronts, inside a caller's own Krylov loop
        _case("apply_poisson_32_f64", op="apply", problem="poisson", nx=32, ny=32, prec="f64", hss=-1),
        # a small whole solve in FP64 with compressed fronts (Poisson, 64 x 64 cells)
        _case("solve_poisson_64_f64", problem="poisson", nx=64, ny=64, prec="f64"),
        # a large application that streams the exact FP64 factor once
        _case("apply_helmholtz_p2_256_f64", op="apply", p=2, nx=256, ny=256, k=40.0, prec="f64", hss=-1),
        # a block of 32 right-hand sides on one FP64 factor, ragged grid
        _case("apply_multi_helmholtz_113x87_f64", op="apply_multi", nx=113, ny=87, k=25.0, prec="f64", hss=-1, nrhs=32),
        # many right-hand sides one after another on the kept mixed-precision factor: one of them
        _case("solve_helmholtz_p2_256_f32", p=2, nx=256, ny=256, k=40.0),
        # a new mid-sized system on odd, ragged grids: factor and solve
        _case("factor_solve_helmholtz_129x75_f32", op="factor_solve", nx=129, ny=75, k=30.0),
        # the main workload, both precisions: a new 256 x 256 P2 Helmholtz matrix, compressed fronts
        _case("factor_solve_helmholtz_p2_256_f32", op="factor_solve", p=2, nx=256, ny=256, k=40.0),
        _case("factor_solve_helmholtz_p2_256_f64", op="factor_solve", p=2, nx=256, ny=256, k=40.0, prec="f64"),
        # the same class at four times the unknowns with exact fronts: the largest dense eliminations
        _case("factor_solve_helmholtz_p2_512_f32_dense", op="factor_solve", p=2, nx=512, ny=512, k=80.0, hss=-1),
        # elastic waves, two components per node, three-part BF16 products
        _case("factor_solve_elastic_192_bf16", op="factor_solve", problem="elastic", nx=192, ny=192, k=0.0,
              prec="bf16", leaf=60),
        # independent uneven problems in one forest, 32 sources each
        _case("batched_helmholtz_16x32_f32", op="batched", nx=64, ny=256, k=0.0, hss=-1, count=16, nrhs=32),
        # full-waveform inversion step: misfit of 8 sources and its gradient with respect to 256 block coefficients
        _case("adjoint_helmholtz_256_f32", op="adjoint", nx=256, ny=256, k=40.0, nrhs=8),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["apply", "apply_multi", "solve", "solve", "factor_solve", "factor_solve", "factor_solve",
                     "batched", "adjoint"])
    c = dict(BASE, op=op)
    if op == "batched":
        c.update(nx=size(48, 96), k=0.0, hss=rng.choice([-1, 4]), count=rng.randint(3, 16), nrhs=rng.choice([7, 16, 32]))
        c.update(ny=size(c["nx"], 200))
        return c
    if op == "adjoint":
        c.update(nx=size(48, 200), nrhs=rng.randint(1, 8))
        c.update(ny=c["nx"], k=0.15 * c["nx"])
        return c
    c["problem"] = rng.choice(["poisson", "helmholtz", "helmholtz", "elastic"])
    c["prec"] = rng.choice(["f64", "f32", "bf16"]) if op in ("solve", "factor_solve") else "f64"
    c["p"] = rng.choice([1, 2]) if c["problem"] != "elastic" else 1
    top = {"elastic": 160, "poisson": 400, "helmholtz": 400}[c["problem"]] // c["p"]
    if c["prec"] == "f64":
        top = top * 3 // 4
    c["nx"], c["ny"] = size(24, top), size(24, top)
    c["hss"] = -1 if op in ("apply", "apply_multi") else rng.choice([-1, 4, 4])
    c["leaf"] = 60 if c["problem"] == "elastic" else 64
    c["nrhs"] = rng.choice([5, 17, 32]) if op == "apply_multi" else 1
    c["k"] = 0.15 * c["p"] * min(c["nx"], c["ny"]) if c["problem"] == "helmholtz" else 0.0
    return c


# ---- discretisation: what the caller's own program brings ---------------------------------------------------


def _element(p, tri):
    """Stiffness, mass (and P1 gradients) of one triangle with the corners ``tri`` by a collapsed Gauss rule."""
    t, w = np.polynomial.legendre.leggauss(4)
    t, w = 0.5 * (t + 1), 0.5 * w
    u, v = np.meshgrid(t, t, indexing="ij")
    x, y, wq = u.ravel(), (v * (1 - u)).ravel(), (np.outer(w, w) * (1 - u)).ravel()
    lam = np.stack([1 - x - y, x, y], 1)
    dl = np.array([[-1.0, -1.0], [1.0, 0.0], [0.0, 1.0]])
    if p == 1:
        val, grad = lam, np.broadcast_to(dl, (x.size, 3, 2))
    else:
        pairs = ((0, 1), (1, 2), (2, 0))
        val = np.concatenate([lam * (2 * lam - 1), np.stack([4 * lam[:, i] * lam[:, j] for i, j in pairs], 1)], 1)
        grad = np.concatenate([(4 * lam - 1)[:, :, None] * dl, np.stack(
            [4 * (lam[:, j, None] * dl[i] + lam[:, i, None] * dl[j]) for i, j in pairs], 1)], 1)
    J = np.stack([tri[1] - tri[0], tri[2] - tri[0]], 1)
    det = abs(np.linalg.det(J))
    g = grad @ np.linalg.inv(J)
    return np.einsum("q,qai,qbi->ab", wq, g, g) * det, np.einsum("q,qa,qb->ab", wq, val, val) * det, g[0]


class Grid:
    """The triangulated nx x ny cell grid: elements, boundary edges, and the CSR pattern their couplings make."""

    def __init__(self, nx, ny, p, ncomp=1, dirichlet=False):
        self.nx, self.ny, self.p, self.nc = nx, ny, p, ncomp
        Lx, Ly = p * nx + 1, p * ny + 1
        dev = "cuda"
        b, a = torch.meshgrid(torch.arange(ny, device=dev), torch.arange(nx, device=dev), indexing="ij")
        a, b = a.reshape(-1), b.reshape(-1)
        at = {s: (p * (a + s[0]), p * (b + s[1])) for s in ((0, 0), (1, 0), (1, 1), (0, 1))}
        tris = []
        for corners in (((0, 0), (1, 0), (1, 1)), ((0, 0), (1, 1), (0, 1))):
            pts = [at[s] for s in corners]
            if p == 2:
                pts += [((pts[i][0] + pts[j][0]) // 2, (pts[i][1] + pts[j][1]) // 2) for i, j in ((0, 1), (1, 2), (2, 0))]
            tris.append(torch.stack([y * Lx + x for x, y in pts], 1))
        self.elem = torch.stack(tris, 1).reshape(2 * nx * ny, -1)
        self.cell = torch.stack([a, b], 1).repeat_interleave(2, 0)
        hx, hy = 1.0 / nx, 1.0 / ny
        c = {s: np.array([s[0] * hx, s[1] * hy]) for s in at}
        self.ref = [_element(p, [c[s] for s in q]) for q in (((0, 0), (1, 0), (1, 1)), ((0, 0), (1, 1), (0, 1)))]
        ex, ey = torch.arange(nx, device=dev), torch.arange(ny, device=dev)
        off = range(0, p + 1) if p == 1 else (0, 2, 1)
        sides = [(torch.stack([j * Lx + p * ex + o for o in off], 1), torch.stack([ex, ex * 0 + min(j, ny - 1)], 1), hx, 1)
                 for j in (0, p * ny)] + \
                [(torch.stack([(p * ey + o) * Lx + i for o in off], 1), torch.stack([ey * 0 + min(i, nx - 1), ey], 1), hy, 0)
                 for i in (0, p * nx)]
        self.edge = torch.cat([s[0] for s in sides])
        self.edge_cell = torch.cat([s[1] for s in sides])
        self.edge_len = torch.cat([torch.full((s[0].shape[0],), s[2], dtype=torch.float64, device=dev) for s in sides])
        self.edge_normal = torch.cat([torch.full((s[0].shape[0],), s[3], device=dev) for s in sides])
        t, w = np.polynomial.legendre.leggauss(4)
        t, w = 0.5 * (t + 1), 0.5 * w
        eb = np.stack([1 - t, t], 1) if p == 1 else np.stack([(1 - t) * (1 - 2 * t), t * (2 * t - 1), 4 * t * (1 - t)], 1)
        self.edge_mass = torch.from_numpy(np.einsum("q,qa,qb->ab", w, eb, eb)).cuda()
        nodes = torch.arange(Lx * Ly, device=dev)
        xy = torch.stack([nodes % Lx, nodes // Lx], 1)
        keep = torch.ones(Lx * Ly, dtype=torch.bool, device=dev)
        if dirichlet:
            keep = (xy[:, 0] > 0) & (xy[:, 0] < Lx - 1) & (xy[:, 1] > 0) & (xy[:, 1] < Ly - 1)
        new = torch.where(keep, torch.cumsum(keep, 0) - 1, -1)
        self.n = int(keep.sum()) * ncomp
        self.lattice = xy[keep].repeat_interleave(ncomp, 0)
        self.xy = self.lattice.to(torch.float64) / torch.tensor([p * nx, p * ny], dtype=torch.float64, device=dev)

        def dofs(e):
            d = new[e]
            return d if ncomp == 1 else (ncomp * d[:, :, None] + torch.arange(ncomp, device=dev)).reshape(e.shape[0], -1)

        self.edof, self.gdof = dofs(self.elem), dofs(self.edge)
        rows = torch.cat([d.repeat_interleave(d.shape[1], 1).reshape(-1) for d in (self.edof, self.gdof)])
        cols = torch.cat([d.repeat(1, d.shape[1]).reshape(-1) for d in (self.edof, self.gdof)])
        self.used = (rows >= 0) & (cols >= 0)
        key, self.order = torch.sort((rows * self.n + cols)[self.used], stable=True)
        uniq, inv, cnt = torch.unique_consecutive(key, return_inverse=True, return_counts=True)
        self.nnz = uniq.numel()
        start = torch.cumsum(cnt, 0) - cnt
        self.slot = inv * int(cnt.max()) + torch.arange(key.numel(), device=dev) - start[inv]
        self.width = int(cnt.max())
        self.col = (uniq % self.n).to(torch.int32)
        self.rowptr = torch.searchsorted(uniq, torch.arange(self.n + 1, device=dev) * self.n).to(torch.int32)

    def per_element(self, i):
        """The two triangles' reference matrices, element after element."""
        m = torch.from_numpy(np.stack([self.ref[0][i], self.ref[1][i]])).cuda()
        return m.repeat(self.nx * self.ny, 1, 1)

    def assemble(self, ke, kg):
        """CSR values of the element matrices ``ke`` and edge matrices ``kg``, summed in a fixed order."""
        dt = torch.promote_types(ke.dtype, kg.dtype)
        v = torch.cat([ke.reshape(-1).to(dt), kg.reshape(-1).to(dt)])[self.used][self.order]
        out = torch.zeros(self.nnz * self.width, dtype=dt, device="cuda")
        out[self.slot] = v
        return out.reshape(self.nnz, self.width).sum(1)

    def tree(self, leaf):
        return ndhss.ndhss_build_tree(*self.host(), leaf)

    def host(self):
        return (np.ascontiguousarray(self.lattice.to(torch.int32).cpu().numpy()), self.rowptr.cpu().numpy(),
                self.col.cpu().numpy())


def _blocks(cells, nx, ny, nb):
    return (cells[:, 0] * nb // nx) * nb + cells[:, 1] * nb // ny


def _helmholtz_values(g, k, m, blk, eblk):
    """Complex symmetric Helmholtz values for block-wise squared slowness m (impedance on all sides)."""
    ke = g.per_element(0) - (k * k) * m[blk][:, None, None] * g.per_element(1)
    kg = -1j * k * (torch.sqrt(m)[eblk] * g.edge_len)[:, None, None] * g.edge_mass
    return g.assemble(ke, kg)


def _sources(g, rng, nrhs):
    """Gaussian point sources of width 0.02 at random places, one per right-hand side: (n, nrhs)."""
    at = torch.from_numpy(rng.uniform(0.1, 0.9, size=(nrhs, 2))).cuda()
    d2 = ((g.xy[:, None, :] - at[None]) ** 2).sum(2)
    return torch.exp(-d2 / (2 * 0.02 ** 2)) / (g.nx * g.ny * g.p ** 2)


def _system(c, rng):
    """Grid, device CSR values and right-hand sides (n, nrhs) of one problem."""
    nx, ny, p = c["nx"], c["ny"], c["p"]
    if c["problem"] == "poisson":
        g = Grid(nx, ny, p, dirichlet=True)
        vals = g.assemble(g.per_element(0), torch.zeros(g.gdof.shape[0], g.gdof.shape[1] ** 2, dtype=torch.float64, device="cuda"))
        return g, vals, torch.from_numpy(rng.uniform(-1, 1, size=(g.n, c["nrhs"]))).cuda() / (nx * ny)
    if c["problem"] == "elastic":
        g = Grid(nx, ny, p, ncomp=2)
        mid = (g.cell.to(torch.float64) + 0.5) / torch.tensor([nx, ny], dtype=torch.float64, device="cuda")

        def field():
            """A sum of 16 Fourier modes with values in [1, 4], per element."""
            kk, ph, am = rng.integers(1, 5, size=(16, 2)), rng.uniform(0, 2 * np.pi, 16), rng.uniform(0.5, 1, 16)
            f = sum(float(am[j]) * torch.cos(2 * np.pi * (mid @ torch.tensor(kk[j], dtype=torch.float64, device="cuda")) + float(ph[j]))
                    for j in range(16)) / float(am.sum())
            return 2.5 + 1.5 * f

        la, mu = field(), field()
        omega = 2 * np.pi * float(mu.min().sqrt()) * min(nx, ny) / 8
        parts = []
        for K, M, gr in g.ref:
            area = 0.5 / (nx * ny)
            div = gr.reshape(6)                                   # div of (node, component) basis functions
            eps = np.zeros((6, 2, 2))
            for a in range(3):
                for q in range(2):
                    e = np.zeros((2, 2))
                    e[q] = gr[a]
                    eps[2 * a + q] = 0.5 * (e + e.T)
            parts.append((area * np.outer(div, div), 2 * area * np.einsum("aij,bij->ab", eps, eps), np.kron(M, np.eye(2))))
        kl, km, mm = (torch.from_numpy(np.stack([parts[0][i], parts[1][i]])).cuda().repeat(nx * ny, 1, 1) for i in range(3))
        ke = la[:, None, None] * kl + mu[:, None, None] * km - omega ** 2 * mm
        ce = 2 * (g.edge_cell[:, 1] * nx + g.edge_cell[:, 0])
        cp, cs = torch.sqrt(la + 2 * mu)[ce], torch.sqrt(mu[ce])
        nrm = torch.nn.functional.one_hot(g.edge_normal, 2).to(torch.float64)
        comp = cp[:, None] * nrm + cs[:, None] * (1 - nrm)        # per edge and component
        kg = torch.einsum("ab,ec,cd->eacbd", g.edge_mass, comp * g.edge_len[:, None],
                          torch.eye(2, dtype=torch.float64, device="cuda"))
        kg = -1j * omega * kg.reshape(g.edge.shape[0], -1)
        return g, g.assemble(ke, kg), _sources(g, rng, c["nrhs"]).to(torch.complex128)
    g = Grid(nx, ny, p)
    m = torch.from_numpy(rng.uniform(0.3, 1.0, size=64)).cuda()
    vals = _helmholtz_values(g, c["k"], m, _blocks(g.cell, nx, ny, 8), _blocks(g.edge_cell, nx, ny, 8))
    return g, vals, _sources(g, rng, c["nrhs"]).to(torch.complex128)


def _opts(c):
    return ndhss.make_factor_opts(prec=PREC[c["prec"]], hss_levels=c["hss"], eps_hss=1e-6,
                                  beta=60 if c["problem"] == "elastic" else 64)


def _vtype(vals):
    return ndhss.NDHSS_C128 if vals.is_complex() else ndhss.NDHSS_R64


def _adjoint_inputs(c, seed):
    """A block model, its true and starting coefficients, sources, receivers and data-shaped targets."""
    rng = np.random.default_rng([seed, 1])
    nx, nb = c["nx"], 16
    g = Grid(nx, nx, 1)
    m = torch.from_numpy(rng.uniform(0.3, 1.0, size=nb * nb)).cuda()
    B = _sources(g, rng, c["nrhs"]).to(torch.complex128)
    rec = torch.nonzero(g.lattice[:, 1] == int(0.9 * nx)).reshape(-1)
    d = torch.from_numpy(rng.normal(size=(rec.numel(), c["nrhs"])) + 1j * rng.normal(size=(rec.numel(), c["nrhs"]))).cuda()
    return g, nb, m, B, rec, 1e-3 * d


def _batch(c, seed):
    """``count`` uneven Helmholtz problems with grids in nx .. ny cells, 10 points on the shortest wavelength."""
    got = []
    sizes = np.random.default_rng([c["count"], c["nx"], c["ny"]])   # the meshes are the case's, the rest the seed's
    for s in range(c["count"]):
        nx, ny = (int(v) for v in sizes.integers(c["nx"], c["ny"] + 1, size=2))
        rng = np.random.default_rng([seed, s])
        omega = 2 * np.pi * min(nx, ny) / 10
        g = Grid(nx, ny, 1)
        m = torch.from_numpy(rng.uniform(1.0, 3.0, size=64)).cuda() ** -2.0
        vals = _helmholtz_values(g, omega, m, _blocks(g.cell, nx, ny, 8), _blocks(g.edge_cell, nx, ny, 8))
        got.append((g, vals, _sources(g, rng, c["nrhs"]).to(torch.complex128)))
    return got


def prepare(case, seed):
    c = dict(BASE, **case)
    s = SimpleNamespace(op=c["op"])
    if c["op"] == "adjoint":
        g, nb, m, B, s.rec, s.d = _adjoint_inputs(c, seed)
        blk, eblk = _blocks(g.cell, g.nx, g.ny, nb), _blocks(g.edge_cell, g.nx, g.ny, nb)
        _, rowptr, col = g.host()

        def assemble(mb):
            v = _helmholtz_values(g, c["k"], torch.from_numpy(mb).cuda(), blk, eblk)
            return SimpleNamespace(shape=(g.n, g.n), nnz=g.nnz, indptr=rowptr, indices=col, data=v.cpu().numpy())

        mass, emass = g.per_element(1), g.edge_len[:, None, None] * g.edge_mass
        s.model = autograd.HelmholtzBlockModel(
            g.tree(c["leaf"]), assemble, c["k"], g.edof.cpu().numpy(), mass.cpu().numpy(), blk.cpu().numpy(),
            g.gdof.cpu().numpy(), emass.cpu().numpy(), eblk.cpu().numpy(), nb * nb, opts=_opts(c), tol=TOL)
        s.m, s.B = m.requires_grad_(), B.requires_grad_()
        return s
    if c["op"] == "batched":
        probs = _batch(c, seed)
        s.tree = ndhss.ndhss_build_tree_batched([g.host() for g, _, _ in probs], c["leaf"])
        off = np.concatenate([[0], np.cumsum([g.n for g, _, _ in probs])])
        eoff = np.concatenate([[0], np.cumsum([g.nnz for g, _, _ in probs])])
        s.off = off.astype(np.int64)
        s.rowptr = torch.cat([g.rowptr[(0 if i == 0 else 1):] + int(eoff[i]) for i, (g, _, _) in enumerate(probs)])
        s.col = torch.cat([g.col + int(off[i]) for i, (g, _, _) in enumerate(probs)])
        s.vals = torch.cat([v for _, v, _ in probs])
        s.B = torch.cat([b for _, _, b in probs]).t().contiguous()
        s.X = torch.zeros_like(s.B)
        s.opts = _opts(c)
        return s
    g, s.vals, b = _system(c, np.random.default_rng([seed, 0]))
    s.rowptr, s.col, s.tree, s.opts = g.rowptr, g.col, g.tree(c["leaf"]), _opts(c)
    s.b = b.contiguous() if c["op"] == "apply_multi" else b[:, 0].contiguous()
    s.x = torch.zeros_like(s.b)
    if c["op"] != "factor_solve":
        s.f = ndhss.ndhss_factor(s.tree, _vtype(s.vals), s.rowptr, s.col, s.vals, s.opts)
    return s


def run(s):
    if s.op == "apply":
        return ndhss.ndhss_apply(s.f, s.b, s.x)
    if s.op == "apply_multi":
        return ndhss.ndhss_apply_multi(s.f, s.b, s.x)
    if s.op == "solve":
        ndhss.ndhss_gmres(s.f, s.rowptr, s.col, s.vals, s.b, s.x, tol=TOL)
        return s.x
    if s.op == "factor_solve":
        f = ndhss.ndhss_factor(s.tree, _vtype(s.vals), s.rowptr, s.col, s.vals, s.opts)
        ndhss.ndhss_gmres(f, s.rowptr, s.col, s.vals, s.b, s.x, tol=TOL)
        return s.x
    if s.op == "batched":
        f = ndhss.ndhss_factor(s.tree, ndhss.NDHSS_C128, s.rowptr, s.col, s.vals, s.opts)
        ndhss.ndhss_gmres_batched(f, s.rowptr, s.col, s.vals, s.off, s.B, s.X, tol=TOL)
        return s.X
    X = autograd.HelmholtzSolve.apply(s.m, s.B, s.model)
    J = 0.5 * (X[s.rec] - s.d).abs().square().sum()
    gm, gB = torch.autograd.grad(J, (s.m, s.B))
    return {"X": X.detach(), "grad_m": gm, "grad_B": gB}


# ---- what a pass cannot do without --------------------------------------------------------------------------


def _fronts(nx, ny, p, nc, leaf, dirichlet):
    """(interior, boundary) unknowns of every front of the box nested dissection of the lattice."""
    lo, hx, hy = (1, p * nx, p * ny) if dirichlet else (0, p * nx + 1, p * ny + 1)
    out = []

    def inner(a, b, lim0, lim1):
        """The lattice lines of [a, b) with no neighbour outside it."""
        if a > lim0:
            a += 1 if p == 1 or a % 2 == 0 else 2
        if b < lim1:
            b -= 1 if p == 1 or b % 2 else 2
        return max(0, b - a)

    def edge(x0, x1, y0, y1):
        return nc * ((x1 - x0) * (y1 - y0) - inner(x0, x1, lo, hx) * inner(y0, y1, lo, hy))

    todo = [(lo, hx, lo, hy)]
    while todo:
        x0, x1, y0, y1 = todo.pop()
        n, mb = nc * (x1 - x0) * (y1 - y0), edge(x0, x1, y0, y1)
        if n <= leaf or (x1 - x0 == 1 and y1 - y0 == 1):
            out.append((n - mb, mb))
            continue
        if x1 - x0 >= y1 - y0:
            c = (x0 + x1) >> 1
            kids = [(x0, c, y0, y1), (c, x1, y0, y1)]
        else:
            c = (y0 + y1) >> 1
            kids = [(x0, x1, y0, c), (x0, x1, c, y1)]
        out.append((sum(edge(*k) for k in kids) - mb, mb))
        todo += kids
    return out


def work(case):
    """Bytes: the matrix, the kept factor (dense blocks of its fronts) where there is one, right-hand sides and
    results, once each.  Flops: the elimination of the fronts where the pass factors, and one application per
    right-hand side and sweep over the factor."""
    c = dict(BASE, **case)
    real = c["problem"] == "poisson"
    e, mul = (8, 2) if real else (16, 8)
    fe = e if c["prec"] == "f64" else e // 2
    nc = 2 if c["problem"] == "elastic" else 1
    sizes = [(c["nx"], c["ny"])]
    if c["op"] == "batched":
        r = np.random.default_rng([c["count"], c["nx"], c["ny"]])
        sizes = [tuple(int(v) for v in r.integers(c["nx"], c["ny"] + 1, size=2)) for _ in range(c["count"])]
    n = nnz = fac = elim = 0
    for nx, ny in sizes:
        fr = _fronts(nx, ny, c["p"], nc, c["leaf"], real)
        nn = nc * ((c["p"] * nx - 1) * (c["p"] * ny - 1) if real else (c["p"] * nx + 1) * (c["p"] * ny + 1))
        n, nnz = n + nn, nnz + nn * nc * (7 if c["p"] == 1 else 11.5)
        fac += sum(i * i + 2 * i * b for i, b in fr)
        elim += sum(i ** 3 / 3 + i * i * b + i * b * b for i, b in fr)
    cols = c["nrhs"]
    matrix = nnz * (e + 4) + 4 * n
    if c["op"] in ("apply", "apply_multi"):
        return {"bytes": fac * fe + 2 * n * e * cols, "flops": mul * fac * cols}
    if c["op"] == "solve":
        return {"bytes": matrix + fac * fe + 2 * n * e, "flops": mul * (fac + nnz)}
    vectors = (4 if c["op"] == "adjoint" else 2) * n * e * cols
    return {"bytes": matrix + vectors, "flops": mul * (elim + (2 if c["op"] == "adjoint" else 1) * cols * (fac + nnz))}


# ---- 64-bit results without this package --------------------------------------------------------------------


class _Direct:
    """Block-tridiagonal LU over strips of lattice rows (unknowns are numbered row after row), one refinement step."""

    def __init__(self, g, vals):
        n = g.n
        strip = g.lattice[:, 1] // g.p
        strip = strip - strip[0]
        ns = int(strip[-1]) + 1
        o = torch.searchsorted(strip, torch.arange(ns + 1, device="cuda")).tolist()
        rp = g.rowptr.tolist()
        rows = torch.repeat_interleave(torch.arange(n, device="cuda"), (g.rowptr[1:] - g.rowptr[:-1]).long())
        cols = g.col.long()
        self.A = torch.sparse_csr_tensor(g.rowptr.long(), cols, vals, size=(n, n))
        self.o, self.ns = o, ns
        self.low, self.lu, self.X = [], [], []
        prev = None
        for s in range(ns):
            a, z = rp[o[s]], rp[o[s + 1]]
            lo, hi = o[max(s - 1, 0)], o[min(s + 2, ns)]
            D = torch.zeros(o[s + 1] - o[s], hi - lo, dtype=vals.dtype, device="cuda")
            D[rows[a:z] - o[s], cols[a:z] - lo] = vals[a:z]
            L, M, U = D[:, :o[s] - lo], D[:, o[s] - lo:o[s + 1] - lo].clone(), D[:, o[s + 1] - lo:]
            if s:
                k, Xp = prev
                M[:, k] -= L @ Xp
            lu = torch.linalg.lu_factor(M)
            nz = torch.nonzero((U != 0).any(0)).reshape(-1)
            Xs = torch.linalg.lu_solve(*lu, U[:, nz].contiguous()) if nz.numel() else U[:, nz]
            prev = (nz, Xs)
            self.low.append(L.contiguous())
            self.lu.append(lu)
            self.X.append(prev)

    def _solve(self, b):
        o, y = self.o, []
        for s in range(self.ns):
            r = b[o[s]:o[s + 1]]
            if s:
                r = r - self.low[s] @ y[-1]
            y.append(torch.linalg.lu_solve(*self.lu[s], r.contiguous()))
        for s in range(self.ns - 2, -1, -1):
            k, Xs = self.X[s]
            if k.numel():
                y[s] = y[s] - Xs @ y[s + 1][k]
        return torch.cat(y)

    def __call__(self, b):
        x = self._solve(b)
        return x + self._solve(b - self.A @ x)


def exact(case, seed):
    c = dict(BASE, **case)
    if c["nx"] * c["p"] * c["ny"] * c["p"] > 520 * 520 and c["op"] != "batched":
        return None                                              # the direct solve takes too long
    if c["op"] == "batched":
        return torch.cat([_Direct(g, v)(b) for g, v, b in _batch(c, seed)]).t().contiguous()
    if c["op"] == "adjoint":
        g, nb, m, B, rec, d = _adjoint_inputs(c, seed)
        blk, eblk = _blocks(g.cell, g.nx, g.ny, nb), _blocks(g.edge_cell, g.nx, g.ny, nb)
        solve = _Direct(g, _helmholtz_values(g, c["k"], m, blk, eblk))
        X = solve(B)
        G = torch.zeros_like(X)
        G[rec] = X[rec] - d
        lam = solve(G.conj().resolve_conj()).conj().resolve_conj()

        def forms(dof, mats, b):
            q = torch.einsum("eas,eab,ebs->e", lam[dof].conj(), mats.to(torch.complex128), X[dof])
            return torch.stack([q[b == j].sum() for j in range(nb * nb)])

        qm = forms(g.edof, g.per_element(1), blk)
        qe = forms(g.gdof, g.edge_len[:, None, None] * g.edge_mass, eblk)
        return {"X": X, "grad_m": (c["k"] ** 2 * qm + 0.5j * c["k"] / torch.sqrt(m) * qe).real, "grad_B": lam}
    g, vals, b = _system(c, np.random.default_rng([seed, 0]))
    if c["op"] == "apply_multi":
        return _Direct(g, vals)(b)
    return _Direct(g, vals)(b[:, :1])[:, 0]
