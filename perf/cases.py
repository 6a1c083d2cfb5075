"""Performance cases: what a program does with this solver, through its public calls.

A case is one pass of one of these (every pass works on unit squares or cubes with the boundary of
the bench workload: a plane wave as the Dirichlet trace on x = 0, impedance on the other sides):

  apply   System.apply_local: one operator (T, P^-1 or T^-1 of every subdomain) on a vector of the
          caller's own Krylov loop, taken back in (subdomain, global DOF) order
  sweep   System.sweep: one DDM sweep, every subdomain's GMRES solve and the interface exchange:
          the unit of work of the interface iteration
  setup   System(...) on a kept mesh, its sources and the first preconditioner apply, which
          factorises: what each iterate of a coefficient search pays before it can solve
  solve   System.solve: a whole solve to a given residual
  grad    autograd.solve, a loss on the centre of the domain and its backward pass: assembly,
          forward solve and adjoint solve

`exact` holds plain 64-bit torch/numpy finite elements on the same grids (a direct block-tridiagonal
solve over the columns of cells), independent of the package.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2105_11993_gb300 as thm
from paper_2105_11993_gb300 import autograd


def listed():
    sq = dict(dim=2, ny=0, nz=0, precond="blockdiag", relax=0, problems=0)
    return [
        # the smallest call: a preconditioner apply on the 32x32 order-1 parity problem, launch-bound
        dict(sq, name="pinv_square32_p1", kind="apply", op="PINV", mode="fp64", order=1, nx=32, sx=2, omega=4 * math.pi),
        # the operator and the preconditioner alone at the bench workload's size
        dict(sq, name="T_square256_p2", kind="apply", op="T", mode="fp64", order=2, nx=256, sx=8, omega=40 * math.pi),
        dict(sq, name="pinv_square256_p2", kind="apply", op="PINV", mode="fp64", order=2, nx=256, sx=8, omega=40 * math.pi),
        # the full 2x2 block operator's inverse, ragged: 100 cells over 3 subdomains, not square
        dict(sq, name="tinv_square100x77_p2", kind="apply", op="TINV", mode="fp64", order=2, nx=100, ny=77, sx=3,
             omega=15 * math.pi),
        # a sweep of the bench workload in mixed precision: about 360 of these make its solve
        dict(sq, name="sweep_square256_p2_mixed", kind="sweep", mode="mixed", order=2, nx=256, sx=8, omega=40 * math.pi),
        # the FP64 baseline's sweep, a quarter of the bench domain (4x4 of its subdomains)
        dict(sq, name="sweep_square128_p2_fp64", kind="sweep", mode="fp64", order=2, nx=128, sx=4, omega=20 * math.pi),
        # a 3-D sweep, lowest order, mixed precision, cells of the 64^3 workload at half its side
        dict(sq, name="sweep_cube32_p1_mixed", kind="sweep", dim=3, mode="mixed", order=1, nx=32, ny=32, nz=32, sx=4,
             omega=8 * math.pi),
        # re-assembly and factorisation with new coefficients on the bench mesh, the FP64 factors
        dict(sq, name="setup_square256_p2", kind="setup", mode="fp64", order=2, nx=256, sx=8, omega=40 * math.pi),
        # a small whole solve, FP64: many launches of little work
        dict(sq, name="solve_square32_p1_fp64", kind="solve", mode="fp64", order=1, nx=32, sx=2, omega=4 * math.pi, rtol=1e-10),
        # a whole mixed-precision solve with the bench's options and phase per cell on 2x2 subdomains
        dict(sq, name="solve_square48_p2_mixed", kind="solve", mode="mixed", order=2, nx=48, sx=2, omega=7.5 * math.pi,
             rtol=1e-10, relax=1),
        # a batch of independent problems of uneven size and frequency in one system
        dict(sq, name="batch_sweep_48_p1_mixed", kind="sweep", mode="mixed", order=1, nx=128, sx=0, omega=32 * math.pi,
             problems=48),
        # differentiation in 3-D, the 12^3 gradient check at half its side: forward and adjoint solve
        dict(sq, name="grad_cube6_p1_mixed", kind="grad", dim=3, mode="mixed", order=1, nx=6, ny=6, nz=6, sx=2,
             omega=1.5 * math.pi, rtol=1e-10, relax=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "sweep", "sweep", "sweep", "setup", "solve", "grad"])
    c = dict(kind=kind, dim=2, order=rng.choice([1, 2]), mode=rng.choice(["fp64", "mixed"]), ny=0, nz=0, precond="blockdiag",
             relax=0, problems=0)
    if kind == "apply":
        c.update(op=rng.choice(["T", "PINV", "TINV"]), mode="fp64")
    if kind == "setup":
        c.update(mode="fp64")
    if kind in ("solve", "grad"):
        c.update(rtol=1e-10)
    three = c.get("op") != "TINV" and rng.random() < 0.3
    if three:
        lo, hi = {"apply": (6, 32), "sweep": (6, 32), "setup": (6, 32), "solve": (3, 5), "grad": (3, 4)}[kind]
        n = _log_int(rng, lo, hi)
        c.update(dim=3, order=1, nx=n, ny=max(3, n - rng.randint(0, 3)), nz=max(3, n - rng.randint(0, 3)))
        c["sx"] = max(2 if kind == "sweep" else 1, min(4, round(n / rng.uniform(5, 9))))
    else:
        # whole solves are small: with the Eq. 7 preconditioner their iteration counts make them long
        full = c["order"] == 2 and kind in ("solve", "grad") and rng.random() < 0.4
        lo, hi = {"apply": (12, 256), "sweep": (12, 160), "setup": (12, 256), "solve": (8, 20), "grad": (6, 12)}[kind]
        if full:
            hi *= 4
        c["nx"] = _log_int(rng, lo, hi)
        c["ny"] = max(lo, c["nx"] - rng.randint(0, 9))
        c["sx"] = max(2 if kind == "sweep" else 1, min(8, round(c["nx"] / rng.uniform(14, 34))))
        if full:
            c.update(precond="full", relax=1)
        elif kind == "sweep" and rng.random() < 0.3:
            c.update(order=1, sx=0, nx=rng.randint(24, 96), ny=0, problems=rng.randint(5, 24))
    # phase per cell: from coarse lowest-order (6 cells per wavelength) to well resolved
    c["omega"] = c["nx"] * rng.uniform(0.25, 0.8 if c["order"] == 1 else 0.6)
    return c


# --------------------------------------------------------------------------
# Grids and inputs
# --------------------------------------------------------------------------
class Grid:
    """n cells per side on the unit square or cube in s blocks per side (sizes differ by at most a cell)."""

    def __init__(self, n, s):
        self.n, self.dim = tuple(n), len(n)
        idx = np.indices(self.n[::-1]).reshape(self.dim, -1)[::-1]                # cell i, j(, k), i fastest
        nv = np.array([1, n[0] + 1, (n[0] + 1) * (n[1] + 1)][:self.dim])
        corner = np.indices((2,) * self.dim).reshape(self.dim, -1)[::-1]
        self.cells = (nv @ idx)[:, None] + (nv @ corner)[None, :]
        self.cell_idx = idx
        v = np.indices(tuple(m + 1 for m in self.n[::-1])).reshape(self.dim, -1)[::-1]
        self.h = [1.0 / m for m in self.n]
        self.coords = np.ascontiguousarray((v * np.array(self.h)[:, None]).T)
        blk = [idx[a] * s // self.n[a] for a in range(self.dim)]
        self.cell_sub = (blk[0] + s * blk[1] + (s * s * blk[2] if self.dim == 3 else 0)).astype(np.int32)
        self.bfaces, self.btag = [], []
        for a in range(self.dim):
            for end in (0, 1):
                c = self.cells[idx[a] == end * (self.n[a] - 1)]
                f = c[:, corner[a] == end]
                self.bfaces.append(f)
                self.btag.append(np.full(len(f), thm.TAG_DIRICHLET if (a, end) == (0, 0) else thm.TAG_IMPEDANCE, np.uint8))
        self.bfaces, self.btag = np.concatenate(self.bfaces), np.concatenate(self.btag)


def _problems(case, seed):
    """[(grid, mu^-1 per cell, omega)]: one problem, or a batch of uneven ones."""
    r = np.random.default_rng([7, seed])
    if case["problems"]:
        sizes = np.random.default_rng(case["problems"] * 1000 + case["nx"])       # the mesh is the case's, not the seed's
        out = []
        for _ in range(case["problems"]):
            n = int(sizes.integers(16, case["nx"] + 1))
            g = Grid((n, n), -(-n // 32))
            om = min(float(r.uniform(2 * math.pi, max(8.0, case["omega"]))), 1.0 * n)
            out.append((g, np.exp(0.3 * r.standard_normal(n * n)), om))
        return out
    n = (case["nx"], case["ny"] or case["nx"], case["nz"])[:case["dim"]]
    g = Grid(n, case["sx"])
    if case["dim"] == 2 and case["order"] == 2:                                     # constant on 16x16-cell tiles
        t = r.uniform(0.5, 2.0, (-(-n[1] // 16), -(-n[0] // 16)))
        mu = t[g.cell_idx[1] // 16, g.cell_idx[0] // 16]
    elif case["dim"] == 2:
        mu = np.exp(0.3 * r.standard_normal(len(g.cells)))
    else:                                                                           # smooth in space
        k = r.integers(1, 4, (6, 3)) * math.pi
        x = [(g.cell_idx[a] + 0.5) * g.h[a] for a in range(3)]
        w = sum(r.standard_normal() * np.cos(k[q, 0] * x[0]) * np.cos(k[q, 1] * x[1]) * np.cos(k[q, 2] * x[2]) for q in range(6))
        mu = np.exp(0.3 * w / w.std())
    return [(g, np.ascontiguousarray(mu), float(case["omega"]))]


def _vector(n, seed, k):
    r = torch.Generator(device="cuda").manual_seed(seed * 10 + k)
    return torch.randn(n, dtype=torch.complex128, device="cuda", generator=r)


def _pol(dim):
    return np.eye(dim)[1].astype(np.complex128), np.eye(dim)[0]


def prepare(case, seed):
    probs = _problems(case, seed)
    pol, d = _pol(case["dim"])
    if case["problems"]:
        mesh, _ = thm.Mesh.batch([g for g, _, _ in probs], case["order"])
        omega = np.array([w for _, _, w in probs])
    else:
        mesh = thm.Mesh.from_workload(probs[0][0], case["order"])
        omega = probs[0][2]
    mu = torch.tensor(np.concatenate([m for _, m, _ in probs]), device="cuda")
    st = dict(case=case, mesh=mesh, mu=mu, omega=omega, pol=pol, dir=d)
    if case["kind"] == "grad":
        g = probs[0][0]
        st["mask"] = torch.tensor(_centre_mask(g, case["order"]), device="cuda")
        st["mu"].requires_grad_(True)
        st["omega"] = torch.tensor(omega, dtype=torch.float64, device="cuda", requires_grad=True)
        return st
    sysg = thm.System(mesh, mu, omega, 1.0, pol, d)
    if case["kind"] == "sweep":
        st["g"] = 1e-2 * _vector(sysg.n_iface, seed, 1)
    if case["kind"] in ("apply", "setup"):
        st["x"] = _vector(sysg.n_local, seed, 2)
    if case["kind"] in ("apply", "setup", "sweep"):
        gd, sub = sysg.local_dofs()
        st["order"] = torch.tensor(np.lexsort((gd, sub)), device="cuda")            # to (subdomain, global DOF) order
        if "x" in st:
            x = torch.empty_like(st["x"])
            x[st["order"]] = st["x"]
            st["x"] = x
    if case["kind"] != "setup":
        st["sys"] = sysg
    return st


_OPS = {"T": thm.OP_T, "PINV": thm.OP_PINV, "TINV": thm.OP_TINV}


def run(st):
    c = st["case"]
    if c["kind"] == "apply":
        return st["sys"].apply_local(_OPS[c["op"]], st["x"], mode=c["mode"])[st["order"]]
    if c["kind"] == "setup":
        s = thm.System(st["mesh"], st["mu"], st["omega"], 1.0, st["pol"], st["dir"])
        return s.local_sources()[st["order"]], s.apply_local(thm.OP_PINV, st["x"], mode=c["mode"])[st["order"]]
    if c["kind"] == "sweep":
        g, u, _ = st["sys"].sweep(st["g"], with_sources=True, mode=c["mode"], inner_tol=1e-12, precond=c["precond"])
        return g, u[st["order"]]
    if c["kind"] == "solve":
        return st["sys"].solve(mode=c["mode"], rtol=c["rtol"], relax=c["relax"], precond=c["precond"])[0]
    st["mu"].grad = st["omega"].grad = None
    u = autograd.solve(st["mesh"], st["mu"], st["omega"], 1.0, st["pol"], st["dir"], mode=c["mode"], rtol=c["rtol"],
                       relax=c["relax"], precond=c["precond"])
    loss = (st["mask"] * (u.real ** 2 + u.imag ** 2)).sum()
    loss.backward()
    return u.detach(), st["mu"].grad, st["omega"].grad


# --------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------
def _sizes(case):
    """(local DOFs, stored entries of the operators) over all problems, from the grid alone."""
    dofs = nnz = 0
    for g, _, _ in _problems(case, 0):
        n = np.array(g.n, float)
        if g.dim == 3:
            e = 3 * n.prod() + n[0] * n[1] + n[1] * n[2] + n[0] * n[2] + n.sum()
            dofs += e
            nnz += 33 * e                                        # an edge couples to the edges of its 4 cells
        else:
            e = 2 * n.prod() + n.sum()
            dofs += e if case["order"] == 1 else 2 * e + 4 * n.prod()
            nnz += 7 * e if case["order"] == 1 else 20 * 2 * e + 12 * 4 * n.prod()
    return dofs, nnz


def work(case):
    """One read of the inputs and the operator's entries and one write of the outputs; for iterations,
    that much per operator apply with a typical count of them (an FP64 or FP32 entry each)."""
    dofs, nnz = _sizes(case)
    b = 4 if case["mode"] == "mixed" else 8
    steps = {"apply": 1, "setup": 1, "sweep": 40, "solve": 40 * 60, "grad": 2 * 40 * 60}[case["kind"]]
    if case["precond"] == "full":
        steps = max(1, steps // 20)
    return {"bytes": steps * (nnz * b + 2 * dofs * 2 * b), "flops": steps * 4.0 * nnz}


# --------------------------------------------------------------------------
# 64-bit values, independent of the package
# --------------------------------------------------------------------------
def _numbering(g, order):
    """cell DOFs: edges in lexicographic (lo, hi) order; order 2: 2e, 2e + 1, then 4 bubbles a cell.
    (On these grids every local edge runs from its lower to its higher vertex id: all signs are +1.)"""
    le = [(0, 1), (2, 3), (0, 2), (1, 3)] if g.dim == 2 else \
        [(0, 1), (2, 3), (4, 5), (6, 7), (0, 2), (1, 3), (4, 6), (5, 7), (0, 4), (1, 5), (2, 6), (3, 7)]
    nv = len(g.coords)
    key = np.stack([g.cells[:, a] * nv + g.cells[:, b] for a, b in le], 1)
    edges, inv = np.unique(key, return_inverse=True)
    inv = inv.reshape(key.shape)
    if order == 1:
        return inv, len(edges), edges, 1
    bub = 2 * len(edges) + 4 * np.arange(len(g.cells))[:, None] + np.arange(4)
    both = np.stack([2 * inv, 2 * inv + 1], 2).reshape(len(inv), -1)
    return np.concatenate([both, bub], 1), 2 * len(edges) + 4 * len(g.cells), edges, 2


def _centre_mask(g, order):
    cd, n, _, _ = _numbering(g, order)
    inside = np.all([(g.cell_idx[a] >= g.n[a] // 3) & (g.cell_idx[a] < g.n[a] - g.n[a] // 3) for a in range(g.dim)], axis=0)
    m = np.zeros(n)
    m[cd[inside].ravel()] = 1.0
    return m


def _element(g, order):
    """Curl-curl and mass matrices of a cell (all cells of a grid are alike), Gauss quadrature."""
    x, w = np.polynomial.legendre.leggauss(5)
    x, w = 0.5 * (x + 1), 0.5 * w
    P = np.stack(np.meshgrid(*[x] * g.dim, indexing="ij")).reshape(g.dim, -1)
    W = np.prod(np.stack(np.meshgrid(*[w] * g.dim, indexing="ij")).reshape(g.dim, -1), 0)
    z, one = np.zeros_like(P[0]), np.ones_like(P[0])
    vals, curls = [], []
    q, dq = (lambda t: t * (1 - t)), (lambda t: 1 - 2 * t)
    if g.dim == 2:
        s, t = P
        wh = [((1 - t, z), one), ((t, z), -one), ((z, 1 - s), -one), ((z, s), one)]
        gr = [(dq(s) * (1 - t), -q(s)), (dq(s) * t, q(s)), (-q(t), dq(t) * (1 - s)), (q(t), dq(t) * s)]
        for k in range(4):
            vals.append(wh[k][0]); curls.append((wh[k][1],))
            if order == 2:
                vals.append(gr[k]); curls.append((z,))
        if order == 2:
            vals += [(q(t) * (1 - s), z), (q(t) * s, z), (z, q(s) * (1 - t)), (z, q(s) * t)]
            curls += [(-dq(t) * (1 - s),), (-dq(t) * s,), (dq(s) * (1 - t),), (dq(s) * t,)]
    else:
        for a in range(3):
            b, c = [k for k in range(3) if k != a]
            for ec in (0, 1):
                for eb in (0, 1):
                    Lb, Lc = (P[b] if eb else 1 - P[b]), (P[c] if ec else 1 - P[c])
                    v, k = [z, z, z], [z, z, z]
                    v[a] = Lb * Lc
                    db, dc = (2 * eb - 1) * Lc, (2 * ec - 1) * Lb              # derivatives along b and c
                    sg = 1 if (a, b, c) in ((0, 1, 2), (2, 0, 1)) else -1
                    k[b], k[c] = sg * dc, -sg * db
                    vals.append(tuple(v)); curls.append(tuple(k))
    V = np.array([[f / g.h[a] for a, f in enumerate(v)] for v in vals])
    det = math.prod(g.h)
    C = np.array([[f * (g.h[a] if g.dim == 3 else 1.0) / det for a, f in enumerate(k)] for k in curls])
    A = np.einsum("iap,jap,p->ij", C, C, W) * det
    M = np.einsum("iap,jap,p->ij", V, V, W) * det
    return A, M


class Exact:
    """Matrices and DDM pieces of one problem as triplets, on the CPU and GPU alike."""

    def __init__(self, g, order, mu, omega):
        self.g, self.order, self.mu, self.omega = g, order, mu, omega
        self.cd, self.n, edges, self.epd = _numbering(g, order)
        self.A, self.M = _element(g, order)
        self.col = np.full(self.n, 1 << 30)                                         # first cell column of a DOF
        np.minimum.at(self.col, self.cd, g.cell_idx[0][:, None])
        nv = len(g.coords)
        lo, hi = edges // nv, edges % nv
        on = np.flatnonzero((g.coords[lo, 0] == 0) & (g.coords[hi, 0] == 0))
        self.dirichlet = np.zeros(self.n, bool)
        self.uD = np.zeros(self.n, complex)
        ed = (self.epd * on[:, None] + np.arange(self.epd)).ravel()
        self.dirichlet[ed] = True
        along_y = (g.coords[hi[on], 1] - g.coords[lo[on], 1]) > 0                   # E_inc = (0, 1, 0) on x = 0
        self.uD[self.epd * on[along_y]] = g.h[1]
        self._edges, self._nv = edges, nv
        # faces: the outer ones but x = 0 (kind 1), those between subdomains (kind 2), as vertex lists
        c = np.indices((2,) * g.dim).reshape(g.dim, -1)[::-1]
        self.faces = []                                                             # (normal axis, vertices, cell, other cell)
        step = [1, g.n[0], g.n[0] * g.n[1]][:g.dim]
        ids = np.arange(len(g.cells))
        for a in range(g.dim):
            for end in (0, 1):
                if (a, end) == (0, 0):
                    continue
                k = ids[g.cell_idx[a] == end * (g.n[a] - 1)]
                self.faces.append((a, g.cells[k][:, c[a] == end], k, np.full(len(k), -1)))
            k = ids[g.cell_idx[a] < g.n[a] - 1]
            k = k[g.cell_sub[k] != g.cell_sub[k + step[a]]]
            self.faces.append((a, g.cells[k][:, c[a] == 1], k, k + step[a]))

    def face_triplets(self, a, v):
        """(rows, cols, values) [faces, entries] of the tangential mass of faces normal to a."""
        eid = lambda p, q: np.searchsorted(self._edges, p * self._nv + q)  # noqa: E731
        h = [self.g.h[k] for k in range(self.g.dim) if k != a]
        if self.g.dim == 2:
            e = self.epd * eid(v[:, 0], v[:, 1])
            d = np.stack([e + k for k in range(self.epd)], 1)
            return d, d, np.broadcast_to(np.array([1.0, 1.0 / 3.0])[:self.epd] / h[0], d.shape)
        ea = [eid(v[:, 0], v[:, 1]), eid(v[:, 2], v[:, 3])]                         # along the first tangent
        eb = [eid(v[:, 0], v[:, 2]), eid(v[:, 1], v[:, 3])]
        r, c, x = [], [], []
        for pair, f in ((ea, h[1] / h[0]), (eb, h[0] / h[1])):
            for i in (0, 1):
                for j in (0, 1):
                    r.append(pair[i]); c.append(pair[j]); x.append(np.full(len(v), f * (1 / 3 if i == j else 1 / 6)))
        return np.stack(r, 1), np.stack(c, 1), np.stack(x, 1)

    def operator(self, cells=None, transmission=False, real=False):
        """Triplets of K over the given cells (all: the global matrix), plus the Sigma terms."""
        cells = np.arange(len(self.g.cells)) if cells is None else cells
        cd = self.cd[cells]
        ke = self.mu[cells][:, None, None] * self.A - self.omega ** 2 * self.M
        k = cd.shape[1]
        r, c, x = [np.repeat(cd, k, 1).ravel()], [np.tile(cd, (1, k)).ravel()], [ke.reshape(-1).astype(complex)]
        if not real:
            mine = np.zeros(len(self.g.cells), bool)
            mine[cells] = True
            for a, v, c0, c1 in self.faces:
                outer = c1 < 0
                keep = (outer & mine[c0]) | (~outer & transmission & (mine[c0] | mine[np.maximum(c1, 0)]))
                fr, fc, fx = self.face_triplets(a, v[keep])
                r.append(fr.ravel()); c.append(fc.ravel()); x.append(1j * self.omega * fx.ravel())
        return np.concatenate(r), np.concatenate(c), np.concatenate(x)

    def subs(self):
        out = []
        for s in range(int(self.g.cell_sub.max()) + 1):
            cells = np.flatnonzero(self.g.cell_sub == s)
            d = np.unique(self.cd[cells])
            out.append((cells, d[~self.dirichlet[d]]))
        return out

    def apply(self, trip, u):
        """Matrix (triplets over global DOFs) times u."""
        r, c, x = trip
        p = x * u[c]
        return np.bincount(r, p.real, self.n) + 1j * np.bincount(r, p.imag, self.n)

    def solve(self, trip, free, rhs):
        """Solves the rows and columns `free` of the triplet matrix: dense LU over the columns of cells."""
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        order = free[np.argsort(self.col[free], kind="stable")]
        pos = np.full(self.n, -1)
        pos[order] = np.arange(len(order))
        col = self.col[order]
        first = np.searchsorted(col, np.arange(col.min(), col.max() + 2))
        r, c, x = trip
        keep = (pos[r] >= 0) & (pos[c] >= 0)
        r, c, x = pos[r[keep]], pos[c[keep]], x[keep]
        blk = np.searchsorted(first, np.arange(len(order)), side="right") - 1
        by = np.argsort(blk[r], kind="stable")
        r, c, x = r[by], c[by], x[by]
        at = np.searchsorted(blk[r], np.arange(len(first)))
        b = torch.tensor(rhs[order], device=dev)
        nb = len(first) - 1
        S, U, y = [], [], []
        for i in range(nb):
            p, q, e = first[i], first[i + 1], first[min(i + 2, nb)]
            sl = slice(at[i], at[i + 1])
            lo = first[max(i - 1, 0)]
            D = torch.zeros((q - p) * (e - lo), dtype=torch.complex128, device=dev)
            D.index_add_(0, torch.tensor((r[sl] - p) * (e - lo) + c[sl] - lo, device=dev), torch.tensor(x[sl], device=dev))
            D = D.view(q - p, e - lo)
            Lo, Di, Up = D[:, :p - lo], D[:, p - lo:q - lo], D[:, q - lo:]
            rh = b[p:q]
            if i:
                Di = Di - Lo @ U[-1]
                rh = rh - Lo @ y[-1]
            X = torch.linalg.solve(Di, torch.cat([Up, rh[:, None]], 1))
            U.append(X[:, :-1].contiguous()); y.append(X[:, -1].contiguous())
        for i in range(nb - 2, -1, -1):
            y[i] = y[i] - U[i] @ y[i + 1]
        out = np.zeros(self.n, complex)
        out[order] = torch.cat(y).cpu().numpy()
        return out


def _exact_sweep(E, g, at):
    """One sweep of one problem; its interface entries start at `at` in g.  -> (g_out, u, entries)"""
    subs = E.subs()
    pairs = {}
    for a, v, c0, c1 in E.faces:
        for f in np.flatnonzero(c1 >= 0):
            s0, s1 = int(E.g.cell_sub[c0[f]]), int(E.g.cell_sub[c1[f]])
            pairs.setdefault((s0, s1), []).append((a, f)); pairs.setdefault((s1, s0), []).append((a, f))
    info, n = {}, at
    for key in sorted(pairs):
        tr = []
        for a in sorted({a for a, _ in pairs[key]}):
            v = next(v for b, v, _, c1 in E.faces if b == a and len(c1) and c1[0] >= 0)
            tr.append(E.face_triplets(a, v[[f for b, f in pairs[key] if b == a]]))
        tr = tuple(np.concatenate([t[k].ravel() for t in tr]) for k in range(3))
        d = np.unique(tr[0])
        d = d[~E.dirichlet[d]]
        info[key] = (n, d, tr)
        n += len(d)
    sols, u = [], []
    for s, (cells, free) in enumerate(subs):
        T = E.operator(cells, transmission=True)
        rhs = -E.apply(T, E.uD)
        for (i, j), (o, d, _) in info.items():
            if i == s:
                rhs[d] += g[o:o + len(d)]
        x = E.solve(T, free, rhs)
        sols.append(x + E.uD)
        u.append(x[free])
    out = np.zeros(n - at, complex)
    for (i, j), (o, d, tr) in info.items():
        back, d2, _ = info[(j, i)]
        out[o - at:o - at + len(d)] = -g[back:back + len(d2)] + 2j * E.omega * E.apply(tr, sols[j])[d]
    return out, np.concatenate(u), n


def exact(case, seed):
    if case["kind"] in ("solve", "grad") and math.prod(max(1, case[k]) for k in ("nx", "ny", "nz")) > 6000:
        return None
    probs = [Exact(g, case["order"], mu, w) for g, mu, w in _problems(case, seed)]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] in ("apply", "setup"):
        E = probs[0]
        subs = E.subs()
        n = sum(len(f) for _, f in subs)
        x = _vector(n, seed, 2).cpu().numpy()
        y, src, o = [], [], 0
        op = "PINV" if case["kind"] == "setup" else case["op"]
        for cells, free in subs:
            xs = np.zeros(E.n, complex)
            xs[free] = x[o:o + len(free)]
            o += len(free)
            A = E.operator(cells, transmission=True, real=op == "PINV")
            y.append(E.apply(A, xs)[free] if op == "T" else E.solve(A, free, xs)[free])
            if case["kind"] == "setup":
                src.append(-E.apply(E.operator(cells, transmission=True), E.uD)[free])
        y = torch.tensor(np.concatenate(y), device=dev)
        return (torch.tensor(np.concatenate(src), device=dev), y) if case["kind"] == "setup" else y
    if case["kind"] == "sweep":
        gs, us, at = [], [], 0
        g = 1e-2 * _vector(_interface_entries(probs), seed, 1).cpu().numpy()
        for E in probs:
            go, u, at = _exact_sweep(E, g, at)
            gs.append(go); us.append(u)
        return torch.tensor(np.concatenate(gs), device=dev), torch.tensor(np.concatenate(us), device=dev)
    u = []
    for E in probs:
        K = E.operator()
        free = np.flatnonzero(~E.dirichlet)
        u.append(E.solve(K, free, -E.apply(K, E.uD)) + E.uD)
    u = np.concatenate(u)
    if case["kind"] == "solve":
        return torch.tensor(u, device=dev)
    E = probs[0]
    a = _centre_mask(E.g, E.order) * u.conj()
    lam = E.solve(K, free, np.where(E.dirichlet, 0, a))
    gmu = -2 * np.real(np.einsum("ci,ij,cj->c", lam[E.cd], E.A, u[E.cd]))
    # dK/domega = -2 omega M + i M_Gamma (K's parts); the trace on x = 0 does not depend on omega
    unit = Exact(E.g, E.order, 0 * E.mu, 1.0)                                        # -M + i M_Gamma
    minus_m = unit.apply(unit.operator(real=True), u)
    gw = -2 * np.real(lam @ (2 * E.omega * minus_m + unit.apply(unit.operator(), u) - minus_m))
    return torch.tensor(u, device=dev), torch.tensor(gmu, device=dev), torch.tensor(float(gw), dtype=torch.float64, device=dev)


def _interface_entries(probs):
    n = 0
    for E in probs:
        pairs = {}
        for a, v, c0, c1 in E.faces:
            k = np.flatnonzero(c1 >= 0)
            if len(k) == 0:
                continue
            r = E.face_triplets(a, v[k])[0]
            for f in range(len(k)):
                s0, s1 = int(E.g.cell_sub[c0[k[f]]]), int(E.g.cell_sub[c1[k[f]]])
                pairs.setdefault((s0, s1), set()).update(int(d) for d in r[f])
        n += 2 * sum(int((~E.dirichlet[sorted(p)]).sum()) for p in pairs.values())
    return n
