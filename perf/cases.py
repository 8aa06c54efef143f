"""Workloads for timing the solver through its public entry points.

Two sorts of case: whole calls (angles or loads in, fields or gradients out), and the blocks that a
solve is made of (one application of the interface operator F or of its preconditioner P^-1), which
`DDH.apply_dual_operator` exposes to programs that run a Krylov method of their own.

A case is a dict: `kind` names the call, `n` the squares per side of the (base) grid, `p` the
degree, `rhs` the right-hand sides of one call, `kh` the wavenumber times the element size (0 for
Poisson), `precision` "fp64" or "mixed", `eps_hi` the upper end of the seeded permittivity draw
U[1, eps_hi], `medium` the seed of that draw.  The seed given to `prepare` draws what changes from
call to call: incident angles, loads, dual vectors.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import workloads as W
from paper_1808_04713_gb300 import ddh
from paper_1808_04713_gb300.autograd import PlaneWaveSolve, PointEval

TOL = 1e-10          # relative residual of FP64 solves (the library's default)
TOL_MIXED = 1e-12    # of mixed solves: one outer iteration past 1e-10, well clear of either threshold
POINTS = 32          # observation points of the lens objective, on x = 0.9


def listed():
    return [
        # Table 2 of the paper (p = 3, N = 64, l = 2): the smallest calls, where launches and host
        # round trips are the whole cost
        _case("poisson_8", "poisson", n=8, p=3, l=2),
        # one plane wave on 16 x 16 squares, plain FP64: the usual first problem (latency)
        _case("plane_16_fp64", "solve", n=16, p=16, kh=6.25),
        # scattering with absorbing layers on every side and volume loads, plain FP64
        _case("pml_32_fp64", "pml", n=32, p=12, kh=1.25, rhs=8, l=3),
        # a batch of plane waves through a random medium: the mixed form, at its full size
        _case("random_64_mixed", "solve", n=64, p=20, kh=6.25, rhs=8, eps_hi=2.0, medium=4, precision="mixed"),
        # the same medium on a quarter of the elements in plain FP64
        _case("random_32_fp64", "solve", n=32, p=20, kh=6.25, rhs=8, eps_hi=2.0, medium=4),
        # hanging nodes, degrees 8 to 24, a batch of angles, mixed form
        _case("disk_16_mixed", "disk", n=16, p=24, kh=4.6875, rhs=16, precision="mixed"),
        # one step of a lens design: set eps, factor, solve, adjoint solve, gradients in eps and k
        _case("lens_24_step", "step", n=24, p=16, kh=200.0 / 48, eps_hi=4.0, medium=5),
        # one application of the interface operator: small and single, then batched, FP64 and
        # complex64, uniform and with hanging nodes and mixed degrees
        _case("operator_16_fp64", "operator", n=16, p=16, kh=6.25),
        _case("operator_64_fp64", "operator", n=64, p=20, kh=6.25, rhs=8, eps_hi=2.0, medium=4),
        _case("operator_64_mixed", "operator", n=64, p=20, kh=6.25, rhs=8, eps_hi=2.0, medium=4, precision="mixed"),
        _case("operator_disk_fp64", "operator_disk", n=16, p=24, kh=4.6875, rhs=13),
        # one application of the Dirichlet preconditioner
        _case("precond_64_fp64", "precond", n=64, p=20, kh=6.25, rhs=8, eps_hi=2.0, medium=4),
    ]


def draw(rng):
    kind = rng.choice(["poisson", "solve", "solve", "pml", "disk", "step", "operator", "operator", "operator_disk",
                       "precond"])
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    medium = rng.randrange(1, 1000)
    if kind == "poisson":
        p = rng.randint(3, 20)
        return _case(None, kind, n=log(3, 32), p=p, rhs=log(1, 16), l=rng.randint(1, 2))
    if kind in ("disk", "operator_disk"):
        return _case(None, kind, n=rng.randint(5, 16), p=rng.randint(10, 24), kh=round(rng.uniform(2.2, 4.7), 3),
                     rhs=log(1, 16), medium=medium, precision=rng.choice(["fp64", "mixed"]))
    p = rng.randint(8, 22)
    # kh from 2.2: just above the criterion's step to l = 1 the method itself needs hundreds of iterations
    if kind == "pml":
        return _case(None, kind, n=log(8, 40), p=p, kh=round(rng.uniform(1.0, 1.5), 3), rhs=log(1, 8), l=3)
    n = log(4, 24 if kind == "step" else 60)
    rhs = log(1, 2 if kind == "step" else 16)
    while n * n * p * p * rhs > 60 * 60 * 20 * 20 * 8:
        rhs -= 1
    eps_hi = round(rng.uniform(1.0, 2.0), 3)
    precision = "fp64" if kind in ("step", "precond") else rng.choice(["fp64", "mixed"])
    top = 0.3 * p
    if kind == "step" or (kind == "solve" and precision == "fp64"):
        # plain FP64 solves stay below the first element resonance (kh sqrt(eps) = 4.44), where an
        # unlucky draw of the medium alone puts 1e-10 out of their reach
        top = min(top, 4.2 / math.sqrt(eps_hi))
    return _case(None, kind, n=n, p=p, kh=round(rng.uniform(2.2, top), 3), rhs=rhs, eps_hi=eps_hi, medium=medium,
                 precision=precision)


def _case(name, kind, n, p, kh=0.0, rhs=1, eps_hi=1.0, medium=1, precision="fp64", l=0):
    c = dict(kind=kind, n=n, p=p, kh=kh, rhs=rhs, eps_hi=eps_hi, medium=medium, precision=precision, l=l)
    return c if name is None else dict(name=name, **c)


# ------------------------------------------------------------------ problems
def _k(case):
    return case["kh"] * case["n"]


def _mesh(case):
    """(leaves, degrees, permittivity or rho) of a case."""
    n, p = case["n"], case["p"]
    if case["kind"] in ("disk", "operator_disk"):
        # the disk r < 0.25 refined two levels, eps = 4 inside, degrees U{8..p}
        lv = W.disk_leaves(n, 0.25, 2)
        c = W.leaf_centres(n, lv)
        eps = np.where((c[:, 0] - 0.5) ** 2 + (c[:, 1] - 0.5) ** 2 < 0.25 ** 2, 4.0, 1.0)
        return lv, np.random.default_rng(case["medium"]).integers(8, p + 1, size=len(lv)).astype(np.int32), eps
    lv = W.uniform_leaves(n)
    if case["kind"] == "poisson":
        return lv, np.full(n * n, p, np.int32), 10.0 ** ((lv[:, 1] - lv[:, 2]) / 4.0 * min(1.0, 8.0 / n))
    eps = np.random.default_rng(case["medium"]).uniform(1.0, case["eps_hi"], size=n * n)
    return lv, np.full(n * n, p, np.int32), eps


def _stretch(case):
    """PML factors per element: layers two elements thick on every side, sigma = k."""
    lv, n = W.uniform_leaves(case["n"]), case["n"]
    st = 1.0 - 1.0j
    return tuple(np.where((lv[:, a] < 2) | (lv[:, a] >= n - 2), st, 1.0) for a in (1, 2))


class _Solver:
    """A factored context on a stream of its own, as a program keeps it between calls."""

    def __init__(self, case):
        lv, p, coef = _mesh(case)
        self.stream = torch.cuda.Stream()
        self.ddh = ddh.DDH(0, stream=self.stream)
        self.eps = coef
        self.ddh.set_mesh(case["n"], lv, p)
        mixed = case["precision"] == "mixed"
        opts = dict(tol=TOL, l_override=case["l"], precision=ddh.PREC_MIXED_FP32 if mixed else ddh.PREC_FP64)
        if case["kind"] == "poisson":
            self.ddh.set_poisson(coef)
        else:
            self.ddh.set_coefficients(_k(case), coef)
            if case["kind"] == "pml":
                self.ddh.set_pml(*_stretch(case))
                self.ddh.set_boundary(ddh.BOUNDARY_DIRICHLET)
                opts["dual_stop"] = 1              # the paper's stopping rule
        with torch.cuda.stream(self.stream):
            self.ddh.factor(**opts)


_kept: dict = {}


def _solver(case):
    """The context of this problem; only the latest is kept, so the card holds one factorisation."""
    key = tuple(sorted((a, b) for a, b in case.items() if a != "name"))
    if key not in _kept:
        _kept.clear()
        _kept[key] = _Solver(case)
    return _kept[key]


def prepare(case, seed):
    if case["kind"] == "step":
        # the design loop hands new permittivities to the context at each step and factors anew
        lv, p, eps = _mesh(case)
        stream = torch.cuda.Stream()
        s = ddh.DDH(0, stream=stream)
        s.set_mesh(case["n"], lv, p)
        rng = np.random.default_rng(seed)
        eps = eps * (1.0 + 1e-3 * rng.standard_normal(len(eps)))
        pts = np.stack([np.full(POINTS, 0.9), np.linspace(0.4, 0.6, POINTS)], axis=1)
        return dict(kind="step", ddh=s, stream=stream, points=pts, thetas=_angles(case, rng),
                    eps=torch.tensor(eps, dtype=torch.float64), k=torch.tensor(_k(case), dtype=torch.float64))
    sv = _solver(case)
    st = dict(kind=case["kind"], ddh=sv.ddh, stream=sv.stream, precision=case["precision"])
    rng = np.random.default_rng(seed)
    if case["kind"] in ("solve", "disk"):
        st["thetas"] = _angles(case, rng)
        return st
    with torch.cuda.stream(sv.stream):
        if case["kind"] in ("poisson", "pml"):
            st["loads"] = _loads(case, seed, sv.ddh.n_local)
        else:
            st["v"] = _dual(case, seed, sv.ddh.info().n_dual)
    torch.cuda.synchronize()
    return st


def _angles(case, rng):
    return rng.uniform(0.0, 2.0 * math.pi, size=case["rhs"])


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _loads(case, seed, n_local):
    lo = 0.0 if case["kind"] == "poisson" else -1.0
    x = torch.rand((case["rhs"], n_local), generator=_generator(seed), device="cuda", dtype=torch.float64)
    return (lo + (1.0 - lo) * x).to(torch.complex128)


def _dual(case, seed, n_dual):
    x = torch.randn((case["rhs"], n_dual, 2), generator=_generator(seed), device="cuda", dtype=torch.float64)
    return torch.view_as_complex(x)


def run(state):
    s, kind = state["ddh"], state["kind"]
    with torch.cuda.stream(state["stream"]):
        if kind in ("solve", "disk"):
            mixed = state["precision"] == "mixed"
            return s.solve(s.rhs_planewave(state["thetas"]), tol=TOL_MIXED if mixed else TOL)[0]
        if kind in ("poisson", "pml"):
            return s.solve(state["loads"], tol=TOL)[0] if kind == "poisson" else \
                s.solve(state["loads"], tol=TOL, stats=False)[0]
        if kind == "step":
            eps = state["eps"].clone().requires_grad_()
            k = state["k"].clone().requires_grad_()
            u = PlaneWaveSolve.apply(eps, k, s, state["thetas"], TOL)
            J = (PointEval.apply(u, s, state["points"]).abs() ** 2).sum()
            J.backward()
            return {"field": u.detach(), "J": J.detach(), "eps": eps.grad, "k": k.grad}
        mixed = state["precision"] == "mixed"
        y = s.apply_dual_operator(1 if kind == "precond" else 0, state["v"],
                                  precision=ddh.PREC_MIXED_FP32 if mixed else ddh.PREC_FP64)
        # the complex64 form computes complex64 digits, and a program keeps them as such
        return y.to(torch.complex64) if mixed else y


# ------------------------------------------------------------------ floors
def _primal(case):
    """Primal constraints per edge: given, or the paper's dispersion criterion."""
    if case["l"]:
        return case["l"]
    kh = case["kh"] * math.sqrt(float(np.max(_mesh(case)[2])))
    return max(1, math.floor(0.5 * (kh + kh ** (1.0 / 3.0) - 1.0)) + 1)


def work(case):
    """Bytes and operations of one pass.  A block reads its element matrices and its vectors once.
    A whole call reads the same matrices and its loads once, writes its fields once, and applies the
    operator at least once per right-hand side (how often is the method's own affair)."""
    lv, p, _ = _mesh(case)
    p = p.astype(float)
    l, R = _primal(case), case["rhs"]
    fp = 16 if case["precision"] == "fp64" else 8
    nE, nT = 4.0 * np.maximum(p - l, 0), 4.0 * l
    dual = 16.0 * R * float(np.sum(nE)) / 2
    if case["kind"] == "precond":
        # one real matrix per degree, shared by all elements
        return {"bytes": 2 * dual + 8.0 * float(np.sum(np.unique(nE) ** 2)), "flops": 4.0 * R * float(np.sum(nE ** 2))}
    flops = 8.0 * R * float(np.sum(nE ** 2 + 2 * nE * nT))
    mats = fp * float(np.sum(nE ** 2 + nE * nT))
    if case["kind"].startswith("operator"):
        return {"bytes": mats + 2 * dual, "flops": flops}
    fields = 16.0 * R * float(np.sum((p + 1) ** 2))
    interior = 16.0 * R * float(np.sum((p - 1) ** 3))      # recovery of the element interiors
    both = 2 if case["kind"] in ("step", "poisson", "pml") else 1
    return {"bytes": mats + both * fields, "flops": (2 if case["kind"] == "step" else 1) * (flops + interior)}


# ------------------------------------------------------------------ 64-bit values
def exact(case, seed):
    """What `run` returns, from dense element matrices and a block-tridiagonal direct solve over the
    grid lines, refined.  None for hanging nodes: their slaved unknowns would take a second
    implementation of the constraints."""
    if case["kind"] in ("disk", "operator_disk"):
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    with torch.no_grad():
        if case["kind"] in ("operator", "precond"):
            l, n, p = _primal(case), case["n"], case["p"]
            v = _dual(case, seed, 2 * n * (n - 1) * max(0, p - l))
            return _exact_precond(case, l, v, dev) if case["kind"] == "precond" else _exact_operator(case, l, v, dev)
        n, p = case["n"], case["p"]
        grid = _Grid(n, p, p, dev, dirichlet=case["kind"] in ("poisson", "pml"))
        rng = np.random.default_rng(seed)
        eps = _mesh(case)[2]
        if case["kind"] == "step":
            eps = eps * (1.0 + 1e-3 * rng.standard_normal(len(eps)))
        direct = _Direct(case, grid, eps)
        if case["kind"] in ("poisson", "pml"):
            b = _loads(case, seed, n * n * (p + 1) ** 2).reshape(case["rhs"], n * n, -1)
            return grid.swap(direct.solve(grid.swap(b))).reshape(case["rhs"], -1)
        thetas, k, h2 = _angles(case, rng), _k(case), 0.5 / n
        b, db = _impedance_loads(grid, k, thetas)
        ut = direct.solve(b)
        u = grid.swap(ut)
        if case["kind"] == "solve":
            return u.reshape(case["rhs"], -1)
        Ev = _point_rows(grid, np.stack([np.full(POINTS, 0.9), np.linspace(0.4, 0.6, POINTS)], axis=1))
        y = u.reshape(len(thetas), -1) @ Ev.T
        lt = direct.solve(grid.swap(((2.0 * y.conj()) @ Ev).reshape(u.shape)))
        mass = (lt * (ut @ grid.MM)).sum(dim=(0, 2)).real * h2 * h2
        robin = sum((lt * (ut @ grid.R[s]) * grid.on_boundary[:, s, None]).sum() for s in range(4))
        gk = (2.0 * k * (mass * torch.as_tensor(eps, device=dev)).sum() + (1j * h2 * robin).real
              + (lt * db).sum().real)
        return {"field": u.reshape(case["rhs"], -1), "J": (y.abs() ** 2).sum(), "eps": (k * k * mass).cpu(),
                "k": gk.cpu()}


class _Grid:
    """n x n squares of degree p on the basis (1 + x)/2, (1 - x)/2, N_2 .. N_p, where N_m are the
    integrated Legendre polynomials, and the numbering of its vertices and of the edge bubbles
    2 .. top by grid lines: strip j holds line j's vertices and horizontal edges and the vertical
    edges above it.  Unknown g is row g % L of strip g // L."""

    def __init__(self, n, p, top, dev, dirichlet=False):
        self.n, self.p, self.top, self.dev = n, p, top, dev
        t, w = np.polynomial.legendre.leggauss(p + 2)
        N, dN = _basis(p, t)
        c = lambda a: torch.as_tensor(a, device=dev, dtype=torch.complex128)  # noqa: E731
        M, K = (N * w) @ N.T, (dN * w) @ dN.T
        self.MK, self.KM, self.MM = c(np.kron(M, K)), c(np.kron(K, M)), c(np.kron(M, M))
        B = np.eye(p + 1)
        B[:2, :2] = np.array([[1.0, 1.0], [1.0, -1.0]]) / math.sqrt(2.0)
        self.B2 = c(np.kron(B, B))
        pick = [np.diag(np.eye(p + 1)[a]) for a in (1, 0)]     # the function that is 1 at x = -1, +1
        self.R = [c(np.kron(M, pick[0])), c(np.kron(M, pick[1])), c(np.kron(pick[0], M)), c(np.kron(pick[1], M))]
        # slots of an element: corners, then the bubbles of the sides x1 = -1, x1 = 1, x2 = -1, x2 = 1
        q = p + 1
        self.corners = [a + q * b for b in (0, 1) for a in (0, 1)]
        self.side = lambda s, m: [1 + q * m, 0 + q * m, m + q * 1, m + q * 0][s]  # noqa: E731
        self.inner = [a + q * b for b in range(2, q) for a in range(2, q)]
        self.skel = self.corners + [self.side(s, m) for s in range(4) for m in range(2, top + 1)]
        nb = top - 1
        self.L = L = (n + 1) + n * nb + (n + 1) * nb
        i, j = np.arange(n)[None, :], np.arange(n)[:, None]
        vert = lambda a, b: b * L + a  # noqa: E731
        hor = lambda a, b: b * L + (n + 1) + a * nb  # noqa: E731
        ver = lambda a, b: b * L + (n + 1) + n * nb + a * nb  # noqa: E731
        cols = [vert(i + 1 - a, j + 1 - b) for b in (0, 1) for a in (0, 1)]
        for first in (ver(i, j), ver(i + 1, j), hor(i, j), hor(i, j + 1)):
            cols += [first + k for k in range(nb)]
        self.glob = torch.as_tensor(np.stack([np.broadcast_to(x, (n, n)) for x in cols], axis=2), device=dev)
        edge = [np.broadcast_to(x, (n, n)) for x in (i == 0, i == n - 1, j == 0, j == n - 1)]
        self.on_boundary = torch.as_tensor(np.stack([e.ravel() for e in edge], axis=1), device=dev).to(torch.complex128)
        # unknowns that are fixed at zero: those of a Dirichlet boundary and the last strip's unused ones
        fixed = np.zeros(((n + 1), L), bool)
        fixed[n, (n + 1) + n * nb:] = True
        if dirichlet:
            fixed[[0, n], : (n + 1) + n * nb] = True
            fixed[:, [0, n]] = True
            fixed[:, (n + 1) + n * nb: (n + 1) + n * nb + nb] = True
            fixed[:, L - nb:] = True
        self.fixed = torch.as_tensor(fixed, device=dev)

    def swap(self, v):
        """N basis <-> the basis of this class (its own inverse)."""
        return v.to(self.dev) @ self.B2

    def elements(self, case, eps, j):
        """Matrices of the elements of row j."""
        n, kind = self.n, case["kind"]
        at = slice(j * n, (j + 1) * n)
        e = torch.as_tensor(np.asarray(eps)[at], device=self.dev).to(torch.complex128)[:, None, None]
        if kind == "poisson":
            return e * (self.MK + self.KM)
        k, h2 = _k(case), 0.5 / n
        pa = pb = s12 = torch.ones_like(e)
        if kind == "pml":
            s1, s2 = (torch.as_tensor(s[at], device=self.dev)[:, None, None] for s in _stretch(case))
            pa, pb, s12 = s2 / s1, s1 / s2, s1 * s2
        A = pa * self.MK + pb * self.KM - (k * h2) ** 2 * e * s12 * self.MM
        if kind != "pml":
            for s in range(4):
                A = A - (1j * k * h2) * self.on_boundary[at, s, None, None] * self.R[s]
        return A


def _basis(p, t):
    """Values and derivatives [p+1, len(t)] of (1 + t)/2, (1 - t)/2 and N_2 .. N_p at t."""
    t = np.asarray(t, dtype=float)
    P = np.zeros((p + 1, t.size))
    P[0], P[1] = 1.0, t
    for m in range(2, p + 1):
        P[m] = ((2 * m - 1) * t * P[m - 1] - (m - 1) * P[m - 2]) / m
    P *= np.sqrt(np.arange(p + 1) + 0.5)[:, None]              # orthonormal
    g = np.array([1.0] + [1.0 / math.sqrt((2 * i + 1) * (2 * i - 1)) for i in range(1, p + 1)])
    N, dN = np.zeros_like(P), np.zeros_like(P)
    N[0], N[1], dN[0], dN[1] = 0.5 * (1 + t), 0.5 * (1 - t), 0.5, -0.5
    for m in range(2, p + 1):
        N[m], dN[m] = g[m] * P[m] - g[m - 1] * P[m - 2], P[m - 1]
    return N, dN


class _Strips:
    """Block-tridiagonal complex symmetric system over the strips of a grid, with refinement."""

    def __init__(self, grid):
        n, L = grid.n, grid.L
        self.grid = grid
        self.D = torch.zeros((n + 1, L, L), dtype=torch.complex128, device=grid.dev)
        self.U = torch.zeros((n, L, L), dtype=torch.complex128, device=grid.dev)

    def add(self, j, S):
        L = self.grid.L
        g = self.grid.glob[j] - j * L
        Z = torch.zeros((2 * L, 2 * L), dtype=S.dtype, device=S.device)
        Z.index_put_((g[:, :, None].expand_as(S), g[:, None, :].expand_as(S)), S, accumulate=True)
        self.D[j] += Z[:L, :L]
        self.D[j + 1] += Z[L:, L:]
        self.U[j] += Z[:L, L:]

    def factor(self):
        n, L, fx = self.grid.n, self.grid.L, self.grid.fixed
        free = (~fx).to(self.D.dtype)
        self.D *= free[:, :, None] * free[:, None, :]
        self.D.diagonal(dim1=1, dim2=2)[fx] = 1.0
        self.U *= free[:n, :, None] * free[1:, None, :]
        self.lu, self.G, S = [], [], self.D[0]
        for j in range(n + 1):
            self.lu.append(torch.linalg.lu_factor(S))
            if j < n:
                self.G.append(torch.linalg.lu_solve(*self.lu[j], self.U[j]))
                S = self.D[j + 1] - self.U[j].T @ self.G[j]
        self.free = free

    def _once(self, r):
        n = self.grid.n
        y = [r[0]]
        for j in range(n):
            y.append(r[j + 1] - self.G[j].T @ y[j])
        x = [None] * (n + 1)
        for j in range(n, -1, -1):
            x[j] = torch.linalg.lu_solve(*self.lu[j], y[j])
            if j < n:
                x[j] = x[j] - self.G[j] @ x[j + 1]
        return torch.stack(x)

    def solve(self, r):
        r = r * self.free[:, :, None]
        x = torch.zeros_like(r)
        for _ in range(4):
            res = r - self.D @ x
            res[:-1] -= self.U @ x[1:]
            res[1:] -= self.U.transpose(1, 2) @ x[:-1]
            x = x + self._once(res)
        return x

    def gather(self, x):
        """[strips, L, R] -> [R, elements, skeleton]."""
        return x.reshape(-1, x.shape[2])[self.grid.glob.reshape(self.grid.n ** 2, -1)].permute(2, 0, 1)

    def scatter(self, f):
        """The transpose of gather, summed."""
        n, L = self.grid.n, self.grid.L
        out = torch.zeros(((n + 1) * L, f.shape[0]), dtype=f.dtype, device=f.device)
        out.index_add_(0, self.grid.glob.reshape(-1), f.permute(1, 2, 0).reshape(-1, f.shape[0]))
        return out.reshape(n + 1, L, -1)


class _Direct:
    """The conforming problem with its element interiors condensed."""

    def __init__(self, case, grid, eps):
        self.grid, self.strips = grid, _Strips(grid)
        I, S = grid.inner, grid.skel
        self.lu, self.X = [], []
        for j in range(grid.n):
            A = grid.elements(case, eps, j)
            lu = torch.linalg.lu_factor(A[:, I][:, :, I])
            X = torch.linalg.lu_solve(*lu, A[:, I][:, :, S])
            self.strips.add(j, A[:, S][:, :, S] - A[:, S][:, :, I] @ X)
            self.lu.append(lu)
            self.X.append(X)
        self.X = torch.cat(self.X)
        self.strips.factor()

    def solve(self, b):
        g = self.grid
        bI = b[:, :, g.inner].permute(1, 2, 0)
        w = torch.cat([torch.linalg.lu_solve(*self.lu[j], bI[j * g.n:(j + 1) * g.n]) for j in range(g.n)])
        f = b[:, :, g.skel] - (self.X.transpose(1, 2) @ bI).permute(2, 0, 1)
        uS = self.strips.gather(self.strips.solve(self.strips.scatter(f)))
        u = torch.zeros_like(b)
        u[:, :, g.skel] = uS
        u[:, :, g.inner] = (w - self.X @ uS.permute(1, 2, 0)).permute(2, 0, 1)
        return u


def _impedance_loads(grid, k, thetas):
    """Loads [R, elements, slots] of g = du/dn - i k u for plane waves exp(i k d.x), and d/dk of them."""
    n, p = grid.n, grid.p
    h = 1.0 / n
    t, w = np.polynomial.legendre.leggauss(p + 40)
    N, _ = _basis(p, t)
    out = np.zeros((2, len(thetas), n * n, (p + 1) ** 2), complex)
    mid = (np.arange(n)[:, None] + 0.5 * (1.0 + t)) * h
    for r, th in enumerate(thetas):
        c, s = math.cos(th), math.sin(th)
        for side, (dn, x, y) in enumerate([(-c, 0.0, mid), (c, 1.0, mid), (-s, mid, 0.0), (s, mid, 1.0)]):
            ph = x * c + y * s
            wave = np.exp(1j * k * ph) * 1j * (dn - 1.0)
            el = [np.arange(n) * n, np.arange(n) * n + n - 1, np.arange(n), np.arange(n) + n * (n - 1)][side]
            slots = [([1, 0][side] + (p + 1) * np.arange(p + 1)) if side < 2 else
                     (np.arange(p + 1) + (p + 1) * [1, 0][side - 2])][0]
            for d, g in enumerate((k * wave, (1.0 + 1j * k * ph) * wave)):
                out[d, r, el[:, None], slots[None, :]] += 0.5 * h * ((g * w) @ N.T)
    return tuple(torch.as_tensor(o, device=grid.dev) for o in out)


def _point_rows(grid, xy):
    """Rows of the evaluation at points, on the N basis [points, n_local]."""
    n, p = grid.n, grid.p
    i, j = (np.minimum(n - 1, np.floor(xy[:, a] * n).astype(int)) for a in (0, 1))
    N1, N2 = (_basis(p, 2.0 * (xy[:, a] * n - b) - 1.0)[0] for a, b in ((0, i), (1, j)))
    out = np.zeros((len(xy), n * n, (p + 1) ** 2), complex)
    for m in range(len(xy)):
        out[m, j[m] * n + i[m]] = np.outer(N2[:, m], N1[:, m]).ravel()
    return grid.swap(torch.as_tensor(out)).reshape(len(xy), -1)


def _dual_slots(n, p, l, dev):
    """Row of the interface vector and its sign for every edge bubble l+1..p of every element side
    (-1 and 0 on the boundary): edges in the order of the elements below and left of them, the
    vertical one first; + on that element, - on the other."""
    row = np.full((n, n, 4), -1)
    sign = np.zeros((n, n, 4))
    at = 0
    for j in range(n):
        for i in range(n):
            for side, other, ok in ((1, (j, i + 1, 0), i < n - 1), (3, (j + 1, i, 2), j < n - 1)):
                if ok:
                    row[j, i, side] = row[other] = at
                    sign[j, i, side], sign[other] = 1.0, -1.0
                    at += p - l
    full = np.where(row[..., None] >= 0, row[..., None] + np.arange(p - l), -1).reshape(n * n, -1)
    return torch.as_tensor(full, device=dev), torch.as_tensor(np.repeat(sign.reshape(n * n, 4), p - l, axis=1), device=dev)


def _jump(row, sign, x, n_dual):
    out = torch.zeros((x.shape[0], n_dual + 1), dtype=x.dtype, device=x.device)
    return out.index_add_(1, torch.where(row < 0, n_dual, row).reshape(-1), (x * sign).flatten(1))[:, :n_dual]


def _exact_operator(case, l, v, dev):
    """F v = C A^-1 C^T v: element matrices condensed on the edges, the vertices and the bubbles up to
    l continuous, the others joined by the rows of C only."""
    n, p = case["n"], case["p"]
    grid = _Grid(n, p, l, dev)
    eps = _mesh(case)[2]
    row, sign = _dual_slots(n, p, l, dev)
    v = v.to(dev)
    r = torch.where(row < 0, 0.0, sign) * v[:, row.clamp(min=0)]              # [R, elements, E]
    I, T = grid.inner, grid.skel
    Es = [grid.side(s, m) for s in range(4) for m in range(l + 1, p + 1)]
    strips, xE, Y = _Strips(grid), [], []
    for j in range(n):
        A = grid.elements(case, eps, j)
        TE = T + Es
        S = A[:, TE][:, :, TE] - A[:, TE][:, :, I] @ torch.linalg.solve(A[:, I][:, :, I], A[:, I][:, :, TE])
        t, lu = len(T), torch.linalg.lu_factor(S[:, len(T):, len(T):])
        xE.append(torch.linalg.lu_solve(*lu, r[:, j * n:(j + 1) * n].permute(1, 2, 0)))
        Y.append(torch.linalg.lu_solve(*lu, S[:, t:, :t]))
        strips.add(j, S[:, :t, :t] - S[:, :t, t:] @ Y[-1])
    strips.factor()
    xE, Y = torch.cat(xE).permute(2, 0, 1), torch.cat(Y)
    f = -(Y.transpose(1, 2) @ r.permute(1, 2, 0)).permute(2, 0, 1)
    xT = strips.gather(strips.solve(strips.scatter(f)))
    xE = xE - (Y @ xT.permute(1, 2, 0)).permute(2, 0, 1)
    return _jump(row, sign, xE, v.shape[1])


def _exact_precond(case, l, v, dev):
    """P^-1 v = (1/4) C S C^T v with S the stiffness condensed on the edge bubbles above l."""
    n, p = case["n"], case["p"]
    grid = _Grid(n, p, l, dev)
    row, sign = _dual_slots(n, p, l, dev)
    A, I = grid.MK + grid.KM, grid.inner
    Es = [grid.side(s, m) for s in range(4) for m in range(l + 1, p + 1)]
    S = A[Es][:, Es] - A[Es][:, I] @ torch.linalg.solve(A[I][:, I], A[I][:, Es])
    v = v.to(dev)
    x = (torch.where(row < 0, 0.0, sign) * v[:, row.clamp(min=0)]) @ S
    return 0.25 * _jump(row, sign, x, v.shape[1])
