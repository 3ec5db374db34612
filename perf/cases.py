"""Timed cases of the FETI-DP library: the calls a user's program makes, over the sizes it makes them at.

Whole calls take a lattice description from the host through setup and solve (what one load analysis,
one step of a design loop or one batch costs); the operator calls are what a program with its own
Krylov loop makes on a context that it keeps.  Lattices follow the generators of
``paper_2308_11371_gb300.workloads``: 2D frame-and-diagonal cells with a column-graded radius and a
bent macro map, 3D body-centred-cubic cells with either a hard mask graded along x (bend + twist, the
benchmark's lattice) or a sigmoid mask with per-cell random radii (the design-gradient lattice).
``exact`` assembles the same finite elements in plain float64 torch / numpy.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2308_11371_gb300 import autograd, binding
from paper_2308_11371_gb300 import workloads as W

PRECISION = {"fp64": binding.FETIDP_FP64, "mixed": binding.FETIDP_MIXED_BF16}


def _case(name, op, precision, cells, elems, mask, n_rb, loads):
    nx, ny, nz = cells
    c = {"op": op, "precision": precision, "nx": nx, "ny": ny, "nz": nz, "elems": elems, "mask": mask,
         "n_rb": n_rb, "loads": loads}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest lattice of the tests and of the smoke run, default precision: latency and launches
        _case("solve_2d_4x4_fp64", "solve", "fp64", (4, 4, 0), 8, "frame", 2, 1),
        # a mid-size 2D analysis of odd shape in the default precision
        _case("solve_2d_24x17_fp64", "solve", "fp64", (24, 17, 0), 10, "graded_frame", 32, 1),
        # the 2D benchmark lattice, mixed precision
        _case("solve_2d_64x64_mixed", "solve", "mixed", (64, 64, 0), 16, "graded_frame", 32, 1),
        # the 3D benchmark cell, six load cases: a corner in the default precision, a larger one mixed
        _case("solve_3d_4x4x2_fp64", "solve", "fp64", (4, 4, 2), 6, "graded_bcc", 16, 6),
        _case("solve_3d_8x8x4_mixed", "solve", "mixed", (8, 8, 4), 6, "graded_bcc", 32, 6),
        # one step of a design loop: compliance and its gradient in every cell's radius, forward and backward
        _case("design_3d_12x12x6_mixed", "design", "mixed", (12, 12, 6), 6, "sigmoid_bcc", 16, 1),
        # four uneven lattices solved together, random radii under the hard mask, three load cases
        _case("batch_3d_mixed", "batch", "mixed", (4, 3, 2), 6, "random_bcc", 64, 3),
        # the inner Krylov operators (Eqs. 48, 49) on kept contexts: large 3D with six load cases, odd 3D
        # with one, 2D at the benchmark's size, and the default precision
        _case("apply_F_3d_16x16x8_mixed", "apply_F", "mixed", (16, 16, 8), 6, "sigmoid_bcc", 16, 6),
        _case("precond_3d_9x7x5_mixed", "precond", "mixed", (9, 7, 5), 6, "sigmoid_bcc", 16, 1),
        _case("precond_2d_64x64_mixed", "precond", "mixed", (64, 64, 0), 16, "graded_frame", 32, 1),
        _case("apply_F_3d_8x8x4_fp64", "apply_F", "fp64", (8, 8, 4), 6, "sigmoid_bcc", 16, 6),
        # the outer saddle-point operator (Eq. 16), FP64 in both precisions, three load cases
        _case("apply_A_3d_12x12x6", "apply_A", "mixed", (12, 12, 6), 6, "sigmoid_bcc", 16, 3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cells(rng, dim, lo, hi, most):
    """Cell counts between lo and hi per axis, at most ``most`` cells, no axis over six times another."""
    while True:
        c = [_log_int(rng, lo, hi) for _ in range(dim)]
        if math.prod(c) <= most and max(c) <= 6 * min(c):
            return tuple(c + [0] * (3 - dim))


def draw(rng):
    op = rng.choice(("solve", "solve", "design", "batch", "apply_F", "precond", "apply_A"))
    precision = rng.choice(("fp64", "mixed"))
    if op == "batch":
        return _case("", op, "mixed", (rng.randint(2, 4), rng.randint(2, 4), rng.randint(1, 2)), 6, "random_bcc", 64,
                     rng.randint(1, 3))
    if op in ("solve", "apply_F", "precond") and rng.random() < 0.4:
        cells = _cells(rng, 2, 3, 64 if precision == "mixed" else 40, 4096)
        return _case("", op, precision, cells, rng.randint(4, 16), "graded_frame", 48, 1)
    loads = rng.randint(1, 6)
    if op == "solve" and precision == "mixed" and rng.random() < 0.5:
        return _case("", op, precision, _cells(rng, 3, 2, 12, 300), 6, "graded_bcc", 32, loads)
    elems = rng.choice((4, 5, 6, 6))
    if op in ("solve", "design"):
        most = 24 if precision == "fp64" else 512
    else:
        most = 256 if precision == "fp64" else 2048
    return _case("", op, precision, _cells(rng, 3, 2, 16, most), elems, "sigmoid_bcc", 16, loads)


# ---------------------------------------------------------------- inputs
def _loads(dim, count):
    unit = [tuple(float(i == c) for i in range(dim)) for c in range(dim)]
    if dim == 2:
        return [W.Load(W.LOAD_TRACTION, (0.0, -1.0), axis=0, side=1)][:count]
    faces = [W.Load(W.LOAD_TRACTION, unit[c], axis=2, side=1) for c in (2, 0, 1)]
    return (faces + [W.Load(W.LOAD_BODY, unit[c]) for c in (2, 0, 1)])[:count]


def _problem(case, seed, cells=None):
    rng = np.random.default_rng(seed)
    nx, ny, nz = cells or (case["nx"], case["ny"], case["nz"])
    mask = case["mask"]
    if nz == 0:
        graded = mask == "graded_frame"
        r = (0.1 if graded else 0.12) + (0.05 if graded else 0.0) * np.sin(2.0 * np.pi * (np.arange(nx) + 0.5) / nx)
        return W.LatticeProblem(
            dim=2, cells=(nx, ny, 1), elems=case["elems"], r_cell=np.tile(r, ny), mask_kind=W.MASK_FRAME_DIAG,
            map_kind=W.MAP_BEND_2D, map_params=(rng.uniform(0.0, nx / 16.0), float(nx)), loads=_loads(2, case["loads"]),
            clamp_axis=0, clamp_side=0, n_rb=case["n_rb"])
    n = nx * ny * nz
    if mask == "graded_bcc":
        r = np.tile(0.15 + 0.15 * (np.arange(nx) + 0.5) / nx, ny * nz)
        kind, params = W.MAP_BEND_TWIST_3D, (rng.uniform(0.0, nx / 8.0), float(nx),
                                             rng.uniform(0.0, np.pi / 8.0) * nx / 32.0, ny / 2.0, nz / 2.0)
    elif mask == "random_bcc":
        r = rng.uniform(0.15, 0.3, size=n)
        g1, g2 = rng.uniform(-0.2, 0.2, size=2)
        kind, params = W.MAP_SHEAR_BEND_3D, (rng.uniform(0.0, nx / 8.0), float(nx), float(g1), float(g2))
    else:
        r, kind, params = rng.uniform(0.15, 0.3, size=n), W.MAP_IDENTITY, ()
    return W.LatticeProblem(
        dim=3, cells=(nx, ny, nz), elems=case["elems"], r_cell=r,
        mask_kind=W.MASK_BCC_SIGMOID if mask == "sigmoid_bcc" else W.MASK_BCC_HARD, map_kind=kind,
        map_params=tuple(params), loads=_loads(3, case["loads"]), clamp_axis=2, clamp_side=0, n_rb=case["n_rb"])


def _batch_cells(case):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    return [(nx, ny, 1), (max(2, nx - 1), ny, nz), (nx, max(2, ny - 1), 1), (2, 2, nz)]


def _vector(shape, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return torch.randn(*shape, generator=gen, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    state = {"op": case["op"], "precision": PRECISION[case["precision"]]}
    if case["op"] == "batch":
        state["problem"] = [_problem(case, 4 * seed + b, cells) for b, cells in enumerate(_batch_cells(case))]
        return state
    problem = state["problem"] = _problem(case, seed)
    if case["op"] == "solve":
        return state
    if case["op"] == "design":
        state["r"] = torch.tensor(problem.r_cell, dtype=torch.float64, device="cuda", requires_grad=True)
        state["weights"] = torch.linspace(1.0, 2.0, case["loads"], dtype=torch.float64, device="cuda")
        return state
    solver = state["solver"] = binding.Solver(problem, precision=state["precision"])
    state["x"] = _vector((solver.n_rhs, solver.n_tot if case["op"] == "apply_A" else solver.L), seed)
    return state


def run(state):
    op = state["op"]
    if op in ("solve", "batch"):
        solver = binding.Solver(state["problem"], precision=state["precision"])
        u, lam, _ = solver.solve()
        solver.close()
        return {"u": u, "lam": lam}
    if op == "design":
        r = state["r"]
        c = autograd.cell_compliance(r, state["problem"], precision=state["precision"])
        (g,) = torch.autograd.grad(c @ state["weights"], r)
        return {"compliance": c.detach(), "gradient": g}
    return {"y": getattr(state["solver"], op)(state["x"])}


# ---------------------------------------------------------------- work that no implementation can do without
def _sizes(cells, e):
    """DOF per cell by class, Gauss points, macro-tensor entries, cells and multiplier rows of a lattice."""
    nx, ny, nz = cells
    d = 2 if nz == 0 else 3
    counts = [nx, ny] + ([nz] if d == 3 else [])
    n = d * (e + 1) ** d
    ni, npr = d * (e - 1) ** d, d * 2 ** d
    nd = n - ni - npr
    N = math.prod(counts)
    # rows at a node: its cells - 1, at a clamped node: its cells; summed as (copies) - (free interface nodes)
    ax = 0 if d == 2 else 2
    g = [c * e + 1 for c in counts]
    interior, vertex = (e - 1) ** d * N, math.prod(c + 1 for c in counts)
    iface = math.prod(g) - interior - vertex
    flat = [k for k in range(d) if k != ax]
    clamped = math.prod(g[k] for k in flat) - math.prod(counts[k] + 1 for k in flat)
    L = N * nd - d * (iface - clamped)
    return {"d": d, "n": n, "nd": nd, "np": npr, "nr": n - npr, "N": N, "L": L, "gp": (2 * e) ** d,
            "nc": 10 if d == 2 else 45, "pairs": (3 * e + 1) ** d, "vertices": vertex}


def _shape(case, cells=None):
    return _sizes(cells or (case["nx"], case["ny"], case["nz"]), case["elems"])


def work(case):
    s, m, k = _shape(case), case["loads"], case["n_rb"]
    w = 8 if case["precision"] == "fp64" else 4
    op = case["op"]
    if op in ("apply_F", "precond"):
        # every cell's symmetric n_d x n_d operator once (n_rb principal ones where those are fewer bytes),
        # the multipliers in and out, and for F the corner coupling n_d x n_p
        tri = s["nd"] * (s["nd"] + 1) // 2
        operators = min(s["N"] * tri * w, k * tri * w + s["N"] * k * 8)
        corner = s["N"] * s["nd"] * s["np"] * w if op == "apply_F" else 0
        flops = 2.0 * m * s["N"] * (s["nd"] ** 2 + (2 * s["nd"] * s["np"] if op == "apply_F" else 0))
        return {"bytes": operators + corner + 16 * m * s["L"], "flops": flops}
    if op == "apply_A":
        # x and y once, one modulus per Gauss point; the sparse cell stiffness as multiply-adds
        ntot = s["N"] * s["nr"] + s["d"] * s["vertices"] + s["L"]
        return {"bytes": 16 * m * ntot + 8 * s["N"] * s["gp"], "flops": 2.0 * m * s["N"] * s["d"] ** 2 * s["pairs"]}
    # whole calls: u and lambda out; the principal inverses, the projection traces of every cell
    # against the principal pairs (Eq. 42), and at least ten applications of the two inner operators
    shapes = [s] if op != "batch" else [_shape(case, c) for c in _batch_cells(case)]
    N, L = sum(q["N"] for q in shapes), sum(q["L"] for q in shapes)
    k = min(k, N)
    flops = k * float(s["nr"]) ** 3 + 2.0 * N * s["gp"] * s["nc"] * k * (k + 1) + 40.0 * m * N * s["nd"] ** 2
    return {"bytes": 8 * m * (N * s["n"] + L) + 8 * N, "flops": flops}


# ---------------------------------------------------------------- the same quantities in plain float64
_GAUSS = (0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0))
_DENSE_DOF = 25000      # largest lattice whose assembled system is factorised densely


class _Lattice:
    """Finite elements of one lattice in float64: cell stiffness products, loads, multiplier rows."""

    def __init__(self, p):
        self.p, self.d, self.e = p, p.dim, p.elems
        d, e = self.d, self.e
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.counts = [int(c) for c in p.cells[:d]]
        self.N = math.prod(self.counts)
        self.cell_ijk = np.stack(np.unravel_index(np.arange(self.N), self.counts[::-1])[::-1], 1)
        self.nodes = (e + 1) ** d
        self.node_ijk = np.stack(np.unravel_index(np.arange(self.nodes), [e + 1] * d)[::-1], 1)
        el = np.stack(np.unravel_index(np.arange(e ** d), [e] * d)[::-1], 1)
        self.el = el
        self.bits = np.array([[(A >> k) & 1 for k in range(d)] for A in range(2 ** d)])
        step = np.array([(e + 1) ** k for k in range(d)])
        self.conn = torch.tensor((el[:, None, :] + self.bits[None]) @ step, device=self.dev)   # [nel, 2^d]
        on = ((self.node_ijk == 0) | (self.node_ijk == e)).sum(1)
        cls = np.where(on == d, 2, np.where(on > 0, 1, 0))
        order = np.concatenate([np.flatnonzero(cls == q) for q in range(3)])
        self.local = torch.tensor((order[:, None] * d + np.arange(d)).ravel(), device=self.dev)   # (i, d, p) -> natural
        self.cls = cls
        self.r = torch.tensor(np.asarray(p.r_cell), device=self.dev, dtype=torch.float64)
        self.field = [self._gauss(gp) for gp in range(2 ** d)]

    def _t(self, a):
        return torch.tensor(np.asarray(a), device=self.dev, dtype=torch.float64)

    def _jacobian(self, xi):
        """dx/dxi at lattice coordinates xi [..., d]."""
        p, d = self.p, self.d
        J = torch.zeros(*xi.shape[:-1], d, d, device=self.dev, dtype=torch.float64)
        J[...] = torch.eye(d, device=self.dev, dtype=torch.float64)
        q = p.map_params
        if p.map_kind == W.MAP_BEND_2D:
            J[..., 1, 0] = q[0] * math.pi / q[1] * torch.cos(math.pi * xi[..., 0] / q[1])
        elif p.map_kind == W.MAP_SHEAR_BEND_3D:
            J[..., 0, 2], J[..., 1, 2] = q[2], q[3]
            J[..., 2, 0] = q[0] * math.pi / q[1] * torch.cos(math.pi * xi[..., 0] / q[1])
        elif p.map_kind == W.MAP_BEND_TWIST_3D:
            a, length, tau, yc, zc = q
            th = tau * xi[..., 0] / length
            c, s = torch.cos(th), torch.sin(th)
            dy, dz = xi[..., 1] - yc, xi[..., 2] - zc
            J[..., 1, 0] = tau / length * (-s * dy - c * dz)
            J[..., 2, 0] = tau / length * (c * dy - s * dz) + a * math.pi / length * torch.cos(math.pi * xi[..., 0] / length)
            J[..., 1, 1], J[..., 1, 2], J[..., 2, 1], J[..., 2, 2] = c, -s, s, c
        return J

    def _distance(self, eta):
        if self.d == 2:
            x, y = eta[..., 0], eta[..., 1]
            parts = [x, 1 - x, y, 1 - y, (x - y).abs() / math.sqrt(2.0), (x + y - 1).abs() / math.sqrt(2.0)]
        else:
            parts = []
            for q in range(4):
                a = self._t([1.0 if q == k + 1 else 0.0 for k in range(3)])
                axis = (1.0 - 2.0 * a) / math.sqrt(3.0)
                w = eta - a
                parts.append((w - (w @ axis)[..., None] * axis).norm(dim=-1))
        return torch.stack(parts).min(0).values

    def _gauss(self, gp):
        """Shape gradients [2^d, d], inverse Jacobian, weight and modulus with its radius derivative."""
        p, d, e = self.p, self.d, self.e
        t = [_GAUSS[b] for b in self.bits[gp]]
        dn = np.empty((2 ** d, d))
        for A, off in enumerate(self.bits):
            for a in range(d):
                dn[A, a] = e * math.prod((1 if off[k] else -1) if k == a else (t[k] if off[k] else 1 - t[k]) for k in range(d))
        eta = self._t((self.el + np.array(t)) / e)
        J = self._jacobian(self._t(self.cell_ijk)[:, None, :] + eta[None])
        dist, r = self._distance(eta)[None], self.r[:, None]
        if p.mask_kind == W.MASK_BCC_SIGMOID:
            sg = torch.sigmoid((r - dist) / p.mask_width)
            E = p.E_void + (p.E_solid - p.E_void) * sg
            dE = (p.E_solid - p.E_void) * sg * (1 - sg) / p.mask_width
        else:
            E = p.E_void + (p.E_solid - p.E_void) * (dist <= r).to(torch.float64)
            dE = torch.zeros_like(E)
        wdet = (0.5 / e) ** d * torch.linalg.det(J)
        return self._t(dn), torch.linalg.inv(J), wdet, E, dE

    def _gradient(self, u, dn, Ji):
        """Physical displacement gradient [N, nel, i, k] of cell fields u [N, nodes, d]."""
        return torch.einsum("cnai,ab,cnbk->cnik", u[:, self.conn], dn, Ji)

    def _stress(self, H):
        nu = self.p.nu
        lam, mu = nu / ((1 + nu) * (1 - 2 * nu)), 0.5 / (1 + nu)
        trace = H.diagonal(dim1=-2, dim2=-1).sum(-1)
        return lam * trace[..., None, None] * torch.eye(self.d, device=self.dev, dtype=H.dtype) + mu * (H + H.mT)

    def apply_K(self, u):
        """K_s u_s of every cell, natural order [N, n]."""
        u = u.reshape(self.N, self.nodes, self.d)
        y = torch.zeros_like(u)
        for dn, Ji, wdet, E, _ in self.field:
            S = self._stress(self._gradient(u, dn, Ji)) * (wdet * E)[..., None, None]
            fe = torch.einsum("cnik,ab,cnbk->cnai", S, dn, Ji)
            y.index_add_(1, self.conn.reshape(-1), fe.reshape(self.N, -1, self.d))
        return y.reshape(self.N, -1)

    def gradient(self, u):
        """-u^T dK_s/dr_s u of every cell [N]."""
        u = u.reshape(self.N, self.nodes, self.d)
        g = torch.zeros(self.N, device=self.dev, dtype=torch.float64)
        for dn, Ji, wdet, _, dE in self.field:
            H = self._gradient(u, dn, Ji)
            g -= ((self._stress(H) * H).sum((-2, -1)) * wdet * dE).sum(1)
        return g

    def load(self, load):
        """f_s of every cell, natural order [N, n] (Eq. 5b)."""
        d, e = self.d, self.e
        f = torch.zeros(self.N, self.nodes, d, device=self.dev, dtype=torch.float64)
        direction = self._t(load.direction[:d])
        body = load.kind == W.LOAD_BODY
        free = [k for k in range(d) if body or k != load.axis]
        el = np.arange(len(self.el)) if body else np.flatnonzero(self.el[:, load.axis] == (e - 1 if load.side else 0))
        on = np.ones(self.N, bool) if body else self.cell_ijk[:, load.axis] == (self.counts[load.axis] - 1 if load.side else 0)
        cells = torch.tensor(np.flatnonzero(on), device=self.dev)
        for fg in range(2 ** len(free)):
            t = np.full(d, float(load.side))
            for q, k in enumerate(free):
                t[k] = _GAUSS[(fg >> q) & 1]
            xi = self._t(self.cell_ijk[on])[:, None, :] + self._t((self.el[el] + t) / e)[None]
            J = self._jacobian(xi)[..., free]
            meas = (0.5 / e) ** len(free) * torch.sqrt(torch.linalg.det(J.mT @ J))
            for A, off in enumerate(self.bits):
                Nv = math.prod(t[k] if off[k] else 1 - t[k] for k in range(d))
                if Nv == 0.0:
                    continue
                fe = (meas * Nv)[..., None] * direction
                part = torch.zeros(len(cells), self.nodes, d, device=self.dev, dtype=torch.float64)
                part.index_add_(1, self.conn[torch.tensor(el, device=self.dev)][:, A], fe)
                f[cells] += part
        return f.reshape(self.N, -1)

    def rows(self):
        """Multiplier rows in order: flat cell-node indices (first copy, second copy or -1) of each node row."""
        d, e, p = self.d, self.e, self.p
        g = np.stack(np.unravel_index(np.arange(math.prod(c * e + 1 for c in self.counts)),
                                      [c * e + 1 for c in self.counts][::-1])[::-1], 1)
        on = (g % e == 0).sum(1)
        g = g[(on > 0) & (on < d)]
        clamp = self.counts[p.clamp_axis] * e if p.clamp_side else 0
        first, second = [], []
        cstep, nstep = np.cumprod([1] + self.counts[:-1]), np.array([(e + 1) ** k for k in range(d)])
        for gc in g:
            cand = [[q for q in ((v // e - 1, v // e) if v % e == 0 else (v // e,)) if 0 <= q < c] for v, c in zip(gc, self.counts)]
            own = sorted((int(np.dot(c, cstep)), c) for c in np.stack(np.meshgrid(*cand, indexing="ij"), -1).reshape(-1, d).tolist())
            flat = [s * self.nodes + int(np.dot(gc - np.array(c) * e, nstep)) for s, c in own]
            if gc[p.clamp_axis] == clamp:
                first += flat
                second += [-1] * len(flat)
            else:
                first += flat[:-1]
                second += flat[1:]
        return torch.tensor(first, device=self.dev), torch.tensor(second, device=self.dev)

    def jump(self, u):
        """B u of cell fields [N, n]: [L]."""
        first, second = self.rows()
        u = u.reshape(-1, self.d)
        z = u[first].clone()
        two = second >= 0
        z[two] -= u[second[two]]
        return z.reshape(-1)

    def jump_T(self, lam):
        """B^T lambda: cell fields [N, n]."""
        first, second = self.rows()
        lam = lam.reshape(-1, self.d)
        u = torch.zeros(self.N * self.nodes, self.d, device=self.dev, dtype=torch.float64)
        u.index_add_(0, first, lam)
        two = second >= 0
        u.index_add_(0, second[two], -lam[two])
        return u.reshape(self.N, -1)

    def _global(self):
        """Global DOF of every cell DOF [N, n] and the mask of free ones."""
        e, d = self.e, self.d
        dims = [c * e + 1 for c in self.counts]
        step = np.cumprod([1] + dims[:-1])
        gi = self.cell_ijk[:, None, :] * e + self.node_ijk[None]
        gdof = (gi @ step)[..., None] * d + np.arange(d)
        clamp = self.counts[self.p.clamp_axis] * e if self.p.clamp_side else 0
        free = np.ones((math.prod(dims), d), bool)
        all_ijk = np.unravel_index(np.arange(math.prod(dims)), dims[::-1])[::-1]
        free[all_ijk[self.p.clamp_axis] == clamp] = False
        return (torch.tensor(gdof.reshape(self.N, -1), device=self.dev), torch.tensor(free.ravel(), device=self.dev))

    def corners(self):
        """Positions of the primal DOF: flat cell DOF -> primal number (-1: clamped), and their count."""
        d, counts = self.d, self.counts
        corner = np.flatnonzero(self.cls == 2)
        vdims = [c + 1 for c in counts]
        vstep = np.cumprod([1] + vdims[:-1])
        ijk = np.stack(np.unravel_index(np.arange(math.prod(vdims)), vdims[::-1])[::-1], 1)
        clamp = counts[self.p.clamp_axis] if self.p.clamp_side else 0
        free = ijk[:, self.p.clamp_axis] != clamp
        num = np.where(free, np.cumsum(free) - 1, -1)
        v = (self.cell_ijk[:, None, :] + (self.node_ijk[corner] // self.e)[None]) @ vstep
        prim = np.where(num[v] >= 0, num[v], -1)
        flat = (np.arange(self.N)[:, None] * self.nodes + corner)
        return torch.tensor(flat.ravel(), device=self.dev), torch.tensor(prim.ravel(), device=self.dev), int(free.sum())

    def apply_A(self, x):
        """The saddle-point operator of Eq. 16 on (u_R in (i, d) order, u_P, lambda)."""
        d, n = self.d, self.nodes * self.d
        flat, prim, nv = self.corners()
        nr = n - d * 2 ** d
        uR, uP, lam = x[:self.N * nr].reshape(self.N, nr), x[self.N * nr:self.N * nr + nv * d], x[self.N * nr + nv * d:]
        u = torch.zeros(self.N, n, device=self.dev, dtype=torch.float64)
        u[:, self.local[:nr]] = uR
        uc = u.reshape(-1, d)
        ok = prim >= 0
        uc[flat[ok]] = uP.reshape(nv, d)[prim[ok]]
        remaining = torch.zeros_like(u)
        remaining[:, self.local[:nr]] = uR
        y = self.apply_K(u)
        yP = torch.zeros(nv, d, device=self.dev, dtype=torch.float64)
        yP.index_add_(0, prim[ok], y.reshape(-1, d)[flat[ok]])
        yR = (y + self.jump_T(lam))[:, self.local[:nr]]
        return torch.cat([yR.reshape(-1), yP.reshape(-1), self.jump(remaining)])

    def solve(self):
        """u [loads, N, n] and lambda [loads, L] of the assembled system."""
        gdof, free = self._global()
        ndof, n = free.numel(), self.nodes * self.d
        nd = self.d * 2 ** self.d
        K = torch.zeros(ndof, ndof, device=self.dev, dtype=torch.float64)
        dof = (self.conn[..., None] * self.d + torch.arange(self.d, device=self.dev)).reshape(-1, nd)
        eye = torch.eye(nd, device=self.dev, dtype=torch.float64).reshape(nd, 2 ** self.d, self.d)
        for dn, Ji, wdet, E, _ in self.field:
            H = torch.einsum("xai,ab,cnbk->cnxik", eye, dn, Ji)
            S = self._stress(H) * (wdet * E)[..., None, None, None]
            Ke = torch.einsum("cnxik,cnyik->cnxy", S, H)
            g = gdof[:, dof]                                           # [N, nel, nd]
            K.view(-1).index_add_(0, (g[..., :, None] * ndof + g[..., None, :]).reshape(-1), Ke.reshape(-1))
        f = [self.load(ld) for ld in self.p.loads]
        rhs = torch.zeros(ndof, len(f), device=self.dev, dtype=torch.float64)
        for q, fs in enumerate(f):
            rhs[:, q].index_add_(0, gdof.reshape(-1), fs.reshape(-1))
        keep = torch.nonzero(free).ravel()
        sol = torch.zeros_like(rhs)
        A = K[keep][:, keep]
        del K
        chol = torch.linalg.cholesky(A)
        x = torch.cholesky_solve(rhs[keep], chol)
        for _ in range(3):                                            # iterative refinement
            x += torch.cholesky_solve(rhs[keep] - A @ x, chol)
        sol[keep] = x
        u = torch.stack([sol[:, q][gdof] for q in range(len(f))])
        first, second = self.rows()
        lams = []
        for q, fs in enumerate(f):
            r = (fs - self.apply_K(u[q])).reshape(-1, self.d)          # = B^T lambda on the copies
            lam = r[first].clone()
            chain = torch.nonzero(second >= 0).ravel().tolist()
            fl, sl = first.tolist(), second.tolist()
            lam = lam.cpu()
            for row in chain:                                          # rows of a chain follow each other
                if row > 0 and sl[row - 1] == fl[row]:
                    lam[row] += lam[row - 1]
            lams.append(lam.reshape(-1).to(self.dev))
        return f, u, torch.stack(lams)


def exact(case, seed):
    op = case["op"]
    if op in ("apply_F", "precond", "batch"):
        return None       # the reduced-order operators have no definition apart from the reduced basis
    if op == "apply_A":
        if _shape(case)["N"] * _shape(case)["gp"] > 2_000_000:
            return None
        lat = _Lattice(_problem(case, seed))
        s = _shape(case)
        free = s["vertices"] - math.prod(c + 1 for c in lat.counts[:2])
        x = _vector((case["loads"], s["N"] * s["nr"] + 3 * free + s["L"]), seed).to(lat.dev)
        return {"y": torch.stack([lat.apply_A(v) for v in x])}
    dof = _sizes((case["nx"], case["ny"], case["nz"]), case["elems"])["d"] * math.prod(
        c * case["elems"] + 1 for c in (case["nx"], case["ny"], case["nz"]) if c)
    if dof > _DENSE_DOF:
        return None
    lat = _Lattice(_problem(case, seed))
    f, u, lam = lat.solve()
    if op == "solve":
        return {"u": u, "lam": lam}
    c = torch.stack([(fs * us).sum() for fs, us in zip(f, u)])
    w = torch.linspace(1.0, 2.0, case["loads"], dtype=torch.float64, device=lat.dev)
    return {"compliance": c, "gradient": sum(w[q] * lat.gradient(u[q]) for q in range(len(f)))}
