"""The work that users of this library have it do, as cases to time.

A case is one pass through the public calls: factorize new values on an
analysed pattern and solve (``solve``), solve again with a factor that is kept
(``kept``), a batch of small systems (``batch``), or the differentiable solve
and log-determinant forward and backward (``diff``).  The analysis is what a
program makes once per pattern and keeps, so states of one pattern share it.
"""
import functools
import math

import numpy as np
import torch

from paper_1405_2636_gb300 import spx
from paper_1405_2636_gb300.autograd import SparseSPD

DEV = "cuda"


def _solve(name, op, nx, ny, nz, method, precision, nrhs, ordering="grid", max_width=64, kind="solve"):
    return {"name": name, "kind": kind, "op": op, "nx": nx, "ny": ny, "nz": nz, "method": method,
            "precision": precision, "nrhs": nrhs, "ordering": ordering, "max_width": max_width}


def listed():
    return [
        # The smallest system of the workloads: one right-hand side, latency alone.
        _solve("laplace2d_31_fp64", "laplace", 31, 31, 1, "llt", "fp64", 1),
        # A general sparse matrix with every option at its default: graph
        # ordering, panels up to 128 wide, an FP64 factor.
        _solve("diffusion_defaults_fp64", "diffusion", 40, 36, 33, "llt", "fp64", 1, "graph", 0),
        # The main workload, in plain FP64 and in mixed precision with
        # refinement to a backward error of 1e-12.
        _solve("diffusion_64_fp64", "diffusion", 64, 64, 64, "llt", "fp64", 16),
        _solve("diffusion_64_tf32", "diffusion", 64, 64, 64, "llt", "tf32", 16),
        # An ordinary ragged box, ordered as a graph, single precision and a
        # few right-hand sides.
        _solve("diffusion_ragged_fp32", "diffusion", 53, 47, 39, "llt", "fp32", 5, "graph"),
        # Elasticity: three unknowns a node, 27-point coupling, BF16 updates.
        _solve("elasticity_28_bf16", "elasticity", 28, 28, 28, "llt", "bf16", 1),
        # A symmetric indefinite (quasi-definite) system.
        _solve("quasidefinite_32_fp64", "quasidefinite", 32, 32, 32, "ldlt", "fp64", 16),
        # One unsymmetric system (upwinded convection-diffusion), refined.
        _solve("convection_lu_fp32", "convection", 121, 97, 1, "lu", "fp32", 3),
        # Time stepping: the factor is kept, one right-hand side a step.
        _solve("kept_factor_48_fp64", "diffusion", 48, 48, 48, "llt", "fp64", 1, kind="kept"),
        # Thousands of small unsymmetric systems of uneven size in one launch,
        # and a handful of smaller ones in FP64.
        {"name": "batch_4096_fp32", "kind": "batch", "count": 4096, "k_lo": 12, "k_hi": 80, "precision": "fp32"},
        {"name": "batch_24_fp64", "kind": "batch", "count": 24, "k_lo": 5, "k_hi": 40, "precision": "fp64"},
        # Training through a solve and a log-determinant: loss, and gradients
        # with respect to the matrix values and the right-hand side.
        {"name": "diff_48", "kind": "diff", "nx": 48, "ny": 48, "nz": 48},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any call, method, precision, ordering and panel width,
    box sides spread over the range of the listed ones."""
    kind = rng.choice(["solve", "solve", "solve", "solve", "kept", "batch", "diff"])
    precision = rng.choice(["fp64", "fp32", "tf32", "bf16"])
    if kind == "batch":
        lo = rng.randint(2, 40)
        return {"kind": "batch", "count": _log_int(rng, 1, 2048), "k_lo": lo, "k_hi": rng.randint(lo, 80),
                "precision": rng.choice(["fp64", "fp32"])}
    # a cube side of the wanted size, each axis up to a third off it
    side = math.exp(rng.uniform(math.log(8), math.log(42)))
    nx, ny, nz = (max(4, min(64, int(side * rng.uniform(0.75, 1.33)))) for _ in range(3))
    if kind == "diff":
        return {"kind": "diff", "nx": nx, "ny": ny, "nz": nz}
    op = rng.choice(["laplace", "diffusion", "diffusion", "elasticity", "quasidefinite", "convection"])
    method = {"quasidefinite": "ldlt", "convection": "lu"}.get(op, "llt")
    if op in ("laplace", "convection"):                     # plane problems: 20 .. 300 a side
        nx, ny = (max(8, _log_int(rng, 20, 300)) for _ in range(2))
        nz = 1
        if op == "convection":                              # the sides of the convection workloads
            nx, ny = max(12, nx // 2), max(12, ny // 2)
    if op in ("elasticity", "quasidefinite"):
        f = 0.6 if op == "elasticity" else 0.75
        nx, ny, nz = (max(4, int(f * k)) for k in (nx, ny, nz))
    width = rng.choice([64, 64, 48, 0]) if method != "ldlt" else rng.choice([64, 48])
    return {k: v for k, v in _solve("", op, nx, ny, nz, method, precision, rng.choice([1, 2, 3, 5, 8, 16, 20]),
                                    rng.choice(["grid", "graph"]), width, kind).items() if k != "name"}


# ---------------------------------------------------------------------------
# Patterns (host) and values (device).  Node (x, y, z) is x + nx (y + ny z); the
# neighbours of a node are its stencil's offsets in ascending order of node
# number, so that a column's stored entries come out sorted.
# ---------------------------------------------------------------------------
def _dof(op):
    return {"elasticity": 3, "quasidefinite": 2}.get(op, 1)


def _offsets(op, nz):
    o = [(dx, dy, dz) for dz in ((-1, 0, 1) if nz > 1 else (0,)) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    return o if op == "elasticity" else [d for d in o if sum(map(abs, d)) <= 1]


def _stencil(op, nx, ny, nz):
    """(neighbour node or -1) per node and offset, and the offsets."""
    off = _offsets(op, nz)
    n = nx * ny * nz
    i = np.arange(n, dtype=np.int64)
    x, y, z = i % nx, i // nx % ny, i // (nx * ny)
    nb = np.empty((n, len(off)), np.int64)
    for s, (dx, dy, dz) in enumerate(off):
        ok = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz >= 0) & (z + dz < nz)
        nb[:, s] = np.where(ok, i + dx + nx * (dy + ny * dz), -1)
    return nb, off


def _csc(nb, dof):
    """(colptr, rowind) of the stencil with dof unknowns a node."""
    ok = nb >= 0
    count = np.repeat(ok.sum(1) * dof, dof)
    colptr = np.zeros(len(count) + 1, np.int64)
    np.cumsum(count, out=colptr[1:])
    rows = nb[:, None, :, None] * dof + np.arange(dof)              # node, column dof, offset, row dof
    rows = np.broadcast_to(rows, (nb.shape[0], dof) + rows.shape[2:])
    keep = np.broadcast_to(ok[:, None, :, None], rows.shape)
    return colptr, rows[keep].astype(np.int32)


def _rand(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 1)
    return g


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _uniform(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _diffusion_slots(nb, off, kappa):
    """Node, offset: 7-point diffusion, face coefficient the mean of two nodes'."""
    face = 0.5 * (kappa[:, None] + torch.where(nb >= 0, kappa[nb.clamp(min=0)], kappa[:, None]))
    c = off.index((0, 0, 0))
    face[:, c] = 0.0
    v = -face
    v[:, c] = face.sum(1)
    return v


def _values(op, nx, ny, nz, g):
    """The stored values of a new matrix, in the order of _csc."""
    nb_h, off = _stencil(op, nx, ny, nz)
    nb = torch.from_numpy(nb_h).to(DEV)
    n, ns = nb.shape
    c = off.index((0, 0, 0))
    if op == "laplace":                       # 4 on the diagonal, a shift that varies by a node
        v = torch.full((n, ns), -1.0, device=DEV, dtype=torch.float64)
        v[:, c] = (4.0 if nz == 1 else 6.0) + _uniform(g, 0.5e-2, 1.5e-2, n)
    elif op == "diffusion":                   # node coefficients exp(g), g ~ N(0, 1)
        v = _diffusion_slots(nb, off, torch.exp(_normal(g, n)))
    elif op == "convection":                  # first-order upwind, mesh Peclet number ~ U(0, 10)
        v = _convection_slots(n, off, _uniform(g, 0.0, 10.0, 1), _uniform(g, 0.0, 2 * math.pi, 1))[0]
    elif op == "quasidefinite":               # [[K, B^T], [B, -C]] per pair of nodes
        K = _diffusion_slots(nb, off, torch.exp(_normal(g, n)))
        C = 0.1 * _diffusion_slots(nb, off, torch.exp(_normal(g, n)))
        B = _uniform(g, -0.5, 0.5, n, ns)     # B[j, s]: row p of the neighbour, column u of j
        opp = torch.tensor([off.index(tuple(-d for d in o)) for o in off], device=DEV)
        Bt = B[nb.clamp(min=0), opp[None, :]]
        v = torch.stack([torch.stack([K, Bt], -1), torch.stack([B, -C], -1)], -2)
    else:                                     # elasticity: K = R diag(mu) R^T per pair, mu ~ logU[1, 1e3]
        def coupling():
            q = _normal(g, n, 4)
            w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
            R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                             2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                             2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).view(n, 3, 3)
            K = (R * torch.exp(_uniform(g, 0.0, math.log(1e3), n, 1, 3))) @ R.transpose(1, 2)
            return 0.5 * (K + K.transpose(1, 2))
        v = torch.zeros(n, ns, 3, 3, device=DEV, dtype=torch.float64)
        for s, o in enumerate(off):
            if o[::-1] <= (0, 0, 0):
                continue
            K, Kb = coupling(), coupling()    # with the node ahead (or the boundary), and a boundary behind
            t = off.index(tuple(-d for d in o))
            v[:, s] = -K
            behind = nb[:, t].clamp(min=0)
            v[:, t] = -K[behind]
            v[:, c] += K + torch.where((nb[:, t] >= 0)[:, None, None], K[behind], Kb)
    if v.dim() == 2:
        return v[nb >= 0]
    d = v.shape[2]
    v = v.permute(0, 3, 1, 2)                 # node, column dof, offset, row dof
    return v[(nb >= 0)[:, None, :, None].expand(n, d, ns, d)].contiguous()


def _convection_slots(n, off, peclet, theta):
    """System, node, offset: entry (neighbour, node) of the upwinded operator."""
    wx, wy = 2 * peclet * torch.cos(theta), 2 * peclet * torch.sin(theta)
    v = torch.empty(len(peclet), n, len(off), device=DEV, dtype=torch.float64)
    for s, (dx, dy, _) in enumerate(off):
        w = wx * dx + wy * dy                 # the row is the neighbour: downwind rows look back at this node
        v[:, :, s] = (4.0 + wx.abs() + wy.abs() if dx == dy == 0 else -1.0 - w.clamp(min=0))[:, None]
    return v


@functools.lru_cache(maxsize=1)
def _pattern(op, nx, ny, nz):
    return _csc(_stencil(op, nx, ny, nz)[0], _dof(op))


def _analyze(case):
    op, nx, ny, nz = case["op"], case["nx"], case["ny"], case["nz"]
    opts = {"max_width": case["max_width"], "ordering": spx.SPX_ORDER_GRAPH}
    if case["ordering"] == "grid":
        opts.update(ordering=spx.SPX_ORDER_GRID, grid=(nx, ny, nz), dof=_dof(op))
    return spx.analyze(*_pattern(op, nx, ny, nz), case["method"], **opts)


def _sides(case):
    """Grid side of each system: uneven, the same for every seed."""
    return [int(k) for k in np.random.default_rng([4, 2]).integers(case["k_lo"], case["k_hi"] + 1, size=case["count"])]


@functools.lru_cache(maxsize=1)
def _plan(key):
    """What a program keeps for a pattern: made once, used for all its values."""
    case = dict(key)
    if case["kind"] == "batch":
        sides = _sides(case)
        pat = {k: _csc(_stencil("convection", k, k, 1)[0], 1) for k in set(sides)}
        return spx.batch_analyze([pat[k] for k in sides], grids=[(k, k, 1) for k in sides],
                                 ordering=spx.SPX_ORDER_GRID, max_width=64)
    if case["kind"] == "diff":
        dims = (case["nx"], case["ny"], case["nz"])
        return SparseSPD(*_pattern("diffusion", *dims), ordering=spx.SPX_ORDER_GRID, grid=dims, max_width=64)
    return _analyze(case)


def _plan_of(case):
    return _plan(tuple(sorted((k, v) for k, v in case.items() if k != "name")))


def _batch_values(case, seed):
    sides = np.array(_sides(case))
    g = _rand(seed)
    peclet, theta = _uniform(g, 0.0, 10.0, len(sides)), _uniform(g, 0.0, 2 * math.pi, len(sides))
    nnz = 5 * sides * sides - 4 * sides
    start = torch.from_numpy(np.concatenate([[0], np.cumsum(nnz)[:-1]])).to(DEV)
    vals = torch.empty(int(nnz.sum()), device=DEV, dtype=torch.float64)
    groups = {}
    for k in sorted(set(sides.tolist())):
        s = torch.from_numpy(np.nonzero(sides == k)[0]).to(DEV)
        nb, off = _stencil("convection", k, k, 1)
        v = _convection_slots(k * k, off, peclet[s], theta[s])[:, torch.from_numpy(nb >= 0).to(DEV)]
        vals[(start[s][:, None] + torch.arange(v.shape[1], device=DEV)).reshape(-1)] = v.reshape(-1)
        groups[k] = (s, v)
    rhs = _uniform(g, -1.0, 1.0, int((sides * sides).sum()))
    return vals, rhs, groups


def prepare(case, seed):
    if case["kind"] == "batch":
        vals, rhs, _ = _batch_values(case, seed)
        return {"kind": "batch", "plan": _plan_of(case), "values": vals, "B": rhs, "precision": case["precision"],
                "refine": spx.default_refine(tol=1e-10) if case["precision"] == "fp32" else None}
    op = case.get("op", "diffusion")
    g = _rand(seed)
    vals = _values(op, case["nx"], case["ny"], case["nz"], g)
    n = case["nx"] * case["ny"] * case["nz"] * _dof(op)
    if case["kind"] == "diff":
        return {"kind": "diff", "plan": _plan_of(case), "values": vals, "b": _normal(g, n), "w": _normal(g, n)}
    nrhs = case["nrhs"]
    B = _uniform(g, -1.0, 1.0, nrhs, n).t() if nrhs > 1 else _uniform(g, -1.0, 1.0, n)
    state = {"kind": case["kind"], "values": vals, "B": B, "precision": case["precision"]}
    if case["kind"] == "kept":                # each state its own factor
        state["plan"] = _analyze(case)
        state["plan"].factorize(vals, case["precision"])
    else:
        state["plan"] = _plan_of(case)
    return state


def run(state):
    plan = state["plan"]
    if state["kind"] == "batch":
        X, _ = plan.run(state["values"], state["B"], precision=state["precision"], refine=state["refine"])
        return X
    if state["kind"] == "diff":
        v = state["values"].clone().requires_grad_()        # values a step's coefficients have just given
        b = state["b"].clone().requires_grad_()
        x, logdet = plan.solve(v, b), plan.logdet(v)
        gv, gb = torch.autograd.grad((state["w"] * x).sum() + logdet, (v, b))
        return {"x": x.detach(), "logdet": logdet.detach(), "grad_values": gv, "grad_b": gb}
    if state["kind"] == "solve":
        plan.factorize(state["values"], state["precision"])
    X, info = plan.solve(state["B"])
    return {"X": X, "converged": info["converged"]}


def work(case):
    """Factorization flops counted from the symbolic structure, and the solves';
    the values, right-hand sides, solutions and the factor once each (the
    factor twice more where only the solve is timed, a read a sweep)."""
    plan = _plan_of(case)
    if case["kind"] == "batch":
        i = plan.info()
        item = 4 if case["precision"] == "fp32" else 8
        return {"bytes": 8 * i["nnz_total"] + 16 * i["n_total"] + item * 2 * i["nnz_l_total"],
                "flops": i["flops"] + 4 * i["nnz_l_total"]}
    i = (plan.handle if case["kind"] == "diff" else plan).info()
    if case["kind"] == "diff":                # two solves, log det, and the selected inverse at twice the factorization
        return {"bytes": 8 * (2 * i["nnz_a"] + 4 * i["n"]) + 16 * i["nnz_l"], "flops": 3 * i["flops"] + 8 * i["nnz_l"]}
    item = 8 if case["precision"] == "fp64" else 4
    lu = 2 if case["method"] == "lu" else 1
    solve = 4 * lu * i["nnz_l"] * case["nrhs"]
    if case["kind"] == "kept":
        return {"bytes": 2 * item * lu * i["nnz_l"] + 16 * i["n"] * case["nrhs"], "flops": solve}
    return {"bytes": 8 * i["nnz_a"] + 16 * i["n"] * case["nrhs"] + item * lu * i["nnz_l"], "flops": i["flops"] + solve}


# ---------------------------------------------------------------------------
# The same results in 64 bits by plain torch: block elimination plane by plane
# (a grid stencil couples only neighbouring planes), then a step of refinement.
# ---------------------------------------------------------------------------
class _Planes:
    def __init__(self, colptr, rowind, vals, planes):
        self.m, self.nb = vals.shape[0], planes
        self.n = len(colptr) - 1
        self.bs = self.n // planes
        self.vals = vals
        self.col = torch.from_numpy(np.repeat(np.arange(self.n), np.diff(colptr))).to(DEV)
        self.row = torch.from_numpy(np.asarray(rowind, np.int64)).to(DEV)
        order = torch.arange(len(rowind), device=DEV)
        self.at = {}
        rb, cb = self.row // self.bs, self.col // self.bs
        for d in (-1, 0, 1):                  # block row - block column
            e = order[rb - cb == d]
            s = torch.bincount(cb[e], minlength=planes).cpu().tolist()
            self.at[d] = list(torch.split(e, s))
        self.lu, self.W, self.logdet = [], [], 0.0
        S = self._dense(0, 0)
        for k in range(planes):
            lu, piv = torch.linalg.lu_factor(S)
            self.lu.append((lu, piv))
            self.logdet = self.logdet + lu.diagonal(dim1=-2, dim2=-1).abs().log().sum(-1)
            if k + 1 < planes:
                self.W.append(torch.linalg.lu_solve(lu, piv, self._dense(-1, k + 1)))
                S = self._dense(0, k + 1) - self._below(k, self.W[k])

    def _dense(self, d, k):
        e = self.at[d][k]
        D = torch.zeros(self.m, self.bs, self.bs, device=DEV, dtype=torch.float64)
        D[:, self.row[e] % self.bs, self.col[e] % self.bs] = self.vals[:, e]
        return D

    def _below(self, k, Y):
        """A's block under plane k, times Y."""
        e = self.at[1][k]
        out = torch.zeros_like(Y)
        for p in torch.split(e, max(1, 50_000_000 // (self.m * Y.shape[-1]))):
            out.index_add_(1, self.row[p] % self.bs, self.vals[:, p, None] * Y[:, self.col[p] % self.bs])
        return out

    def _once(self, B):
        b = B.reshape(self.m, self.nb, self.bs, -1)
        y, x = [], [None] * self.nb
        for k in range(self.nb):
            r = b[:, k] - (self._below(k - 1, y[k - 1]) if k else 0.0)
            y.append(torch.linalg.lu_solve(*self.lu[k], r))
        x[-1] = y[-1]
        for k in range(self.nb - 2, -1, -1):
            x[k] = y[k] - self.W[k] @ x[k + 1]
        return torch.cat(x, 1)

    def solve(self, B):
        """B: system, unknown, right-hand side."""
        X = self._once(B)
        for _ in range(2):
            R = B.clone()
            for p in torch.split(torch.arange(len(self.row), device=DEV), max(1, 50_000_000 // (self.m * B.shape[-1]))):
                R.index_add_(1, self.row[p], -self.vals[:, p, None] * X[:, self.col[p]])
            X = X + self._once(R)
        return X

    def inverse_on_pattern(self):
        """(A^-1)(j, i) of every stored entry (i, j), A symmetric."""
        out = torch.zeros_like(self.vals)
        eye = torch.eye(self.bs, device=DEV, dtype=torch.float64).expand(self.m, -1, -1)
        Z = None
        for k in range(self.nb - 1, -1, -1):
            Zkk = torch.linalg.lu_solve(*self.lu[k], eye)
            if Z is not None:
                off = -self.W[k] @ Z          # plane k, plane k + 1
                for d, c in ((1, k), (-1, k + 1)):
                    e = self.at[d][c]
                    r, q = self.row[e] % self.bs, self.col[e] % self.bs
                    out[:, e] = off[:, q, r] if d == 1 else off[:, r, q]
                Zkk = Zkk - off @ self.W[k].transpose(1, 2)
            e = self.at[0][k]
            out[:, e] = Zkk[:, self.row[e] % self.bs, self.col[e] % self.bs]
            Z = Zkk
        return out


def exact(case, seed):
    if case["kind"] == "batch":
        _, rhs, groups = _batch_values(case, seed)
        sides = np.array(_sides(case))
        first = np.concatenate([[0], np.cumsum(sides * sides)[:-1]])
        X = torch.empty_like(rhs)
        for k, (s, v) in groups.items():
            at = torch.from_numpy(first).to(DEV)[s][:, None] + torch.arange(k * k, device=DEV)
            P = _Planes(*_csc(_stencil("convection", k, k, 1)[0], 1), v, k)
            X[at.reshape(-1)] = P.solve(rhs[at][:, :, None]).reshape(-1)
        return X
    op, (nx, ny, nz) = case.get("op", "diffusion"), (case[k] for k in ("nx", "ny", "nz"))
    g = _rand(seed)
    vals = _values(op, nx, ny, nz, g)
    colptr, rowind = _pattern(op, nx, ny, nz)
    n = len(colptr) - 1
    P = _Planes(colptr, rowind, vals[None], nz if nz > 1 else ny)
    if case["kind"] == "diff":
        b, w = _normal(g, n), _normal(g, n)
        x, lam = P.solve(torch.stack([b, w], 1)[None])[0].unbind(1)
        gv = P.inverse_on_pattern()[0] - lam[P.row] * x[P.col]
        return {"x": x, "logdet": P.logdet[0], "grad_values": gv, "grad_b": lam}
    nrhs = case["nrhs"]
    B = _uniform(g, -1.0, 1.0, nrhs, n).t() if nrhs > 1 else _uniform(g, -1.0, 1.0, n)
    X = P.solve(B.reshape(1, n, -1))[0]
    return {"X": X if nrhs > 1 else X[:, 0], "converged": None}
