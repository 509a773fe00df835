"""The work that a user of this framework has it do, as cases with sizes.

A case names a matrix family, its sizes, the number of value sets and the call made on
them.  The families are the ones of the benchmark and the tests: bordered 2-D grids,
bands, spatio-temporal precisions with dense covariate rows, and 3-D FEM operators.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) the analysed plan and the inputs, on the GPU
    run(state)          one pass through the public entry points, and its outputs
    work(case)          bytes and FP64 operations of one pass
    exact(case, seed)   what run returns, from plain torch in 64 bits (block tridiagonal
                        elimination in the input's own order, the dense rows last)
"""
import math

import numpy as np
import torch

from paper_2609_29765_gb300 import api

F64 = torch.float64


def listed():
    return [
        # one small precision matrix at a time: an optimiser's step on a 2-D field, latency only
        {"name": "grid2d_plain", "family": "grid2d", "nx": 32, "ny": 32, "border": 2, "nb": 64, "route": "auto",
         "batch": 1, "nrhs": 1, "op": "separate"},
        # the same pattern captured in a CUDA graph, a few dozen hyperparameter sets per replay
        {"name": "grid2d_graph", "family": "grid2d", "nx": 32, "ny": 32, "border": 2, "nb": 64, "route": "semisparse",
         "batch": 64, "nrhs": 1, "op": "graph"},
        # a sweep over hyperparameter sets on one small pattern: factor, logdet and solve of each
        {"name": "grid2d_batch", "family": "grid2d", "nx": 32, "ny": 32, "border": 2, "nb": 64, "route": "auto",
         "batch": 1024, "nrhs": 1, "op": "separate"},
        # one long band (an SPDE field on a line), one value set: the chain of block columns
        {"name": "band_plain", "family": "band", "n": 50000, "bw": 200, "nb": 128, "route": "auto",
         "batch": 1, "nrhs": 1, "op": "fused"},
        # the benchmark's step on a quarter of its length: factorize, logdet and solve of 64 value sets
        {"name": "band_batch", "family": "band", "n": 50000, "bw": 200, "nb": 128, "route": "auto",
         "batch": 64, "nrhs": 1, "op": "fused"},
        # a narrow band with posterior marginals: the factor and the selected inverse on its pattern
        {"name": "band_marginals", "family": "band", "n": 50000, "bw": 20, "nb": 32, "route": "auto",
         "batch": 16, "nrhs": 1, "op": "marginals"},
        # samples or predictions from a factor in hand: many right-hand sides
        {"name": "band_rhs", "family": "band", "n": 50000, "bw": 200, "nb": 128, "route": "auto",
         "batch": 1, "nrhs": 16, "op": "rhs"},
        # logdets of a spatio-temporal precision at several hyperparameter sets
        {"name": "stcov_batch", "family": "stcov", "nx": 30, "ny": 30, "nt": 25, "border": 20, "nb": 64,
         "route": "auto", "batch": 16, "nrhs": 1, "op": "logdet"},
        # the full-size spatio-temporal precision (n = 180,020), one evaluation with its solve
        {"name": "stcov_full", "family": "stcov", "nx": 60, "ny": 60, "nt": 50, "border": 20, "nb": 64,
         "route": "auto", "batch": 1, "nrhs": 1, "op": "fused"},
        # training: the gradient of logdet(Q) - x'Qx with respect to the values of Q
        {"name": "stcov_grad", "family": "stcov", "nx": 20, "ny": 20, "nt": 10, "border": 20, "nb": 64,
         "route": "auto", "batch": 64, "nrhs": 1, "op": "grad"},
        # FEM operators of three sizes in one launch
        {"name": "fem_mixed", "family": "fem", "g0": 16, "g1": 24, "g2": 32, "nb": 64, "route": "dense",
         "batch": 8, "nrhs": 1, "op": "mixed"},
        # one larger FEM operator: factorize and solve
        {"name": "fem_plain", "family": "fem", "g0": 48, "nb": 64, "route": "auto", "batch": 1, "nrhs": 1,
         "op": "fused"},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    kind = rng.choice(["grid2d", "band", "band", "stcov", "stcov", "fem"])
    if kind == "grid2d":
        nx, ny = rng.randint(15, 60), rng.randint(15, 60)
        op = rng.choice(["separate", "separate", "graph", "fused", "grad"])
        return {"family": "grid2d", "nx": nx, "ny": ny, "border": rng.randint(0, 5),
                "nb": rng.choice([32, 64, 64, 128]), "route": rng.choice(["auto", "auto", "semisparse"]),
                "batch": max(1, min(_log(rng, 1, 1024), 1100000 // (nx * ny))), "nrhs": rng.randint(1, 3), "op": op}
    if kind == "band":
        n, bw = _log(rng, 2000, 50000), _log(rng, 15, 220)
        op = rng.choice(["fused", "fused", "separate", "marginals", "rhs"])
        top = 20000000 if op == "marginals" else 300000000
        return {"family": "band", "n": n, "bw": bw, "nb": 128 if bw >= 80 else rng.choice([32, 64, 96, 128]),
                "route": rng.choice(["auto", "auto", "dense"]),
                "batch": max(1, min(_log(rng, 1, 64), top // (n * bw))), "nrhs": rng.randint(1, 8), "op": op}
    if kind == "stcov":
        op = rng.choice(["logdet", "fused", "grad"])
        nx, ny, nt = rng.randint(9, 32), rng.randint(9, 32), rng.randint(6, 30)
        if nx * ny * nt <= 6000:
            op = "grad"
        top = 24 if nx * ny * nt <= 6000 else 8 if op != "grad" else 3
        return {"family": "stcov", "nx": nx, "ny": ny, "nt": nt, "border": rng.randint(0, 20), "nb": 64,
                "route": rng.choice(["auto", "auto", "semisparse"]), "batch": _log(rng, 1, top), "nrhs": 1, "op": op}
    if rng.random() < 0.5:
        return {"family": "fem", "g0": rng.randint(9, 18), "g1": rng.randint(12, 24), "g2": rng.randint(16, 30),
                "nb": rng.choice([32, 64, 64, 96]), "route": rng.choice(["dense", "semisparse", "auto"]),
                "batch": _log(rng, 1, 8), "nrhs": 1, "op": "mixed"}
    return {"family": "fem", "g0": rng.randint(20, 44), "nb": rng.choice([64, 64, 128]),
            "route": rng.choice(["auto", "dense"]), "batch": 1, "nrhs": rng.randint(1, 3),
            "op": rng.choice(["fused", "logdet"])}


# ---- patterns: lower CSC with the diagonal, rows ascending in each column -----------------
_STENCILS = {
    "grid2d": [(0, 0, 0), (1, 0, 0), (0, 1, 0)],
    "fem": [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1)],
    "stcov": [(0, 0, 0), (1, 0, 0), (-1, 1, 0), (0, 1, 0), (1, 1, 0)] +
             [(dx, dy, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)],
}


class _Pattern:
    """colptr, rowind and lattice coordinates of one matrix; entry e is (row[e], col[e]), and
    pick[e] its place in the [columns, slots] array of candidates the values are made in."""

    def __init__(self, family, dims, border):
        if family == "band":
            n, bw = dims
            j = np.arange(n, dtype=np.int64)
            rows = j[:, None] + np.arange(bw + 1, dtype=np.int64)[None, :]
            live = rows < n
            self.block, self.nf, self.coords, self.stencil = bw, n, None, None
        else:
            nx, ny, nz = dims
            nf = nx * ny * nz
            j = np.arange(nf, dtype=np.int64)
            x, y, z = j % nx, (j // nx) % ny, j // (nx * ny)
            off = _STENCILS[family]
            rows = np.empty((nf, len(off) + border), dtype=np.int64)
            live = np.ones((nf, len(off) + border), dtype=bool)
            for s, (dx, dy, dz) in enumerate(off):
                rows[:, s] = j + dx + nx * (dy + ny * dz)
                live[:, s] = (x + dx >= 0) & (x + dx < nx) & (y + dy >= 0) & (y + dy < ny) & (z + dz < nz)
            rows[:, len(off):] = nf + np.arange(border)
            c = np.stack([x, y, z], axis=1).astype(np.float64)
            self.coords = np.vstack([c, np.full((border, 3), np.nan)])
            self.block, self.nf, self.stencil = (nx if nz == 1 else nx * ny), nf, off
        self.border = border
        self.n = self.nf + border
        pick = np.flatnonzero(live.ravel())
        r, col = rows.ravel()[pick], np.repeat(np.arange(self.nf, dtype=np.int64), rows.shape[1])[pick]
        tail = np.arange(self.nf, self.n, dtype=np.int64)  # the dense rows' own columns: a diagonal each
        self.row, self.col = np.concatenate([r, tail]), np.concatenate([col, tail])
        self.colptr = np.zeros(self.n + 1, dtype=np.int64)
        np.cumsum(np.bincount(self.col, minlength=self.n), out=self.colptr[1:])
        self.pick, self.slots, self.live = pick, rows.shape[1], live
        self.dims = dims

    def plan(self, case):
        natural = self.coords is None
        return api.Plan(self.n, self.colptr, self.row, coords=self.coords, nb=case["nb"], route=case["route"],
                        ordering="natural" if natural else "nd")


def _patterns(case):
    f = case["family"]
    if f == "band":
        return [_Pattern(f, (case["n"], case["bw"]), 0)]
    if f == "grid2d":
        return [_Pattern(f, (case["nx"], case["ny"], 1), case["border"])]
    if f == "stcov":
        return [_Pattern(f, (case["nx"], case["ny"], case["nt"]), case["border"])]
    return [_Pattern(f, (case[k],) * 3, 0) for k in ("g0", "g1", "g2") if k in case]


# ---- values [batch, nnz] on the GPU, from the seed alone ----------------------------------
def _finish(p, v, border_diag=None):
    """[batch, columns, slots] candidates (and the dense rows' diagonals) -> [batch, nnz]."""
    out = v.reshape(v.shape[0], -1)[:, torch.as_tensor(p.pick, device=v.device)]
    return out.contiguous() if border_diag is None else torch.cat([out, border_diag], dim=1).contiguous()


def _values(case, p, gen):
    dev, B = "cuda", case["batch"]

    def uniform(lo, hi, *shape):
        return torch.rand(*shape, generator=gen, device=dev, dtype=F64) * (hi - lo) + lo

    live = torch.as_tensor(p.live, device=dev)
    if case["family"] == "band":
        # off-diagonals U(-1, 1) 0.5 / bw, diagonal 1 + the row's absolute sum
        bw = p.slots - 1
        v = uniform(-0.5 / bw, 0.5 / bw, B, p.nf, p.slots) * live
        s = v[:, :, 1:].abs().sum(dim=2)
        for d in range(1, p.slots):
            s[:, d:] += v[:, : p.nf - d, d].abs()
        v[:, :, 0] = 1.0 + s
        return _finish(p, v)
    nx, ny, nz = p.dims
    off, m = p.stencil, len(p.stencil)
    v = torch.zeros(B, p.nf, p.slots, dtype=F64, device=dev)
    if case["family"] == "fem":
        # 7-point graph Laplacian with lognormal(0, 1) conductances + 1e-3 I
        c = torch.exp(torch.randn(B, p.nf, m, generator=gen, device=dev, dtype=F64)) * live
        v[:, :, 0] = 1e-3
        for s in range(1, m):
            step = off[s][0] + nx * (off[s][1] + ny * off[s][2])
            v[:, :, s] = -c[:, :, s]
            v[:, :, 0] += c[:, :, s]
            v[:, step:, 0] += c[:, : p.nf - step, s]
        return _finish(p, v)
    if case["family"] == "grid2d":
        # tau (5-point Dirichlet Laplacian + shift I), tau and shift differing by value set
        tau, shift = torch.exp(uniform(-2.3, 2.3, B, 1)), torch.exp(uniform(-4.6, 0.0, B, 1))
        v[:, :, 0] = tau * (4.0 + shift)
        v[:, :, 1:m] = -tau[:, :, None]
    else:
        # tau AR1(rho) (x) (kappa^2 + T) (x) (kappa^2 + T), T = tridiag(-1, 2, -1); theta log-uniform
        tau, rho, kap = (torch.exp(uniform(math.log(a), math.log(b), B, 1))
                         for a, b in ((0.1, 10.0), (0.05, 0.95), (0.05, 2.0)))
        t = torch.arange(p.nf, device=dev) // (nx * ny)
        inner = ((t > 0) & (t < nz - 1)).to(F64)[None, :]
        d = 2.0 + kap * kap
        for s, (dx, dy, dt) in enumerate(off):
            v[:, :, s] = tau * (-rho if dt else 1.0 + rho * rho * inner) * (-1.0 if dx else d) * (-1.0 if dy else d)
    if not p.border:
        return _finish(p, v)
    # dense covariate rows N(0, 0.01^2); both diagonals raised by the absolute sums
    b = 0.01 * torch.randn(B, p.nf, p.border, generator=gen, device=dev, dtype=F64)
    v[:, :, 0] += b.abs().sum(dim=2)
    v[:, :, m:] = b
    return _finish(p, v, 1.0 + b.abs().sum(dim=1))


def _inputs(case, seed):
    """Patterns, values of each and right-hand sides of the first."""
    ps = _patterns(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) * 7919 + 17)
    vals = [_values(case, p, gen) for p in ps]
    rhs = torch.randn(case["batch"], case["nrhs"], ps[0].n, generator=gen, device="cuda", dtype=F64)
    return ps, vals, rhs


def prepare(case, seed):
    ps, vals, rhs = _inputs(case, seed)
    plans = [p.plan(case) for p in ps]
    for q in plans:
        q.upload()
    st = {"op": case["op"], "plan": plans[0], "values": vals[0], "b": rhs}
    if case["op"] == "graph":
        st["graph"] = api.GraphedFactorize(plans[0], case["batch"])
    elif case["op"] == "rhs":
        st["factor"] = plans[0].factorize(vals[0])
    elif case["op"] == "mixed":
        st["group"] = api.Group(plans, [case["batch"]] * len(plans))
        st["values"] = vals
    elif case["op"] == "grad":
        st["values"] = vals[0].requires_grad_(True)
        st["x"] = rhs[:, 0].contiguous()
    return st


def run(st):
    op, plan, values = st["op"], st["plan"], st["values"]
    if op == "fused":
        fac, x = plan.factorize_solve(values, st["b"])
        return {"L": fac.data, "info": fac.info, "logdet": fac.logdet(), "x": x}
    if op == "separate":
        fac = plan.factorize(values)
        return {"L": fac.data, "info": fac.info, "logdet": fac.logdet(), "x": fac.solve(st["b"])}
    if op == "logdet":
        fac = plan.factorize(values)
        return {"L": fac.data, "info": fac.info, "logdet": fac.logdet()}
    if op == "graph":
        g = st["graph"]
        return {"logdet": g(values), "L": g.factor, "info": g.info}
    if op == "marginals":
        fac = plan.factorize(values)
        return {"L": fac.to_csc(), "info": fac.info, "logdet": fac.logdet(), "sigma": fac.selinv().to_csc()}
    if op == "rhs":
        return {"x": st["factor"].solve(st["b"])}
    if op == "mixed":
        facs = st["group"].factorize(values)
        return {"L": [f.data for f in facs], "info": [f.info for f in facs], "logdet": [f.logdet() for f in facs]}
    j = api.logdet(values, plan) - api.quad_form(values, st["x"], plan)
    (g,) = torch.autograd.grad(j.sum(), values)
    return {"value": j.detach(), "grad": g}


def work(case):
    """sum_j c_j^2 per factorization, twice that for a selected inverse, 4 nnz(L) per solve;
    every value, factor entry, right-hand side, solution and gradient once."""
    byts = flops = 0.0
    op, B = case["op"], case["batch"]
    for p in _patterns(case):
        i = p.plan(case).info
        nnz_a, nnz_l, fl, n = float(i["nnzA"]), float(i["nnzL"]), float(i["flops_alg"]), float(p.n)
        if op != "rhs":
            flops += B * fl
            byts += B * 8 * nnz_a
            if op != "grad":
                byts += B * 8 * nnz_l
        if op == "rhs":
            byts += B * 8 * nnz_l
        if op in ("fused", "separate", "rhs"):
            flops += B * case["nrhs"] * 4 * nnz_l
            byts += B * case["nrhs"] * 16 * n
        if op == "marginals":
            flops += B * 2 * fl
            byts += B * 8 * nnz_l
        if op == "grad":
            flops += B * (2 * fl + 8 * nnz_a)
            byts += B * 8 * (nnz_a + n)
    return {"bytes": byts, "flops": flops}


# ---- the same in plain torch, 64 bits -----------------------------------------------------
# In its own order each field is block tridiagonal (a grid row, a plane, a time step, or bw
# consecutive variables per block); the dense rows are eliminated last through their Schur
# complement.
class _Blocks:
    def __init__(self, p, vals):
        B, m = vals.shape[0], p.block
        nk = -(-p.nf // m)
        dev = vals.device
        row, col = torch.as_tensor(p.row, device=dev), torch.as_tensor(p.col, device=dev)
        field = (row < p.nf) & (col < p.nf)
        self.D = torch.zeros(B, nk, m, m, dtype=F64, device=dev)
        self.E = torch.zeros(B, max(nk - 1, 1), m, m, dtype=F64, device=dev)  # block (k + 1, k)
        pad = torch.arange(p.nf, nk * m, device=dev)
        self.D[:, -1, pad % m, pad % m] = 1.0
        same = field & (row // m == col // m)
        r, c = row[same], col[same]
        self.D[:, c // m, r % m, c % m] = vals[:, same]
        self.D[:, c // m, c % m, r % m] = vals[:, same]
        nxt = field & (row // m == col // m + 1)
        r, c = row[nxt], col[nxt]
        self.E[:, c // m, r % m, c % m] = vals[:, nxt]
        self.Bd = self.C = None
        if p.border:
            d = (row >= p.nf) & (col < p.nf)
            self.Bd = torch.zeros(B, nk * m, p.border, dtype=F64, device=dev)
            self.Bd[:, col[d], row[d] - p.nf] = vals[:, d]
            self.C = torch.diag_embed(vals[:, (row >= p.nf) & (col >= p.nf)])
        self.p, self.m, self.nk = p, m, nk

    def factor(self):
        """D[k] <- L_kk, E[k] <- L_(k+1,k); W = T^{-1} B and the border's own factor."""
        for k in range(self.nk):
            if k:
                self.D[:, k] -= self.E[:, k - 1] @ self.E[:, k - 1].mT
            self.D[:, k] = torch.linalg.cholesky(self.D[:, k])
            if k + 1 < self.nk:
                self.E[:, k] = torch.linalg.solve_triangular(self.D[:, k].mT, self.E[:, k], upper=True, left=False)
        ld = self.D.diagonal(dim1=2, dim2=3).log().sum(dim=(1, 2))
        if self.C is not None:
            self.W = self._field_solve(self.Bd)
            self.Cf = torch.linalg.cholesky(self.C - self.Bd.mT @ self.W)
            ld = ld + self.Cf.diagonal(dim1=1, dim2=2).log().sum(dim=1)
        self.logdet = 2.0 * ld
        return self

    def _field_solve(self, b):
        y = b.reshape(b.shape[0], self.nk, self.m, -1).clone()
        for k in range(self.nk):
            if k:
                y[:, k] -= self.E[:, k - 1] @ y[:, k - 1]
            y[:, k] = torch.linalg.solve_triangular(self.D[:, k], y[:, k], upper=False)
        for k in range(self.nk - 1, -1, -1):
            if k + 1 < self.nk:
                y[:, k] -= self.E[:, k].mT @ y[:, k + 1]
            y[:, k] = torch.linalg.solve_triangular(self.D[:, k].mT, y[:, k], upper=True)
        return y.reshape(b.shape[0], self.nk * self.m, -1)

    def solve(self, b):
        """b [batch, nrhs, n] -> x of the same shape."""
        nf, pad = self.p.nf, self.nk * self.m - self.p.nf
        f = torch.nn.functional.pad(b[:, :, :nf], (0, pad)).mT.contiguous()
        x = self._field_solve(f)
        if self.C is None:
            return x[:, :nf].mT.contiguous()
        z = torch.cholesky_solve(b[:, :, nf:].mT - self.Bd.mT @ x, self.Cf)
        return torch.cat([(x - self.W @ z)[:, :nf].mT, z.mT], dim=2).contiguous()

    def sigma(self):
        """The inverse on the pattern of A, [batch, nnz] in its order."""
        m, dev = self.m, self.D.device
        eye = torch.eye(m, dtype=F64, device=dev).expand(self.D.shape[0], m, m)
        S, T = torch.empty_like(self.D), torch.empty_like(self.E)
        for k in range(self.nk - 1, -1, -1):
            Li = torch.linalg.solve_triangular(self.D[:, k], eye, upper=False)
            S[:, k] = Li.mT @ Li
            if k + 1 < self.nk:
                G = self.E[:, k] @ Li  # L_(k+1,k) L_kk^{-1}
                T[:, k] = -S[:, k + 1] @ G
                S[:, k] -= G.mT @ T[:, k]
        row, col = torch.as_tensor(self.p.row, device=dev), torch.as_tensor(self.p.col, device=dev)
        nf = self.p.nf
        out = torch.empty(self.D.shape[0], row.numel(), dtype=F64, device=dev)
        bord = row >= nf
        r, c = row.clamp(max=nf - 1), col.clamp(max=nf - 1)
        same = (r // m == c // m) & ~bord
        nxt = (r // m == c // m + 1) & ~bord
        out[:, same] = S[:, c[same] // m, r[same] % m, c[same] % m]
        out[:, nxt] = T[:, c[nxt] // m, r[nxt] % m, c[nxt] % m]
        if self.C is not None:
            Ci = torch.cholesky_inverse(self.Cf)
            V = self.W @ Ci
            f = ~bord
            out[:, f] += (V[:, row[f]] * self.W[:, col[f]]).sum(dim=2)
            d = bord & (col < nf)
            out[:, d] = -V[:, col[d], row[d] - nf]
            out[:, bord & (col >= nf)] = Ci.diagonal(dim1=1, dim2=2)
        return out

    def lower(self):
        """L on the pattern of A where the natural order gives no fill (a full band)."""
        row, col = torch.as_tensor(self.p.row, device=self.D.device), torch.as_tensor(self.p.col, device=self.D.device)
        m = self.m
        same = row // m == col // m
        out = torch.empty(self.D.shape[0], row.numel(), dtype=F64, device=self.D.device)
        out[:, same] = self.D[:, col[same] // m, row[same] % m, col[same] % m]
        out[:, ~same] = self.E[:, col[~same] // m, row[~same] % m, col[~same] % m]
        return out


def exact(case, seed):
    ps, vals, rhs = _inputs(case, seed)
    op = case["op"]
    zero = torch.zeros(case["batch"], dtype=torch.int32, device="cuda")
    fs = [_Blocks(p, v).factor() for p, v in zip(ps, vals)]
    f, p, v = fs[0], ps[0], vals[0]
    if op == "mixed":
        return {"L": [None] * len(fs), "info": [zero] * len(fs), "logdet": [q.logdet for q in fs]}
    if op == "grad":
        x = rhs[:, 0]
        row, col = torch.as_tensor(p.row, device="cuda"), torch.as_tensor(p.col, device="cuda")
        two = torch.where(row == col, 1.0, 2.0).to(F64)
        xx = two * x[:, row] * x[:, col]
        return {"value": f.logdet - (v * xx).sum(dim=1), "grad": two * f.sigma() - xx}
    if op == "marginals":
        return {"L": f.lower(), "info": zero, "logdet": f.logdet, "sigma": f.sigma()}
    if op == "rhs":
        return {"x": f.solve(rhs)}
    out = {"L": None, "info": zero, "logdet": f.logdet}
    if op in ("fused", "separate"):
        out["x"] = f.solve(rhs)
    return out
