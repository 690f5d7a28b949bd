"""The work a user of this library has it do, as timed cases.

Every case goes through the public calls of ``paper_1703_01325_gb300.bilu`` (or
``adjoint``) on reservoir-style block matrices: cells of an nx x ny x nz grid in
natural order, b unknowns per cell, a 7- or 27-point block stencil, lognormal
permeability (sigma = 1) and a small accumulation term (0.01) -- the recipe of
``reservoir.py``, drawn here on the GPU so that large inputs are made quickly.

``op`` says which call a case makes:

  apply, apply_f32                  the preconditioner apply M^{-1} r
  factor, factor_f32                the numeric ILU(k) factorization
  spmv, spmv_f32, spmv_f32x         the block SpMV
  setup                             a new mesh: device symbolic phase, upload, factorization
  solve, solve_f32prec, solve_mixed, gmres
                                    a whole preconditioned solve to a true relative residual of 1e-12
  grad                              forward and backward of the differentiable solve

``exact`` repeats a case in plain torch FP64: the ILU(k) pattern of a grid from
the fill-path theorem, the factorization and the triangular solves level by
level, whole systems by a block-Jacobi BiCGSTAB.
"""
from __future__ import annotations

import math

import torch

from paper_1703_01325_gb300 import bilu as B
from paper_1703_01325_gb300.adjoint import BlockILUSolver
from paper_1703_01325_gb300.reservoir import grid_pattern, stencil_offsets

DEV = "cuda"
F64 = torch.float64
SIGMA, ACCUM = 1.0, 0.01
TOL, MAXIT = 1e-12, 1500


def _case(name, op, dims, b, k, stencil=7):
    nx, ny, nz = dims
    c = {"op": op, "nx": nx, "ny": ny, "nz": nz, "stencil": stencil, "b": b, "k": k}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the preconditioner on a small model: every launch and hand-off counts
        _case("apply_16x16x8_b3_k1", "apply", (16, 16, 8), 3, 1),
        # the preconditioner on the benchmark's grid: the call a solve spends its time in
        _case("apply_128x128x64_b3_k1", "apply", (128, 128, 64), 3, 1),
        # the single-precision preconditioner on the grid of the precision comparison
        _case("apply_f32_96x96x48_b4_k1", "apply_f32", (96, 96, 48), 4, 1),
        # wide rows: a 27-point stencil with two levels of fill (up to 60 blocks a row)
        _case("apply_27pt_80x80x40_b3_k2", "apply", (80, 80, 40), 3, 2, 27),
        # odd extents, more components, no fill
        _case("apply_61x47x33_b5_k0", "apply", (61, 47, 33), 5, 0),
        # new matrix values on a known mesh: every Newton step factors again
        _case("factor_96x96x48_b3_k1", "factor", (96, 96, 48), 3, 1),
        # the single-precision factorization, odd extents, two levels of fill
        _case("factor_f32_61x47x33_b4_k2", "factor_f32", (61, 47, 33), 4, 2),
        # the operator itself on the benchmark's grid
        _case("spmv_128x128x64_b3", "spmv", (128, 128, 64), 3, 0),
        # a new mesh: symbolic phase, schedules and factorization
        _case("setup_64x64x32_b3_k1", "setup", (64, 64, 32), 3, 1),
        # a small system solved from start to end
        _case("solve_16x16x8_b3_k1", "solve", (16, 16, 8), 3, 1),
        # FP64 BiCGSTAB with the single-precision preconditioner
        _case("solve_f32prec_96x96x48_b4_k1", "solve_f32prec", (96, 96, 48), 4, 1),
        # parameter estimation: the solve and its adjoint, gradients of values and right-hand side
        _case("grad_64x64x32_b3_k1", "grad", (64, 64, 32), 3, 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["apply"] * 5 + ["apply_f32"] * 3 + ["factor"] * 3 + ["factor_f32"] * 2 +
                    ["spmv", "spmv", "spmv_f32", "spmv_f32x", "setup", "solve", "solve_f32prec", "solve_mixed",
                     "gmres", "grad"])
    whole = op in ("solve", "solve_f32prec", "solve_mixed", "gmres", "grad")
    while True:
        stencil = 27 if op != "apply_f32" and rng.random() < 0.2 else 7
        dims = (_log_int(rng, 9, 150), _log_int(rng, 7, 140), _log_int(rng, 5, 80))
        b = rng.choice([1, 2, 3, 3, 4, 5] if whole else [1, 2, 2, 3, 3, 3, 4, 4, 5, 6, 7, 8])
        k = 0 if op.startswith("spmv") else rng.choice([0, 1, 1, 2])
        if op == "gmres":  # restarts stall on weaker preconditioners
            b, k = min(b, 3), max(k, 1)
        cells = dims[0] * dims[1] * dims[2]
        blocks = stencil * (1, 2, 3.5)[k]  # of a row of P', about
        # no costlier than the largest listed case of its kind
        most = 30_000 * 49 if op == "gmres" else 130_000 * 130 if whole or op == "setup" else 1_050_000 * 126
        if cells * blocks * b * b <= most and cells >= 400:
            break
    return _case(None, op, dims, b, k, stencil)


# ---- inputs ----------------------------------------------------------------


def _grid(case):
    """Offsets (sorted by the column they address), their validity per cell and the cells' coordinates."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    c = torch.arange(nx * ny * nz, device=DEV)
    return (c % nx, (c // nx) % ny, c // (nx * ny)), (nx, ny, nz)


def _inside(xyz, dims, off):
    ok = None
    for q, d, o in zip(xyz, dims, off):
        if o:
            t = (q + o >= 0) & (q + o < d)
            ok = t if ok is None else ok & t
    return torch.ones_like(xyz[0], dtype=torch.bool) if ok is None else ok


def _lin(dims, off):
    return off[0] + dims[0] * (off[1] + dims[1] * off[2])


def _stencil(case):
    xyz, dims = _grid(case)
    offs = stencil_offsets(case["stencil"])
    return xyz, dims, offs, torch.stack([_inside(xyz, dims, o) for o in offs], 1)


def _values(case, seed):
    """A's blocks as a dense (cells, offsets, b, b) array [.., r, c] (zero where there is no neighbour), the
    validity mask and the right-hand side."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    b = case["b"]
    xyz, dims, offs, ok = _stencil(case)
    n = xyz[0].numel()
    K = torch.exp(SIGMA * torch.randn(n, generator=g, device=DEV, dtype=F64))
    A = torch.rand((n, len(offs), b, b), generator=g, device=DEV, dtype=F64)
    A.mul_(0.2).sub_(0.1)
    A += torch.eye(b, device=DEV, dtype=F64)  # I + 0.1 R
    cell = torch.arange(n, device=DEV)
    mid = offs.index((0, 0, 0))
    total = torch.zeros(n, device=DEV, dtype=F64)
    for q, o in enumerate(offs):
        if q == mid:
            continue
        kd = K[(cell + _lin(dims, o)).clamp(0, n - 1)]
        T = torch.where(ok[:, q], 2 * K * kd / (K + kd), 0.0)
        total += T
        A[:, q].mul_(-T[:, None, None])
    A[:, mid].mul_(ACCUM)
    A[:, mid] += total[:, None, None] * torch.eye(b, device=DEV, dtype=F64)
    rhs = torch.rand(n * b, generator=g, device=DEV, dtype=F64) * 2 - 1
    return A, ok, rhs


def _flat(blocks):
    """Blocks [.., r, c] as the library stores them: column by column, one after another."""
    return blocks.transpose(-1, -2).contiguous().view(-1)


def _system(case, seed):
    A, ok, rhs = _values(case, seed)
    rp, ci = grid_pattern(case["nx"], case["ny"], case["nz"], case["stencil"])
    return rp, ci, _flat(A[ok]), rhs


def prepare(case, seed):
    op, b, k = case["op"], case["b"], case["k"]
    n = case["nx"] * case["ny"] * case["nz"]
    rp, ci, vals, rhs = _system(case, seed)
    s = {"op": op, "n": n, "b": b, "k": k, "rhs": rhs, "vals": vals}
    if op == "setup":
        return {**s, "rp": rp, "ci": ci}
    if op == "grad":
        s["solver"] = BlockILUSolver(n, b, rp, ci, k, tol=TOL, maxit=MAXIT)
        s["solver"].transposed()
        g = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
        s["weight"] = torch.rand(n * b, generator=g, device=DEV, dtype=F64) + 0.5
        return s
    if op.startswith("spmv"):
        s["rp"], s["ci"] = (torch.from_numpy(a).to(DEV) for a in (rp, ci))
        if op != "spmv":
            s["vals"] = B.bilu_convert_f32(vals)
        if op == "spmv_f32x":
            s["rhs"] = rhs.float()
        return s
    s["P"] = B.bilu_symbolic_gpu(n, rp, ci, k, row_capacity=256).upload()
    if op == "factor":
        s["work"] = B.workspace(s["P"].factor_workspace_bytes(b))
        s["F"] = B.new_factors(s["P"], b)
        return s
    if op == "factor_f32":
        s["work"] = B.workspace(s["P"].factor_workspace_bytes(b))
        return s
    if op == "apply_f32":
        # single-precision factors a program keeps: the same bits whatever computed them
        s["F"] = _factors(case, seed).float()
    else:
        s["F"], _ = B.bilu_factor(s["P"], b, vals)
    if op in ("apply", "apply_f32"):
        s["work"] = B.workspace(s["P"].apply_workspace_bytes(b))
        s["x"] = torch.empty_like(rhs)
        del s["vals"]
        return s
    s["A"] = (n, b, *(torch.from_numpy(a).to(DEV) for a in (rp, ci)), vals)
    if op in ("solve_f32prec", "solve_mixed"):
        s["F"] = B.bilu_convert_f32(s["F"])
    if op == "solve_mixed":
        s["vals32"] = B.bilu_convert_f32(vals)
        s["work"] = B.workspace(s["P"].bicgstab_mixed_workspace_bytes(b))
    elif op != "gmres":
        s["work"] = B.workspace(s["P"].bicgstab_workspace_bytes(b))
    return s


def run(s):
    op, b, P = s["op"], s["b"], s.get("P")
    if op == "apply":
        return B.bilu_apply(P, b, s["F"], s["rhs"], x=s["x"], work=s["work"])
    if op == "apply_f32":
        return B.bilu_apply_f32(P, b, s["F"], s["rhs"], x=s["x"], work=s["work"])
    if op == "factor":
        return B.bilu_factor(P, b, s["vals"], factors=s["F"], work=s["work"])[0]
    if op == "factor_f32":
        return B.bilu_factor_f32(P, b, s["vals"], work=s["work"])[0]
    if op == "spmv":
        return B.bsr_spmv(s["n"], b, s["rp"], s["ci"], s["vals"], s["rhs"])
    if op == "spmv_f32":
        return B.bsr_spmv_f32(s["n"], b, s["rp"], s["ci"], s["vals"], s["rhs"])
    if op == "spmv_f32x":
        return B.bsr_spmv_f32x(s["n"], b, s["rp"], s["ci"], s["vals"], s["rhs"])
    if op == "setup":
        new = B.bilu_symbolic_gpu(s["n"], s["rp"], s["ci"], s["k"]).upload()
        return B.bilu_factor(new, b, s["vals"])[0]
    if op == "solve":
        return B.bicgstab_solve(P, s["A"], s["F"], s["rhs"], tol=TOL, maxit=MAXIT, work=s["work"])[0]
    if op == "solve_f32prec":
        return B.bicgstab_solve_f32prec(P, s["A"], s["F"], s["rhs"], tol=TOL, maxit=MAXIT, work=s["work"])[0]
    if op == "solve_mixed":
        return B.bicgstab_solve_mixed(P, s["A"], s["vals32"], s["F"], s["rhs"], tol=TOL, maxit=MAXIT,
                                      work=s["work"])[0]
    if op == "gmres":
        return B.gmres_solve(P, s["A"], s["F"], s["rhs"], tol=TOL, maxit=MAXIT)[0]
    if op == "grad":
        v = s["vals"].detach().requires_grad_(True)
        r = s["rhs"].detach().requires_grad_(True)
        x = s["solver"].solve(v, r)
        gv, gr = torch.autograd.grad(((s["weight"] * x) ** 2).sum(), (v, r))
        return {"x": x.detach(), "grad_vals": gv, "grad_rhs": gr}
    raise ValueError(op)


def _counts(case):
    """(blocks of A, strictly lower blocks of P', strictly upper blocks of P'), from the interior row's fill."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    a = sum(max(0, nx - abs(o[0])) * max(0, ny - abs(o[1])) * max(0, nz - abs(o[2]))
            for o in stencil_offsets(case["stencil"]))
    if case["op"].startswith("spmv"):
        return a, 0, 0
    low = sum(max(0, nx - abs(o[0])) * max(0, ny - abs(o[1])) * max(0, nz - abs(o[2]))
              for o in _fill_offsets(case)[0])
    return a, low, low


def _fill_offsets(case):
    """Offsets of an interior row's strictly lower and strictly upper blocks of P' (fill-path theorem: (i, j) is
    kept at level k iff a path of at most k + 1 stencil steps leads from i to j through cells numbered below both),
    in ascending column order, and the paths to each."""
    dims = (case["nx"], case["ny"], case["nz"])
    steps = [o for o in stencil_offsets(case["stencil"]) if o != (0, 0, 0)]
    paths = {}
    # partial paths through cells numbered below the start: [offset, cells passed]
    partial = [((0, 0, 0), ())]
    for _ in range(case["k"] + 1):
        longer = []
        for at, via in partial:
            for st in steps:
                to = tuple(p + q for p, q in zip(at, st))
                if to == (0, 0, 0) or any(abs(t) >= d for t, d in zip(to, dims)):
                    continue
                end = _lin(dims, to)
                if all(_lin(dims, v) < min(0, end) for v in via):
                    paths.setdefault(to, set()).add(via)
                if end < 0:
                    longer.append((to, via + (to,)))
        partial = longer
    offs = sorted(paths, key=lambda o: _lin(dims, o))
    return [o for o in offs if _lin(dims, o) < 0], [o for o in offs if _lin(dims, o) > 0], paths


def work(case):
    op, b, n = case["op"], case["b"], case["nx"] * case["ny"] * case["nz"]
    a, low, up = _counts(case)
    bb = b * b
    pat, vec = 4 * (n + 1), 8 * n * b
    mat = a * (8 * bb + 4) + pat
    fac = (low + up) * (8 * bb + 4) + 8 * n * bb + 2 * pat
    fac32 = fac - 4 * (low + up + n) * bb
    flops_apply, flops_spmv = 2 * bb * (low + up + n), 2 * bb * a
    # per row and pivot: one b x b product, and one for each block of the pivot's upper row that is kept (about half)
    flops_factor = 2 * b * bb * low * (1 + (up / max(n, 1)) / 2) + 2 * b * bb * (n + up)
    moved, flops = {
        "apply": (fac + 2 * vec, flops_apply),
        "apply_f32": (fac32 + 2 * vec, flops_apply),
        "factor": (mat + fac, flops_factor),
        "factor_f32": (mat + fac32, flops_factor),
        "setup": (mat + fac, flops_factor),
        "spmv": (mat + 2 * vec, flops_spmv),
        "spmv_f32": (mat - 4 * bb * a + 2 * vec, flops_spmv),
        "spmv_f32x": (mat - 4 * bb * a + vec + vec // 2, flops_spmv),
        "solve": (mat + fac + 2 * vec, 2 * (flops_apply + flops_spmv)),
        "solve_f32prec": (mat + fac32 + 2 * vec, 2 * (flops_apply + flops_spmv)),
        "solve_mixed": (mat + fac32 + 2 * vec, 2 * (flops_apply + flops_spmv)),
        "gmres": (mat + fac + 2 * vec, flops_apply + flops_spmv),
        "grad": (2 * (mat + fac) + 8 * bb * a + 4 * vec, 4 * (flops_apply + flops_spmv) + flops_factor),
    }[op]
    return {"bytes": moved, "flops": flops}


# ---- the same in plain FP64 ------------------------------------------------


class _Ilu:
    """ILU(k) of a case's matrix by slots: block (cell, cell + offset) of every cell at once, zero where there is none."""

    def __init__(self, case, A, ok):
        b = case["b"]
        xyz, dims = _grid(case)
        n = xyz[0].numel()
        self.n, self.b = n, b
        self.low, self.up, paths = _fill_offsets(case)
        inside = {}

        def there(o):
            if o not in inside:
                inside[o] = _inside(xyz, dims, o)
            return inside[o]

        def mask(o):
            m = torch.zeros(n, dtype=torch.bool, device=DEV)
            for via in paths[o]:
                t = there(o)
                for v in via:
                    t = t & there(v)
                m |= t
            return m

        self.cell = torch.arange(n, device=DEV)
        self.lin = {o: _lin(dims, o) for o in self.low + self.up}
        self.m = {o: mask(o) for o in self.low + self.up}
        stencil = {o: q for q, o in enumerate(stencil_offsets(case["stencil"]))}
        zero = lambda: torch.zeros((n, b, b), device=DEV, dtype=F64)  # noqa: E731
        self.F = {o: (A[:, stencil[o]] * ok[:, stencil[o], None, None]) if o in stencil else zero()
                  for o in self.low + self.up}
        self.D = A[:, stencil[(0, 0, 0)]].clone()
        self._factor()

    def _levels(self, offs):
        lvl = torch.zeros(self.n, dtype=torch.int32, device=DEV)
        if not offs:
            return [self.cell]
        at = [(self.cell + self.lin[o]).clamp(0, self.n - 1) for o in offs]
        while True:
            old = lvl
            for _ in range(16):
                for o, p in zip(offs, at):
                    lvl = torch.maximum(lvl, torch.where(self.m[o], lvl[p] + 1, 0))
            if torch.equal(old, lvl):
                break
        order = torch.argsort(lvl, stable=True)
        return list(torch.split(order, torch.bincount(lvl).tolist()))

    def _factor(self):
        self.inv = torch.zeros_like(self.D)
        self.levels = self._levels(self.low)
        zero = (0, 0, 0)
        for I in self.levels:
            for s in self.low:
                p = (I + self.lin[s]).clamp(0, self.n - 1)
                lip = self.F[s][I] @ self.inv[p]
                self.F[s][I] = lip
                for u in self.up:
                    t = tuple(x + y for x, y in zip(s, u))
                    if t == zero:
                        self.D[I] -= lip @ self.F[u][p]
                    elif t in self.F:
                        self.F[t][I] -= (lip @ self.F[u][p]) * self.m[t][I][:, None, None]
            self.inv[I] = torch.linalg.inv_ex(self.D[I])[0]
        for u in self.up:
            self.F[u] = self.inv @ self.F[u]

    def flat(self):
        """The factors in the library's order: L, D^{-1}, U', rows and columns ascending."""
        def part(offs):
            if not offs:
                return torch.zeros(0, device=DEV, dtype=F64)
            return _flat(torch.stack([self.F[o] for o in offs], 1)[torch.stack([self.m[o] for o in offs], 1)])
        return torch.cat([part(self.low), _flat(self.inv), part(self.up)])

    def apply(self, r):
        x = r.view(self.n, self.b).clone()
        for offs, levels in ((self.low, self.levels), (self.up, self._levels(self.up))):
            for I in levels:
                for o in offs:
                    p = (I + self.lin[o]).clamp(0, self.n - 1)
                    x[I] -= (self.F[o][I] @ x[p].unsqueeze(-1)).squeeze(-1)
            if offs is self.low:
                x = (self.inv @ x.unsqueeze(-1)).squeeze(-1)
        return x.reshape(-1)

    def rounded(self):
        self.F = {o: f.float().double() for o, f in self.F.items()}
        self.inv = self.inv.float().double()
        return self


def _factors(case, seed):
    A, ok, _ = _values(case, seed)
    return _Ilu(case, A, ok).flat()


class _Plain:
    """A by slots: products with it, and solutions by a block-Jacobi BiCGSTAB restarted from the true residual."""

    def __init__(self, case, A, ok):
        _, dims, offs, _ = _stencil(case)
        n, b = A.shape[0], case["b"]
        cell = torch.arange(n, device=DEV)
        self.at = torch.stack([(cell + _lin(dims, o)).clamp(0, n - 1) for o in offs], 1)
        self.n, self.b, self.ok = n, b, ok
        A = A * ok[:, :, None, None]
        self.rows = A.permute(0, 2, 1, 3).reshape(n, b, -1).contiguous()
        self.inv = torch.linalg.inv(A[:, offs.index((0, 0, 0))])
        back = [offs.index(tuple(-x for x in o)) for o in offs]
        self.T = lambda: _Plain(case, torch.stack(
            [A[self.at[:, q], back[q]].transpose(-1, -2) for q in range(len(offs))], 1), ok)

    def mul(self, x):
        return (self.rows * x.view(self.n, self.b)[self.at].reshape(self.n, 1, -1)).sum(-1).view(-1)

    def solve(self, rhs):
        pre = lambda v: (self.inv * v.view(self.n, 1, self.b)).sum(-1).view(-1)  # noqa: E731
        x, goal, best = torch.zeros_like(rhs), 1e-15 * rhs.norm(), math.inf
        for _ in range(12):
            r = rhs - self.mul(x)
            now = float(r.norm())
            if now <= goal or now > 0.5 * best:
                break
            best, rh = now, r
            d, rho, alpha, omega = torch.zeros_like(x), 1.0, 1.0, 1.0
            v = p = torch.zeros_like(x)
            least, keep = torch.dot(r, r), d
            for it in range(2000):
                rho, last = torch.dot(rh, r), rho
                p = r + (rho / last) * (alpha / omega) * (p - omega * v)
                ph = pre(p)
                v = self.mul(ph)
                alpha = rho / torch.dot(rh, v)
                q = r - alpha * v
                sh = pre(q)
                t = self.mul(sh)
                omega = torch.dot(t, q) / torch.dot(t, t)
                d = d + alpha * ph + omega * sh
                r = q - omega * t
                rr = torch.dot(r, r)
                keep = torch.where(rr < least, d, keep)
                least = torch.minimum(rr, least)
                if it % 20 == 19 and not float(rr) > (1e-9 * now) ** 2:
                    break
            x = x + keep
        return x


def exact(case, seed):
    op, b = case["op"], case["b"]
    if not op.startswith("spmv") and op in ("apply", "factor", "factor_f32", "setup", "apply_f32"):
        low, up, _ = _fill_offsets(case)
        if len(low) > 12:
            return None  # thousands of products on each level: minutes
    A, ok, rhs = _values(case, seed)
    if op.startswith("spmv"):
        if op != "spmv":
            A = A.float().double()
        return _Plain(case, A, ok).mul(rhs.float().double() if op == "spmv_f32x" else rhs)
    if op in ("factor", "factor_f32", "setup"):
        return _Ilu(case, A, ok).flat()
    if op == "apply":
        return _Ilu(case, A, ok).apply(rhs)
    if op == "apply_f32":
        return _Ilu(case, A, ok).rounded().apply(rhs)
    M = _Plain(case, A, ok)
    x = M.solve(rhs)
    if op != "grad":
        return x
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
    w = torch.rand(x.numel(), generator=g, device=DEV, dtype=F64) + 0.5
    lam = M.T().solve(2 * w * w * x)
    L, X = lam.view(-1, b), x.view(-1, b)
    outer = -(L[:, None, :, None] * X[M.at][:, :, None, :])
    return {"x": x, "grad_vals": _flat(outer[ok]), "grad_rhs": lam}
