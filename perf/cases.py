"""Workloads of this library as its users run them, each through the public
entry points (``native.Solver``, ``native.BatchSolver``, ``adjoint.sparse_solve``).

Two kinds of solve are used. A *budgeted* solve runs 20 iterations of a steady
convection-diffusion system and returns the iterate with its residual history:
the solver as a smoother or an inner step, and the form in which two correct
implementations can be compared number by number (past a few dozen iterations
BiCGStab on these systems amplifies any change of rounding). A *converged*
solve runs to its tolerance on a system where the number of iterations does
not hang on the rounding: an implicit time step (the operator plus ``sigma``
on the diagonal) or a diagonally dominant random matrix. Its right-hand side
is A x* with a known x*, so x* is the exact answer.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1612_01395_gb300 import adjoint, native, problems

BUDGET = 20   # iterations of a budgeted solve


def listed():
    return [
        # The smallest calls: a 2-D steady system of 4096 unknowns in CSR form, solved to full
        # accuracy (a coarse problem, or one of many in an outer loop): latency and launches count.
        dict(name="small_2d_csr", kind="solve", form="csr", method="pipelined", nx=64, ny=64, nz=1, sigma=0.0,
             rtol=1e-10, budget=0, replace=50, its=121),
        # The same in 3-D with odd sides, stencil form, by standard BiCGStab.
        dict(name="small_3d_standard", kind="solve", form="stencil", method="standard", nx=17, ny=15, nz=13,
             sigma=0.0, rtol=1e-10, budget=0, replace=0, its=43),
        # Ordinary 2-D work: 52 k unknowns, 5-point CSR rows, with residual replacement.
        dict(name="mid_2d_csr", kind="solve", form="csr", method="pipelined", nx=301, ny=173, nz=1, sigma=0.0,
             rtol=0.0, budget=BUDGET, replace=10, its=BUDGET),
        # Ordinary 3-D work on a ragged grid: 491 k unknowns, matrix-free.
        dict(name="mid_3d_stencil", kind="solve", form="stencil", method="pipelined", nx=97, ny=83, nz=61, sigma=0.0,
             rtol=0.0, budget=BUDGET, replace=0, its=BUDGET),
        # The benchmark's system (16.7 M unknowns) in stencil form, by both methods.
        dict(name="large_3d_stencil", kind="solve", form="stencil", method="pipelined", nx=256, ny=256, nz=256,
             sigma=0.0, rtol=0.0, budget=BUDGET, replace=50, its=BUDGET),
        dict(name="large_3d_standard", kind="solve", form="stencil", method="standard", nx=256, ny=256, nz=256,
             sigma=0.25, rtol=1e-8, budget=0, replace=0, its=43),
        # The benchmark's system as an assembled matrix: one implicit time step to 1e-8.
        dict(name="large_3d_csr", kind="solve", form="csr", method="pipelined", nx=256, ny=256, nz=256, sigma=0.25,
             rtol=1e-8, budget=0, replace=50, its=44),
        # Jacobi-preconditioned solve of an unstructured system whose rows differ in scale.
        dict(name="jacobi_random_csr", kind="jacobi", n=200003, row_lo=8, row_hi=32, rtol=1e-10, its=10),
        # Mixed precision to a true residual of 1e-10, matrix-free and assembled (FP32 values).
        dict(name="mixed_3d_stencil", kind="mixed", form="stencil", values="f32", nx=192, ny=192, nz=192, sigma=0.25,
             rtol=1e-10, its=66),
        dict(name="mixed_3d_csr", kind="mixed", form="csr", values="f32", nx=193, ny=160, nz=131, sigma=0.25,
             rtol=1e-10, its=66),
        # The batch of the benchmark: 512 random systems of 1 k to 64 k unknowns in one launch.
        dict(name="batched_512", kind="batched", nsys=512, nmin=1000, nmax=64000, row_lo=8, row_hi=32, rtol=1e-8,
             its=21),
        # Forward and backward through a differentiable solve: 1024^2, a velocity per cell.
        dict(name="adjoint_2d", kind="adjoint", nx=1024, ny=1024, sigma=0.25, rtol=1e-12, its=65),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, dim, lo, hi):
    """Sides of a grid of about log-uniform(lo, hi) points, each side off the mean by up to 30 %."""
    side = _log(rng, lo, hi) ** (1.0 / dim)
    s = [max(3, int(side * math.exp(rng.uniform(-0.3, 0.3)))) for _ in range(dim)]
    while s[0] * s[1] * (s[2] if dim == 3 else 1) > hi:
        s = [max(3, int(0.95 * v)) for v in s]
    return s[0], s[1], s[2] if dim == 3 else 1


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "jacobi", "mixed", "batched", "adjoint"])
    if kind == "solve":
        nx, ny, nz = _grid(rng, rng.choice([2, 3]), 1000, 14000000)
        method = rng.choice(["pipelined", "pipelined", "standard"])
        steady = rng.random() < 0.5
        return dict(kind=kind, form=rng.choice(["csr", "stencil"]), method=method, nx=nx, ny=ny, nz=nz,
                    sigma=0.0 if steady else 0.25, rtol=0.0 if steady else 1e-8, budget=BUDGET if steady else 0,
                    replace=rng.choice([0, 10, 50]) if method == "pipelined" else 0, its=BUDGET if steady else 43)
    if kind == "jacobi":
        lo = rng.randint(3, 12)
        return dict(kind=kind, n=_log(rng, 2000, 500000), row_lo=lo, row_hi=rng.randint(lo, 32), rtol=1e-10, its=12)
    if kind == "mixed":
        nx, ny, nz = _grid(rng, 3, 8000, 7077888)
        form = rng.choice(["csr", "stencil"])
        return dict(kind=kind, form=form, values="f32" if form == "stencil" else rng.choice(["f32", "bf16"]), nx=nx,
                    ny=ny, nz=nz, sigma=0.25, rtol=1e-10, its=66)
    if kind == "batched":
        lo, small = rng.randint(4, 12), _log(rng, 300, 4000)
        return dict(kind=kind, nsys=_log(rng, 16, 320), nmin=small, nmax=_log(rng, 4 * small, 64000), row_lo=lo,
                    row_hi=rng.randint(lo, 32), rtol=1e-8, its=24)
    nx, ny, _ = _grid(rng, 2, 4096, 1048576)
    return dict(kind=kind, nx=nx, ny=ny, sigma=0.25, rtol=1e-12, its=65)


# ---- inputs, made on the GPU from the seed alone -------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) + 1))
    return g


def _uniform(g, n):
    return 2.0 * torch.rand(n, dtype=torch.float64, device="cuda", generator=g) - 1.0


def _stencil(nx, ny, nz, sigma):
    """First-order upwind convection-diffusion scaled by h^2 (velocity 10, 10 in 2-D; 20 sin y,
    20 cos z, 20 sin x in 3-D), plus sigma on the diagonal."""
    h = 1.0 / (max(nx, ny, nz) + 1)
    at = lambda m: (np.arange(m) + 1) * h   # noqa: E731
    lower = lambda c: -1.0 - h * np.maximum(c, 0.0)   # noqa: E731
    upper = lambda c: -1.0 - h * np.maximum(-c, 0.0)   # noqa: E731
    size = lambda c: 2.0 + h * np.abs(c)   # noqa: E731
    c = [problems.Coef(value=0.0) for _ in range(7)]
    if nz == 1:
        cx, cy = np.full(ny, 10.0), np.full(nx, 10.0)
        c[problems.C] = problems.Coef(table=size(cx) + sigma, stride=(0, 1, 0), table2=size(cy), stride2=(1, 0, 0))
        along_s, stride_s = cy, (1, 0, 0)
    else:
        cx, cy, cz = 20.0 * np.sin(at(ny)), 20.0 * np.cos(at(nz)), 20.0 * np.sin(at(nx))
        plane = (size(cy)[:, None] + size(cx)[None, :] + sigma).ravel()   # index j + ny k
        c[problems.C] = problems.Coef(table=plane, stride=(0, 1, ny), table2=size(cz), stride2=(1, 0, 0))
        c[problems.B] = problems.Coef(table=lower(cz), stride=(1, 0, 0))
        c[problems.T] = problems.Coef(table=upper(cz), stride=(1, 0, 0))
        along_s, stride_s = cy, (0, 0, 1)
    c[problems.W] = problems.Coef(table=lower(cx), stride=(0, 1, 0))
    c[problems.E] = problems.Coef(table=upper(cx), stride=(0, 1, 0))
    c[problems.S] = problems.Coef(table=lower(along_s), stride=stride_s)
    c[problems.N] = problems.Coef(table=upper(along_s), stride=stride_s)
    return problems.Stencil(nx=nx, ny=ny, nz=nz, coefs=c)


def _on_grid(coef, nx, ny, nz):
    """A coefficient as a (nz, ny, nx) view on the device."""
    def view(table, stride):
        t = torch.as_tensor(table, dtype=torch.float64, device="cuda")
        return torch.as_strided(t, (nz, ny, nx), (stride[2], stride[1], stride[0]))
    if coef.table is None:
        return torch.full((1, 1, 1), coef.value, dtype=torch.float64, device="cuda").expand(nz, ny, nx)
    v = view(coef.table, coef.stride)
    return v if coef.table2 is None else v + view(coef.table2, coef.stride2)


def _apply(fields, shape, u):
    """y = A u by slices."""
    nx, ny, nz = shape
    u = u.reshape(nz, ny, nx)
    y = fields[problems.C] * u
    for d, axis, step in ((problems.W, 2, -1), (problems.E, 2, 1), (problems.S, 1, -1), (problems.N, 1, 1),
                          (problems.B, 0, -1), (problems.T, 0, 1)):
        m = u.shape[axis]
        if m < 2:
            continue
        to, frm = (1, 0) if step < 0 else (0, 1)
        y.narrow(axis, to, m - 1).addcmul_(fields[d].narrow(axis, to, m - 1), u.narrow(axis, frm, m - 1))
    return y.reshape(-1)


def _assemble(fields, shape):
    """The stencil as CSR arrays on the device, columns ascending."""
    nx, ny, nz = shape
    n = nx * ny * nz
    i = torch.arange(nx, device="cuda").view(1, 1, nx)
    j = torch.arange(ny, device="cuda").view(1, ny, 1)
    k = torch.arange(nz, device="cuda").view(nz, 1, 1)
    masks = []
    for d in problems.CSR_ORDER:
        di, dj, dk = problems.OFFSETS[d]
        m = ((i + di >= 0) & (i + di < nx)) & ((j + dj >= 0) & (j + dj < ny)) & ((k + dk >= 0) & (k + dk < nz))
        masks.append((d, di + nx * (dj + ny * dk), m.reshape(-1)))
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(sum(m.to(torch.int32) for _, _, m in masks), 0, out=rowptr[1:])
    nnz = int(rowptr[-1])
    col = torch.empty(nnz, dtype=torch.int32, device="cuda")
    val = torch.empty(nnz, dtype=torch.float64, device="cuda")
    pos = rowptr[:-1].clone()
    rows = torch.arange(n, dtype=torch.int32, device="cuda")
    for d, off, m in masks:
        p = pos[m]
        col[p] = rows[m] + off
        val[p] = fields[d].reshape(-1)[m]
        pos += m
    return SimpleNamespace(n=n, nnz=nnz, rowptr=rowptr.to(torch.int32), col=col, val=val)


def _random_rows(g, offsets, row_lo, row_hi):
    """Random systems one after another (rows offsets[s]..offsets[s+1] are system s): row_lo to row_hi
    N(0, 1) entries a row at uniform columns, the diagonal 1.1 times their absolute sum; columns local
    to the system and ascending. Returns rowptr (int64), row of each entry, col, val."""
    total = int(offsets[-1])
    first = torch.as_tensor(offsets, device="cuda")
    sizes = first[1:] - first[:-1]
    system = torch.repeat_interleave(torch.arange(len(offsets) - 1, device="cuda"), sizes)
    counts = torch.randint(row_lo, row_hi + 1, (total,), device="cuda", generator=g)
    rows = torch.repeat_interleave(torch.arange(total, device="cuda"), counts)
    m = rows.numel()
    n_of, local = sizes[system], torch.arange(total, device="cuda") - first[:-1][system]
    u = torch.rand(m, dtype=torch.float64, device="cuda", generator=g)
    cols = (u * (n_of[rows] - 1)).to(torch.int64)
    del u
    cols += cols >= local[rows]
    vals = torch.randn(m, dtype=torch.float64, device="cuda", generator=g)
    diag = 1.1 * torch.zeros(total, dtype=torch.float64, device="cuda").index_add_(0, rows, vals.abs())
    key = torch.cat([rows * 2 ** 20 + cols, torch.arange(total, device="cuda") * 2 ** 20 + local])
    del rows, cols
    key, order = torch.sort(key)
    val = torch.cat([vals, diag])[order]
    del vals, order
    rowptr = torch.zeros(total + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(counts + 1, 0, out=rowptr[1:])
    return rowptr, key >> 20, (key & (2 ** 20 - 1)).to(torch.int32), val, first[:-1][system]


def _sizes(case):
    """Sizes of a batch: log-uniform between nmin and nmax, largest first."""
    f = (np.arange(case["nsys"]) + 0.5) / case["nsys"]
    return np.rint(case["nmin"] * (case["nmax"] / case["nmin"]) ** f).astype(np.int64)[::-1].copy()


def _problem(case, seed):
    """The system of a grid case and its known solution: (stencil, fields, shape, x*, b)."""
    shape = (case["nx"], case["ny"], case.get("nz", 1))
    st = _stencil(*shape, case["sigma"])
    fields = [_on_grid(c, *shape) for c in st.coefs]
    xs = _uniform(_generator(seed), st.n)
    return st, fields, shape, xs, _apply(fields, shape, xs)


def _cell_problem(case, seed):
    """The adjoint's system: a velocity c ~ U[0, 50] per cell in both directions. Returns its fields,
    shape, x*, b, the adjoint solution lambda* and the gradient A^T lambda* that it belongs to."""
    shape = (case["nx"], case["ny"], 1)
    n = shape[0] * shape[1]
    g = _generator(seed)
    h = 1.0 / (max(shape) + 1)
    hc = (25.0 * h * (_uniform(g, n) + 1.0)).reshape(1, shape[1], shape[0])
    one, none = torch.full_like(hc, -1.0), torch.zeros_like(hc)
    fields = [None] * 7
    fields[problems.C] = 4.0 + 2.0 * hc + case["sigma"]
    fields[problems.W] = fields[problems.S] = -1.0 - hc
    fields[problems.E] = fields[problems.N] = one
    fields[problems.B] = fields[problems.T] = none
    xs, lam = _uniform(g, n), _uniform(g, n)
    # A^T has the mirrored entries: its west entry at a cell is A's east entry at the west neighbour
    roll = lambda f, axis, by: torch.roll(f, by, axis)   # noqa: E731
    ft = [fields[problems.C], roll(fields[problems.E], 2, 1), roll(fields[problems.W], 2, -1),
          roll(fields[problems.N], 1, 1), roll(fields[problems.S], 1, -1), none, none]
    return fields, shape, xs, _apply(fields, shape, xs), lam, _apply(ft, shape, lam)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "mixed"):
        st, fields, shape, _, b = _problem(case, seed)
        low = None
        if case["form"] == "csr":
            A = _assemble(fields, shape)
            solver = native.Solver.from_csr(A)
            if kind == "mixed":
                low = A.val.to(torch.float32 if case["values"] == "f32" else torch.bfloat16)
        else:
            solver = native.Solver.from_stencil(st)
        return dict(case=case, solver=solver, b=b, low=low)
    if kind == "jacobi":
        A, _, b = _jacobi_problem(case, seed)
        return dict(case=case, solver=native.Solver.from_csr(A, prec=native.PBCG_PREC_JACOBI), b=b)
    if kind == "batched":
        batch, _, b = _batch_problem(case, seed)
        return dict(case=case, solver=native.BatchSolver(batch), b=b)
    fields, shape, xs, b, _, gx = _cell_problem(case, seed)
    A = _assemble(fields, shape)
    return dict(case=case, structure=adjoint.CSRStructure(A.rowptr, A.col), values=A.val.requires_grad_(),
                b=b.requires_grad_(), target=xs - gx)


def _jacobi_problem(case, seed):
    g = _generator(seed)
    n = case["n"]
    rowptr, rows, col, val, _ = _random_rows(g, np.array([0, n]), case["row_lo"], case["row_hi"])
    val *= (10.0 ** _uniform(g, n))[rows]   # rows scaled by 0.1 to 10
    xs = _uniform(g, n)
    b = torch.zeros_like(xs).index_add_(0, rows, val * xs[col.long()])
    return SimpleNamespace(n=n, nnz=val.numel(), rowptr=rowptr.to(torch.int32), col=col, val=val), xs, b


def _batch_problem(case, seed):
    g = _generator(seed)
    offsets = np.concatenate([[0], np.cumsum(_sizes(case))])
    rowptr, rows, col, val, first = _random_rows(g, offsets, case["row_lo"], case["row_hi"])
    xs = _uniform(g, int(offsets[-1]))
    b = torch.zeros_like(xs).index_add_(0, rows, val * xs[col + first[rows]])
    batch = SimpleNamespace(nsys=case["nsys"], total_rows=int(offsets[-1]), row_offset=torch.as_tensor(offsets),
                            rowptr=rowptr.to(torch.int32), col=col, val=val)
    return batch, xs, b


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        if case["budget"]:
            x, _, hist = state["solver"].solve(state["b"], rtol=0.0, maxit=case["budget"],
                                               replace_period=case["replace"], method=case["method"], history=True,
                                               fixed_iters=case["budget"])
            return x, hist
        return state["solver"].solve(state["b"], rtol=case["rtol"], maxit=2000, replace_period=case["replace"],
                                     method=case["method"])[0]
    if kind == "jacobi":
        return state["solver"].solve(state["b"], rtol=case["rtol"], maxit=2000, replace_period=50)[0]
    if kind == "mixed":
        low = native.PBCG_VALUES_BF16 if case["values"] == "bf16" else native.PBCG_VALUES_F32
        return state["solver"].solve_mixed(state["b"], state["low"], lowp_type=low, rtol=case["rtol"],
                                           inner_rtol=1e-4 if case["values"] == "f32" else 1e-2)[0]
    if kind == "batched":
        x = torch.zeros_like(state["b"])
        state["solver"].launch(state["b"], x, rtol=case["rtol"], maxit=1000, replace_period=50)
        return x
    x = adjoint.sparse_solve(state["values"], state["b"], state["structure"], rtol=case["rtol"])
    gv, gb = torch.autograd.grad(x, (state["values"], state["b"]), x.detach() - state["target"])
    return x.detach(), gv, gb


# ---- what a pass needs ---------------------------------------------------------------------------

ON_CHIP = 100e6   # bytes of vectors and matrix that stay on the chip from one iteration to the next


def work(case):
    """Operations: 2 per stored entry and product with A, 2 per recurrence and dot product term
    (Algorithm 9: 13 and 8 a row and iteration; Algorithm 7: 6 and 6), two products an iteration.
    Bytes: the vectors that the iteration's two (Algorithm 7: three) sweeps have to read and write
    (23 and 19) and the matrix for each product; a system that fits on the chip is read once."""
    kind, its = case["kind"], case["its"]
    if kind in ("solve", "mixed", "adjoint"):
        n = case["nx"] * case["ny"] * case.get("nz", 1)
        nnz = (5 if case.get("nz", 1) == 1 else 7) * n
    elif kind == "jacobi":
        n = case["n"]
        nnz = n * (1 + (case["row_lo"] + case["row_hi"]) / 2)
    else:
        n = int(_sizes(case).sum())
        nnz = n * (1 + (case["row_lo"] + case["row_hi"]) / 2)
    standard = case.get("method") == "standard"
    real = 4 if kind == "mixed" else 8
    stored = 0 if case.get("form") == "stencil" else nnz * (4 + (2 if case.get("values") == "bf16" else real)) + 4 * n
    vectors = (19 if standard else 24 if kind == "jacobi" else 23) * real * n
    flops = its * (4 * nnz + (24 if standard else 42) * n)
    resident = stored + (8 if standard else 12) * real * n
    system = resident if kind != "batched" else resident / case["nsys"]
    moved = its * (2 * stored + vectors) if system > ON_CHIP else stored + 3 * real * n
    scale = 2 if kind == "adjoint" else 1   # forward and backward
    return {"bytes": float(scale * moved), "flops": float(scale * flops)}


def tolerance(case):
    """Four times the distance seen to the same in 64 bits: of a budgeted solve's iterate and history
    (2.3e-10, where replacements amplify the rounding; 1e-13 elsewhere), and of a converged one's x to
    x*, which is what the stopping tolerance leaves (1.7e-7 at 1e-8, 2.5e-8 at 1e-10 on the worst
    conditioned system, 2e-11 for the refinement and 2.3e-11 for the adjoint, whose gradients multiply
    two solutions; smaller grids and coarser values up to ten times these)."""
    if case["kind"] == "solve" and case["budget"]:
        return {"rel": 1e-9}
    if case["kind"] in ("mixed", "adjoint"):
        return {"rel": 1e-9}
    return {"rel": 1e-7 if case["rtol"] <= 1e-10 else 1e-6}


# ---- the same in plain torch ---------------------------------------------------------------------

def _bicgstab(apply, b, its):
    """Standard BiCGStab from x0 = 0 in 64 bits; in exact arithmetic every form of the method, with or
    without residual replacement, has these iterates."""
    x, r = torch.zeros_like(b), b.clone()
    r0, p, rho, hist = r.clone(), r.clone(), torch.dot(r, r), [r.norm()]
    for _ in range(its):
        s = apply(p)
        alpha = rho / torch.dot(r0, s)
        q = r - alpha * s
        y = apply(q)
        omega = torch.dot(q, y) / torch.dot(y, y)
        x += alpha * p + omega * q
        r = q - omega * y
        hist.append(r.norm())
        rho, last = torch.dot(r0, r), rho
        p = r + (alpha / omega) * (rho / last) * (p - omega * s)
    return x, torch.stack(hist)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "mixed"):
        _, fields, shape, xs, b = _problem(case, seed)
        if kind == "solve" and case["budget"]:
            return _bicgstab(lambda u: _apply(fields, shape, u), b, case["budget"])
        return xs
    if kind == "jacobi":
        return _jacobi_problem(case, seed)[1]
    if kind == "batched":
        return _batch_problem(case, seed)[1]
    fields, shape, xs, _, lam, _ = _cell_problem(case, seed)
    A = _assemble(fields, shape)
    rows = torch.repeat_interleave(torch.arange(A.n, device="cuda"), (A.rowptr[1:] - A.rowptr[:-1]).long())
    return xs, -lam[rows] * xs[A.col.long()], lam
