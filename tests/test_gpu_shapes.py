"""The dispatch lines of the solvers (needs a GB300): the on-chip cluster, the
wide kernel above 700k rows, the FP32 groups of rows, and what their sums do
with zeros and non-finite values. Bars as in the parity tests: residual norms
within 1e-8 relative and x within 1e-9 of the FP64 oracle over the first
iterations; the transposes are compared exactly."""
import numpy as np
import pytest

import oracle
from paper_1612_01395_gb300 import native
from paper_1612_01395_gb300 import problems as P

pytestmark = pytest.mark.gpu
K = 10


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def grid_stencil(nx, ny, nz):
    """Upwind convection-diffusion on any nx x ny x nz grid."""
    c = [P.Coef(value=0.0) for _ in range(7)]
    c[P.C] = P.Coef(table=6.3 + 0.01 * np.arange(ny), stride=(0, 1, 0), table2=0.02 * np.arange(nx), stride2=(1, 0, 0))
    c[P.W], c[P.E] = P.Coef(value=-1.1), P.Coef(value=-0.9)
    c[P.S] = P.Coef(table=-1.0 - 0.001 * np.arange(nx), stride=(1, 0, 0))
    c[P.N] = P.Coef(value=-1.0)
    if nz > 1:
        c[P.B], c[P.T] = P.Coef(value=-1.05), P.Coef(value=-0.95)
    return P.Stencil(nx=nx, ny=ny, nz=nz, coefs=c)


def check(solver, A, b, method):
    ref = (oracle.pbicgstab if method == "pipelined" else oracle.bicgstab)(A, b, rtol=0.0, maxit=K, fixed_iters=K)
    x, info, hist = solver.solve(dev(b), rtol=0.0, maxit=K, fixed_iters=K, method=method, history=True)
    h = hist.cpu().numpy()
    assert np.max(np.abs(h - ref.hist[:K + 1]) / ref.hist[:K + 1]) <= 1e-8
    assert np.linalg.norm(x.cpu().numpy() - ref.x) <= 1e-9 * np.linalg.norm(ref.x)
    x2, _ = solver.solve(dev(b), rtol=0.0, maxit=K, fixed_iters=K, method=method)
    np.testing.assert_array_equal(x.cpu().numpy(), x2.cpu().numpy())
    return info


@pytest.mark.parametrize("method", ["pipelined", "standard"])
@pytest.mark.parametrize("form", ["csr", "stencil"])
@pytest.mark.parametrize("dims", [(7, 1, 1), (33, 1, 1), (5, 7, 3), (31, 33, 1), (64, 64, 1), (69, 71, 1), (15, 15, 15)])
def test_small_systems_on_chip(dims, form, method):
    """One row a CTA and less, ragged last CTAs, one and several rows a thread."""
    st = grid_stencil(*dims)
    A = P.stencil_to_csr(st)
    s = native.Solver.from_csr(A) if form == "csr" else native.Solver.from_stencil(st)
    b = oracle.spmv(A, P.splitmix64_uniform(7, A.n))
    if A.n > 100:
        assert check(s, A, b, method)["cluster"] > 0
    x, info = s.solve(dev(b), rtol=1e-12, maxit=400, method=method)
    assert info["status"] == native.PBCG_OK and info["cluster"] > 0
    assert np.linalg.norm(b - oracle.spmv(A, x.cpu().numpy())) <= 1e-11 * np.linalg.norm(b)
    s.close()


def test_on_chip_entries_that_do_not_fit_their_cta():
    """The first rows hold most of the entries: their CTA reads them from global memory."""
    n = 640
    a = np.eye(n) * 40.0
    a[:20] += np.where(np.arange(n) % 2 == 0, 0.01, -0.013)
    a[np.arange(1, n), np.arange(n - 1)] += -1.0
    A = P.dense_to_csr(a)
    assert A.nnz <= 24576
    s = native.Solver.from_csr(A)
    for method in ("pipelined", "standard"):
        x, info = s.solve(dev(A.to_dense() @ np.linspace(-1, 1, n)), rtol=1e-12, maxit=200, method=method)
        assert info["cluster"] > 0 and info["status"] == native.PBCG_OK
        assert np.max(np.abs(x.cpu().numpy() - np.linspace(-1, 1, n))) <= 1e-10
    s.close()


@pytest.mark.parametrize("method", ["pipelined", "standard"])
@pytest.mark.parametrize("prec", [native.PBCG_PREC_NONE, native.PBCG_PREC_JACOBI])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 256, 257, 1283])
def test_short_rows_and_pairs_of_rows_on_a_grid(n, prec, method):
    """Rows of 1 to 11 entries (averaging under 6) around the chunk of five, on
    one and two blocks: no, one, an odd and an even number of rows a thread."""
    a = np.zeros((n, n))
    for i in range(n):
        for k in range(1 + (7 * i) % 11 if i % 3 == 0 else 1 + i % 6):
            a[i, (i + k * k * 5) % n] = -0.1 - 0.01 * k
        a[i, i] = 3.0 + 0.001 * (i % 17)
    A = P.dense_to_csr(a)
    assert A.nnz <= 6 * n
    s = native.Solver.from_csr(A, prec=prec)
    b = oracle.spmv(A, P.splitmix64_uniform(3, n))
    for grid in (1, 2):
        x, info = s.solve(dev(b), rtol=1e-12, maxit=200, method=method, cluster=-1, grid=grid)
        assert info["status"] == native.PBCG_OK and info["cluster"] == 0
        # off-diagonal sums are at most 1.55, so |A^-1| <= 1 / 1.45 in the maximum norm;
        # 4: the true residual against the recursive one that ended the solve
        assert np.max(np.abs(x.cpu().numpy() - P.splitmix64_uniform(3, n))) <= 4 * 1e-12 * np.linalg.norm(b) / 1.45
    s.close()


@pytest.mark.parametrize("method", ["pipelined", "standard"])
@pytest.mark.parametrize("form", ["csr", "stencil"])
@pytest.mark.parametrize("dims", [(100, 100, 70), (83, 89, 95), (839, 837, 1)])
def test_wide_sums_above_their_line(dims, form, method):
    """700 000 rows (the last below the line), 701 765 and 702 243 ragged ones; the
    solution is zero on half of the grid, so products vanish and sums cancel."""
    st = grid_stencil(*dims)
    A = P.stencil_to_csr(st)
    x = P.splitmix64_uniform(3, A.n)
    x[: A.n // 2] = 0.0
    s = native.Solver.from_csr(A) if form == "csr" else native.Solver.from_stencil(st)
    info = check(s, A, oracle.spmv(A, x), method)
    assert info["block"] == (512 if A.n > 700000 else 256)
    s.close()


@pytest.fixture(scope="module")
def wide_reference():
    """The oracle's first iterations on a system of `dims`, once per method and options."""
    done = {}

    def get(dims, method, prec, replace):
        st = grid_stencil(*dims)
        if dims not in done:
            A = P.stencil_to_csr(st)
            x = P.splitmix64_uniform(3, A.n)
            x[: A.n // 2] = 0.0
            done[dims] = A, oracle.spmv(A, x)
        A, b = done[dims]
        key = dims, method, prec, replace
        if key not in done:
            args = dict(rtol=0.0, maxit=K, fixed_iters=K)
            if method == "pipelined":
                args["replace_period"] = replace
            run = getattr(oracle, ("p" if method == "pipelined" else "") + "bicgstab" + ("_prec" if prec else ""))
            done[key] = run(A, oracle.jacobi_minv(A), b, **args) if prec else run(A, b, **args)
        return st, A, b, done[key]
    return get


@pytest.mark.parametrize("method,replace", [("pipelined", 0), ("pipelined", 4), ("standard", 0)])
@pytest.mark.parametrize("prec", [native.PBCG_PREC_JACOBI, native.PBCG_PREC_NONE])
@pytest.mark.parametrize("form", ["csr", "stencil"])
@pytest.mark.parametrize("dims", [(83, 89, 95), (839, 837, 1)])
def test_wide_sums_of_preconditioned_and_replaced_iterations(wide_reference, dims, form, prec, method, replace):
    """Algorithms 10 and 11, and residual replacement, with the dot products in integers.
    The Jacobi 2-D system falls by 12 orders in these iterations, where the two methods'
    oracles differ by 1e-4 of the last norms: besides 1e-8 of itself, a norm may differ by
    1e-13 of the first, a few hundred roundings of vectors of that size."""
    st, A, b, ref = wide_reference(dims, method, prec, replace)
    s = native.Solver.from_csr(A, prec=prec) if form == "csr" else native.Solver.from_stencil(st, prec=prec)
    x, info, hist = s.solve(dev(b), rtol=0.0, maxit=K, fixed_iters=K, method=method, replace_period=replace, history=True)
    assert info["block"] == 512 and info["n_replacements"] == (K // replace if replace else 0)
    h = hist.cpu().numpy()
    assert np.all(np.abs(h - ref.hist[:K + 1]) <= 1e-8 * ref.hist[:K + 1] + 1e-13 * ref.hist[0])
    assert np.linalg.norm(x.cpu().numpy() - ref.x) <= 1e-9 * np.linalg.norm(ref.x)
    s.close()


def test_wide_sums_report_non_finite_values():
    st = grid_stencil(100, 100, 71)
    s = native.Solver.from_stencil(st)
    b = P.splitmix64_uniform(1, st.n)
    for bad in (np.nan, np.inf):
        b[12345] = bad
        for method in ("pipelined", "standard"):
            _, info = s.solve(dev(b), rtol=1e-8, maxit=20, method=method)
            assert info["status"] == native.PBCG_NONFINITE
    b[:] = 0.0
    x, info = s.solve(dev(b), rtol=1e-8, maxit=20)
    assert info["status"] == native.PBCG_OK and info["iters"] == 0 and not x.any()
    s.close()


@pytest.mark.parametrize("dims", [(8, 9, 1), (6, 5, 4), (7, 3, 5), (4, 4, 4), (1, 9, 3), (2, 2, 2), (64, 3, 2), (65, 5, 3),
                                  (66, 4, 5), (67, 3, 4)])
def test_fp32_groups_of_rows(dims):
    """x-lines of every length modulo 4, lines shorter than a group among them:
    the refinement reaches 1e-12 and repeats bit for bit."""
    st = grid_stencil(*dims)
    A = P.stencil_to_csr(st)
    b = oracle.spmv(A, P.splitmix64_uniform(2, A.n))
    s = native.Solver.from_stencil(st)
    x, info = s.solve_mixed(dev(b), None, rtol=1e-12, inner_rtol=1e-3)
    x2, _ = s.solve_mixed(dev(b), None, rtol=1e-12, inner_rtol=1e-3)
    assert info["status"] == native.PBCG_OK
    assert np.linalg.norm(b - oracle.spmv(A, x.cpu().numpy())) <= 1e-11 * np.linalg.norm(b)
    np.testing.assert_array_equal(x.cpu().numpy(), x2.cpu().numpy())
    s.close()


@pytest.mark.parametrize("bad", [np.nan, -np.inf, 1e300])
@pytest.mark.parametrize("dims", [(8, 9, 1), (5, 6, 4), (6, 5, 4), (7, 3, 5), (1, 9, 3), (64, 3, 2)])
def test_fp32_groups_drop_the_entries_outside_the_grid(dims, bad):
    """West and east entries at the ends of an x-line belong to no neighbour: what
    the tables (or, on lines of one node, the constants) hold there changes nothing."""
    nx = dims[0]
    out = {}
    for fill in (0.0, bad):
        st = grid_stencil(*dims)
        west, east = -1.1 - 0.01 * np.arange(nx), -0.9 + 0.01 * np.arange(nx)
        west[0] = east[-1] = fill
        st.coefs[P.W] = P.Coef(table=west, stride=(1, 0, 0))
        st.coefs[P.E] = P.Coef(table=east, stride=(1, 0, 0)) if nx > 1 else P.Coef(value=fill)
        s = native.Solver.from_stencil(st)
        x, info = s.solve_mixed(dev(P.splitmix64_uniform(4, st.n)), None, rtol=1e-12, inner_rtol=1e-3)
        assert info["status"] == native.PBCG_OK
        out[fill == 0.0] = x.cpu().numpy(), info["inner_iters"]
        s.close()
    np.testing.assert_array_equal(out[True][0], out[False][0])
    assert out[True][1] == out[False][1]


@pytest.mark.parametrize("dims", [(1, 9, 3), (1, 64, 50), (1, 1, 37), (1, 30, 1), (1, 203, 301)])
def test_fp32_sweeps_of_x_lines_of_one_node(dims):
    """The same system, bit for bit, as on the grid without that axis."""
    out = []
    for drop in range(2 if dims[1] > 1 else 3):
        nx, ny, nz = (dims + (1, 1))[drop:drop + 3]
        along = {1: (0, 1, 0), 2: (0, 0, 1)}   # the strides of the first grid's axes y and z
        move = lambda st: (st + (0, 0))[drop:drop + 3]   # noqa: E731
        coefs = [P.Coef(value=0.0) for _ in range(7)]
        coefs[P.C] = P.Coef(table=6.3 + 0.01 * np.arange(dims[1]), stride=move(along[1]),
                            table2=0.02 * np.arange(dims[2]), stride2=move(along[2]))
        back = P.Coef(table=-1.0 - 0.001 * np.arange(dims[1]), stride=move(along[1]))
        pairs = [(P.W, P.E), (P.S, P.N), (P.B, P.T)]
        for axis, (lo, hi) in enumerate([(back, P.Coef(value=-0.9)), (P.Coef(value=-1.05), P.Coef(value=-0.95))]):
            to = axis + 1 - drop
            if to >= 0:
                coefs[pairs[to][0]], coefs[pairs[to][1]] = lo, hi
        st = P.Stencil(nx=nx, ny=ny, nz=nz, coefs=coefs)
        s = native.Solver.from_stencil(st)
        x, info = s.solve_mixed(dev(P.splitmix64_uniform(4, st.n)), None, rtol=1e-12, inner_rtol=1e-3)
        assert info["status"] == native.PBCG_OK
        out.append((x.cpu().numpy(), info["inner_iters"]))
        s.close()
    for x, iters in out[1:]:
        np.testing.assert_array_equal(x, out[0][0])
        assert iters == out[0][1]


@pytest.mark.parametrize("values", ["f32", "bf16"])
@pytest.mark.parametrize("n", [2, 33, 64, 257, 5001, 90001])
def test_fp32_sweeps_of_long_rows(n, values):
    """Rows dealt to the blocks in runs: odd numbers of pairs, blocks without a row, several rounds."""
    import torch
    A = P.random_sparse(n, seed=n, nnz_lo=min(9, n), nnz_hi=min(21, n))
    b = oracle.spmv(A, P.splitmix64_uniform(2, n))
    s = native.Solver.from_csr(A)
    low = torch.from_numpy(A.val).cuda().to(torch.float32 if values == "f32" else torch.bfloat16)
    kind = native.PBCG_VALUES_F32 if values == "f32" else native.PBCG_VALUES_BF16
    for grid in (0, 3, 608):
        solve = lambda: s.solve_mixed(dev(b), low, lowp_type=kind, rtol=1e-12, inner_rtol=1e-2, grid=grid)   # noqa: E731
        x, info = solve()
        assert info["status"] == native.PBCG_OK
        assert np.linalg.norm(b - oracle.spmv(A, x.cpu().numpy())) <= 1e-11 * np.linalg.norm(b)
        np.testing.assert_array_equal(x.cpu().numpy(), solve()[0].cpu().numpy())
    s.close()


@pytest.mark.parametrize("dims", [(3, 2, 1), (37, 41, 5), (2500, 2000, 1), (2501, 2000, 1), (171, 171, 171)])
def test_stencil_spmv_on_both_sides_of_its_line(dims):
    """5,000,000 rows (the last with loads in place), 5,002,000 and 5,000,211: the bits of the assembled matrix."""
    st = grid_stencil(*dims)
    x = dev(P.splitmix64_uniform(5, st.n))
    s, c = native.Solver.from_stencil(st), native.Solver.from_csr(P.stencil_to_csr(st))
    np.testing.assert_array_equal(s.spmv(x).cpu().numpy(), c.spmv(x).cpu().numpy())
    s.close()
    c.close()


@pytest.mark.parametrize("n", [0, 1, 4094, 4095, 4096, 12289])
def test_transpose_row_pointers_at_the_tiles_of_the_scan(n):
    import torch
    rng = np.random.default_rng(n)
    counts = rng.integers(0, 4, n) if n else np.zeros(0, dtype=int)
    rp = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    nnz = int(rp[-1])
    col = rng.integers(0, max(n, 1), nnz).astype(np.int32)
    val = rng.standard_normal(nnz)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()   # noqa: E731
    drp, dcol, dval = t(rp), t(col if nnz else np.zeros(1, np.int32)), t(val if nnz else np.zeros(1))
    trp = torch.empty(n + 1, dtype=torch.int32, device="cuda")
    tcol, tval = torch.empty_like(dcol), torch.empty_like(dval)
    wb = native.pbicgstab_transpose_work_bytes(n)
    work = torch.empty(wb // 4 + 64, dtype=torch.int32, device="cuda")
    rc = native.pbicgstab_csr_transpose(n, nnz, drp.data_ptr(), dcol.data_ptr(), dval.data_ptr(), trp.data_ptr(),
                                        tcol.data_ptr(), tval.data_ptr(), work.data_ptr(), wb,
                                        torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert rc == native.PBCG_OK
    expect = np.concatenate([[0], np.cumsum(np.bincount(col, minlength=n))]) if n else np.zeros(1)
    np.testing.assert_array_equal(trp.cpu().numpy(), expect)
    rows = np.repeat(np.arange(n), counts)
    order = np.lexsort((rows, col))
    np.testing.assert_array_equal(tcol.cpu().numpy()[:nnz], rows[order])
