"""The one-launch solve over the device (the route spx_solve takes for CSR
systems of rows of similar length from about a thousand to three hundred
thousand rows) against the CPU oracle's residual and against the general path,
which a pinned SpMV kernel keeps: same status, about the same iterations, same
solution; at the sizes where the partition changes (one, two and four rows per
thread, the largest system, a ragged last block), for every solver and
precision, and for the ends of a solve other than convergence."""
import threading

import numpy as np
import pytest

import oracle
from paper_2103_10116_gb300 import synth
from tests._helpers import residual_limit

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def spx():
    from paper_2103_10116_gb300 import spx as s
    s.load()
    return s


@pytest.fixture(scope="module")
def ctx(spx):
    c = spx.spx_ctx_create(0)
    yield c
    torch.cuda.synchronize()
    spx.spx_ctx_destroy(c)


def _t(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _both(spx, ctx, mat, b, solver, precision, tol, maxit=20000, x0=None, fmt="csr", precond=None):
    """(info, x) by the automatic route, solved twice (equal bits), and by the general path."""
    rp, col, val = mat
    f32 = precision == "f32"
    dt = torch.float32 if f32 else torch.float64
    out = []
    for pinned in (False, True):
        A = spx.spx_matrix_create(ctx, fmt, _t(rp), _t(col), _t(val).to(dt),
                                  flags=spx.SPX_MIXED_SHADOW if precision == "mixed" else 0)
        if pinned:
            kernel = {"csr": (spx.SPX_KERNEL_CSR_ROWS, 0), "coo": (spx.SPX_KERNEL_COO, 216)}.get(fmt, (spx.SPX_KERNEL_ELL, 1))
            spx.spx_matrix_set_kernel(A, *kernel)
        bt = _t(b).to(dt)
        xs = []
        for _ in range(1 if pinned else 2):
            x = torch.zeros_like(bt) if x0 is None else _t(x0).to(dt)
            info = spx.spx_solve(ctx, A, bt, x, solver, tol, maxit, precision=precision, precond=precond)
            xs.append(x.double().cpu().numpy())
        if not pinned:
            assert np.array_equal(xs[0], xs[1], equal_nan=True)  # no dependence on timing
        out.append((info, xs[0]))
        spx.spx_matrix_destroy(A)
    return out


# blocks of 152 SMs: one row per thread up to 77 824 rows, two up to 155 648, four up to 311 296
# (the next size takes the general path); the smallest sizes of each solver and precision
SIZES = [("bicgstab", "f64", 513), ("cgs", "f32", 1021), ("cg", "mixed", 1283), ("cg", "f64", 12289), ("cg", "f32", 16387),
         ("bicgstab", "mixed", 5003), ("cgs", "mixed", 20011), ("cg", "f64", 77825), ("bicgstab", "f32", 77791),
         ("cgs", "f64", 155649), ("cg", "mixed", 155649), ("bicgstab", "f64", 311296), ("cg", "f64", 311297)]


@pytest.mark.parametrize("solver,precision,n", SIZES)
def test_sizes_against_oracle_and_general_path(spx, ctx, solver, precision, n):
    mat = synth.ragged_laplace2d(n, 0.2)
    xs = synth.uniform_vector(n, seed=n)
    b = oracle.spmv_csr(*mat, xs)
    tol = 1e-4 if precision == "f32" else 1e-10
    (info, x), (ginfo, gx) = _both(spx, ctx, mat, b, solver, precision, tol)
    assert info.status == ginfo.status == spx.SPX_CONVERGED
    assert info.relres_true <= tol
    # refinement cycles and CGS's squared polynomial amplify the order of the sums
    slack = max(4, ginfo.iterations // (5 if precision == "mixed" and solver != "cg" else 10))
    assert abs(info.iterations - ginfo.iterations) <= slack, (info, ginfo)
    if precision != "f32":  # (an FP32 residual is of the FP32-rounded system)
        r = np.linalg.norm(b - oracle.spmv_csr(*mat, x)) / np.linalg.norm(b)
        assert r <= residual_limit(*mat, b, x, tol)
    # both residuals are below tol: the solutions differ by at most 2 tol ||A^-1|| ||b||, ||A^-1|| <= 1 / shift
    assert np.linalg.norm(x - gx) <= 2.5 * tol / 0.2 * np.linalg.norm(b)


@pytest.mark.parametrize("solver,precision", [("bicgstab", "f64"), ("cgs", "f64"), ("bicgstab", "mixed"), ("bicgstab", "f32")])
def test_long_rows(spx, ctx, solver, precision):
    """Rows of 8 to 32 random columns: full and partial chunks of eight entries."""
    n = 9001
    mat = synth.DiagDomFamily(n, seed=5).matrix(n)
    xs = synth.uniform_vector(n, seed=2)
    b = oracle.spmv_csr(*mat, xs)
    tol = 1e-5 if precision == "f32" else 1e-10
    (info, x), (ginfo, _) = _both(spx, ctx, mat, b, solver, precision, tol)
    assert info.status == ginfo.status == spx.SPX_CONVERGED and info.relres_true <= tol
    assert abs(info.iterations - ginfo.iterations) <= max(3, ginfo.iterations // 10)
    # the diagonal is twice the sum of the others' magnitudes: ||A^-1||_inf <= 1 / min(diag / 2)
    assert np.linalg.norm(x - xs) <= 1e3 * tol * np.linalg.norm(xs)


@pytest.mark.parametrize("fmt", ["ell", "coo", "hyb"])
@pytest.mark.parametrize("solver,precision", [("cg", "f64"), ("cg", "mixed"), ("bicgstab", "f64"), ("cgs", "mixed"), ("bicgstab", "f32")])
@pytest.mark.parametrize("n", [1, 33, 4099, 90001])
def test_other_formats(spx, ctx, n, solver, precision, fmt):
    """ELL (HYB without overflow included) and COO fill the same slices: ragged rows, empty ones beside them."""
    mat = synth.ragged_laplace2d(n, 0.2) if solver == "cg" or n < 40 else synth.DiagDomFamily(n, seed=5).matrix(n)
    if fmt == "hyb" and solver != "cg" and n >= 40:
        pytest.skip("overflow entries: the general path")
    b = oracle.spmv_csr(*mat, synth.uniform_vector(n, seed=3))
    tol = 1e-5 if precision == "f32" else 1e-10
    (info, x), (ginfo, gx) = _both(spx, ctx, mat, b, solver, precision, tol, fmt=fmt)
    assert info.status == ginfo.status == spx.SPX_CONVERGED and info.relres_true <= tol
    assert abs(info.iterations - ginfo.iterations) <= max(4, ginfo.iterations // 5)
    if precision != "f32":
        assert np.linalg.norm(b - oracle.spmv_csr(*mat, x)) / np.linalg.norm(b) <= residual_limit(*mat, b, x, tol)


def _graded(n, solver, seed):
    """S A S with S spread over a decade, so that Jacobi matters; the diagonal of every fifth row in two entries."""
    rp, col, val = synth.ragged_laplace2d(n, 0.2) if solver == "cg" or n < 40 else synth.DiagDomFamily(n, seed=5).matrix(n)
    row = np.repeat(np.arange(n), np.diff(rp))
    s = 10.0 ** np.random.default_rng(seed).uniform(-0.5, 0.5, n)
    val = s[row] * val * s[col]
    twice = (col == row) & (row % 5 == 0)
    count = 1 + twice.astype(np.int64)
    at = np.repeat(np.arange(len(col)), count)
    out = np.zeros(n + 1, np.int32)
    out[1:] = np.cumsum(np.bincount(row, weights=count, minlength=n))
    return out, col[at].astype(np.int32), val[at] / count[at]


@pytest.mark.parametrize("fmt", ["csr", "ell", "coo"])
@pytest.mark.parametrize("solver", ["cg", "bicgstab", "cgs"])
@pytest.mark.parametrize("precision", ["f64", "f32", "mixed"])
@pytest.mark.parametrize("n", [1, 33, 4099, 90001])
def test_jacobi(spx, ctx, n, solver, precision, fmt):
    """Jacobi in the launch: as on the general path, over storages, one and two rows per thread."""
    mat = _graded(n, solver, seed=n)
    b = oracle.spmv_csr(*mat, synth.uniform_vector(n, seed=3))
    tol = 1e-4 if precision == "f32" else 1e-10
    (info, x), (ginfo, gx) = _both(spx, ctx, mat, b, solver, precision, tol, fmt=fmt, precond="jacobi")
    assert info.status == ginfo.status == spx.SPX_CONVERGED and info.relres_true <= tol
    assert abs(info.iterations - ginfo.iterations) <= max(4, ginfo.iterations // 5), (info, ginfo)
    if precision != "f32":
        assert np.linalg.norm(b - oracle.spmv_csr(*mat, x)) / np.linalg.norm(b) <= residual_limit(*mat, b, x, tol)


@pytest.mark.parametrize("precision", ["f64", "f32", "mixed"])
@pytest.mark.parametrize("solver", ["cg", "bicgstab", "cgs"])
def test_jacobi_other_ends(spx, ctx, solver, precision):
    """Without a diagonal M is I; b = 0, the iteration limit and a NaN as on the general path."""
    n = 5003
    mat = _graded(n, "cg", seed=1)
    b = synth.uniform_vector(n, seed=4)
    (info, x), (ginfo, _) = _both(spx, ctx, mat, np.zeros(n), solver, precision, 1e-4, x0=b, precond="jacobi")
    assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations) == (spx.SPX_CONVERGED, 0)
    assert not x.any()
    (info, x), (ginfo, gx) = _both(spx, ctx, mat, b, solver, precision, 1e-14, maxit=5, precond="jacobi")
    assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations) == (spx.SPX_MAX_ITER, 5)
    # five iterations of one recurrence in two orders of summation
    eps = 2.0 ** -53 if precision == "f64" else 2.0 ** -24
    assert np.linalg.norm(x - gx) <= 1e4 * eps * np.linalg.norm(gx)
    bn = b.copy()
    bn[n // 2] = np.nan
    (info, x), (ginfo, _) = _both(spx, ctx, mat, bn, solver, precision, 1e-4, maxit=5, precond="jacobi")
    assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations)
    shift = (np.arange(n + 1, dtype=np.int32), ((np.arange(n) + 1) % n).astype(np.int32), np.ones(n))  # r . A r = 0
    e = np.zeros(n)
    e[3] = 1.0
    (info, _), (ginfo, _) = _both(spx, ctx, shift, e, solver, precision, 1e-4, maxit=50, precond="jacobi")
    assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations)


@pytest.mark.parametrize("solver", ["cg", "bicgstab", "cgs"])
@pytest.mark.parametrize("precision", ["f64", "f32", "mixed"])
def test_other_ends(spx, ctx, solver, precision):
    """b = 0, an initial guess, the iteration limit, a breakdown and a NaN end as on the general path."""
    n = 17001
    mat = synth.ragged_laplace2d(n, 0.2)
    b = synth.uniform_vector(n, seed=4)
    tol = 1e-4 if precision == "f32" else 1e-10

    (info, x), (ginfo, _) = _both(spx, ctx, mat, np.zeros(n), solver, precision, tol, x0=b)
    assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations) == (spx.SPX_CONVERGED, 0)
    assert not x.any()

    xs = synth.uniform_vector(n, seed=6)
    rhs = oracle.spmv_csr(*mat, xs)
    (info, x), (ginfo, _) = _both(spx, ctx, mat, rhs, solver, precision, tol, x0=xs * (1 + 1e-3))
    assert info.status == ginfo.status == spx.SPX_CONVERGED
    assert abs(info.iterations - ginfo.iterations) <= max(4, ginfo.iterations // 5)

    (info, x), (ginfo, gx) = _both(spx, ctx, mat, b, solver, precision, 1e-14, maxit=7)
    assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations) == (spx.SPX_MAX_ITER, 7)
    # seven iterations of one recurrence in two orders of summation
    eps = 2.0 ** -53 if precision == "f64" else 2.0 ** -24
    assert np.linalg.norm(x - gx) <= 1e4 * eps * np.linalg.norm(gx)

    # skew-symmetric, integers: r . A r is exactly 0 in the first iteration
    i = np.arange(n)
    rows = np.concatenate([i[1:], i[:-1]])
    cols = np.concatenate([i[:-1], i[1:]])
    vals = np.concatenate([-np.ones(n - 1), np.ones(n - 1)])
    order = np.lexsort((cols, rows))
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(rows, minlength=n))
    skew = (rp, cols[order].astype(np.int32), vals[order])
    bi = (np.arange(n) % 3 - 1).astype(np.float64)
    if precision != "mixed" or solver == "cg":  # (refinement scales the residual: not integers any more)
        (info, _), (ginfo, _) = _both(spx, ctx, skew, bi, solver, precision, tol, maxit=50)
        assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations) == (spx.SPX_BREAKDOWN, 0)

    bn = b.copy()
    bn[n // 2] = np.nan
    (info, x), (ginfo, _) = _both(spx, ctx, mat, bn, solver, precision, tol, maxit=5)
    assert info.status == ginfo.status and info.iterations == ginfo.iterations
    assert np.isnan(x).any() or info.iterations == 0


def test_mixed_cg_iteration_limit(spx, ctx):
    """A limit that falls on the iteration after which the FP32 residual is below tol but the FP64 one is not: the
    solve ends there, as on the general path."""
    n = 5003
    mat = synth.ragged_laplace2d(n, 0.2)
    b = _t(oracle.spmv_csr(*mat, synth.uniform_vector(n, seed=3)))
    A = spx.spx_matrix_create(ctx, "csr", *(_t(a) for a in mat), flags=spx.SPX_MIXED_SHADOW)
    solve = lambda tol, k: spx.spx_solve(ctx, A, b, torch.zeros_like(b), "cg", tol, k, precision="mixed")
    for tol in (1e-7, 1e-12, 4e-16, 3e-16, 2e-16, 1.5e-16, 1e-16):  # the last ones about what FP64 can reach
        full = solve(tol, 200).iterations
        for k in range(max(1, full - 40), full):
            info = solve(tol, k)
            assert (info.status, info.iterations) == (spx.SPX_MAX_ITER, k), (tol, info)
    spx.spx_matrix_destroy(A)


def test_pending_error_is_reported(spx, ctx):
    """A wait that gave up on this context before the solve is reported by it, as on the general path, and cleared."""
    n = 5003
    mat = synth.ragged_laplace2d(n, 0.2)
    A = spx.spx_matrix_create(ctx, "csr", *(_t(a) for a in mat))
    b, x = _t(synth.uniform_vector(n, seed=3)), torch.zeros(n, dtype=torch.float64, device=DEV)
    spx.spx_selftest_wait_timeout(ctx, 0)
    with pytest.raises(spx.SpxError) as ei:
        spx.spx_solve(ctx, A, b, x, "bicgstab", 1e-10, 1000)
    assert ei.value.status == spx.SPX_ERR_TIMEOUT
    assert spx.spx_solve(ctx, A, b, x, "bicgstab", 1e-10, 1000).status == spx.SPX_CONVERGED
    spx.spx_matrix_destroy(A)


@pytest.mark.parametrize("fmt", ["csr", "ell", "coo"])
@pytest.mark.parametrize("n", [300, 5003, 40009])
def test_unknown_precision_is_refused(spx, ctx, n, fmt):
    mat = synth.ragged_laplace2d(n, 0.2)
    A = spx.spx_matrix_create(ctx, fmt, _t(mat[0]), _t(mat[1]), _t(mat[2]).float())
    b, x = _t(synth.uniform_vector(n, seed=3)).float(), torch.zeros(n, dtype=torch.float32, device=DEV)
    with pytest.raises(spx.SpxError) as ei:
        spx.spx_solve(ctx, A, b, x, "cg", 1e-4, 1000, precision=7)
    assert ei.value.status == spx.SPX_ERR_INVALID
    spx.spx_matrix_destroy(A)


@pytest.mark.parametrize("solver,precision,n,precond", [
    ("cg", "f64", 40009, None), ("cg", "mixed", 97336, None), ("cg", "f32", 200003, None), ("bicgstab", "f64", 90001, None),
    ("cgs", "mixed", 70001, None), ("cg", "mixed", 160001, "jacobi"), ("cg", "f64", 250007, None)])
def test_contexts_at_once(spx, solver, precision, n, precond):
    """Solves of several contexts and threads at once give the bits of the solve alone: with others running, a solve
    takes the kernel with fewer registers (three of these sizes at four rows per thread, one of them FP64)."""
    mat = synth.ragged_laplace2d(n, 0.2)
    dt = torch.float32 if precision == "f32" else torch.float64
    b = _t(oracle.spmv_csr(*mat, synth.uniform_vector(n, seed=n))).to(dt)
    tol = 1e-4 if precision == "f32" else 1e-9
    args = [_t(mat[0]), _t(mat[1]), _t(mat[2]).to(dt)]
    flags = spx.SPX_MIXED_SHADOW if precision == "mixed" else 0
    torch.cuda.synchronize()

    def solves(out, count):
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            c = spx.spx_ctx_create(0, stream=st, allocator="cuda")
            A = spx.spx_matrix_create(c, "csr", *args, flags=flags)
            for _ in range(count):
                x = torch.zeros_like(b)
                info = spx.spx_solve(c, A, b, x, solver, tol, 20000, precision=precision, precond=precond)
                out.append((info.status, info.iterations, x.cpu().numpy()))
            spx.spx_matrix_destroy(A)
            spx.spx_ctx_destroy(c)

    alone = []
    solves(alone, 1)
    assert alone[0][0] == spx.SPX_CONVERGED
    outs = [[] for _ in range(6)]
    threads = [threading.Thread(target=solves, args=(o, 4)) for o in outs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for o in outs:
        assert len(o) == 4
        for status, iterations, x in o:
            assert (status, iterations) == alone[0][:2] and np.array_equal(x, alone[0][2])
