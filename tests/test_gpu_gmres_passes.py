"""GMRES's Gram-Schmidt passes where they can go wrong: every number of basis
vector groups (1, 8, 9, 16, 17, 24, 25 and 31 vectors), systems of less than a
tile, whole tiles and ragged last tiles, a solution vector that is not 16-byte
aligned, a matrix whose first pass cancels nearly all of the new vector (the
second pass runs), and matrices scaled far from 1.

The reference is the definition: after k steps of one cycle x minimises
||b - A x|| over the Krylov space span(b, A b, ..., A^(k-1) b), computed here in
numpy with a twice-orthogonalised basis and a dense least-squares solve."""
import numpy as np
import pytest

import oracle
from paper_2103_10116_gb300 import synth

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


def _optimum(mat, b, k):
    """min ||b - A x|| over the k-dimensional Krylov space of b, relative to ||b||."""
    V = [b / np.linalg.norm(b)]
    AV = []
    for _ in range(k):
        w = oracle.spmv_csr(*mat, V[-1])
        AV.append(w.copy())
        Q = np.array(V)
        for _ in range(2):
            w = w - Q.T @ (Q @ w)
        if np.linalg.norm(w) <= 1e-13 * np.linalg.norm(AV[-1]):
            break  # the space is invariant
        V.append(w / np.linalg.norm(w))
    M = np.array(AV).T
    y = np.linalg.lstsq(M, b, rcond=None)[0]
    return np.linalg.norm(b - M @ y) / np.linalg.norm(b)


def _relres(spx, ctx, mat, b, k, dt, offset=0):
    rp, col, val = mat
    A = spx.spx_matrix_create(ctx, "csr", _t(rp), _t(col), _t(val).to(dt))
    n = b.shape[0]
    x = torch.zeros(n + offset, dtype=dt, device=DEV)[offset:]
    bt = _t(b).to(dt)
    info = spx.spx_solve_fixed(ctx, A, bt, x, "gmres", k, restart=k, precision="f64" if dt == torch.float64 else "f32")
    spx.spx_matrix_destroy(A)
    assert info.iterations <= k
    return np.linalg.norm(b - oracle.spmv_csr(rp, col, val, x.double().cpu().numpy())) / np.linalg.norm(b)


def _problem(n):
    """n x n leading block of an upwind convection-diffusion matrix (nonsymmetric)."""
    rp, col, val = synth.convdiff3d_upwind(int(np.ceil(n ** (1 / 3))) + 1)
    keep_rows = np.repeat(np.arange(rp.shape[0] - 1), np.diff(rp))
    keep = (keep_rows < n) & (col < n)
    rows, col, val = keep_rows[keep], col[keep], val[keep]
    out = np.zeros(n + 1, np.int32)
    out[1:] = np.cumsum(np.bincount(rows, minlength=n))
    return out, col.astype(np.int32), val


# FP64 tiles of 64 and 128 rows, FP32 of 128 and 256: below one, exactly whole tiles, ragged
@pytest.mark.parametrize("k", [1, 8, 9, 16, 17, 24, 25, 31])
@pytest.mark.parametrize("n", [50, 1024, 20011])
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
def test_residual_is_the_minimum(spx, ctx, n, k, dt):
    mat = _problem(n)
    b = synth.uniform_vector(n, seed=n + k)
    best = _optimum(mat, b, k)
    got = _relres(spx, ctx, mat, b, k, dt)
    # (FP32 also rounds A, b and x: k + 8 roundings of ||A|| ||x||, ||A|| <= 14 and ||x|| a few ||b||)
    eps = 2.0 ** -53 if dt == torch.float64 else 2.0 ** -24
    assert got <= best * (1 + 1e3 * eps * k) + 200 * (k + 8) * eps, (got, best)
    if dt == torch.float64 and k in (9, 31):  # x at an odd 8-byte address
        off = _relres(spx, ctx, mat, b, k, dt, offset=1)
        assert abs(off - got) <= 1e-12


def _gmres(A, b, k, passes):
    """Relative residual of k steps with classical Gram-Schmidt in the arrays' precision, `passes` passes a step."""
    V = [b / np.linalg.norm(b)]
    H = np.zeros((k + 1, k))
    for j in range(k):
        w, Q = A @ V[j], np.array(V)
        for _ in range(passes):
            h = Q @ w
            w = w - Q.T @ h
            H[:j + 1, j] += h
        H[j + 1, j] = np.linalg.norm(w)
        V.append(w / np.linalg.norm(w))
    e = np.zeros(k + 1)
    e[0] = np.linalg.norm(b)
    x = np.array(V[:k]).T @ np.linalg.lstsq(H, e, rcond=None)[0].astype(A.dtype)
    A, b, x = (v.astype(np.float64) for v in (A, b, x))
    return np.linalg.norm(b - A @ x) / np.linalg.norm(b)


@pytest.mark.parametrize("dt,alpha", [(torch.float64, 1e8), (torch.float32, 1e4)])
def test_second_pass(spx, ctx, dt, alpha):
    """A = Laplacian + alpha b v^T: every A v_j is along v_0 = b but for a part of 1 / alpha, and the Laplacian keeps the
    convergence slow.  With one pass the basis is lost, and the residual stays at ten times the limit or more."""
    n, k = 2000, 30
    rp, col, val = synth.laplace2d_5pt(40, 50)
    A = np.zeros((n, n))
    A[np.repeat(np.arange(n), np.diff(rp)), col] = val
    rng = np.random.default_rng(1)
    b = rng.uniform(-1.0, 1.0, n)
    b *= np.sqrt(n) / np.linalg.norm(b)
    A[:, np.arange(100, n, 400)] += alpha * b[:, None] * rng.uniform(0.5, 1.0, 5)
    A, b = (v.astype(np.float64 if dt == torch.float64 else np.float32) for v in (A, b))
    limit = 1.5 * _gmres(A.astype(np.float64), b.astype(np.float64), k, 2)
    assert _gmres(A, b, k, 1) >= 10 * limit
    rp = np.concatenate([[0], np.cumsum((A != 0).sum(1))]).astype(np.int32)
    rows, cols = np.nonzero(A)
    got = _relres(spx, ctx, (rp, cols.astype(np.int32), A[rows, cols].astype(np.float64)), b.astype(np.float64), k, dt)
    assert got <= limit, (got, limit)


@pytest.mark.parametrize("scale", [1e-13, 1e13])
def test_scaled_fp32(spx, ctx, scale):
    """Products of entries of the unnormalised basis stay in FP32's range however A is scaled."""
    n, k = 4097, 17
    rp, col, val = _problem(n)
    b = synth.uniform_vector(n, seed=9)
    a = _relres(spx, ctx, (rp, col, val), b, k, torch.float32)
    c = _relres(spx, ctx, (rp, col, val * scale), b, k, torch.float32)
    assert abs(a - c) <= 200 * (k + 8) * 2.0 ** -24, (a, c)


@pytest.mark.parametrize("first,rest", [(1e-14, 1e4), (1e-4, 1e14), (1e10, 1e-7)])
def test_norms_far_apart_fp32(spx, ctx, first, rest):
    """A maps e1 -> first e2, e2 -> rest e3, e3 -> rest (e1 + e3), in n / 3 equal blocks: the stored basis vectors'
    norms lie rest / first = 1e18 or 1e-17 apart, and raw products of their entries leave FP32's range."""
    blocks = 1000
    i = 3 * np.arange(blocks)
    rows = np.concatenate([i, i + 1, i + 2, i + 2])
    cols = np.concatenate([i + 2, i, i + 1, i + 2])
    vals = np.concatenate([np.full(blocks, v) for v in (rest, first, rest, rest)])
    order = np.lexsort((cols, rows))
    rp = np.zeros(3 * blocks + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(rows, minlength=3 * blocks))
    A = spx.spx_matrix_create(ctx, "csr", _t(rp), _t(cols[order].astype(np.int32)), _t(vals[order]).float())
    b = np.zeros(3 * blocks)
    b[i] = 1.0
    x = torch.zeros(3 * blocks, dtype=torch.float32, device=DEV)
    spx.spx_solve_fixed(ctx, A, _t(b).float(), x, "gmres", 3, restart=3, precision="f32")
    spx.spx_matrix_destroy(A)
    # A x = b: x = (0, -1, 1) / rest, to the roundings of three steps, row by row of A: the error of e1's coefficient
    # weighs `first`, that of the others `rest`
    err = x.double().cpu().numpy() - np.tile([0.0, -1.0, 1.0], blocks) / rest
    err[i] *= first / rest
    assert np.abs(err).max() * rest <= 100 * 2.0 ** -24, err[:3] * rest
