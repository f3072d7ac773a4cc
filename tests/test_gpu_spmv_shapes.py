"""Products at the edges of two kernels' shapes against the CPU oracle, row by row:
ELL slabs taken four at a time (every remainder of the width, ragged last
warps), and row-block CSR tiles of 32 rows with two threads per row (FP64, 16 or
more entries a row on average: odd lengths, empty rows, part tiles)."""
import numpy as np
import pytest

import oracle
from paper_2103_10116_gb300 import synth
from tests._helpers import TOL, assert_spmv_close

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


def _random(lens, seed):
    n = len(lens)
    rng = np.random.default_rng(seed)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    return rp, rng.integers(0, n, rp[-1]).astype(np.int32), rng.standard_normal(rp[-1])


def _check(spx, ctx, mat, fmt, dt, rows_per_thread=0):
    rp, col, val = mat
    n = rp.shape[0] - 1
    key = "f64" if dt == torch.float64 else "f32"
    r = (lambda a: a) if key == "f64" else (lambda a: a.astype(np.float32).astype(np.float64))
    xh, yh = synth.uniform_vector(n, 1), synth.uniform_vector(n, 2)
    ref, bound = oracle.spmv_csr(rp, col, r(val), r(xh)), oracle.spmv_absbound(rp, col, r(val), r(xh))
    A = spx.spx_matrix_create(ctx, fmt, _t(rp), _t(col), _t(val).to(dt))
    if rows_per_thread:
        spx.spx_matrix_set_kernel(A, spx.SPX_KERNEL_ELL, rows_per_thread)
    y = torch.full((n,), float("nan"), dtype=dt, device=DEV)
    spx.spx_spmv(ctx, A, _t(xh).to(dt), y)
    assert_spmv_close(y.double().cpu().numpy(), ref, bound, TOL[key])
    y = _t(yh).to(dt)
    spx.spx_spmv_axpby(ctx, A, -0.5, _t(xh).to(dt), 2.0, y)
    assert_spmv_close(y.double().cpu().numpy(), -0.5 * ref + 2.0 * r(yh), 0.5 * bound + 2.0 * np.abs(yh), TOL[key])
    spx.spx_matrix_destroy(A)


@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("n", [1, 31, 257, 70001])
@pytest.mark.parametrize("width", [1, 2, 3, 4, 5, 7, 8, 9])
def test_ell_widths(spx, ctx, width, n, dt):
    lens = np.random.default_rng(width).integers(0, width + 1, n)
    lens[-1] = width
    _check(spx, ctx, _random(lens, n), "ell", dt)


@pytest.mark.parametrize("n", [1, 31, 32, 33, 319, 320, 321, 50001])
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
def test_row_block_small_tiles(spx, ctx, n, dt):
    lens = np.random.default_rng(n).integers(9, 33, n)
    lens[:: 7] = 32
    if n > 64:
        lens[40:44] = 0
    lens[0] = 16
    mat = _random(lens, n)
    assert np.mean(lens) >= 16 and lens.max() <= 2 * np.mean(lens) + 8  # the automatic choice: row-block, two threads
    _check(spx, ctx, mat, "csr", dt)


@pytest.mark.parametrize("m", [49, 70])
@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
def test_row_block_matrix_copies(spx, ctx, m, dt):
    """Matrices of 24, 36, 73 and 109 MB (FP32, FP64 by size): the copies' hint changes at half of L2."""
    _check(spx, ctx, synth.stencil3d_27pt(m), "csr", dt)


@pytest.mark.parametrize("dt,rows", [(torch.float64, 2), (torch.float32, 2), (torch.float32, 4), (torch.float32, 0)])
@pytest.mark.parametrize("width", [1, 2, 3, 4, 5, 6, 7, 9])
def test_ell_several_rows_per_thread(spx, ctx, width, dt, rows):
    """The last slabs two and one at a time; 0: the automatic choice for as many rows (two in FP32)."""
    n = 257 if rows else 90001
    lens = np.random.default_rng(width).integers(0, width + 1, n)
    lens[-1] = width
    _check(spx, ctx, _random(lens, n), "ell", dt, rows)


@pytest.mark.parametrize("m,dt", [(46, torch.float64), (50, torch.float64), (67, torch.float32), (70, torch.float32),
                                  (80, torch.float32)])
def test_ell_matrix_loads(spx, ctx, m, dt):
    """Matrices of 32, 41, 65, 74 and 111 MB: plain loads; evict-first ones; those at one row per thread in FP32."""
    _check(spx, ctx, synth.stencil3d_27pt(m), "ell", dt)
