"""CG on one thread-block cluster with matrix and vectors on chip, against the
general path (which a pinned SpMV kernel keeps) and the oracle's residual: where
the rows per thread change (1, 2, 4), blocks without rows, the largest system of
the route, rows of more than one chunk of eight entries, slices that do not fit
(the other routes take those), and the ends of a solve other than convergence."""
import numpy as np
import pytest

import oracle
from paper_2103_10116_gb300 import synth
from tests._helpers import residual_limit
from tests.test_gpu_grid_solve import _both, ctx, spx  # noqa: F401  (fixtures)

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _mat(name):
    return synth.stencil3d_27pt(int(name[4:])) if str(name).startswith("pt27") else synth.ragged_laplace2d(name, 0.2)


# 16 blocks of 256 threads: one row per thread up to 4096 rows, two up to 8192, four up to 16 384
@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("name", [1, 17, 255, 4096, 4097, 8192, 8193, 14335, 14336, 16384, 16385, "pt2715", "pt2722"])
def test_sizes(spx, ctx, name, precision):  # noqa: F811
    mat = _mat(name)
    n = mat[0].shape[0] - 1
    xs = synth.uniform_vector(n, seed=n)
    b = oracle.spmv_csr(*mat, xs)
    tol = 1e-4 if precision == "f32" else 1e-10
    (info, x), (ginfo, gx) = _both(spx, ctx, mat, b, "cg", precision, tol)
    assert info.status == ginfo.status == spx.SPX_CONVERGED and info.relres_true <= tol
    assert abs(info.iterations - ginfo.iterations) <= max(3, ginfo.iterations // 10)
    if precision == "f64":
        assert np.linalg.norm(b - oracle.spmv_csr(*mat, x)) / np.linalg.norm(b) <= residual_limit(*mat, b, x, tol)
    # smallest eigenvalue at least 0.2 (ragged) and 27 - 3^3 cos^3-like above 0.2 up to 22^3: 27 - (1 + 2 cos(pi/23))^3
    lam = 0.2 if not str(name).startswith("pt27") else 27 - (1 + 2 * np.cos(np.pi / (int(name[4:]) + 1))) ** 3
    assert np.linalg.norm(x - gx) <= 2.5 * tol / lam * np.linalg.norm(b)


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("n", [300, 9001])
def test_other_ends(spx, ctx, n, precision):  # noqa: F811
    mat = synth.ragged_laplace2d(n, 0.2)
    b = synth.uniform_vector(n, seed=4)
    tol = 1e-4 if precision == "f32" else 1e-10
    (info, x), _ = _both(spx, ctx, mat, np.zeros(n), "cg", precision, tol, x0=b)
    assert (info.status, info.iterations) == (spx.SPX_CONVERGED, 0) and not x.any()
    (info, x), (ginfo, gx) = _both(spx, ctx, mat, b, "cg", precision, 1e-14, maxit=7)
    assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations) == (spx.SPX_MAX_ITER, 7)
    eps = 2.0 ** -53 if precision == "f64" else 2.0 ** -24
    assert np.linalg.norm(x - gx) <= 1e4 * eps * np.linalg.norm(gx)
    bn = b.copy()
    bn[n // 2] = np.nan
    (info, x), (ginfo, _) = _both(spx, ctx, mat, bn, "cg", precision, tol, maxit=5)
    assert info.status == ginfo.status and info.iterations == ginfo.iterations and np.isnan(x).any()
    zero = (np.zeros(n + 1, np.int32), np.zeros(1, np.int32)[:0], np.zeros(0))  # no entries: p . A p = 0
    (info, _), (ginfo, _) = _both(spx, ctx, zero, b, "cg", precision, tol)
    assert (info.status, info.iterations) == (ginfo.status, ginfo.iterations) == (spx.SPX_BREAKDOWN, 0)
