"""The batched kernel's product for long rows (several lanes per row), taken system
by system: rows of 0 to 70 entries, systems of one row to several rounds of a
block, every block size, solver and precision, beside short-row systems in one
batch; each result is the same bits whatever the others of its batch are."""
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


def _dominant(n, lo, hi, seed, symmetric):
    """Strictly diagonally dominant rows of about lo..hi entries, some of the diagonal alone."""
    rng = np.random.default_rng(seed)
    d = {}
    for i in range(n):
        m = 0 if i % 50 == 7 else int(rng.integers(lo, hi + 1)) // (2 if symmetric else 1)
        for j in rng.integers(0, n, m):
            if j != i:
                v = rng.standard_normal()
                d[(i, int(j))] = v
                if symmetric:
                    d[(int(j), i)] = v
    s = np.zeros(n)
    for (i, j), v in d.items():
        s[i] += abs(v)
    for i in range(n):
        d[(i, i)] = 2 * s[i] + 1
    keys = sorted(d)
    rp = np.zeros(n + 1, np.int32)
    for i, _ in keys:
        rp[i + 1] += 1
    return np.cumsum(rp).astype(np.int32), np.array([j for _, j in keys], np.int32), np.array([d[k] for k in keys])


def _solve(spx, ctx, mats, bs, solver, precision, tol):
    f32 = precision == "f32"
    dt = torch.float32 if f32 else torch.float64
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    ro = np.concatenate([[0], np.cumsum([m[0].shape[0] - 1 for m in mats])])
    no = np.concatenate([[0], np.cumsum([m[1].shape[0] for m in mats])])
    B = spx.spx_batch_create(ctx, ro, no, t(np.concatenate([m[0] for m in mats])), t(np.concatenate([m[1] for m in mats])),
                             t(np.concatenate([m[2] for m in mats])).to(dt),
                             flags=spx.SPX_MIXED_SHADOW if precision == "mixed" else 0)
    b = t(np.concatenate(bs)).to(dt)
    x = torch.zeros_like(b)
    infos = spx.spx_batch_solve(ctx, B, b, x, len(mats), solver, tol, 2000, precision)
    spx.spx_batch_destroy(B)
    xh = x.double().cpu().numpy()
    return infos, [xh[ro[k]:ro[k + 1]] for k in range(len(mats))]


# the mean size sets the block: 128 threads up to 1500 rows, 256 up to 4000, 512 above
@pytest.mark.parametrize("big", [300, 3001, 9001])
@pytest.mark.parametrize("solver", ["cg", "bicgstab", "cgs"])
@pytest.mark.parametrize("precision", ["f64", "f32", "mixed"])
def test_wide_systems(spx, ctx, big, solver, precision):
    sym = solver == "cg"
    mats = [_dominant(n, 14, 70, n, sym) for n in (1, 31, 33, 257)] + [synth.ragged_laplace2d(500, 0.5)]
    if big > 1000:  # rows of 20 to 32 without the slow generator
        fam = synth.DiagDomFamily(big, seed=3).matrix(big)
        mats = [synth.stencil3d_27pt(int(round(big ** (1 / 3)))) if sym else fam] * 3 + [synth.ragged_laplace2d(big, 0.5)]
    tol = 1e-4 if precision == "f32" else 1e-10
    xs = [synth.uniform_vector(m[0].shape[0] - 1, seed=k) for k, m in enumerate(mats)]
    bs = [oracle.spmv_csr(*m, v) for m, v in zip(mats, xs)]
    infos, got = _solve(spx, ctx, mats, bs, solver, precision, tol)
    for m, b, i, x in zip(mats, bs, infos, got):
        assert i.status == spx.SPX_CONVERGED, i
        r = np.linalg.norm(b - oracle.spmv_csr(*m, x)) / np.linalg.norm(b)
        # FP32 solves the FP32-rounded system: rounding A, b and x moves the residual by a few
        # 2^-24 of || |A||x| || / ||b||, which dominance keeps below 4
        assert r <= tol * 1.001 + (16 * 2.0 ** -24 if precision == "f32" else 0.0), (r, i)
    alone_infos, alone = _solve(spx, ctx, mats[:1], bs[:1], solver, precision, tol)
    if big > 1000:  # the same block size alone: the same bits
        assert np.array_equal(alone[0], got[0]) and alone_infos[0].iterations == infos[0].iterations
        _, alone = _solve(spx, ctx, mats[-1:], bs[-1:], solver, precision, tol)  # short rows, without the others
        assert np.array_equal(alone[0], got[-1])


@pytest.mark.parametrize("precision,line", [("f64", 512), ("f32", 768), ("mixed", 768)])
@pytest.mark.parametrize("solver", ["cg", "bicgstab"])
def test_size_line(spx, ctx, solver, precision, line):
    """Systems of long rows around the size from which they take several lanes per row, beside each other."""
    mats = [_dominant(n, 14, 70, n, solver == "cg") for n in (line - 1, line, line + 1, line + 33)]
    tol = 1e-4 if precision == "f32" else 1e-10
    bs = [oracle.spmv_csr(*m, synth.uniform_vector(m[0].shape[0] - 1, seed=k)) for k, m in enumerate(mats)]
    infos, got = _solve(spx, ctx, mats, bs, solver, precision, tol)
    for k, (m, b, i, x) in enumerate(zip(mats, bs, infos, got)):
        assert i.status == spx.SPX_CONVERGED, i
        r = np.linalg.norm(b - oracle.spmv_csr(*m, x)) / np.linalg.norm(b)
        assert r <= tol * 1.001 + (16 * 2.0 ** -24 if precision == "f32" else 0.0), (r, i)  # (as above)
        _, alone = _solve(spx, ctx, mats[k:k + 1], bs[k:k + 1], solver, precision, tol)
        assert np.array_equal(alone[0], x)
