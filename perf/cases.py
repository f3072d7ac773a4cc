"""The work a program has this library do, as cases that can be timed.

Every case goes through the public entry points of the Python binding (the
names of the C ABI), or through the serving class on top of them:

  spmv     y = A x (or y = alpha A x + beta y) with a matrix kept on the device
  noalloc  y = A x from the caller's own CSR arrays, nothing allocated
  solve    one system with CG, BiCGSTAB, CGS or GMRES(30) on a resident matrix
  batch    many small independent systems in one call
  serve    a burst of requests on host arrays through the request server

The matrices are the families the library's generators name (2D and 3D
Laplacians, the 27-point stencil, upwind convection-diffusion, power-law rows,
diagonally dominant random rows, ragged 2D Laplacians), built here with torch
on the device because host generation of millions of rows takes seconds.
Right-hand sides are b = A x* with x* ~ U[-1, 1] from the seed, so the exact
solution of every system is x*.
"""
import math

import numpy as np
import torch

from paper_2103_10116_gb300 import spx
from paper_2103_10116_gb300.serving import Server

DEV = "cuda:0"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest call: one product of the 64 x 64 Laplacian, where latency and launch cost are all there is
        {"name": "spmv_lap2d_64_csr_f64", "kind": "spmv", "family": "lap2d", "m": 64, "format": "csr",
         "dtype": "f64", "axpby": False},
        # a million-row stencil product, the format and type most solvers run on
        {"name": "spmv_27pt_100_csr_f64", "kind": "spmv", "family": "pt27", "m": 100, "format": "csr",
         "dtype": "f64", "axpby": False},
        # two million ragged rows of random columns in single precision, stored as coordinates
        {"name": "spmv_powerlaw_2m_coo_f32", "kind": "spmv", "family": "powerlaw", "m": 2_000_000, "format": "coo",
         "dtype": "f32", "axpby": False},
        # a product inside a loop that may not allocate, an odd size of some tens of thousands of rows
        {"name": "noalloc_7pt_41_f64", "kind": "noalloc", "family": "lap3d", "m": 41, "dtype": "f64"},
        # the smallest solve: the 64 x 64 Laplacian to 1e-10
        {"name": "cg_lap2d_64_f64", "kind": "solve", "family": "lap2d", "m": 64, "format": "csr", "solver": "cg",
         "precision": "f64", "precond": "none", "block": 0, "tol": 1e-10},
        # an ordinary solve: a stencil of 97 336 rows in mixed precision to 1e-8
        {"name": "cg_7pt_46_mixed", "kind": "solve", "family": "lap3d", "m": 46, "format": "csr", "solver": "cg",
         "precision": "mixed", "precond": "none", "block": 0, "tol": 1e-8},
        # an ordinary nonsymmetric solve: 30 001 rows of about 20 random columns
        {"name": "bicgstab_diagdom_30001_f64", "kind": "solve", "family": "diagdom", "m": 30_001, "format": "csr",
         "solver": "bicgstab", "precision": "f64", "precond": "none", "block": 0, "tol": 1e-10},
        # a large SPD solve: 7-point Poisson on 128^3
        {"name": "cg_7pt_128_f64", "kind": "solve", "family": "lap3d", "m": 128, "format": "csr", "solver": "cg",
         "precision": "f64", "precond": "none", "block": 0, "tol": 1e-10},
        # the largest nonsymmetric solve: GMRES(30) on convection-diffusion, 128^3
        {"name": "gmres_convdiff_128_f64", "kind": "solve", "family": "convdiff", "m": 128, "format": "csr",
         "solver": "gmres", "precision": "f64", "precond": "none", "block": 0, "tol": 1e-10},
        # a preconditioned solve in the other common storage: strong upwinding, ELL, block-Jacobi of 8 rows
        {"name": "bicgstab_bj8_peclet_101_ell", "kind": "solve", "family": "peclet", "m": 101, "format": "ell",
         "solver": "bicgstab", "precision": "f64", "precond": "block_jacobi", "block": 8, "tol": 1e-10},
        # thousands of small uneven systems in one call
        {"name": "batch_cg_4096_f64", "kind": "batch", "count": 4096, "nmax": 10_000, "solver": "cg",
         "precision": "f64", "tol": 1e-10},
        # a burst of served requests, half stencils (CG), half random rows (BiCGSTAB), 1e3 to 1e5 rows
        {"name": "serve_48_mixed", "kind": "serve", "count": 48, "nmax": 100_000, "tol": 1e-8},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, family, rows):
    """A size parameter of `family` with about 1e3 .. rows rows, spread over the logarithm."""
    n = _logint(rng, 1000, rows)
    if family == "lap2d":
        return max(16, int(round(n ** 0.5)))
    if family in ("lap3d", "pt27", "convdiff", "peclet"):
        return max(10, int(round(n ** (1.0 / 3.0))))
    return n


def draw(rng):
    kind = rng.choices(["spmv", "noalloc", "solve", "batch", "serve"], [8, 2, 8, 3, 1])[0]
    if kind == "spmv":
        family = rng.choice(["lap2d", "lap3d", "pt27", "powerlaw", "diagdom"])
        rows = {"pt27": 1_000_000, "diagdom": 1_000_000}.get(family, 2_000_000)
        # (column-major padding does not hold heavy-tailed rows: those take HYB)
        fmt = rng.choice(["csr", "coo", "hyb"] if family == "powerlaw" else ["csr", "ell", "coo", "hyb"])
        return {"kind": kind, "family": family, "m": _size(rng, family, rows), "format": fmt,
                "dtype": rng.choice(["f64", "f32"]), "axpby": rng.random() < 0.25}
    if kind == "noalloc":
        family = rng.choice(["lap2d", "lap3d", "pt27", "powerlaw"])
        return {"kind": kind, "family": family, "m": _size(rng, family, 1_000_000),
                "dtype": rng.choice(["f64", "f32"])}
    if kind == "solve":
        family = rng.choice(["lap2d", "lap3d", "pt27", "convdiff", "peclet", "diagdom"])
        solver = "cg" if family in ("lap2d", "lap3d", "pt27") else rng.choice(["bicgstab", "cgs", "gmres"])
        # 2D grids need iterations in proportion to their side: up to 300 x 300, the others up to 128^3
        rows = {"lap2d": 90_000, "diagdom": 1_000_000, "pt27": 1_000_000}.get(family, 2_097_152)
        precision = rng.choice(["f64", "mixed", "f32"] if family == "diagdom" else ["f64", "f64", "mixed"])
        precond = rng.choice(["none", "none", "none", "jacobi", "block_jacobi"])
        return {"kind": kind, "family": family, "m": _size(rng, family, rows),
                "format": rng.choice(["csr", "csr", "csr", "ell", "coo"]), "solver": solver, "precision": precision,
                "precond": precond, "block": rng.choice([4, 8, 16]) if precond == "block_jacobi" else 0,
                "tol": 1e-5 if precision == "f32" else 1e-10}
    if kind == "batch":
        precision = rng.choice(["f64", "mixed", "f32"])
        return {"kind": kind, "count": _logint(rng, 16, 4096), "nmax": _logint(rng, 300, 10_000),
                "solver": rng.choice(["cg", "cg", "bicgstab"]), "precision": precision,
                "tol": 1e-4 if precision == "f32" else 1e-10}
    return {"kind": kind, "count": _logint(rng, 12, 60), "nmax": _logint(rng, 5_000, 100_000), "tol": 1e-8}


# ------------------------------------------------------------------ matrices (row lengths, columns, values)
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000 + salt)
    return g


def _stencil(shape, offsets, weights):
    """Constant-coefficient stencil with Dirichlet boundary on a grid, last axis fastest, columns ascending."""
    n = math.prod(shape)
    strides = [math.prod(shape[d + 1:]) for d in range(len(shape))]
    order = sorted(range(len(offsets)), key=lambda k: sum(o * s for o, s in zip(offsets[k], strides)))
    i = torch.arange(n, device=DEV, dtype=torch.int32)
    coord = [(i // strides[d]) % shape[d] for d in range(len(shape))]
    cols = torch.empty(n, len(order), dtype=torch.int32, device=DEV)
    valid = torch.ones(n, len(order), dtype=torch.bool, device=DEV)
    for k, o in enumerate(order):
        cols[:, k] = i + sum(q * s for q, s in zip(offsets[o], strides))
        for d, q in enumerate(offsets[o]):
            if q:
                valid[:, k] &= coord[d] >= 1 if q < 0 else coord[d] < shape[d] - 1
    w = torch.tensor([weights[k] for k in order], dtype=torch.float64, device=DEV).expand(n, len(order))
    return valid.sum(1), cols[valid], w[valid]


def _axis_offsets(dims):
    return [(0,) * dims] + [tuple(s if a == d else 0 for a in range(dims)) for d in range(dims) for s in (-1, 1)]


def _upwind(m, peclet):
    h = 1.0 / (m + 1)
    c = h * peclet / math.sqrt(3.0)
    return _stencil((m, m, m), _axis_offsets(3), [6.0 + 3.0 * c] + [-1.0 - c, -1.0] * 3)


def _random_rows(n, lens, seed, sort_cols=True):
    """Uniform random columns for rows of the given lengths, ascending within a row."""
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), lens)
    cols = torch.randint(0, n, rows.shape, device=DEV, generator=_gen(seed, 1))
    key = torch.sort(rows * n + cols)[0]
    return rows, key - rows * n


def _powerlaw(n, seed):
    """Row lengths min(20000, floor(x_m U^(-2/3))) with x_m fitted to a mean of 16; N(0, 1) values."""
    g = (1.0 - torch.rand(n, device=DEV, dtype=torch.float64, generator=_gen(seed, 2))) ** (-1.0 / 1.5)
    cap = min(20_000, n)
    lo, hi = 1.0, 16.0
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if float(torch.floor(mid * g).clamp_(max=cap).mean()) < 16.0 else (lo, mid)
    lens = torch.floor(hi * g).clamp_(max=cap).long()
    _, cols = _random_rows(n, lens, seed)
    vals = torch.randn(cols.shape, device=DEV, dtype=torch.float64, generator=_gen(seed, 3))
    return lens, cols.int(), vals


def _diagdom(n, seed):
    """8 to 32 entries a row: the diagonal, twice the sum of the others' magnitudes, and N(0, 1) values in random columns."""
    lens = torch.randint(8, 33, (n,), device=DEV, generator=_gen(seed, 4))
    rows, cols = _random_rows(n, lens, seed)
    vals = torch.randn(cols.shape, device=DEV, dtype=torch.float64, generator=_gen(seed, 5))
    first = torch.cumsum(lens, 0) - lens
    vals[first] = 0.0
    total = torch.segment_reduce(vals.abs(), "sum", lengths=lens, unsafe=True)
    cols[first] = torch.arange(n, device=DEV)  # the diagonal is stored first
    vals[first] = 2.0 * total + 1.0
    return lens, cols.int(), vals


def _matrix(case, seed):
    """(row lengths int64, columns int32, values float64) on the device."""
    f, m = case["family"], case["m"]
    if f == "lap2d":
        return _stencil((m, m), _axis_offsets(2), [4.0] + [-1.0] * 4)
    if f == "lap3d":
        return _stencil((m, m, m), _axis_offsets(3), [6.0] + [-1.0] * 6)
    if f == "pt27":
        offs = [(a, b, c) for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
        return _stencil((m, m, m), offs, [26.0 if o == (0, 0, 0) else -1.0 for o in offs])
    if f == "convdiff":
        return _upwind(m, 10.0)
    if f == "peclet":
        return _upwind(m, 10.0 * (m + 1))  # cell Peclet number 10
    if f == "powerlaw":
        return _powerlaw(m, seed)
    return _diagdom(m, seed)


def _row_ptr(lens):
    rp = torch.zeros(lens.numel() + 1, dtype=torch.int32, device=DEV)
    rp[1:] = torch.cumsum(lens, 0)
    return rp


def _product(lens, cols, vals, x):
    """A x in 64 bits, each row summed on its own (the same bits every time)."""
    return torch.segment_reduce(vals.double() * x.double()[cols.long()], "sum", lengths=lens, unsafe=True)


def _uniform(n, seed, salt):
    return torch.rand(n, device=DEV, dtype=torch.float64, generator=_gen(seed, salt)) * 2.0 - 1.0


def _rows(case):
    return case["m"] ** {"lap2d": 2, "lap3d": 3, "pt27": 3, "convdiff": 3, "peclet": 3}.get(case["family"], 1)


def _nnz(case):
    f, m = case["family"], case["m"]
    if f == "lap2d":
        return 5 * m * m - 4 * m
    if f in ("lap3d", "convdiff", "peclet"):
        return 7 * m ** 3 - 6 * m * m
    if f == "pt27":
        return (3 * m - 2) ** 3
    return (16 if f == "powerlaw" else 20) * m


def _batch_matrix(case, seed):
    """Ragged 2D Laplacians plus a shift, as one block-diagonal matrix: (sizes, row lengths, local columns, values,
    first rows, system of each row).  The sizes go by the case, the shifts by the seed."""
    sizes = torch.randint(100, case["nmax"] + 1, (case["count"],), device=DEV, generator=_gen(case["nmax"], 6))
    shift = torch.rand(case["count"], device=DEV, dtype=torch.float64, generator=_gen(seed, 6)) * 0.99 + 0.01
    sysid = torch.repeat_interleave(torch.arange(case["count"], device=DEV), sizes)
    off = torch.cumsum(sizes, 0) - sizes
    i = torch.arange(sysid.numel(), device=DEV) - off[sysid]
    n = sizes[sysid]
    nx = torch.sqrt(n.double()).round().long()
    cand = torch.stack([i - nx, i - 1, i, i + 1, i + nx], 1)
    ok = torch.stack([i >= nx, i % nx != 0, i >= 0, ((i + 1) % nx != 0) & (i + 1 < n), i + nx < n], 1)
    vals = torch.full(cand.shape, -1.0, dtype=torch.float64, device=DEV)
    vals[:, 2] = 4.0 + shift[sysid]
    return sizes, ok.sum(1), cand[ok].int(), vals[ok], off, sysid


# ------------------------------------------------------------------ states
class State:
    """What a program holds: its context, matrix (or batch, or server) and vectors."""

    def __init__(self, case):
        self.case = case
        self.ctx = spx.spx_ctx_create(0)
        self.A = self.B = self.server = None

    def __del__(self):
        if self.server is not None:
            self.server.close()
        if self.A is not None:
            spx.spx_matrix_destroy(self.A)
        if self.B is not None:
            spx.spx_batch_destroy(self.B)
        spx.spx_ctx_destroy(self.ctx)


def _served(case, seed):
    """The burst's systems: (row lengths, columns, values, x*, solver), stencils and random rows in turn.  The sizes
    go by the case, the random rows and the solutions by the seed."""
    rng = np.random.default_rng(case["nmax"])
    out = []
    for k in range(case["count"]):
        n = int(round(math.exp(rng.uniform(math.log(1000), math.log(case["nmax"])))))
        if k % 2 == 0:
            sub = {"family": "lap3d", "m": max(10, int(round(n ** (1.0 / 3.0))))}
        else:
            sub = {"family": "diagdom", "m": n}
        lens, cols, vals = _matrix(sub, seed * 100 + k)
        xs = _uniform(lens.numel(), seed * 100 + k, 7)
        out.append((lens, cols, vals, xs, "cg" if k % 2 == 0 else "bicgstab"))
    return out


def prepare(case, seed):
    st = State(case)
    kind = case["kind"]
    if kind == "serve":
        st.server = Server(st.ctx, max_slots=16)
        st.requests = []
        for lens, cols, vals, xs, solver in _served(case, seed):
            b = _product(lens, cols, vals, xs)
            st.requests.append(tuple(a.cpu().numpy() for a in (_row_ptr(lens), cols, vals, b)) + (solver,))
        return st
    if kind == "batch":
        f32 = case["precision"] == "f32"
        sizes, lens, cols, vals, off, sysid = _batch_matrix(case, seed)
        xs = _uniform(sysid.numel(), seed, 7)
        b = _product(lens, cols + off[sysid].repeat_interleave(lens), vals, xs)
        # row pointers restart at 0 in every system, which holds size + 1 of them
        ends = torch.cumsum(lens, 0)
        nnz_off = torch.zeros(case["count"] + 1, dtype=torch.int64, device=DEV)
        nnz_off[1:] = ends[off + sizes - 1]
        row_off = torch.zeros_like(nnz_off)
        row_off[1:] = torch.cumsum(sizes, 0)
        rp = torch.zeros(sysid.numel() + case["count"], dtype=torch.int32, device=DEV)
        rp[torch.arange(sysid.numel(), device=DEV) + sysid + 1] = (ends - nnz_off[sysid]).int()
        dt = torch.float32 if f32 else torch.float64
        st.B = spx.spx_batch_create(st.ctx, row_off.cpu().numpy(), nnz_off.cpu().numpy(), rp, cols, vals.to(dt),
                                    flags=spx.SPX_MIXED_SHADOW if case["precision"] == "mixed" else 0)
        st.b, st.x = b.to(dt), torch.zeros(sysid.numel(), dtype=dt, device=DEV)
        return st
    lens, cols, vals = _matrix(case, seed)
    n = lens.numel()
    rp = _row_ptr(lens)
    if kind == "solve":
        dt = torch.float32 if case["precision"] == "f32" else torch.float64
        st.b = _product(lens, cols, vals, _uniform(n, seed, 7)).to(dt)
        st.A = spx.spx_matrix_create(st.ctx, case["format"], rp, cols, vals.to(dt),
                                     flags=spx.SPX_MIXED_SHADOW if case["precision"] == "mixed" else 0)
        st.x = torch.zeros(n, dtype=dt, device=DEV)
        return st
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    st.x, st.y = _uniform(n, seed, 7).to(dt), _uniform(n, seed, 8).to(dt)
    if kind == "noalloc":
        st.rp, st.cols, st.vals = rp, cols, vals.to(dt)
    else:
        st.A = spx.spx_matrix_create(st.ctx, case["format"], rp, cols, vals.to(dt))
    return st


def run(st):
    c = st.case
    if c["kind"] == "spmv":
        if c["axpby"]:
            spx.spx_spmv_axpby(st.ctx, st.A, 0.5, st.x, 0.25, st.y)
        else:
            spx.spx_spmv(st.ctx, st.A, st.x, st.y)
        return st.y
    if c["kind"] == "noalloc":
        spx.spx_spmv_csr_noalloc(st.rp, st.cols, st.vals, st.x, st.y)
        return st.y
    if c["kind"] == "solve":
        st.x.zero_()
        spx.spx_solve(st.ctx, st.A, st.b, st.x, c["solver"], c["tol"], 20_000, restart=30, precision=c["precision"],
                      precond=None if c["precond"] == "none" else c["precond"], block_size=c["block"] or 8)
        return st.x
    if c["kind"] == "batch":
        st.x.zero_()
        spx.spx_batch_solve(st.ctx, st.B, st.b, st.x, c["count"], c["solver"], c["tol"], 20_000, c["precision"])
        return st.x
    s = st.server
    ids = [s.submit(rp, col, val, b, solver=solver, tol=c["tol"], precision="mixed")
           for rp, col, val, b, solver in st.requests]
    s.drain()
    return [s.results.pop(i)["x"] for i in ids]


# ------------------------------------------------------------------ what a pass needs, and how exact it is
def _vector_bytes(solver, v, n):
    """Vector traffic of one iteration, each vector an update needs read or written once: CG x, r, p, q;
    BiCGSTAB x, r, r^, p, v, s, t; CGS x, r, r^, p, u, q, v; GMRES(30) half the basis twice."""
    return v * n * {"cg": 9, "bicgstab": 16, "cgs": 16, "gmres": 35}[solver]


def _vector_flops(solver, n):
    """Flops of one iteration's dots and updates (an FMA counts 2)."""
    return n * {"cg": 10, "bicgstab": 24, "cgs": 19, "gmres": 65}[solver]


def _iterations(case):
    """About how many iterations a solve takes (seen at the sizes of the library's own measurements)."""
    f, m, s = case["family"], case["m"], case["solver"]
    if f == "diagdom":
        return 12
    it = {"lap2d": 3.1, "lap3d": 3.3, "pt27": 1.5, "convdiff": 2.1, "peclet": 2.3}[f] * m
    return it * (2.8 if s == "gmres" else 1.0) * (0.8 if case["precond"] == "block_jacobi" else 1.0)


def _system(n, nnz, solver, v, its):
    """Bytes and flops of a solve that streams the matrix and its vectors once per product and update."""
    products = 2 if solver in ("bicgstab", "cgs") else 1
    matrix = nnz * (v + 4) + 4 * (n + 1)
    return {"bytes": its * (products * matrix + _vector_bytes(solver, v, n)),
            "flops": its * (products * 2 * nnz + _vector_flops(solver, n))}


def work(case):
    kind = case["kind"]
    if kind in ("spmv", "noalloc"):
        v = 8 if case["dtype"] == "f64" else 4
        n, nnz = _rows(case), _nnz(case)
        index = 8 * nnz if case.get("format") == "coo" else 4 * nnz + 4 * (n + 1)
        return {"bytes": v * nnz + index + (3 if case.get("axpby") else 2) * v * n, "flops": 2 * nnz}
    if kind == "solve":
        v = 8 if case["precision"] == "f64" else 4  # mixed precision iterates on FP32
        return _system(_rows(case), _nnz(case), case["solver"], v, _iterations(case))
    if kind == "batch":
        v = 8 if case["precision"] == "f64" else 4
        n = case["count"] * (100 + case["nmax"]) // 2
        return _system(n, 5 * n, case["solver"], v, 40 if case["tol"] < 1e-5 else 20)
    n = (case["nmax"] - 1000) / math.log(case["nmax"] / 1000.0) * case["count"] / 2  # half stencils, half random rows
    a, b = _system(n, 7 * n, "cg", 4, 80), _system(n, 20 * n, "bicgstab", 4, 12)
    return {"bytes": a["bytes"] + b["bytes"], "flops": a["flops"] + b["flops"]}


def tolerance(case):
    kind = case["kind"]
    if kind in ("spmv", "noalloc"):
        # (the largest difference was 2e-5 in FP32: one row of thousands of N(0, 1) entries among short ones)
        return {"rel": 1e-15, "max": 2e-13} if case["dtype"] == "f64" else {"rel": 5e-7, "max": 1e-4}
    # a solve ends once its residual is below tol: the error of x is then a part of the matrix's condition times tol.
    # Condition 0.4 m^2 for the Laplacians (convection included) and 0.3 m^2 taken for the 27-point stencil; the part was
    # 0.009 .. 0.025 for CG and 0.3 for GMRES, whose last steps leave the smooth error; four times that is stated.
    if kind == "solve":
        f, m = case["family"], case["m"]
        if f in ("diagdom", "peclet"):
            return {"rel": 40.0 * case["tol"]}
        kappa = (0.3 if f == "pt27" else 0.4) * m * m
        return {"rel": max(10.0, {"cg": 0.1, "gmres": 1.2}.get(case["solver"], 0.4) * kappa) * case["tol"]}
    return {"rel": (40.0 if kind == "batch" else 120.0) * case["tol"]}


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return [s[3] for s in _served(case, seed)]
    if kind == "batch":
        n = int(_batch_matrix(case, seed)[0].sum())
        return _uniform(n, seed, 7)
    if kind == "solve":  # b = A x*: the solution is x*
        return _uniform(_rows(case), seed, 7)
    lens, cols, vals = _matrix(case, seed)
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    x, y = _uniform(lens.numel(), seed, 7).to(dt), _uniform(lens.numel(), seed, 8).to(dt)
    t = _product(lens, cols, vals.to(dt), x)
    return 0.5 * t + 0.25 * y.double() if case.get("axpby") else t
