"""spx_spmv_csr_noalloc where its two routes can go wrong: one tile, whole and
ragged tiles (1024 row ends and nonzeros on the one-launch route), rows that run
over many tiles, empty rows, the size at which the tile map is launched instead,
calls of different sizes and types that follow one another on the scratch they
share, and replays of a captured call.  Against the CPU oracle, row by row."""
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


def _rows(lens, ncols, seed):
    """Rows of the given lengths, random columns, N(0, 1) values."""
    rng = np.random.default_rng(seed)
    rp = np.zeros(len(lens) + 1, np.int32)
    rp[1:] = np.cumsum(lens)
    return rp, rng.integers(0, ncols, rp[-1]).astype(np.int32), rng.standard_normal(rp[-1])


CASES = {
    "one_entry": _rows([1], 1, 0),
    "one_tile": _rows([7] * 128, 128, 1),                 # 128 + 896 = 1024 items: exactly one tile
    "one_tile_and_one": _rows([7] * 127 + [9], 128, 2),   # 1025 or more: a second tile
    "empty_rows": _rows([0, 5, 0, 0, 3] * 700, 3500, 3),
    "one_long_row": _rows([9000], 4000, 4),               # one row over nine tiles
    "long_rows": _rows([3] * 500 + [6000] + [2] * 800 + [5000, 1, 7000] + [0] * 300, 2000, 5),
    "all_tiles": synth.powerlaw(60000, mean=16, max_len=6000, seed=6),
    "stencil": synth.laplace3d_7pt(41),
    "map_route": synth.laplace3d_7pt(64),                 # 2.07 M items: more tiles than the device holds blocks
}


def _call(spx, name, dt, seed):
    rp, col, val = CASES[name]
    n = rp.shape[0] - 1
    ncols = max(n, int(col.max()) + 1)
    xh = synth.uniform_vector(ncols, seed)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
    args = t(rp), t(col), t(val).to(dt), t(xh).to(dt)
    y = torch.full((n,), float("nan"), dtype=dt, device=DEV)
    spx.spx_spmv_csr_noalloc(*args, y, ncols=ncols)
    return args, y, xh


def _check(name, dt, xh, y):
    rp, col, val = CASES[name]
    r = (lambda a: a.astype(np.float32).astype(np.float64)) if dt == torch.float32 else (lambda a: a)
    ref, bound = oracle.spmv_csr(rp, col, r(val), r(xh)), oracle.spmv_absbound(rp, col, r(val), r(xh))
    assert_spmv_close(y.double().cpu().numpy(), ref, bound, TOL["f32" if dt == torch.float32 else "f64"])


@pytest.mark.parametrize("dt", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", sorted(CASES))
def test_sizes(spx, name, dt):
    _, y, xh = _call(spx, name, dt, 3)
    _check(name, dt, xh, y)


def test_calls_in_a_row(spx):
    """The scratch keeps the previous call's flags and carries: sizes, types and routes follow one another unsynchronised."""
    order = [("long_rows", torch.float64), ("map_route", torch.float32), ("one_long_row", torch.float32),
             ("all_tiles", torch.float64), ("one_long_row", torch.float64), ("map_route", torch.float64),
             ("long_rows", torch.float32), ("one_entry", torch.float64), ("long_rows", torch.float64)]
    out = [(n, dt) + _call(spx, n, dt, k) for k, (n, dt) in enumerate(order)]
    torch.cuda.synchronize()
    side = torch.cuda.Stream()  # then on two streams in turn, each call ordered after the one before
    for k, (n, dt) in enumerate(order):
        with torch.cuda.stream(side if k % 2 else torch.cuda.default_stream()):
            out.append((n, dt) + _call(spx, n, dt, k))
            torch.cuda.current_stream().synchronize()
    for n, dt, _, y, xh in out:
        _check(n, dt, xh, y)


@pytest.mark.parametrize("name", ["long_rows", "all_tiles"])
def test_captured(spx, name):
    args, y, xh = _call(spx, name, torch.float64, 5)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        spx.spx_spmv_csr_noalloc(*args, y, ncols=args[3].numel(), stream=s)
    for seed in (11, 12, 13):
        x2 = synth.uniform_vector(args[3].numel(), seed)
        args[3].copy_(torch.from_numpy(x2))
        y.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        _check(name, torch.float64, x2, y)
        _, y2, xh2 = _call(spx, "map_route", torch.float64, seed)  # a direct call of another size after a replay
        torch.cuda.synchronize()
        _check("map_route", torch.float64, xh2, y2)


@pytest.mark.parametrize("name", ["one_tile_and_one", "long_rows", "map_route"])
def test_after_overlapping_calls(spx, name):
    """What overlapping calls can leave in the scratch (their tile map, carries and flags, a captured call's counts)
    changes no later call: direct ones, on two streams in turn, and the replays of a captured one."""
    args, y, xh = _call(spx, name, torch.float64, 5)
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=s):
        spx.spx_spmv_csr_noalloc(*args, y, ncols=args[3].numel(), stream=s)
    for k in range(4):
        with torch.cuda.stream(s if k % 2 else torch.cuda.default_stream()):
            spx.spx_selftest_noalloc_spoil()
            if k >= 2:
                y.fill_(float("nan"))
                g.replay()
                torch.cuda.synchronize()
                _check(name, torch.float64, xh, y)
            _, y1, xh1 = _call(spx, name, torch.float32, 20 + k)
            _, y2, xh2 = _call(spx, "long_rows", torch.float64, 30 + k)
            torch.cuda.synchronize()
        _check(name, torch.float32, xh1, y1)
        _check("long_rows", torch.float64, xh2, y2)
