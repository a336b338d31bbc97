"""The straight-line time loops and their cell index against the general loop
(needs a GB300).

A call whose cell index is bounded below 2^22 on every path takes the index
from an addition rounded down (the cell itself on a log-spaced grid, a bin of
at most two nodes on another one), inside loops without a bound check; any other
call takes it from a float-to-integer conversion or a binary search, inside
loops that check every step. A grid value that no path can reach (the last time
row, at a maturity inside the time cell before it) moves a call from one to the
other without touching any path: both must then give every path the same
value, bit for bit. As in test_gpu_packed.py, on at most a few hundred paths
the price moves by less than 1e-13 under another summation order and by 1e-8 /
n_paths when one path differs by an ulp. Step counts straddle the blocks of
four steps."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

from .test_gpu_packed import READINGS, TOL

pytestmark = pytest.mark.gpu

CALLS = ["price", "one path per lane", "two paths per lane", "k = 8", "extended", "tangent", "tangent pairs", "vanna",
         "vanna pairs"]


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return lv.load()


def _run(surf, opt, lib, reading, call):
    s = lv.Surface.from_workload(surf, lib)
    s.set_interpolation(reading[0])
    s.set_scheme(reading[1])
    if call in ("two paths per lane", "tangent pairs", "vanna pairs"):
        s.set_paths_per_lane(2)
    elif call != "price":
        s.set_paths_per_lane(1)
    if call == "k = 8":
        s.set_launch(128, 8, 0)
    if call.startswith("tangent"):
        s.set_adjoint_method(lv.LV_ADJ_TANGENT)
    a = (opt.S0, opt.r, opt.K, opt.T, opt.n_steps, opt.n_paths, opt.seed)
    f = {"price": s.price, "extended": s.price_greeks_ext, "vanna": s.price_greeks_vanna,
         "vanna pairs": s.price_greeks_vanna}.get(call, s.price_greeks)
    r = f(*a)
    s.close()
    return r


def _grids():
    """20 x 10 grid, log-spaced; the same values on irregular nodes (bins); on
    nodes with gaps between 1 and 400 of the smallest (up to 512 bins); on two
    spot nodes 0.2 % off a log-spaced grid's, S0 itself a node. The last time
    cell is [8/9, 1] in all of them."""
    surf, _ = W.config_small()
    rng = np.random.Generator(np.random.PCG64(11))
    gaps = rng.uniform(0.4, 1.6, size=19)
    uneven = 50.0 * 4.0 ** (np.concatenate([[0.0], np.cumsum(gaps)]) / gaps.sum())
    tight = np.concatenate([np.linspace(98.0, 102.0, 15), [50.0, 70.0, 130.0, 160.0, 200.0]])
    off = surf.spot.copy()
    off[[7, 12]] *= 1.002
    off[9] = 100.0
    return [("log-spaced", surf.spot), ("irregular", uneven), ("tight around S0", np.sort(tight)),
            ("S0 a node", off)]


@pytest.mark.parametrize("grid", _grids(), ids=[g[0] for g in _grids()])
@pytest.mark.parametrize("n_steps", [1, 3, 5, 8, 41])
@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("reading", READINGS, ids=[r[2] for r in READINGS])
def test_both_loops_give_the_same_paths(reading, call, n_steps, grid, lib):
    if reading[2] != "main reading" and (call.startswith("vanna") or call == "tangent pairs"):
        pytest.skip("main reading only")
    surf, opt = W.config_small()
    surf = W.Surface(grid[1], surf.time, surf.sigma)
    opt = W.Option(**{**opt.__dict__, "T": 0.85, "r": 0.01, "n_steps": n_steps, "n_paths": 97})
    far = W.Surface(surf.spot, surf.time, surf.sigma.copy())
    far.sigma[-1, -1] = 1.0e7                          # unreachable: t_n < 0.85 < 8/9
    got, ref = _run(surf, opt, lib, reading, call), _run(far, opt, lib, reading, call)
    scale = max(abs(ref[0]), 1e-300)
    assert np.isfinite(ref[0]) and abs(got[0] - ref[0]) <= TOL * scale
    if call != "price":
        assert abs(got[1] - ref[1]) <= TOL * max(abs(ref[1]), 1e-300)
        # binary32 bucket sums of 97 paths in another order: a few ulps of the largest
        assert np.max(np.abs(got[2] - ref[2])) <= 1e-6 * max(np.max(np.abs(ref[2])), 1e-300)
