"""Irregular grids with more than two nodes in a bin (needs a GB300): the search among a
bin's cells against the search among all. As in test_gpu_cell_index.py a grid value that no
path can reach moves a call to the latter; the same cells give the same paths, 97 of them,
so the price and Delta agree to 1e-13 and the buckets to a few ulps of the largest.

Grids: nodes a factor 1e-6 apart (one binary32 ulp of a spot is 6e-8) beside wide gaps, a
thousand nodes, a grid within half a percent, whose bins are as narrow as they may be."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

from .test_gpu_cell_index import _run
from .test_gpu_packed import READINGS, TOL

pytestmark = pytest.mark.gpu

CALLS = ["price", "one path per lane", "two paths per lane", "k = 8", "extended", "tangent", "vanna"]


def _grids():
    rng = np.random.Generator(np.random.PCG64(8))
    near = 100.0 * (1.0 + 1e-6 * np.arange(-20, 20))
    return [("forty nodes in a bin", np.sort(np.concatenate([near, [50.0, 70.0, 90.0, 99.0, 101.0, 130.0, 200.0]]))),
            ("a thousand nodes", 50.0 * 4.0 ** np.sort(rng.uniform(0.0, 1.0, size=1000))),
            ("half a percent", 99.75 + 0.5 * np.sort(np.concatenate([[0.0, 1.0], rng.uniform(0.0, 1.0, size=62)])))]


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return lv.load()


def _surfaces(spot):
    rng = np.random.Generator(np.random.PCG64(1))
    sig = 0.2 - 0.05 * np.log(spot / 100.0)[:, None] + rng.uniform(0.0, 1e-7, size=(spot.size, 10))
    far = sig.copy()
    far[-1, -1] = 1.0e7                                # unreachable: t_n < 0.85 < 8/9
    return [W.Surface(spot, np.linspace(0.0, 1.0, 10), s) for s in (sig, far)]


@pytest.mark.parametrize("grid", _grids(), ids=[g[0] for g in _grids()])
@pytest.mark.parametrize("n_steps", [1, 5, 41])
@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("reading", READINGS, ids=[r[2] for r in READINGS])
def test_a_bins_cells_are_all_it_needs(reading, call, n_steps, grid, lib):
    if reading[2] != "main reading" and call == "vanna":
        pytest.skip("main reading only")
    _, opt = W.config_small()
    opt = W.Option(**{**opt.__dict__, "T": 0.85, "r": 0.01, "n_steps": n_steps, "n_paths": 97})
    got, ref = (_run(s, opt, lib, reading, call) for s in _surfaces(grid[1]))
    assert np.isfinite(ref[0]) and abs(got[0] - ref[0]) <= TOL * max(abs(ref[0]), 1e-300)
    if call != "price":
        assert abs(got[1] - ref[1]) <= TOL * max(abs(ref[1]), 1e-300)
        assert np.max(np.abs(got[2] - ref[2])) <= 1e-6 * max(np.max(np.abs(ref[2])), 1e-300)


class _Item:
    surface, stream_id, phi, K, T, n_steps, n_paths = 0, 3, 1, 100.0, 0.85, 41, 97


@pytest.mark.parametrize("grid", _grids(), ids=[g[0] for g in _grids()])
def test_books_and_diagnostics(grid, lib):
    out = []
    for surf in _surfaces(grid[1]):
        s = lv.Surface.from_workload(surf, lib)
        book = lv.Book([s], [_Item()], lib)
        r = np.array(book.run(100.0, 0.01, 7))
        out.append((r, s.debug_paths(100.0, 0.01, 100.0, 0.85, 41, 7, 0, 97)[:3]))
        book.close()
        s.close()
    (r, d), (r1, d1) = out
    assert abs(r[0] - r1[0]) <= TOL * r1[0] and abs(r[1] - r1[1]) <= TOL * abs(r1[1])
    assert np.max(np.abs(r[3:] - r1[3:])) <= 1e-6 * np.max(np.abs(r1[3:]))
    for a, b in zip(d, d1):
        np.testing.assert_array_equal(a, b)
