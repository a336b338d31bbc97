"""Sweeps with checkpoints every 16 or 32 steps: the cell from the bins against the binary
search (needs a GB300). As in test_gpu_cell_index.py a grid value that no path can reach
moves a call from one to the other; the same cells give the same paths, 97 of them, so the
price and Delta agree to 1e-13 and the buckets to a few ulps of the largest."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

from .test_gpu_cell_index import _grids
from .test_gpu_packed import TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return lv.load()


@pytest.mark.parametrize("grid", _grids(), ids=[g[0] for g in _grids()])
@pytest.mark.parametrize("n_steps", [1, 17, 33, 41])
@pytest.mark.parametrize("k", [16, 32])
@pytest.mark.parametrize("method", [lv.LV_ADJ_REVERSE, lv.LV_ADJ_TANGENT])
def test_long_intervals_find_the_same_cells(method, k, n_steps, grid, lib):
    surf, opt = W.config_small()
    r = []
    for far in (False, True):
        sig = surf.sigma.copy()
        if far:
            sig[-1, -1] = 1.0e7                        # unreachable: t_n < 0.85 < 8/9
        s = lv.Surface.from_workload(W.Surface(grid[1], surf.time, sig), lib)
        s.set_adjoint_method(method)
        s.set_launch(128, k, 0)
        r.append(s.price_greeks(opt.S0, 0.01, opt.K, 0.85, n_steps, 97, opt.seed))
        s.close()
    got, ref = r
    for i in (0, 1):
        assert np.isfinite(ref[i]) and abs(got[i] - ref[i]) <= TOL * max(abs(ref[i]), 1e-300)
    assert np.max(np.abs(got[2] - ref[2])) <= 1e-6 * max(np.max(np.abs(ref[2])), 1e-300)
