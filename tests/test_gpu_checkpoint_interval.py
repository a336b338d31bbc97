"""Checkpoints every 16 and 32 steps against every 4 (needs a GB300).

At 16 steps a segment's factors are all held at once; at 32 the segment is run
forward once more for the state before each block of four steps, and its blocks are
swept last to first; at 4 every block has its checkpoint. The states are the same values either way, so each path's x_bar_0
is the same bit for bit: on 97 paths the price and Delta, binary64 sums, agree to
1e-13, and the binary32 bucket sums to a few ulps of the largest (as in
test_gpu_cell_index.py). Step counts lie at the edges of blocks and segments."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return lv.load()


@pytest.mark.parametrize("n_steps", [1, 3, 4, 5, 15, 16, 17, 20, 31, 32, 33, 36, 37, 64, 65, 100])
@pytest.mark.parametrize("kahan", [0, 1])
@pytest.mark.parametrize("k", [16, 32])
def test_long_intervals_sweep_the_same_paths(k, kahan, n_steps, lib):
    surf, opt = W.config_small()
    r = []
    for kk in (4, k):
        s = lv.Surface.from_workload(surf, lib)
        s.set_launch(128, kk, 0)
        s.set_paths_per_lane(1)
        s.set_accumulation(kahan)
        r.append(s.price_greeks(opt.S0, 0.01, opt.K, 0.85, n_steps, 97, opt.seed))
        s.close()
    ref, got = r
    tol = 2.0 ** -22 if kahan else 1e-13               # Kahan: binary32 sums with a carried remainder
    for i in (0, 1):
        assert np.isfinite(ref[i]) and abs(got[i] - ref[i]) <= tol * max(abs(ref[i]), 1e-300)
    assert np.max(np.abs(got[2] - ref[2])) <= 1e-6 * max(np.max(np.abs(ref[2])), 1e-300)
