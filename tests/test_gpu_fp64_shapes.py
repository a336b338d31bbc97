"""The binary64 adjoint's launch shapes (needs a GB300): one path, calls whose
blocks are smaller than 512 threads, several rounds of a block's paths, and a step
count whose tapes hold fewer threads than the SMs take. The oracle's definition in
binary64 at the tolerance of test_gpu_fp64.py (both sides round every step of a
path once or twice, 1e-16 of the state each)."""
import numpy as np
import pytest

import oracle
import workloads as W
from paper_2002_02481_gb300 import build, lv

from .test_gpu_fp64 import TOL, _fp64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return lv.load()


@pytest.mark.parametrize("n_steps, n_paths", [(1, 1), (3, 31), (5, 152 * 32 + 1), (4, 152 * 512 + 77), (8192, 20000)])
def test_launch_shapes(n_steps, n_paths, lib):
    surf, opt = W.config_paper_shape()
    opt = W.Option(**{**opt.__dict__, "n_steps": n_steps, "n_paths": n_paths, "K": 80.0})
    g = _fp64(lib, surf, opt)
    ref = oracle.finalize(oracle.run_sums(surf, opt), opt.n_paths, opt.S0, surf.n_spot * surf.n_time)
    for k in (0, 1):
        assert abs(g[k] - ref[k]) <= TOL * max(abs(ref[k]), 1e-300), (k, g[k], ref[k])
    assert np.max(np.abs(g[3:] - ref[3:])) <= TOL * max(np.max(np.abs(ref[3:])), 1e-300)
