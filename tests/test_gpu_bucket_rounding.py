"""Rounding of the binary32 bucket sums in 512-thread blocks (needs a GB300).

A call of 512 paths per SM runs one 512-thread block per SM, and nothing is
drained before its end: a bucket's binary32 sum takes every live path of the warps that
share it. The same call in 32-thread blocks puts one 32-path tile into a block's
buckets, and the blocks' sums are added in binary64: with a quarter of the paths of a
128-thread block in a sum, that is the reference. A random sum's rounding grows as the
number of its terms, so the reference is off by a quarter of what the 128-thread blocks
are and changes either distance by 3 %. Warps that share a bucket four by four put as
many paths into it as a 128-thread block's do: the two distances have the same
distribution. Sixteen sharing one would be off four times as far.

The geometric mean of the distances' ratio over 72 calls (three grids, 24 seeds): the
logarithm of a distance of two degrees of freedom, as few as a coarse grid's buckets
can have, has a standard deviation of pi / sqrt(24) = 0.64, that of a ratio 0.91 and the
mean of 72 of them 0.107. 1.5 is four of these."""
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


def _grid(n_spot, n_time):
    rng = np.random.Generator(np.random.PCG64(7))
    spot = 50.0 * 4.0 ** np.linspace(0.0, 1.0, n_spot)
    sig = 0.25 - 0.1 * np.log(spot / 100.0)[:, None] + rng.normal(0.0, 0.005, size=(n_spot, n_time))
    return W.Surface(spot, np.linspace(0.0, 1.0, n_time), sig)


GRIDS = [_grid(5, 2), _grid(12, 2), _grid(20, 10)]
CALLS = ["reverse", "tangent", "extended", "vanna"]


def _buckets(surf, opt, lib, call, launch):
    s = lv.Surface.from_workload(surf, lib)
    s.set_paths_per_lane(1)
    if launch:
        s.set_launch(*launch)
    if call == "tangent":
        s.set_adjoint_method(lv.LV_ADJ_TANGENT)
    f = {"extended": s.price_greeks_ext, "vanna": s.price_greeks_vanna}.get(call, s.price_greeks)
    try:
        return np.array(f(opt.S0, opt.r, opt.K, opt.T, opt.n_steps, opt.n_paths, opt.seed)[2]).reshape(-1)
    finally:
        s.close()


@pytest.mark.parametrize("call", CALLS)
def test_wide_blocks_round_as_narrow_ones(call, lib):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _, opt = W.config_small()
    ratios = []
    for surf in GRIDS:
        for seed in range(1, 25):
            o = W.Option(**{**opt.__dict__, "n_steps": 104, "n_paths": 512 * sms, "seed": seed})
            ref = _buckets(surf, o, lib, call, (32, 4, 0))
            wide, narrow = (np.linalg.norm(_buckets(surf, o, lib, call, launch) - ref) for launch in (None, (0, 0, 4)))
            assert narrow > 0.0
            ratios.append(wide / narrow)
    assert np.exp(np.mean(np.log(ratios))) <= 1.5, np.exp(np.mean(np.log(ratios)))


def test_the_cell_the_paths_start_in(lib):
    """15 steps on 95 x 22 nodes, 5,500 paths per SM: three quarters of the vegas' 2-norm is one
    node of the cell of S0, where every path ends its sweep. A binary32 sum of n terms of one
    sign is off by n^1.5. 512-thread blocks sum there by lanes, 32 sums of a 32nd of the terms:
    a 32nd of a 128-thread block's distance. No other node takes more than a third of that one's terms;
    theirs, the same in both, come to less than a fifth (3^-1.5) of it. The reference: the same paths in
    ranges that put one 32-path tile into a 32-thread block, added in binary64. The geometric
    mean of 24 ratios has a spread of 0.91 / sqrt(24) = 0.19 in its logarithm; 0.5 is more than three of
    them from a fifth and from 1."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.Generator(np.random.PCG64(3))
    spot = 50.0 * 4.0 ** np.linspace(0.0, 1.0, 95)
    sig = 0.25 - 0.1 * np.log(spot / 100.0)[:, None] + rng.normal(0.0, 0.005, size=(95, 22))
    surf = W.Surface(spot, np.linspace(0.0, 5.0, 22), sig)
    n, step, ratios = 5500 * sms, 256 * sms, []
    s = lv.Surface.from_workload(surf, lib)
    s.set_launch(32, 4, 0)
    d = torch.zeros(3 + s.IJ, dtype=torch.float64, device="cuda")
    for seed in range(1, 25):
        ref = np.zeros(s.IJ)
        for p in range(0, n, step):
            s.price_greeks_sums_device(100.0, 0.03, 100.0, 4.5, 15, p, min(p + step, n), seed, 0, d.data_ptr())
            ref += d.cpu().numpy()[3:]
        ref /= n
        o = W.Option(S0=100.0, r=0.03, K=100.0, T=4.5, n_steps=15, n_paths=n, seed=seed)
        wide, narrow = (np.linalg.norm(_buckets(surf, o, lib, "reverse", launch) - ref) for launch in (None, (0, 0, 4)))
        ratios.append(wide / narrow)
    s.close()
    assert np.exp(np.mean(np.log(ratios))) <= 0.5, np.exp(np.mean(np.log(ratios)))
