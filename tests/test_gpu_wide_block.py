"""One 512-thread block per SM against several of 128, and the forward-only
kernel at one path per lane against two (needs a GB300).

From 512 paths per SM on, a Greeks call runs one 512-thread block per SM; with
the number of blocks per SM given, it runs 128-thread blocks. A path's
arithmetic is the same in both, only the sums' order changes: the price, Delta,
rho and d V / d T are binary64 sums of at most 2^18 terms, off by less than 2^18 ulp
of the largest partial sum in the worst case and by about sqrt(2^18) ulp, 1e-13, as the
last bits fall; 1e-11 leaves room for terms of both signs. Kahan sums are binary32 with
a carried remainder: two ulps, 2^-22. A bucket takes at most 2^15 binary32 additions
between two drains: sqrt(2^15) half ulps, 1.1e-5 of the largest bucket.

Sizes: 31 and 62 cells per time row (a lane's worth and twice it, less one), one
time node, the first wide call, an odd last tile, and enough batches for every warp to
drain its buckets."""
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


def _grid(n_spot, n_time, uneven):
    rng = np.random.Generator(np.random.PCG64(5))
    gaps = rng.uniform(0.4, 1.6, size=n_spot - 1) if uneven else np.ones(n_spot - 1)
    spot = 50.0 * 4.0 ** (np.concatenate([[0.0], np.cumsum(gaps)]) / gaps.sum())
    return W.Surface(spot, np.linspace(0.0, 1.0, n_time) if n_time > 1 else np.array([0.0]),
                     rng.uniform(0.15, 0.35, size=(n_spot, n_time)))


GRIDS = [("31 cells", _grid(32, 5, False)), ("62 cells, one time node", _grid(63, 1, False)),
         ("2 cells", _grid(3, 2, False)), ("irregular", _grid(20, 10, True))]
PATHS = [512, 513, 1536, 1537]                         # per SM, and one more path than that
CALLS = ["reverse", "reverse, Kahan", "Euler on S", "extended", "tangent", "tangent, Kahan", "vanna"]


def _run(surf, opt, lib, call, ppl, narrow):
    s = lv.Surface.from_workload(surf, lib)
    s.set_paths_per_lane(ppl)
    if narrow:
        s.set_launch(0, 0, 3)
    if call == "Euler on S":
        s.set_scheme(lv.LV_SCHEME_S)
    if call.endswith("Kahan"):
        s.set_accumulation(1)
    if call.startswith("tangent"):
        s.set_adjoint_method(lv.LV_ADJ_TANGENT)
    f = {"extended": s.price_greeks_ext, "vanna": s.price_greeks_vanna}.get(call, s.price_greeks)
    try:
        return f(opt.S0, opt.r, opt.K, opt.T, opt.n_steps, opt.n_paths, opt.seed)
    except lv.LVError as e:            # both ratio methods refuse a path whose factor 1 + g_n vanishes
        assert call.startswith(("tangent", "vanna")) and "1 + g_n" in str(e)
        return e.status
    finally:
        s.close()


@pytest.mark.parametrize("grid", GRIDS, ids=[g[0] for g in GRIDS])
@pytest.mark.parametrize("per_sm", PATHS)
@pytest.mark.parametrize("ppl", [1, 2])
@pytest.mark.parametrize("call", CALLS)
def test_block_width_changes_only_the_order_of_sums(call, ppl, per_sm, grid, lib):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = per_sm * sms if per_sm % 2 == 0 else (per_sm - 1) * sms + 1
    _, opt = W.config_small()
    opt = W.Option(**{**opt.__dict__, "T": 0.85, "r": 0.01, "n_steps": 9, "n_paths": n})
    got, ref = _run(grid[1], opt, lib, call, ppl, False), _run(grid[1], opt, lib, call, ppl, True)
    if isinstance(ref, int) or isinstance(got, int):
        assert got == ref              # the same paths, the same refusal
        return
    tol = 2.0 ** -22 if call.endswith("Kahan") else 1e-11
    for i, (a, b) in enumerate(zip(got, ref)):
        if i == 2:
            assert np.all(np.isfinite(b)) and np.max(np.abs(b)) > 0
            assert np.max(np.abs(a - b)) <= 1.1e-5 * np.max(np.abs(b))
        else:
            assert np.isfinite(b) and abs(a - b) <= tol * abs(b), (i, a, b)


@pytest.mark.parametrize("n_paths", [1, 31, 33, 64, 97, 4096])
@pytest.mark.parametrize("grid", GRIDS, ids=[g[0] for g in GRIDS])
@pytest.mark.parametrize("scheme", [lv.LV_SCHEME_LOG, lv.LV_SCHEME_S])
def test_forward_only_lanes_give_the_same_paths(scheme, grid, n_paths, lib):
    """As in test_gpu_packed.py: binary64 sums of the same payoffs, 1e-13 apart at a few
    hundred paths; 4,096 paths sum to within 64 ulps."""
    _, opt = W.config_small()
    p = []
    for ppl in (1, 2):
        s = lv.Surface.from_workload(grid[1], lib)
        s.set_scheme(scheme)
        s.set_paths_per_lane(ppl)
        p.append(s.price(opt.S0, 0.01, opt.K, 0.85, 9, n_paths, opt.seed)[0])
        s.close()
    assert np.isfinite(p[0]) and abs(p[0] - p[1]) <= 1e-13 * max(abs(p[0]), 1e-300)
