"""The launch shape read back is the one a call runs (needs a GB300): its block and
its grid as the profiler sees them, and results at that shape against the oracle on
a grid whose wide blocks keep 9,900 cells staged."""
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

from . import gpu_common as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    lib = lv.load()
    s = _surface(lib, "price")             # the profiler attaches during its first use and misses launches of it
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]):
        s.price(100.0, 0.01, 100.0, 3.0, 52, 1024, 3)
    s.close()
    return lib


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


CALLS = ["greeks", "price", "tangent", "ln-S weight", "k = 8", "three blocks"]


def _surface(lib, call):
    s = lv.Surface.from_workload(W.config_paper_shape()[0], lib)
    if call == "tangent":
        s.set_adjoint_method(lv.LV_ADJ_TANGENT)
    if call == "ln-S weight":
        s.set_interpolation(lv.LV_INTERP_LOGS)
    if call == "k = 8":
        s.set_launch(0, 8, 0)
    if call == "three blocks":
        s.set_launch(0, 0, 3)
    return s


@pytest.mark.parametrize("per_sm", [8, 512, 2048])
@pytest.mark.parametrize("call", CALLS)
def test_read_back_is_what_runs(call, per_sm, lib, tmp_path):
    import json

    import torch
    sms, n = _sms(), per_sm * _sms()
    s = _surface(lib, call)
    a = (100.0, 0.01, 100.0, 3.0, 52, n, 3)
    f = s.price if call == "price" else s.price_greeks
    f(*a)
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as prof:
        f(*a)
    prof.export_chrome_trace(str(tmp_path / "trace.json"))
    block, k, bps = s.get_call_launch(52, n, call != "price")
    s.close()
    ran = [e["args"] for e in json.loads((tmp_path / "trace.json").read_text())["traceEvents"]
           if e.get("cat") == "kernel" and "_kernel" in e["name"]]
    assert len(ran) == 1
    warps, wide = block // 32, per_sm >= 512 and call not in ("price", "k = 8", "three blocks")
    assert block == (512 if wide else 128) and (not wide or bps == 1)
    assert k == (8 if call == "k = 8" else 4)
    ppl = 1 if call != "price" or per_sm < 200 else 2                  # paths of a lane in a claimed tile
    tiles = -(-n // (32 * ppl))
    assert ran[0]["block"] == [block, 1, 1]
    assert ran[0]["grid"] == [min(bps * sms, -(-tiles // warps)), 1, 1]


def test_wide_blocks_on_a_fine_grid_against_the_oracle(lib):
    """100 x 100 grid at 512 paths per SM: one 512-thread block per SM."""
    surf, opt = W.config_large()
    opt = W.Option(**{**opt.__dict__, "n_steps": 252, "T": 1.0, "n_paths": 512 * _sms()})
    s = G.make_surface(surf, opt, lib)
    assert s.get_call_launch(opt.n_steps, opt.n_paths, True) == (512, 4, 1)
    s.close()
    G.full_parity(surf, opt, lib, label="100x100 grid, wide blocks")
