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


def test_a_block_asked_for_is_kept(lib):
    """128 threads are 128 threads at any path count; 0 is the default's choice."""
    s = _surface(lib, "greeks")
    n = 2048 * _sms()
    assert s.get_call_launch(52, n)[0] == 512
    s.set_launch(128, 4, 0)
    assert s.get_call_launch(52, n)[0] == 128
    s.set_launch(0, 4, 0)
    assert s.get_call_launch(52, n)[0] == 512
    s.close()


def test_tuner_times_the_default_too(lib, tmp_path, monkeypatch):
    """What it keeps is what a later call and a later handle run, and what lv_set_launch makes of its block."""
    monkeypatch.setenv("LV_TUNE_CACHE", str(tmp_path / "tune.txt"))
    n = 2048 * _sms()
    s = _surface(lib, "greeks")
    block, k, _ = s.tune(100.0, 0.01, 100.0, 3.0, 52, n, 3)
    assert block in (0, 64, 128)
    shape = s.get_call_launch(52, n)
    assert shape[0] == (block or 512) and shape[1] == k
    for keep in (lambda t: None, lambda t: (t.set_launch(block, k, 0), t.set_paths_per_lane(s.get_paths_per_lane(52, n)))):
        t = _surface(lib, "greeks")
        keep(t)
        assert t.get_call_launch(52, n) == shape
        t.close()
    s.close()


@pytest.mark.parametrize("line,block", [("128 4 2 0", 512), ("128 4 2 1", 128), ("0 4 2 1", 512), ("64 4 2 0", 64)])
def test_lines_of_a_tune_cache(line, block, lib, tmp_path, monkeypatch):
    """A line of 128 threads that was not timed against 512 leaves a large call the default."""
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("LV_TUNE_CACHE", str(cache))
    s = _surface(lib, "greeks")
    s.tune(100.0, 0.01, 100.0, 3.0, 52, 4096, 3)
    cache.write_text(cache.read_text().split()[0] + f" {line} 1.0\n")
    t = _surface(lib, "greeks")
    assert t.get_call_launch(52, 2048 * _sms())[0] == block
    s.close()
    t.close()


def test_forward_only_calls_keep_half_the_resident_blocks(lib):
    """The search for the blocks per SM that leave the last round fullest stays in the upper half."""
    s = _surface(lib, "price")
    occ = s.get_launch(52, False)[2]
    for tiles in [*range(1, 400, 7), *range(1216, 60000, 97), 32268, 34049, 56048]:
        assert 2 * s.get_call_launch(52, 64 * tiles, False)[2] >= occ, tiles
    s.close()


def test_tangent_ratio_runs_the_same_at_every_interval(lib):
    """It keeps no checkpoints: k = 16 and 32 leave it its cells and its 512-thread blocks."""
    n = 1024 * _sms()
    out = []
    for k in (4, 16, 32):
        s = _surface(lib, "tangent")
        s.set_launch(0, k, 0)
        assert s.get_call_launch(52, n)[0] == 512
        out.append(s.price_greeks(100.0, 0.01, 100.0, 3.0, 52, n, 3))
        s.close()
    for p, d, _ in out[1:]:
        assert abs(p - out[0][0]) <= 1e-12 * p and abs(d - out[0][1]) <= 1e-12 * abs(d)


def test_two_paths_per_lane_from_six_pairs_a_warp(lib):
    s = _surface(lib, "greeks")
    assert [s.get_paths_per_lane(52, n) for n in (6144 * _sms() - 1, 6144 * _sms())] == [1, 2]
    s.close()


@pytest.mark.parametrize("n_time", [80, 84, 88, 100])
def test_grids_around_the_staging_limit(n_time, lib):
    """60 spot nodes: 80 and 84 time rows fit beside four blocks' limit of 55 KB, 88 and 100 are read through L1."""
    opt = W.Option(S0=100.0, r=0.01, K=100.0, T=3.0, n_steps=40, n_paths=2048, seed=6)
    G.full_parity(W.seeded_skew_surface(4, n_spot=60, n_time=n_time), opt, lib, label=f"60 x {n_time}")
