"""The binary64 run on a device with little memory left (needs a GB300).

Its tapes take up to 2 GiB for the threads of the whole chip; where the device has
less, fewer threads take the paths in more rounds. The values are sums of the same
binary64 terms in another order: 77,824 of them, below 1e-11 of the largest sum."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

pytestmark = pytest.mark.gpu


def test_tapes_shrink_to_the_memory_there_is():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    lib = lv.load()
    surf, opt = W.config_small()
    out = []
    for fill in (False, True):
        s = lv.Surface.from_workload(surf, lib)
        d = torch.zeros(3 + s.IJ, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        held = None
        if fill:            # 1 GiB stays free: the tapes of 77,824 threads and 900 steps are 1.8 GiB
            torch.cuda.empty_cache()
            held = torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")
        s.price_greeks_fp64_device(opt.S0, opt.r, opt.K, opt.T, 900, 77824, opt.seed, d.data_ptr())
        torch.cuda.synchronize()
        out.append(d.cpu().numpy())
        del held
        torch.cuda.empty_cache()
        s.close()
    assert np.all(np.isfinite(out[0])) and np.max(np.abs(out[0][3:])) > 0
    for part in (slice(0, 1), slice(1, 2), slice(2, 3), slice(3, None)):
        assert np.max(np.abs(out[1][part] - out[0][part])) <= 1e-11 * np.max(np.abs(out[0][part]))
