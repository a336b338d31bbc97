"""Nothing is lost between a bucket's additions and its drains (needs a GB300).

While one warp takes a bucket's sums others keep adding to it. On a grid of two to
sixteen cells every path adds to the same few buckets, and a call of 2^20 paths drains them
about three times in each of an SM's four arrays, some 2,000 sums in all. The same paths in
ranges of fewer than 512 per SM run one tile a warp and drain nothing; their sums added
in binary64 are the reference. A bucket's binary32 sum takes at most 2^11 additions
between drains and is off by sqrt(2^11) half ulps, 2.7e-6; 2,000 of these that fall
either way leave 6e-8 of the total, 1e-6 with terms of both signs. One lost sum is 5e-4 of a
bucket's total."""
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


@pytest.mark.parametrize("n_spot,n_time", [(3, 2), (5, 5)])
@pytest.mark.parametrize("acc", [lv.LV_ACC_FP64, lv.LV_ACC_KAHAN])
@pytest.mark.parametrize("method", [lv.LV_ADJ_REVERSE, lv.LV_ADJ_TANGENT])
def test_drains_lose_nothing(method, acc, n_spot, n_time, lib):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    spot = 50.0 * 4.0 ** np.linspace(0.0, 1.0, n_spot)
    surf = W.Surface(spot, np.linspace(0.0, 1.0, n_time), np.full((n_spot, n_time), 0.25))
    s = lv.Surface.from_workload(surf, lib)
    s.set_accumulation(acc)
    s.set_adjoint_method(method)
    n, step = 1 << 20, 511 * sms
    args = (100.0, 0.01, 100.0, 1.0, 52)
    d = torch.zeros(3 + s.IJ, dtype=torch.float64, device="cuda")
    ref = np.zeros(3 + s.IJ)
    for p in range(0, n, step):
        s.price_greeks_sums_device(*args, p, min(p + step, n), 9, 0, d.data_ptr())
        ref += d.cpu().numpy()
    s.price_greeks_sums_device(*args, 0, n, 9, 0, d.data_ptr())
    got = d.cpu().numpy()
    s.close()
    top = np.max(np.abs(ref[3:]))
    assert top > 0.0 and np.max(np.abs(got[3:] - ref[3:])) <= 1e-6 * top
