"""Time weights of steps far past a narrow last cell (needs a GB300): the weight is 1
there also where (t - tau_j) / (tau_{j+1} - tau_j) overflows binary64."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gap", [1e-280, 1e-289, 1e-300, 5e-324])
@pytest.mark.parametrize("T", [1.0, 1e30, 1e300])
def test_weight_past_a_narrow_cell(T, gap):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    s = lv.Surface.from_workload(W.Surface(np.array([80.0, 125.0]), np.array([0.0, gap]), np.full((2, 2), 0.2)), lv.load())
    j, v = s.time_table(T, 10)
    s.close()
    assert np.all(j == 0) and v[0] == 0.0 and np.all(v[1:] == 1.0)
