"""The binary64 run on spot nodes whose gaps have no inverse in binary64 (needs a
GB300). Every quantity of a call scales with the spot: nodes, S0 and strike 2^1023 times
smaller give 2^1023 times smaller prices and vegas and the same Delta. Spots near 2^-1020
have an ln S of -707, whose binary64 rounding is 6e-14: over seventeen steps 2.5e-13 of a
spot, ten times that of a payoff at the money, either way on 4,096 paths; prices of 2^-1024
keep 50 bits. 1e-11 covers both."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

pytestmark = pytest.mark.gpu


def test_gaps_without_an_inverse():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    lib = lv.load()
    base = 2.0 ** -1020 * np.array([0.75, 0.875, 0.953125, 1.0, 1.0625, 1.1875, 1.375])
    rng = np.random.Generator(np.random.PCG64(4))
    sig = rng.uniform(0.2, 0.3, size=(7, 4))
    out = []
    for up in (1.0, 2.0 ** 1023):
        spot = base * up
        s = lv.Surface.from_workload(W.Surface(spot, np.linspace(0.0, 1.0, 4), sig), lib)
        d = torch.zeros(3 + s.IJ, dtype=torch.float64, device="cuda")
        s.price_greeks_fp64_device(float(2.0 ** -1020 * 1.03125 * up), 0.01, float(2.0 ** -1020 * up), 1.0, 17, 4096, 3,
                                   d.data_ptr())
        v = d.cpu().numpy()
        s.close()
        out.append((v[0] / up, v[1], v[3:] / up))
    (p, dl, v), (p1, dl1, v1) = out
    assert p1 > 0.0 and abs(p - p1) <= 1e-11 * p1
    assert abs(dl - dl1) <= 1e-11 * abs(dl1)
    assert np.max(np.abs(v1)) > 0.0 and np.max(np.abs(v - v1)) <= 1e-11 * np.max(np.abs(v1))
