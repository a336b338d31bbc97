"""A book whose grids and time table leave no room for the bins of irregular spot
nodes (needs a GB300): it searches for its cells, as every irregular grid did before there
were bins. 100 x 160 nodes and 3,900 steps: about 193 KB at one path per lane without the bins' 8, of 200.

The same option alone: the same paths, so price and Delta are binary64 sums of 256 equal
terms (1e-12), a bucket's binary32 sums of at most 256 paths with at most 3,900 / 160 = 25 steps
in its time row: sqrt(256 * 25) half ulps, 4.8e-6 of the largest."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

pytestmark = pytest.mark.gpu


class _Item:
    surface, stream_id, phi, K, T, n_steps, n_paths = 0, 0, 1, 100.0, 1.0, 3900, 256


def test_book_without_room_for_bins():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    lib = lv.load()
    # the smallest gap is 1/765 of the grid in ln S: 511 bins
    y = np.concatenate([np.arange(97) * 4.0, [385.0, 600.0, 765.0]])
    y[48:52] = [192.0, 193.5, 195.0, 200.0]
    spot = 100.0 * 4.0 ** ((y - 193.0) / 765.0)
    rng = np.random.Generator(np.random.PCG64(2))
    surf = W.Surface(spot, np.linspace(0.0, 1.0, 160), 0.25 + rng.uniform(-1e-3, 1e-3, size=(100, 160)))
    s = lv.Surface.from_workload(surf, lib)
    o = _Item()
    book = lv.Book([s], [o], lib)
    r = np.array(book.run(100.0, 0.01, 5))
    p, d, v = s.price_greeks(100.0, 0.01, o.K, o.T, o.n_steps, o.n_paths, 5)
    book.close()
    s.close()
    assert abs(r[0] - p) <= 1e-12 * p and abs(r[1] - d) <= 1e-12 * abs(d)
    assert np.max(np.abs(r[3:] - v.reshape(-1))) <= 4.8e-6 * np.max(np.abs(v))
