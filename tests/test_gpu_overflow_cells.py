"""Spots above the binary32 range on an irregular grid (needs a GB300).

Every spot at or above the last node lies in the last cell, I - 2, an infinite
one too: a path of the log-Euler scheme passes y = log2 S = 128 and may come back.
The cell from the bin table must be the binary search's there as anywhere. A grid
value that no path can reach (the last time row, at a maturity inside the time cell before
it) moves a call to the search without touching any path, as in test_gpu_cell_index.py,
so both calls sum the same terms: price and Delta in binary64 (4,096 terms in
another order, below 1e-11), each bucket in binary32 sums of at most 32 paths (one warp
a block) with up to 16 flushes each: sqrt(2^9) half ulps, 1.4e-6 of the largest bucket;
4,096 paths in the book's one item: sqrt(2^16) half ulps, 1.6e-5.

Log-Euler: a put struck far below S0 = 2e38 at volatilities of 2 to 2.6 is in the money on
about 600 of 4,096 paths, of which one in ten was above 2^128 on its way. Euler on S, where
no path comes back from infinity: a put just below S0 at volatilities of 0.3 to 0.4, which
keep spots positive; one path in twenty leaves the range."""
import numpy as np
import pytest

import workloads as W
from paper_2002_02481_gb300 import build, lv

from .test_gpu_packed import READINGS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    build.build()
    return lv.load()


def _surface(n_spot, n_time, far=False, seed=3, lo=2.0, hi=2.6):
    rng = np.random.Generator(np.random.PCG64(seed))
    gaps = rng.uniform(0.4, 1.6, size=n_spot - 1)
    spot = 1e36 * 300.0 ** (np.concatenate([[0.0], np.cumsum(gaps)]) / gaps.sum())
    sig = rng.uniform(lo, hi, size=(n_spot, n_time))
    if far:
        sig[-1, -1] = 1.0e7                            # unreachable: t_n < 0.85 < 8/9
    return W.Surface(spot, np.linspace(0.0, 1.0, n_time), sig)


OPT = W.Option(S0=2e38, r=0.01, K=2e36, T=0.85, n_steps=16, n_paths=4096, seed=5, phi=-1)


def _close(got, ref, tol):
    """The same values; where the search's are no numbers (on 100 x 100 rough nodes adjoints
    overflow: S d sigma / d S is above 10), the same ones are none."""
    assert np.isfinite(ref[0]) and ref[0] > 0.0
    np.testing.assert_allclose(got[:2], ref[:2], rtol=1e-11)
    top = np.max(np.abs(ref[2][np.isfinite(ref[2])]))
    assert top > 0.0
    np.testing.assert_allclose(got[2], ref[2], rtol=0.0, atol=tol * top)


@pytest.mark.parametrize("n_spot,n_time", [(5, 10), (20, 10), (100, 100)])
@pytest.mark.parametrize("ppl", [1, 2])
@pytest.mark.parametrize("reading", READINGS, ids=[r[2] for r in READINGS])
def test_infinite_spots_stay_in_the_last_cell(reading, ppl, n_spot, n_time, lib):
    on_s = reading[1] == lv.LV_SCHEME_S
    a = (OPT.S0, OPT.r, 1.9e38 if on_s else OPT.K, OPT.T, OPT.n_steps, OPT.n_paths, OPT.seed)
    out = []
    for far in (False, True):
        s = lv.Surface.from_workload(_surface(n_spot, n_time, far, 3, *((0.3, 0.4) if on_s else (2.0, 2.6))), lib)
        s.set_option_type(-1)
        s.set_interpolation(reading[0])
        s.set_scheme(reading[1])
        s.set_launch(32, 4, 0)
        s.set_paths_per_lane(ppl)
        out.append(s.price_greeks(*a))
        assert abs(s.price(*a)[0] - out[-1][0]) <= 1e-11 * out[-1][0]
        s.close()
    _close(*out, 1.4e-6)


class _Item:
    def __init__(self, surface, stream_id):
        self.surface, self.stream_id, self.phi, self.K, self.T = surface, stream_id, -1, OPT.K, OPT.T
        self.n_steps, self.n_paths = OPT.n_steps, OPT.n_paths


def test_a_book_keeps_such_spots_in_their_own_buckets(lib):
    """Two options on one surface, one on another: as with the binary search on the first."""
    out = []
    for far in (False, True):
        surfs = [lv.Surface.from_workload(_surface(20, 10, far), lib), lv.Surface.from_workload(_surface(7, 3, seed=4), lib)]
        book = lv.Book(surfs, [_Item(0, 0), _Item(1, 1), _Item(0, 2)], lib)
        r = np.array(book.run(OPT.S0, OPT.r, OPT.seed))
        out.append([(r[o], r[o + 1], r[o + 3:o + 3 + n]) for o, n in ((0, 200), (203, 21), (227, 200))])
        book.close()
        [s.close() for s in surfs]
    for got, ref in zip(*out):
        _close(got, ref, 1.6e-5)
