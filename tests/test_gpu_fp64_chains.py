"""The FP64 chains at their edges: segment, group and block boundaries, and
the values that leave the fast forms (prices of 2^52 cents and more, series
that decay below the two-operation division's range, values that turn
negative), each bit for bit against the oracle or the step-by-step path."""
import numpy as np
import pytest
import torch

import oracle
import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

pytestmark = pytest.mark.gpu

EXACT = [0, 1, 2, 4, 5, 6, 8, 9, 10]       # every metric but the two through pow()


def _indicators(close, high, low, dev):
    got = fr.market_indicators(*[torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (close, high, low)])
    torch.cuda.synchronize()
    return got.cpu().numpy()


@pytest.mark.parametrize("T, K", [(7, 31), (8, 32), (9, 33), (63, 2), (64, 3), (65, 64), (128, 65), (193, 5)])
def test_indicator_segment_edges(dev, built_lib, T, K):
    mk = synth.stock_market(T, K, seed=T * 100 + K)
    assert np.array_equal(_indicators(mk.close, mk.high, mk.low, dev), oracle.indicators(mk.close, mk.high, mk.low))


def test_indicator_values_outside_the_fast_forms(dev, built_lib):
    # column 0: prices around 2^52 and 2^53; column 1: one move, then flat for
    # 25,000 days, so the smoothed series decay through 2^-400 and below
    # 2^-1022; column 2: low above high on some days
    T = 25_000
    rng = np.random.default_rng(11)
    close = np.empty((T, 3), np.int64)
    close[:, 0] = (1 << 52) + rng.integers(-(1 << 50), 1 << 53, T)
    close[:, 1] = 7000
    close[:3, 1] = (5000, 9000, 6000)
    close[:, 2] = rng.integers(1, 100_000, T)
    high, low = close + 3, np.maximum(close - 3, 1)
    high[:, 1] = low[:, 1] = close[:, 1]
    high[::5, 2], low[::5, 2] = low[::5, 2], high[::5, 2]
    assert np.array_equal(_indicators(close, high, low, dev), oracle.indicators(close, high, low))
