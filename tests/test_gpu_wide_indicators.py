"""Indicator tables of few days or many assets, whose blocks share their SMs, bit
for bit against the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T, K", [(1, 9), (2, 1000), (31, 17), (32, 700), (33, 5), (64, 611), (65, 610), (128, 333),
                                  (129, 420), (300, 601)])
def test_indicator_tables_of_many_assets(dev, built_lib, T, K):
    mk = synth.stock_market(T, K, seed=T + K)
    got = fr.market_indicators(*[torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (mk.close, mk.high, mk.low)])
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy(), oracle.indicators(mk.close, mk.high, mk.low))
