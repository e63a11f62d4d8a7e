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


@pytest.mark.parametrize("N, T", [(1, 1), (15, 7), (16, 8), (17, 9), (33, 25), (2432, 12), (2433, 17), (2500, 64)])
@pytest.mark.parametrize("values", ["ordinary", "large", "any sign"])
def test_trajectory_metrics_edges_match_oracle(dev, built_lib, N, T, values):
    rng = np.random.default_rng(N * 1000 + T)
    v0 = 100_000_000 if values != "large" else (1 << 45)
    rew = rng.integers(-v0 // 300, v0 // 250, (T, N))
    if values == "large":
        rew[rng.random((T, N)) < 0.1] = 1 << 53       # values pass 2^53
    if values == "any sign":
        rew[rng.random((T, N)) < 0.1] = -(2 * v0)     # values turn negative and back
        rew[rng.random((T, N)) < 0.1] = 3 * v0
    rew[:, ::7] = 0                                   # no move at all: zero variance
    done = (rng.random((T, N)) < 0.05).astype(np.uint8)
    for d in (None, done):
        got = fr.trajectory_metrics(torch.from_numpy(rew).to(dev), None if d is None else torch.from_numpy(d).to(dev),
                                    v0=v0, ann=252.0, gamma=0.99)
        torch.cuda.synchronize()
        g = got.cpu().numpy()
        want = oracle.trajectory_metrics(rew, np.zeros_like(done) if d is None else d, v0, 252.0, 0.99)
        assert np.array_equal(g[:, EXACT], want[:, EXACT], equal_nan=True)
        assert np.allclose(g[:, [3, 7]], want[:, [3, 7]], rtol=1e-13, atol=0, equal_nan=True)


@pytest.mark.parametrize("N, pieces", [(5, (9, 1, 30)), (16, (40,)), (2600, (3, 17, 20))])
def test_replay_of_the_value_log_equals_stepping(ctx, dev, N, pieces):
    # the same actions through env_step give the same accumulators, also where
    # the envs' step counts differ (windows of 3 to 40 seconds, in pieces)
    mk = fr.fr_market_create(ctx, synth.crypto_market(8000, seed=3))
    start = np.arange(N) % 4000 + 3600
    W = 3 + np.arange(N) * 7 % 38
    a, b = (fr.env_create(ctx, mk, start=start, window=W, pmax=3) for _ in range(2))
    dims = (10, 32, 3)
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, 3, seed=4, out_scale=4.0), precision=fr.PREC_BF16,
                             combine=fr.COMBINE_VOTE, out_act=0)
    ma, mb = (torch.empty(N, 3, dtype=torch.float64, device=dev) for _ in range(2))
    for T in pieces:
        act = torch.empty(T, N, dtype=torch.uint8, device=dev)
        fr.rollout(a, ens, T, traj={"act": act}, metrics=ma)
        for t in range(T):
            fr.env_step(b, act[t], fr.ACT_U8_DISCRETE)
        fr.env_metrics(b, mb)
        torch.cuda.synchronize()
        assert torch.equal(ma, mb)
