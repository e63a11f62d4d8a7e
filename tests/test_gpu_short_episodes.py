"""Episode statistics around the line between one thread per env and the warp
pipeline: trajectories against the oracle, and the replay of a rollout's value
log against stepping."""
import numpy as np
import pytest
import torch

import oracle
import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

pytestmark = pytest.mark.gpu

EXACT = [0, 1, 2, 4, 5, 6, 8, 9, 10]       # every metric but the two through pow()


@pytest.mark.parametrize("N, T", [(1, 0), (1, 1), (130, 1), (9728, 4), (9728, 6), (9729, 8), (9729, 30), (20_000, 33),
                                  (20_000, 60), (40_000, 5)])
@pytest.mark.parametrize("values", ["ordinary", "any sign"])
def test_trajectory_metrics_of_few_steps(dev, built_lib, N, T, values):
    rng = np.random.default_rng(N + T)
    v0 = 100_000_000
    rew = rng.integers(-v0 // 300, v0 // 250, (T, N))
    if values == "any sign":
        rew[rng.random((T, N)) < 0.1] = -(2 * v0)     # values turn negative and back
        rew[rng.random((T, N)) < 0.1] = 1 << 53       # and past 2^53
    rew[:, ::7] = 0
    done = (rng.random((T, N)) < 0.05).astype(np.uint8)
    for d in (None, done):
        got = fr.trajectory_metrics(torch.from_numpy(rew).to(dev), None if d is None else torch.from_numpy(d).to(dev),
                                    v0=v0, ann=252.0, gamma=0.99)
        torch.cuda.synchronize()
        g = got.cpu().numpy()
        want = oracle.trajectory_metrics(rew, np.zeros_like(done) if d is None else d, v0, 252.0, 0.99)
        assert np.array_equal(g[:, EXACT], want[:, EXACT], equal_nan=True)
        assert np.allclose(g[:, [3, 7]], want[:, [3, 7]], rtol=1e-13, atol=0, equal_nan=True)


@pytest.mark.parametrize("N, pieces", [(3, (1, 4, 6, 5)), (9000, (1, 10, 13)), (10_000, (20, 12))])
def test_replay_of_a_short_log_equals_stepping(ctx, dev, N, pieces):
    mk = fr.fr_market_create(ctx, synth.crypto_market(8000, seed=3))
    start, W = np.arange(N) % 4000 + 3600, 3 + np.arange(N) * 7 % 38
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


def test_rollout_of_many_envs_in_pieces(ctx, dev):
    # the pieces' replays, one thread per env at this many envs, run beside the
    # next pieces, which take the step counts from the kernel alone
    N, T = 20_000, 256
    mk = fr.fr_market_create(ctx, synth.stock_market(700, 30, seed=3))
    e = synth.stock_envs_cohorts(N, 30, 700, 2 * T, 8, 3)
    dims = (301, 64, 64, 30)
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, 3, seed=3), precision=fr.PREC_BF16)
    out = []
    for split in (False, True):
        env = fr.env_create(ctx, mk, start=e.start, window=e.W, n_assets=e.Ke, bps=e.bps)
        fr.env_set_rollout_split(env, split)
        got = []
        for steps in (T, 130):
            m = torch.empty(N, 3, dtype=torch.float64, device=dev)
            fr.rollout(env, ens, steps, metrics=m)
            st = [torch.empty(N, dtype=t, device=dev) for t in (torch.int64, torch.int32, torch.uint8)]
            fr.env_get_state(env, cash=st[0], steps=st[1], done=st[2])
            got += [m] + st
        torch.cuda.synchronize()
        out.append(got)
    assert all(torch.equal(x, y) for x, y in zip(*out))
