"""Crypto env steps whose observation rows leave a block as one span: batch
sizes around the blocks, and buffers that start and do not start on 16 bytes,
give the same observations, rewards and state."""
import numpy as np
import pytest
import torch

import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 4, 127, 128, 129, 1000])
def test_rows_equal_whatever_the_buffer(ctx, dev, N):
    mk = fr.fr_market_create(ctx, synth.crypto_market(9_000, seed=2))
    rng = np.random.default_rng(N)
    start, W = rng.integers(3600, 8_000, N).astype(np.int32), rng.integers(2, 9, N).astype(np.int32)
    acts = rng.integers(0, 3, (5, N)).astype(np.uint8)
    outs = []
    for off in (0, 1):
        env = fr.env_create(ctx, mk, start=start, window=W, pmax=3, auto_reset=N % 2 == 1)
        buf = torch.full((N * env.D + off + 3,), -7.0, device=dev)
        obs = buf[off:off + N * env.D].view(N, env.D)
        got = []
        for a in acts:
            rew = torch.empty(N, dtype=torch.int64, device=dev)
            done = torch.empty(N, dtype=torch.uint8, device=dev)
            fr.env_step(env, torch.from_numpy(a).to(dev), fr.ACT_U8_DISCRETE, rew=rew, done=done, obs=obs)
            again = torch.empty(N, env.D, device=dev)
            fr.env_observe(env, again)
            torch.cuda.synchronize()
            assert torch.equal(obs, again)
            got += [obs.clone(), rew, done]
        assert (buf[:off] == -7.0).all() and (buf[off + N * env.D:] == -7.0).all()
        m = torch.empty(N, 3, dtype=torch.float64, device=dev)
        fr.env_metrics(env, m)
        torch.cuda.synchronize()
        outs.append(got + [m])
    assert all(torch.equal(x, y) for x, y in zip(*outs))
