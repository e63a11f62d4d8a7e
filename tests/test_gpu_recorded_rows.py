"""Recorded stock rollouts: every observation row, also of envs that start in the
middle of an episode, end or restart inside the rollout, and in rows with a
stride, is the one env_observe gives before the same step."""
import numpy as np
import pytest
import torch

import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ld", [301, 304, 400])
@pytest.mark.parametrize("auto_reset", [False, True])
def test_rows_equal_observations(ctx, dev, ld, auto_reset):
    N = 150
    mk = fr.fr_market_create(ctx, synth.stock_market(200, 30, seed=5))
    e = synth.stock_envs_uneven(N, 30, 200, w_lo=5, w_hi=40, seed=5)
    a, b = (fr.env_create(ctx, mk, start=e.start, window=e.W, n_assets=e.Ke, bps=e.bps, auto_reset=auto_reset)
            for _ in range(2))
    dims = (301, 64, 64, 30)
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, 3, seed=5), precision=fr.PREC_BF16)
    row = torch.empty(N, 301, device=dev)
    for T in (1, 4, 9, 30):
        tr = {"obs": torch.full((T, N, ld), -7.0, device=dev), "act": torch.empty(T, N, 30, device=dev),
              "rew": torch.empty(T, N, dtype=torch.int64, device=dev), "done": torch.empty(T, N, dtype=torch.uint8, device=dev)}
        fr.rollout(a, ens, T, traj=tr)
        for t in range(T):
            fr.env_observe(b, row)
            rew, done = torch.empty(N, dtype=torch.int64, device=dev), torch.empty(N, dtype=torch.uint8, device=dev)
            fr.env_step(b, tr["act"][t], fr.ACT_F32_UNIT, rew=rew, done=done)
            torch.cuda.synchronize()
            assert torch.equal(tr["obs"][t, :, :301], row) and (tr["obs"][t, :, 301:] == -7.0).all()
            assert torch.equal(tr["rew"][t], rew) and torch.equal(tr["done"][t], done)
