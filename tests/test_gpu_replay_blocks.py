"""Replay pushes around the blocks that count and copy their rows: the stored
transitions are the trajectory's valid rows in order."""
import numpy as np
import pytest
import torch

import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N, T", [(1, 1), (31, 1), (32, 1), (33, 3), (257, 2), (4096, 16), (4097, 16), (8192, 9)])
def test_pushed_rows_in_order(ctx, dev, N, T):
    mk = fr.fr_market_create(ctx, synth.crypto_market(8_000, seed=3))
    env = fr.env_create(ctx, mk, start=np.arange(N) % 3000 + 3600, window=T + 2, pmax=3)
    g = torch.Generator(device=dev)
    g.manual_seed(N)
    rows = torch.arange(T * N, device=dev, dtype=torch.float32).view(T, N)
    tr = {"obs": rows[:, :, None] + torch.arange(10, device=dev) * 0.03125,
          "act": torch.randint(0, 3, (T, N), device=dev, generator=g).to(torch.uint8), "rew_f32": -rows,
          "done": (torch.rand(T, N, device=dev, generator=g) < 0.3).to(torch.uint8)}
    tr["done"] = tr["done"].cummax(0).values.contiguous()
    last = -torch.ones(N, 10, device=dev) - torch.arange(N, device=dev)[:, None]
    live0 = (torch.rand(N, device=dev, generator=g) < 0.8).to(torch.uint8)
    tr["done"][:, live0 == 0] = 1
    valid = torch.cat([live0[None] != 0, tr["done"][:-1] == 0]).flatten()
    idx = valid.nonzero().flatten()
    C = max(1, len(idx))
    rb = fr.replay_create(ctx, env, C)
    fr.replay_push(rb, env, tr, T, last, live0=live0)
    assert fr.replay_size(rb)[0] == len(idx)
    if len(idx) == 0:
        return
    nxt = torch.cat([tr["obs"][1:], last[None]])
    s = fr.replay_sample(rb, 2000, seed=5)
    torch.cuda.synchronize()
    at = idx[s["index"]]                                # the k-th stored row is the k-th valid one
    assert torch.equal(s["obs"], tr["obs"].view(-1, 10)[at])
    assert torch.equal(s["next_obs"], nxt.reshape(-1, 10)[at])
    assert torch.equal(s["act"], tr["act"].flatten()[at]) and torch.equal(s["rew"], tr["rew_f32"].flatten()[at])
    assert torch.equal(s["done"], tr["done"].flatten()[at])
