"""The resident-weight actor kernels (narrow networks with every agent in one
CTA, wide ones over CTA pairs) at their tile edges: each width class and agent
count, batch sizes around the row tiles and the waves, observations that bulk
copies can and cannot take, against a float64 evaluation on the same 16-bit
operands; the same bits whatever the batch a row is in; and the narrow rollout
against the unfused path."""
import numpy as np
import pytest
import torch

import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _round16(x, f16):
    """float64 -> the nearest 16-bit operand, as float64."""
    t = torch.from_numpy(np.ascontiguousarray(x)).float()
    return t.to(torch.float16 if f16 else torch.bfloat16).double().numpy()


def _forward16(dims, params, x, f16, tanh):
    """Forward on 16-bit operands in float64, and an elementwise bound of the
    kernels' distance from it: an fp32 sum of K products is off by at most
    (K + 2) U sum |w x| (1 + small), the layer below adds its bound through
    |W|, and a hidden value that lands on the other side of a rounding
    boundary is one 16-bit step (2^-10 or 2^-7 of it) further off."""
    step = 2.0 ** (-10 if f16 else -7)
    layers = synth.unpack_params(dims, params.astype(np.float64))
    x, err = _round16(x, f16), np.zeros(x.shape)
    for i, (W, b) in enumerate(layers):
        W = _round16(W.reshape(dims[i + 1], dims[i]), f16)
        A = np.abs(W).T
        g = (dims[i] + 4) * U * 1.01
        err = g * (np.abs(x) @ A + err @ A + np.abs(b)) + err @ A
        x = x @ W.T + b
        if i + 1 < len(layers):
            x = np.maximum(x, 0.0)
            err = err + np.where(err > 0, step * (np.abs(x) + err), 0.0)
            x = _round16(x, f16)
    if tanh:
        x, err = np.tanh(x), err + 4 * U
    return x, err


# narrow: one CTA holds every agent; wide: one CTA or a pair per agent
NETS = [((10, 128, 128, 3), 5), ((10, 128, 128, 4), 4), ((16, 65, 127, 16), 1), ((1, 16, 16, 1), 2),
        ((301, 256, 256, 30), 3), ((304, 255, 129, 32), 1), ((61, 64, 64, 30), 4), ((17, 128, 200, 17), 2),
        ((10, 144, 96, 3), 5)]


@pytest.mark.parametrize("dims,M", NETS)
@pytest.mark.parametrize("prec", ["fp16", "bf16"])
def test_resident_forward_at_tile_edges(ctx, dev, dims, M, prec):
    f16, tanh = prec == "fp16", int(dims[-1] > 16)
    P = synth.actor_params(dims, M, seed=sum(dims) + M)
    ens = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_FP16 if f16 else fr.PREC_BF16, out_act=tanh)
    rng = np.random.default_rng(7)
    n_max = 20_491                                  # several waves and an odd last tile
    x = rng.standard_normal((n_max, dims[0])).astype(np.float32)
    xd = torch.from_numpy(x).to(dev)
    full = torch.empty(M, n_max, dims[-1], device=dev)
    fr.ensemble_forward(ens, xd, full)
    torch.cuda.synchronize()
    got = full.cpu().numpy().astype(np.float64)
    rows = np.r_[0:150, n_max - 130:n_max]
    for j in range(M):
        want, err = _forward16(dims, P[j], x[rows].astype(np.float64), f16, tanh)
        assert (np.abs(got[j, rows] - want) <= err).all()
    for n in (1, 3, 15, 16, 17, 47, 64, 65, 1000, 2500, 9729):
        y = torch.empty(M, n, dims[-1], device=dev)
        fr.ensemble_forward(ens, xd[:n].contiguous(), y)
        # an observation buffer that does not start on 16 bytes
        z = torch.empty(n * dims[0] + 1, device=dev)[1:].view(n, dims[0])
        z.copy_(xd[:n])
        y2 = torch.full_like(y, -7.0)
        fr.ensemble_forward(ens, z, y2)
        torch.cuda.synchronize()
        assert torch.equal(y, full[:, :n]) and torch.equal(y2, y)
    assert fr.ensemble_device_errors(ens) == 0


@pytest.mark.parametrize("N,M,hidden,auto_reset,prec", [
    (1, 1, 16, False, "fp16"), (17, 5, 128, True, "fp16"), (100, 4, 128, False, "bf16"), (2500, 3, 64, True, "bf16"),
    (9800, 5, 128, False, "fp16")])
def test_narrow_rollout_equals_unfused(ctx, dev, N, M, hidden, auto_reset, prec):
    T = 40
    mk = fr.fr_market_create(ctx, synth.crypto_market(30_000, seed=5))
    e = synth.crypto_envs(N, 30_000, 64, seed=N)
    W = np.random.default_rng(N).integers(2, 64, N).astype(np.int32)       # windows ending inside the rollout
    dims = (10, hidden, hidden, 3)
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=N, out_scale=4.0), out_act=0,
                             precision=fr.PREC_FP16 if prec == "fp16" else fr.PREC_BF16, combine=fr.COMBINE_VOTE)
    out = []
    for path in (fr.PATH_AUTO, fr.PATH_UNFUSED):
        env = fr.env_create(ctx, mk, start=e.start, window=W, pmax=3, init_cash=30_000_000, auto_reset=auto_reset)
        fr.env_set_rollout_path(env, path)
        tr = {"obs": torch.empty(T, N, 10, device=dev), "act": torch.empty(T, N, dtype=torch.uint8, device=dev),
              "rew": torch.empty(T, N, dtype=torch.int64, device=dev), "rew_f32": torch.empty(T, N, device=dev),
              "done": torch.empty(T, N, dtype=torch.uint8, device=dev)}
        m = torch.empty(N, 3, dtype=torch.float64, device=dev)
        fr.rollout(env, ens, T, traj=tr, metrics=m)
        st = {"cash": torch.empty(N, dtype=torch.int64, device=dev), "hold": torch.empty(N, dtype=torch.int32, device=dev),
              "steps": torch.empty(N, dtype=torch.int32, device=dev), "done": torch.empty(N, dtype=torch.uint8, device=dev)}
        fr.env_get_state(env, **st)
        torch.cuda.synchronize()
        out.append({**tr, **st, "metrics": m})
    for k in out[0]:
        assert torch.equal(out[0][k], out[1][k]), k


@pytest.mark.parametrize("dims,M", [((301, 256, 256, 30), 3), ((301, 256, 256, 30), 1), ((304, 255, 129, 32), 4),
                                    ((61, 64, 64, 30), 5), ((61, 64, 64, 17), 2)])
def test_act_equals_forward_then_mean(ctx, dev, dims, M):
    # the agents combined in the forward's own launch, and (past its range) after it
    w = np.random.default_rng(M).random(M).astype(np.float32)
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=M), weights=w, precision=fr.PREC_BF16)
    wt = torch.from_numpy(w).to(dev)
    n_max = 4500
    x = torch.from_numpy(np.random.default_rng(3).standard_normal((n_max, dims[0])).astype(np.float32)).to(dev)
    for n in (1, 8, 16, 17, 47, 48, 49, 1104, 1105, 1199, 2209, 4096, 4097, 4500):
        y = torch.empty(M, n, dims[-1], device=dev)
        act = torch.full((n + 1, dims[-1]), -7.0, device=dev)
        fr.ensemble_forward(ens, x[:n].contiguous(), y)
        fr.ensemble_act(ens, x[:n].contiguous(), act[:n])
        want = y[0].clone()
        for j in range(1, M):
            want = want + wt[j] * (y[j] - y[0])
        torch.cuda.synchronize()
        assert torch.equal(act[:n], want) and (act[n] == -7.0).all()
    assert fr.ensemble_device_errors(ens) == 0


@pytest.mark.parametrize("dims,M,combine", [((301, 256, 256, 30), 3, "mean"), ((10, 128, 128, 3), 5, "vote")])
def test_first_call_inside_a_capture(ctx, dev, dims, M, combine):
    # a new ensemble's first forward and act, captured; replays equal direct calls on other inputs
    vote = combine == "vote"
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=9), precision=fr.PREC_FP16,
                             combine=fr.COMBINE_VOTE if vote else fr.COMBINE_MEAN, out_act=0 if vote else 1)
    n = 70
    x, y = torch.zeros(n, dims[0], device=dev), torch.empty(M, n, dims[-1], device=dev)
    a = torch.empty(n, dtype=torch.uint8, device=dev) if vote else torch.empty(n, dims[-1], device=dev)
    torch.cuda.synchronize()
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=side):
        fr.ensemble_forward(ens, x, y, stream=side)
        fr.ensemble_act(ens, x, a, stream=side)
    for seed in range(3):
        x.copy_(torch.from_numpy(np.random.default_rng(seed).standard_normal((n, dims[0])).astype(np.float32)))
        g.replay()
        y2, a2 = torch.empty_like(y), torch.empty_like(a)
        fr.ensemble_forward(ens, x, y2)
        fr.ensemble_act(ens, x, a2)
        torch.cuda.synchronize()
        assert torch.equal(y, y2) and torch.equal(a, a2)


@pytest.mark.parametrize("explore", [False, True])
def test_narrow_rollout_in_pieces(ctx, dev, explore):
    # 200 steps in three pieces whose replays run beside the next, then 130 in
    # two, equal single launches; and a captured rollout replays them
    N = 700
    mk = fr.fr_market_create(ctx, synth.crypto_market(30_000, seed=6))
    e = synth.crypto_envs(N, 30_000, 500, seed=6)
    W = np.random.default_rng(6).integers(2, 400, N).astype(np.int32)
    ens = fr.ensemble_create(ctx, (10, 64, 128, 3), synth.actor_params((10, 64, 128, 3), 5, seed=6, out_scale=4.0),
                             precision=fr.PREC_FP16, combine=fr.COMBINE_VOTE, out_act=0)

    def run(env, lengths):
        out = []
        for T in lengths:
            m = torch.empty(N, 3, dtype=torch.float64, device=dev)
            fr.rollout(env, ens, T, metrics=m)
            st = [torch.empty(N, dtype=t, device=dev) for t in (torch.int64, torch.int32, torch.int32, torch.uint8)]
            fr.env_get_state(env, cash=st[0], hold=st[1], steps=st[2], done=st[3])
            out += [m] + st
        return out

    envs = []
    for split in (False, True):
        env = fr.env_create(ctx, mk, start=e.start, window=W, pmax=3)
        fr.env_set_rollout_split(env, split)
        if explore:
            fr.env_set_exploration(env, fr.EXPLORE_EPS_GREEDY, eps=0.3, seed=5)
        envs.append(env)
    a, b = run(envs[0], (200, 130)), run(envs[1], (200, 130))
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(a, b))
    if explore:
        return
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    m = torch.empty(N, 3, dtype=torch.float64, device=dev)
    with torch.cuda.graph(g, stream=side):
        fr.env_reset(envs[1], stream=side)
        fr.rollout(envs[1], ens, 200, metrics=m, stream=side)
    for _ in range(2):
        m.fill_(-7.0)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(m, a[0])
