"""The resident-weight actor kernels where their tiles, launches and dispatch
rules have an edge: shapes at the shared-memory limit, weights changed under a
captured call, NaN in large batches."""
import numpy as np
import pytest
import torch

import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth
from test_gpu_resident import _forward16

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(302, 256, 256, 30), (303, 256, 256, 30), (304, 256, 256, 32), (304, 16, 241, 17)])
@pytest.mark.parametrize("prec", ["fp16", "bf16"])
def test_shapes_at_the_shared_memory_limit(ctx, dev, dims, prec):
    # 64-row tiles of the widest inputs and second layers need more than an SM
    # has: batches that would take them run all the same
    M, f16 = 3, prec == "fp16"
    P = synth.actor_params(dims, M, seed=sum(dims))
    ens = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_FP16 if f16 else fr.PREC_BF16)
    n_max = 20_491
    x = np.random.default_rng(7).standard_normal((n_max, dims[0])).astype(np.float32)
    xd = torch.from_numpy(x).to(dev)
    full = torch.empty(M, n_max, dims[-1], device=dev)
    fr.ensemble_forward(ens, xd, full)
    torch.cuda.synchronize()
    got = full.cpu().numpy().astype(np.float64)
    rows = np.r_[0:150, n_max - 130:n_max]
    for j in range(M):
        want, err = _forward16(dims, P[j], x[rows].astype(np.float64), f16, 1)
        assert (np.abs(got[j, rows] - want) <= err).all()
    for n in (1, 17, 1199, 1201, 4500):
        y, act = torch.empty(M, n, dims[-1], device=dev), torch.empty(n, dims[-1], device=dev)
        fr.ensemble_forward(ens, xd[:n].contiguous(), y)
        fr.ensemble_act(ens, xd[:n].contiguous(), act)
        torch.cuda.synchronize()
        w = torch.full((), 1.0 / 3.0, device=dev)
        assert torch.equal(y, full[:, :n])
        assert torch.equal(act, y[0] + w * (y[1] - y[0]) + w * (y[2] - y[0]))
    assert fr.ensemble_device_errors(ens) == 0


@pytest.mark.parametrize("prec", [fr.PREC_BF16, fr.PREC_FP32])
@pytest.mark.parametrize("n", [8, 1500, 4500])
def test_captured_act_follows_new_weights(ctx, dev, n, prec):
    # a replayed act uses the weights set since its capture, at every batch size
    dims, M = (61, 64, 200, 30), 3
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=2), precision=prec)
    x = torch.from_numpy(np.random.default_rng(2).standard_normal((n, dims[0])).astype(np.float32)).to(dev)
    a, b = torch.empty(n, dims[-1], device=dev), torch.empty(n, dims[-1], device=dev)
    torch.cuda.synchronize()
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=side):
        fr.ensemble_act(ens, x, a, stream=side)
    seen = []
    for w in ((0.2, 0.3, 0.5), (0.0, 1.0, 0.0), (0.1, 0.0, 0.9)):
        fr.ensemble_set_weights(ens, np.float32(w))
        g.replay()
        fr.ensemble_act(ens, x, b)
        torch.cuda.synchronize()
        assert torch.equal(a, b)
        seen.append(a.clone())
    assert not torch.equal(seen[0], seen[1]) and not torch.equal(seen[1], seen[2])


@pytest.mark.parametrize("dims", [(61, 64, 200, 30), (10, 64, 64, 3)])
@pytest.mark.parametrize("prec", [fr.PREC_BF16, fr.PREC_FP16])
def test_nan_rows_in_large_batches(ctx, dev, dims, prec):
    # a NaN observation: ensemble_act_noalloc stands for the single-agent kernel
    # (max(x, 0) makes a hidden NaN 0) whatever the batch, ensemble_act and
    # _forward for the large-batch one (it stays) from one tile of 128 rows per SM
    M, n = 2, 128 * ctx.sm_count
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=3), precision=prec)
    x = torch.from_numpy(np.random.default_rng(4).standard_normal((n, dims[0])).astype(np.float32)).to(dev)
    x[5, 1] = float("nan")
    a, few = torch.empty(n, dims[-1], device=dev), torch.empty(100, dims[-1], device=dev)
    big, y = torch.empty_like(a), torch.empty(M, n, dims[-1], device=dev)
    fr.ensemble_act_noalloc(ens, x, a)
    fr.ensemble_act_noalloc(ens, x[:100].contiguous(), few)
    fr.ensemble_act(ens, x, big)
    fr.ensemble_forward(ens, x, y)
    torch.cuda.synchronize()
    assert torch.isfinite(a).all() and torch.equal(a[:100], few)
    keep = torch.arange(n, device=dev) != 5
    assert torch.equal(a[keep], big[keep])
    assert torch.isnan(big[5]).all() and torch.isnan(y[:, 5]).all()


def test_forward_beside_a_fused_rollout(ctx, dev):
    # two kernels whose CTAs work in clusters and hold tensor memory, on two
    # streams at once: the results are those of each alone
    dims, M, n, N, T = (10, 144, 96, 3), 5, 5000, 700, 40
    P = synth.actor_params(dims, M, seed=8, out_scale=4.0)
    ens = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_BF16, out_act=0)
    vote = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_BF16, combine=fr.COMBINE_VOTE, out_act=0)
    mk = fr.fr_market_create(ctx, synth.crypto_market(9_000, seed=8))
    env = fr.env_create(ctx, mk, start=np.arange(N) % 4000 + 3600, window=T + 1, pmax=3)
    x = torch.from_numpy(np.random.default_rng(8).standard_normal((n, dims[0])).astype(np.float32)).to(dev)
    y = [torch.empty(M, n, dims[-1], device=dev) for _ in range(2)]
    m = [torch.empty(N, 3, dtype=torch.float64, device=dev) for _ in range(2)]
    s = [torch.cuda.Stream() for _ in range(2)]
    fr.ensemble_forward(ens, x, y[0])
    torch.cuda.synchronize()
    fr.rollout(env, vote, T, metrics=m[0])
    torch.cuda.synchronize()
    for _ in range(10):
        y[1].fill_(-7.0)
        m[1].fill_(-7.0)
        torch.cuda.synchronize()
        fr.env_reset(env, stream=s[0])
        fr.rollout(env, vote, T, metrics=m[1], stream=s[0])
        for _ in range(20):
            fr.ensemble_forward(ens, x, y[1], stream=s[1])
        torch.cuda.synchronize()
        assert torch.equal(y[0], y[1]) and torch.equal(m[0], m[1])
    assert fr.ensemble_device_errors(ens) == 0 and fr.ensemble_device_errors(vote) == 0


def test_fused_crypto_rollout_of_many_clusters(ctx, dev):
    # 256 columns of tensor memory per CTA and more clusters than the GPU holds
    # at two CTAs per SM: the rollout equals the unfused one
    dims, M, N, T = (10, 144, 96, 3), 5, 12_000, 12
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=8, out_scale=4.0), precision=fr.PREC_BF16,
                             combine=fr.COMBINE_VOTE, out_act=0)
    mk = fr.fr_market_create(ctx, synth.crypto_market(9_000, seed=8))
    out = []
    for path in (fr.PATH_AUTO, fr.PATH_UNFUSED):
        env = fr.env_create(ctx, mk, start=np.arange(N) % 4000 + 3600, window=T + 1, pmax=3)
        fr.env_set_rollout_path(env, path)
        act, m = torch.empty(T, N, dtype=torch.uint8, device=dev), torch.empty(N, 3, dtype=torch.float64, device=dev)
        fr.rollout(env, ens, T, traj={"act": act}, metrics=m)
        torch.cuda.synchronize()
        out.append((act, m))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert fr.ensemble_device_errors(ens) == 0


def test_narrow_rollout_with_room_for_the_log_alone(dev):
    # the step counts of a rollout in pieces are no reason to refuse one: not
    # under a budget with room for the value log alone, nor in a capture of an
    # env whose scratch is that log
    N, T, dims, M = 300, 200, (10, 64, 64, 3), 3

    def setup(budget):
        ctx = fr.fr_ctx_create(0, budget)
        mk = fr.fr_market_create(ctx, synth.crypto_market(9_000, seed=8))
        env = fr.env_create(ctx, mk, start=np.arange(N) % 4000 + 3600, window=T + 1, pmax=3)
        kw = dict(combine=fr.COMBINE_VOTE, out_act=0)
        P = synth.actor_params(dims, M, seed=8, out_scale=4.0)
        ens = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_FP16, **kw)
        x3 = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_BF16X3, **kw)
        return ctx, mk, env, ens, x3, torch.empty(N, 3, dtype=torch.float64, device=dev)

    free = setup(0)
    used = free[0].bytes_in_use
    fr.rollout(free[2], free[3], T, metrics=free[5])
    tight = setup(used + 8 * N * T)
    fr.rollout(tight[2], tight[3], T, metrics=tight[5])
    torch.cuda.synchronize()
    assert torch.equal(free[5], tight[5])
    # captured: the first fused kernel's rollout has made the scratch one value log
    ctx, mk, env, ens, x3, m = setup(0)
    fr.rollout(env, x3, T, metrics=m)
    torch.cuda.synchronize()
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=side):
        fr.env_reset(env, stream=side)
        fr.rollout(env, ens, T, metrics=m, stream=side)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(free[5], m)


def test_first_call_of_a_narrow_mean_ensemble_inside_a_capture(ctx, dev):
    # its forward and its act run different kernels, both prepared with it
    dims, M, n = (10, 128, 128, 3), 2, 70
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=9), precision=fr.PREC_BF16)
    x, y, a = torch.zeros(n, dims[0], device=dev), torch.empty(M, n, 3, device=dev), torch.empty(n, 3, device=dev)
    torch.cuda.synchronize()
    g, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=side):
        fr.ensemble_forward(ens, x, y, stream=side)
        fr.ensemble_act(ens, x, a, stream=side)
    for seed in range(2):
        x.copy_(torch.from_numpy(np.random.default_rng(seed).standard_normal((n, dims[0])).astype(np.float32)))
        g.replay()
        y2, a2 = torch.empty_like(y), torch.empty_like(a)
        fr.ensemble_forward(ens, x, y2)
        fr.ensemble_act(ens, x, a2)
        torch.cuda.synchronize()
        assert torch.equal(y, y2) and torch.equal(a, a2)


@pytest.mark.parametrize("dims,M", [((32, 160, 160, 30), 2), ((36, 200, 40, 17), 3), ((64, 64, 64, 30), 1),
                                    ((100, 256, 129, 30), 2), ((200, 64, 64, 30), 3), ((300, 256, 256, 30), 2)])
@pytest.mark.parametrize("prec", ["fp16", "bf16"])
def test_input_widths_of_whole_quads(ctx, dev, dims, M, prec):
    # rows read 16 bytes at a time: the last quad of the width, packed rows and
    # rows at any address
    f16 = prec == "fp16"
    P = synth.actor_params(dims, M, seed=sum(dims))
    ens = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_FP16 if f16 else fr.PREC_BF16)
    for n in (1, 5, 65, 2500):
        x = np.random.default_rng(n).standard_normal((n, dims[0])).astype(np.float32)
        xd = torch.from_numpy(x).to(dev)
        z = torch.empty(n * dims[0] + 1, device=dev)[1:].view(n, dims[0])
        z.copy_(xd)
        y, y2 = torch.empty(M, n, dims[-1], device=dev), torch.empty(M, n, dims[-1], device=dev)
        fr.ensemble_forward(ens, xd, y)
        fr.ensemble_forward(ens, z, y2)
        torch.cuda.synchronize()
        assert torch.equal(y, y2)
        for j in range(M):
            want, err = _forward16(dims, P[j], x.astype(np.float64), f16, 1)
            assert (np.abs(y[j].cpu().numpy() - want) <= err).all()


@pytest.mark.parametrize("dims,M", [((10, 144, 96, 3), 5), ((61, 64, 64, 30), 8), ((128, 16, 256, 30), 4),
                                    ((304, 129, 256, 30), 8), ((301, 128, 256, 17), 6)])
@pytest.mark.parametrize("prec", [fr.PREC_BF16, fr.PREC_FP16])
def test_large_batches_on_either_kernel(ctx, dev, dims, M, prec):
    # around the lines where large batches change between the resident and the
    # tiled kernel (a wave of tiles more, the last wave nearly empty or full):
    # every row as in a small batch, acts as forward then mean
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=sum(dims)), precision=prec)
    wave = 128 * ctx.sm_count
    x = torch.from_numpy(np.random.default_rng(6).standard_normal((2 * wave + 3, dims[0])).astype(np.float32)).to(dev)
    few = torch.empty(M, 2000, dims[-1], device=dev)
    w = torch.full((), np.float32(1.0 / M).item(), device=dev)
    for n in (wave - 128, wave - 127, wave, wave + 1, 2 * wave - 1, 2 * wave + 3):
        y, act = torch.empty(M, n, dims[-1], device=dev), torch.empty(n, dims[-1], device=dev)
        fr.ensemble_forward(ens, x[:n].contiguous(), y)
        fr.ensemble_act(ens, x[:n].contiguous(), act)
        for r in (0, n - 2000):
            fr.ensemble_forward(ens, x[r:r + 2000].contiguous(), few)
            torch.cuda.synchronize()
            assert torch.equal(y[:, r:r + 2000], few)
        want = y[0].clone()
        for j in range(1, M):
            want = want + w * (y[j] - y[0])
        assert torch.equal(act, want)
    assert fr.ensemble_device_errors(ens) == 0


@pytest.mark.parametrize("dims,M", [((61, 64, 64, 30), 8), ((10, 16, 16, 3), 6), ((301, 256, 256, 30), 4), ((61, 64, 64, 30), 1)])
def test_act_around_its_waves(ctx, dev, dims, M):
    # batch sizes around the line between the agents combined in the forward's
    # launch and after it: the same actions
    w = np.random.default_rng(M).random(M).astype(np.float32)
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=M), weights=w, precision=fr.PREC_BF16)
    wt = torch.from_numpy(w).to(dev)
    x = torch.from_numpy(np.random.default_rng(3).standard_normal((4100, dims[0])).astype(np.float32)).to(dev)
    y = torch.empty(M, 4100, dims[-1], device=dev)
    fr.ensemble_forward(ens, x, y)
    want = y[0].clone()
    for j in range(1, M):
        want = want + wt[j] * (y[j] - y[0])
    for n in (1, *range(96 * 10, 4100, 191), 4095, 4096, 4097):
        act = torch.full((n + 1, dims[-1]), -7.0, device=dev)
        fr.ensemble_act(ens, x[:n].contiguous(), act[:n])
        torch.cuda.synchronize()
        assert torch.equal(act[:n], want[:n]) and (act[n] == -7.0).all()
    assert fr.ensemble_device_errors(ens) == 0
