"""The fp32 actor path at its tile edges: every layer-width class, batch sizes
around the row tiles, against a float64 forward within the rounding bound of
fp32 sums, and the same bits whatever the batch a row is in."""
import numpy as np
import pytest
import torch

import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _forward64(dims, params, x, tanh):
    """float64 forward and the elementwise bound of an fp32 evaluation: a sum
    of K products is off by at most (K + 2) U sum |w x| (1 + small), and the
    error of the layer below passes through |W|."""
    err = np.zeros_like(x)
    layers = synth.unpack_params(dims, params.astype(np.float64))
    for i, (W, b) in enumerate(layers):
        W = W.reshape(dims[i + 1], dims[i])
        g = (dims[i] + 4) * U * 1.01
        mag = np.abs(x) @ np.abs(W).T + np.abs(b)
        err = g * (mag + err @ np.abs(W).T) + err @ np.abs(W).T
        x = x @ W.T + b
        if i + 1 < len(layers):
            x = np.maximum(x, 0.0)
    if tanh:
        x, err = np.tanh(x), err + 4 * U           # tanhf: a few units in the last place of at most 1
    return x, err


@pytest.mark.parametrize("dims", [(301, 256, 256, 30), (10, 128, 128, 3), (304, 129, 65, 33, 1), (1, 256), (37, 32, 31),
                                  (64, 64, 256, 200)])
@pytest.mark.parametrize("tanh", [0, 1])
def test_fp32_forward_at_tile_edges(ctx, dev, dims, tanh):
    M = 2
    P = synth.actor_params(dims, M, seed=sum(dims))
    ens = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_FP32, out_act=tanh)
    rng = np.random.default_rng(5)
    n_max = 10_300                                  # 64-row tiles
    x = rng.standard_normal((n_max, dims[0])).astype(np.float32)
    xd = torch.from_numpy(x).to(dev)
    full = torch.empty(M, n_max, dims[-1], device=dev)
    fr.ensemble_forward(ens, xd, full)
    torch.cuda.synchronize()
    got = full.cpu().numpy()
    rows = np.r_[0:130, n_max - 70:n_max]
    for j in range(M):
        want, err = _forward64(dims, P[j], x[rows].astype(np.float64), tanh)
        assert (np.abs(got[j, rows] - want) <= err).all()
    for n in (1, 15, 16, 17, 31, 33, 63, 64, 65, 300, 2400, 2600, 5000):
        y = torch.empty(M, n, dims[-1], device=dev)
        fr.ensemble_forward(ens, xd[:n].contiguous(), y)
        torch.cuda.synchronize()
        assert torch.equal(y, full[:, :n])
