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
