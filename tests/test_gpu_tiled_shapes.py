"""The single-agent and the tiled large-batch tensor-core kernels on the shapes
that the resident kernels leave to them (two and four layers, wide inputs, more
than 32 outputs; FP8 and split BF16): batches that end inside a warp's rows and
tiles of 128, against a float64 evaluation on the same operands, and the same
bits whatever the batch and the kernel."""
import numpy as np
import pytest
import torch

import paper_2501_10709_gb300 as fr
from paper_2501_10709_gb300 import synth
from test_gpu_resident import _forward16

pytestmark = pytest.mark.gpu

SHAPES = [((320, 256, 256, 30), 3), ((301, 64, 30), 2), ((301, 128, 96, 64, 30), 2), ((61, 80, 256, 33), 2),
          ((500, 256, 256, 200), 1), ((10, 64, 3), 5)]
SIZES = (1, 4, 5, 17, 31, 33, 100, 129, 1000)


@pytest.mark.parametrize("dims,M", SHAPES)
@pytest.mark.parametrize("prec", ["bf16", "fp16"])
def test_shapes_outside_the_resident_kernels(ctx, dev, dims, M, prec):
    f16, tanh = prec == "fp16", int(dims[-1] != 3)
    P = synth.actor_params(dims, M, seed=sum(dims))
    ens = fr.ensemble_create(ctx, dims, P, precision=fr.PREC_FP16 if f16 else fr.PREC_BF16, out_act=tanh)
    n_max = 2 * 128 * ctx.sm_count + 77
    x = np.random.default_rng(7).standard_normal((n_max, dims[0])).astype(np.float32)
    xd = torch.from_numpy(x).to(dev)
    full = torch.empty(M, n_max, dims[-1], device=dev)
    fr.ensemble_forward(ens, xd, full)              # tiled
    for n in SIZES + (128 * ctx.sm_count - 128, 128 * ctx.sm_count - 127):   # single-agent, tiled
        y = torch.full((M, n, dims[-1]), -7.0, device=dev)
        fr.ensemble_forward(ens, xd[:n].contiguous(), y)
        torch.cuda.synchronize()
        assert torch.equal(y, full[:, :n])
    rows = np.r_[0:150, n_max - 130:n_max]
    got = full.cpu().numpy().astype(np.float64)
    for j in range(M):
        want, err = _forward16(dims, P[j], x[rows].astype(np.float64), f16, tanh)
        assert (np.abs(got[j, rows] - want) <= err).all()
    assert fr.ensemble_device_errors(ens) == 0


@pytest.mark.parametrize("dims,M", [((301, 256, 256, 30), 3), ((10, 128, 128, 3), 5), ((61, 64, 33), 2)])
@pytest.mark.parametrize("prec", [fr.PREC_FP8, fr.PREC_BF16X3])
def test_rows_do_not_depend_on_the_batch(ctx, dev, dims, M, prec):
    ens = fr.ensemble_create(ctx, dims, synth.actor_params(dims, M, seed=1), precision=prec)
    xd = torch.from_numpy(np.random.default_rng(7).standard_normal((1000, dims[0])).astype(np.float32)).to(dev)
    if prec == fr.PREC_FP8:
        fr.ensemble_calibrate_sync(ens, xd)
    full = torch.empty(M, 1000, dims[-1], device=dev)
    fr.ensemble_forward(ens, xd, full)
    for n in SIZES:
        y = torch.full((M, n, dims[-1]), -7.0, device=dev)
        fr.ensemble_forward(ens, xd[:n].contiguous(), y)
        torch.cuda.synchronize()
        assert torch.equal(y, full[:, :n])
    assert torch.isfinite(full).all() and fr.ensemble_device_errors(ens) == 0
