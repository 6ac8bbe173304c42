"""abp_bias_readout into device memory comes after the work that the caller
queued before it on the default stream, whatever stream the context uses."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("own_stream", [False, True])
def test_readout_waits_for_the_default_streams_work(own_stream):
    from paper_1609_09833_gb300 import abp

    side = torch.cuda.Stream()  # (not ordered with the default stream by itself)
    ctx = abp.Context(0, stream=side.cuda_stream if own_stream else None)
    try:
        n = 300
        g = ctx.make_grid(synth.grid((0.0, 0.0), (1.0, 1.0), (n, n), (False, False)), abp.ABP_PREC_FP64)
        f = np.zeros((n * n, 4))
        f[:, :3] = np.random.default_rng(3).normal(size=(n * n, 3))
        abp.abp_grid_restore(ctx.handle, g, f.view(np.uint8).reshape(-1))
        dst = torch.empty(n * n, 3, dtype=torch.float64, device="cuda")
        other = torch.ones(64 << 20, device="cuda")
        torch.cuda.synchronize()
        for _ in range(20):  # over a millisecond of work ahead of the fill
            other.mul_(1.0)
        dst.fill_(7.0)
        abp.abp_bias_readout(ctx.handle, g, dst, True, abp.ABP_F64)
        torch.cuda.synchronize()
        assert np.array_equal(dst.cpu().numpy(), f[:, :3])
    finally:
        torch.cuda.synchronize()
        ctx.close()
