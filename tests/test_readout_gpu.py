"""abp_bias_readout against the stored node records (abp_grid_save), converted
here in numpy: value + compensation in FP64, rounded once. Every grid
dimension, both precisions and output types, odd sizes, a grid of several
staging blocks, host and device destinations off their natural alignment."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(2,), (1021,), (3, 2), (129, 257), (5, 3, 7), (113, 109, 117)])
@pytest.mark.parametrize("fp64", [False, True])
def test_readout_equals_the_stored_records(n, fp64):
    from paper_1609_09833_gb300 import abp

    d = len(n)
    ctx = abp.Context(0)
    try:
        prec = abp.ABP_PREC_FP64 if fp64 else abp.ABP_PREC_FP32_COMP
        g = ctx.make_grid(synth.grid((0.0,) * d, (1.0,) * d, n, (False,) * d), prec)
        nodes, w = int(np.prod(n)), 2 if d == 1 else 4
        f = np.random.default_rng(7).normal(size=(nodes, w))
        f[:, 1 + d:] = 0
        if fp64:
            rec, want = f, f[:, :1 + d]
        else:
            hi = f.astype(np.float32)
            rec = np.concatenate([hi, (f - hi).astype(np.float32)], axis=1)
            want = rec[:, :w].astype(np.float64)[:, :1 + d] + rec[:, w:].astype(np.float64)[:, :1 + d]
        abp.abp_grid_restore(ctx.handle, g, np.ascontiguousarray(rec).view(np.uint8).reshape(-1))
        for dtype, t in ((abp.ABP_F64, np.float64), (abp.ABP_F32, np.float32)):
            bytes_ = nodes * (1 + d) * np.dtype(t).itemsize
            host = np.zeros(bytes_ + 3, dtype=np.uint8)
            dev = torch.zeros(bytes_ + 3, dtype=torch.uint8, device="cuda")
            for off in (0, 3):
                host[:], _ = 0, dev.zero_()
                torch.cuda.synchronize()
                abp.abp_bias_readout(ctx.handle, g, host.ctypes.data + off, False, dtype)
                abp.abp_bias_readout(ctx.handle, g, dev.data_ptr() + off, True, dtype)
                for got in (host, dev.cpu().numpy()):
                    assert np.array_equal(got[off:off + bytes_].copy().view(t).reshape(nodes, 1 + d), want.astype(t))
                    assert not got[:off].any() and not got[off + bytes_:].any()
    finally:
        torch.cuda.synchronize()
        ctx.close()
