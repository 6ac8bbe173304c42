"""abp_run with force records of consecutive steps that overlap without
coinciding (0 < |force_step_stride| < atoms): written in step order, as by one
call per step, in every form a call can take."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth
from tests.test_split_gpu import _frames, _specs

pytestmark = pytest.mark.gpu


def _run(abp, specs, frames, mode, stride, chunks, fp64=False):
    ctx = abp.Context(0)
    try:
        ws = ctx.make_walkers(specs, precision=abp.ABP_PREC_FP64 if fp64 else abp.ABP_PREC_FP32_COMP)
        dt = abp.ABP_F64 if fp64 else abp.ABP_F32
        rec = abp.to_records(frames.astype(np.float64) if fp64 else frames).cuda()
        T, A = rec.shape[0], rec.shape[1]
        offs = torch.tensor(synth.offsets_of(specs), dtype=torch.int64, device="cuda")
        # every walker's records in a region of their own, room on both sides
        room = T * abs(stride)
        first = torch.tensor([o + (2 * i + 1) * room for i, o in enumerate(synth.offsets_of(specs))],
                             dtype=torch.int64, device="cuda")
        F = torch.full((A + (2 * len(specs) + 2) * room, 4), 0.25, device="cuda", dtype=rec.dtype)
        t = 0
        for n in chunks:
            abp.abp_run(ctx.handle, ws, rec[t:], dt, offs, A, F, first + t * stride, stride, mode, t, n)
            t += n
        torch.cuda.synchronize()
        return F.cpu().numpy(), [ctx.bias(w) for w in ws]
    finally:
        torch.cuda.synchronize()
        ctx.close()


# (windowed and per-step walkers, two in a batch; short and long calls)
@pytest.mark.parametrize("kind,T,fp64", [("sweep", 5, False), ("sweep", 70, False), ("rmsd", 24, False),
                                         ("pocket_odd", 9, False), ("pocket_tiny", 40, False), ("sweep", 12, True)])
@pytest.mark.parametrize("stride", [1, 3, -2])
def test_overlapping_force_records_are_written_in_step_order(kind, T, fp64, stride):
    from paper_1609_09833_gb300 import abp

    specs = _specs(kind)[:2]
    frames = _frames(specs, T, 9)
    for mode in (abp.ABP_FORCES_OVERWRITE, abp.ABP_FORCES_ACCUMULATE):
        F, G = _run(abp, specs, frames, mode, stride, [T], fp64)
        f, g = _run(abp, specs, frames, mode, stride, [1] * T, fp64)
        assert np.array_equal(F, f) and F.any()
        assert all(np.array_equal(a, b) for a, b in zip(G, g))
