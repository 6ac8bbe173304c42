"""A coordination number of more than 40 A atoms keeps every switch value, also
one below the last place of the value added just before it.

A atoms at r = r0 (switch value 1/2) and at q = (r / r0)^2 = 512 (1 / (1 +
2^27), 1/4 of the last place of 1/2), 8 atoms of each in turn as the warps take
them; B atoms all at the origin. The same with the far atoms out of reach (no
value left) gives the close ones' sum, rounded alike, so the difference is the
far atoms' part alone: 2^-27 a pair to the reciprocal's last place and the
resolution of the sum's low part (2^-48 of ~5000), both below 1e-6 of it."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["short", "split", "split_full", "group"])
@pytest.mark.parametrize("na", [41, 48, 80, 85])
def test_small_switch_values_are_kept(form, na):
    from paper_1609_09833_gb300 import abp

    nb = 301
    nw, T = {"short": (1, 1), "split": (1, 3), "split_full": (900, 3), "group": (1, 1)}[form]
    far = np.arange(na) // 8 % 2 == 1
    sp = {"natoms": na + nb,
          "cvs": [{"type": "coord", "a": np.arange(na), "b": np.arange(na, na + nb), "r0": 0.5, "n": 6, "m": 12}],
          "grid": synth.grid((0.0,), (40000.0,), (64,), (False,)), "hill": synth.hill(0.5, [1000.0], 1000, 15.0)}
    s = []
    for out in (8.0, 30000.0):
        x = np.zeros((na + nb, 3), dtype=np.float32)
        x[:na, 0] = 0.5
        x[:na][far] = (out, out, 0.0)
        ctx = abp.Context(0)
        try:
            if form == "group":
                abp.abp_ctx_tune(ctx.handle, abp.ABP_TUNE_GROUP_THREADS, 128)
            ws = ctx.make_walkers([sp] * nw)
            rec = abp.to_records(np.repeat(x[None], T, axis=0)).cuda()  # the walkers' records are the same ones
            offs = torch.zeros(nw, dtype=torch.int64, device="cuda")
            F = torch.zeros(T, nw * x.shape[0], 4, device="cuda")
            foffs = torch.arange(nw, dtype=torch.int64, device="cuda") * x.shape[0]
            abp.abp_run(ctx.handle, ws, rec, abp.ABP_F32, offs, x.shape[0], F, foffs, nw * x.shape[0],
                        abp.ABP_FORCES_OVERWRITE, 1, T)
            torch.cuda.synchronize()
            s.append(ctx.readout(ws[-1])["s"][0])
        finally:
            torch.cuda.synchronize()
            ctx.close()
    part = far.sum() * nb / (1 + 2.0 ** 27)
    assert abs((s[0] - s[1]) - part) <= 1e-6 * part
