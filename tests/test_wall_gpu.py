"""The CV range wall acts on an FP32 CV's high and low part in every open-loop
form: its gradient against 64 bits on an empty bias.

Bound of |dU/ds / kwall - (s - smax)|, s a COM distance in [3, 4.5), smax = 3,
kwall a power of two: s_hi - smax is exact (Sterbenz), adding s_lo rounds the
difference once (2^-24 of it), and s_hi + s_lo is the distance to well below
2e-8 nm (each weighted offset is summed exactly split into high and low part).
The high part alone is up to 4e-7 nm off here."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu

KWALL, SMAX = 1024.0, 3.0


@pytest.mark.parametrize("form", ["short", "split", "group", "plain", "phased", "windowed", "windowed_mabp"])
def test_wall_gradient_of_a_com_distance(form):
    from paper_1609_09833_gb300 import abp

    na, nb, T = 8, 30, 70
    cvs = [{"type": "com_dist", "a": np.arange(na), "b": np.arange(na, na + nb)}]
    if not form.startswith("windowed"):
        cvs.append({"type": "coord", "a": np.arange(na), "b": np.arange(na, na + nb), "r0": 0.4, "n": 6, "m": 12})
    d = len(cvs)
    g = synth.grid((0.0,) * d, (8.0,) * d, (64,) * d, (False,) * d)
    # no hill before the last step: the grid is empty
    h = synth.mabp_hill([0.3] * d, 3, 0.5, 1.0, stride=1 << 40) if form == "windowed_mabp" else \
        synth.hill(0.5, [0.3] * d, 1 << 40, 15.0)
    sp = {"natoms": na + nb, "cvs": cvs, "grid": g, "hill": synth.with_wall(h, [SMAX] * d, KWALL)}
    if form == "phased":
        sp["shared"] = "g"
    ctx = abp.Context(0)
    try:
        if form == "group":
            abp.abp_ctx_tune(ctx.handle, abp.ABP_TUNE_GROUP_THREADS, 128)
        w = ctx.make_walkers([sp])
        offs = torch.zeros(1, dtype=torch.int64, device="cuda")
        for seed in range(24):
            x = np.random.default_rng(seed).random((T, na + nb, 3)).astype(np.float32)
            x[:, na:] += np.float32(2.1)
            rec = abp.to_records(x).cuda()
            F = torch.zeros_like(rec)
            n = T if form == "split" or form.startswith("windowed") else 1
            if form == "plain":
                abp.abp_step_plain(ctx.handle, w, rec, abp.ABP_F32, offs, F, offs, abp.ABP_FORCES_OVERWRITE, 1)
            else:
                abp.abp_run(ctx.handle, w, rec, abp.ABP_F32, offs, na + nb, F, offs, na + nb,
                            abp.ABP_FORCES_OVERWRITE, 1, n)
            torch.cuda.synchronize()
            y = x[n - 1].astype(np.float64)
            s = np.linalg.norm(y[na:].mean(0) - y[:na].mean(0))
            assert SMAX < s < 4.5
            err = ctx.readout(w[0])["dV"][0] / KWALL - (s - SMAX)
            assert abs(err) <= 2.0 ** -24 * (s - SMAX) + 2e-8, (seed, s, err)
    finally:
        torch.cuda.synchronize()
        ctx.close()
