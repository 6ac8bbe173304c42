"""COM distances of more than 1280 atoms are summed in four parts: the same
bits from one warp, from any number of warps a group and from the forms of
short and long calls; the distance against 64 bits (hi + lo: every weighted
offset is summed with its exact error, 2e-8 nm leaves room for the weights)."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


def _spec(na, nb, cn):
    n = na + nb
    cvs = [{"type": "com_dist", "a": np.arange(na), "b": np.arange(na, n), "pbc": cn, "box": (9.0, 9.0, 9.0)},
           {"type": "com_dist", "a": np.arange(n - 40, n), "b": np.arange(n - 40)}]
    if cn:
        cvs.append({"type": "coord", "a": np.arange(4), "b": np.arange(n - 9, n), "r0": 0.4, "n": 6, "m": 12})
    d = len(cvs)
    g = synth.grid((0.0,) * d, (8.0, 8.0, 40.0)[:d], (20,) * d, (False,) * d)
    return {"natoms": n, "cvs": cvs, "grid": g, "hill": synth.hill(0.5, [synth.bins(g, k, 2.0) for k in range(d)], 3, 9.0)}


def _run(abp, specs, frames, chunks, threads):
    ctx = abp.Context(0)
    try:
        if threads:
            abp.abp_ctx_tune(ctx.handle, abp.ABP_TUNE_GROUP_THREADS, threads)
        ws = ctx.make_walkers(specs)
        rec = abp.to_records(frames).cuda()
        A = rec.shape[1]
        offs = torch.tensor(synth.offsets_of(specs), dtype=torch.int64, device="cuda")
        F = torch.zeros_like(rec)
        t = 0
        for n in chunks:
            abp.abp_run(ctx.handle, ws, rec[t:], abp.ABP_F32, offs, A, F[t:], offs, A, abp.ABP_FORCES_OVERWRITE, t, n)
            t += n
        torch.cuda.synchronize()
        return F.cpu().numpy(), [ctx.bias(w) for w in ws], [ctx.readout(w) for w in ws]
    finally:
        torch.cuda.synchronize()
        ctx.close()


@pytest.mark.parametrize("na,nb", [(640, 640), (640, 641), (1, 1500), (1029, 1001)])
@pytest.mark.parametrize("cn", [False, True])
def test_wide_com_sums_do_not_depend_on_the_form(na, nb, cn):
    from paper_1609_09833_gb300 import abp

    specs, T = [_spec(na, nb, cn)] * 2, 11
    n = na + nb
    x = np.random.default_rng(n).random((T, 2 * n, 3)) * 2.0
    x.reshape(T, 2, n, 3)[:, :, na:, 0] += 2.5
    frames = x.astype(np.float32)
    F, G, S = _run(abp, specs, frames, [T], 0)
    # other group widths change a coordination number's order, so only 128 then
    for chunks, threads in [([1] * T, 0)] + [([T], w) for w in ((128,) if cn else (32, 64, 128, 256))]:
        f, g, s = _run(abp, specs, frames, chunks, threads)
        assert np.array_equal(F, f) and all(np.array_equal(a, b) for a, b in zip(G, g))
        for a, b in zip(S, s):
            assert np.array_equal(a["s"], b["s"]) and np.array_equal(a["dV"], b["dV"]) and a["V"] == b["V"]
    y = frames[-1].astype(np.float64).reshape(2, n, 3)
    for i in range(2):
        v = y[i, na:].mean(0) - y[i, :na].mean(0)
        v -= 9.0 * np.floor(v / 9.0 + 0.5) if cn else 0.0
        u = y[i, :n - 40].mean(0) - y[i, n - 40:].mean(0)
        for got, want in zip(S[i]["s"], (np.linalg.norm(v), np.linalg.norm(u))):
            assert abs(got - want) <= 2e-8
