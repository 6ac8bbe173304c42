"""A dihedral has the same bits in every kernel that evaluates it: short, split,
group and captured open-loop calls (walkers of windows and of coordination
numbers), the closed loop; with narrow hills (the angle in FP64),
wide ones and FP64 grids, with and without a periodic box."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [0.02, 0.1])
@pytest.mark.parametrize("pbc", [False, True])
@pytest.mark.parametrize("kind", ["windows", "fp64", "cn"])
def test_every_form_gives_the_same_dihedral(kind, pbc, sigma):
    from paper_1609_09833_gb300 import abp

    fp64, cn = kind == "fp64", kind == "cn"
    box = (3.1, 2.9, 3.3)
    cvs = [{"type": "dihedral", "a": np.array([3, 0, 2, 5]), "pbc": pbc, "box": box}]
    if cn:
        cvs.append({"type": "coord", "a": np.arange(3), "b": np.arange(3, 8), "r0": 0.4, "n": 6, "m": 12})
    d = len(cvs)
    g = synth.grid((-np.pi, 0.0)[:d], (np.pi, 16.0)[:d], (720, 16)[:d], (True, False)[:d])
    sp = {"natoms": 8, "cvs": cvs, "grid": g, "hill": synth.hill(0.5, [sigma, 2.0][:d], 1000, 12.0)}
    T = 70
    x = np.random.default_rng(8).uniform(-4.0, 4.0, size=(T, 8, 3)).astype(np.float64 if fp64 else np.float32)
    dt = abp.ABP_F64 if fp64 else abp.ABP_F32
    got = {}
    for form in ("short", "long", "group", "captured") + (() if cn else ("closed",)):
        ctx = abp.Context(0)
        try:
            if form == "group":
                abp.abp_ctx_tune(ctx.handle, abp.ABP_TUNE_GROUP_THREADS, 128 if cn else 256)
            w = ctx.make_walkers([sp], precision=abp.ABP_PREC_FP64 if fp64 else abp.ABP_PREC_FP32_COMP)
            field = np.zeros((int(np.prod(g["n"])), 1 + d))
            field[:, 1] = 3.0  # a force on every step, the same at every value of the CV
            ctx.upload_bias(w[0], field)
            rec = abp.to_records(x).cuda()
            F = torch.zeros_like(rec)
            offs = torch.zeros(1, dtype=torch.int64, device="cuda")
            st = np.zeros(1, dtype=np.uint32)

            def run(t, n):
                abp.abp_run(ctx.handle, w, rec[t:], dt, offs, 8, F[t:], offs, 8, abp.ABP_FORCES_OVERWRITE, 1 + t, n)

            if form in ("long", "group"):
                run(0, T)
            elif form == "captured":
                run(0, 1)  # (caches the walker table)
                side = torch.cuda.Stream()
                torch.cuda.synchronize()
                ctx.set_stream(side.cuda_stream)
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=side):
                    run(0, T)
                graph.replay()
                torch.cuda.synchronize()
                ctx.set_stream(torch.cuda.current_stream().cuda_stream)
            else:
                for t in range(T):
                    if form == "short":
                        run(t, 1)
                    else:
                        abp.abp_md_run(ctx.handle, w, rec[t].clone(), dt, offs, synth.md_params(seed=1, mu=0.1), st,
                                       forces=F[t:], force_offsets=offs, step0=1 + t, nsteps=1)
            torch.cuda.synchronize()
            got[form] = (ctx.readout(w[0])["s"][0], F.cpu().numpy())
        finally:
            torch.cuda.synchronize()
            ctx.close()
    for form, (s, F) in got.items():
        assert s == got["short"][0], form
        # (the closed loop adds the look-up's corners in another order)
        assert F.any() and (form == "closed" or np.array_equal(F, got["short"][1])), form
