"""FP64 closed loops of one COM distance in several blocks of steps (the noise
of a block fits 64 MB): coordinates, trajectories, forces, grids, states and
the count of stopped walkers as from one launch over all steps (a captured
call). One walker starts with a non-finite atom, one stops in the second block,
where its first hill is so high that it throws the atoms out of range."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu

NW, ATOMS, T = 150, 255, 160  # 918 kB of noise a step: blocks of 73, 73 and 14 steps


def _md(abp, captured, record):
    specs = []
    for i in range(NW):
        specs.append({"natoms": ATOMS, "cvs": [{"type": "com_dist", "a": np.arange(100), "b": np.arange(100, 210)}],
                      "grid": synth.grid((-2.0,), (4.0,), (512,), (False,)),
                      "hill": synth.hill(1e307 if i == 7 else 0.8, (0.05,), 100, 8.0)})
    x0 = np.random.default_rng(4).uniform(0.0, 1.5, size=(NW * ATOMS, 3))
    x0[:, 0] += (np.arange(NW * ATOMS) % ATOMS >= 100) * 0.8
    x0[3 * ATOMS + 20, 1] = np.nan
    ctx = abp.Context(0)
    try:
        ws = ctx.make_walkers(specs, precision=abp.ABP_PREC_FP64)
        u = np.linspace(0.0, 6.0, 512)
        for w in ws:  # a bias from the first step on
            ctx.upload_bias(w, np.stack([1.0 + np.cos(u), -np.sin(u)], 1))
        x = abp.to_records(x0[None])[0].contiguous().cuda()
        offs = torch.tensor(synth.offsets_of(specs), dtype=torch.int64, device="cuda")
        A = x.shape[0]
        F = torch.full((T if record else 1, A, 4), 0.5, dtype=torch.float64, device="cuda")
        traj = torch.zeros(T, A, 4, dtype=torch.float64, device="cuda") if record else None
        md = synth.md_double_well(seed=3)
        st = np.arange(NW, dtype=np.uint32)

        def call(t, n):
            if record:
                abp.abp_md_run(ctx.handle, ws, x, abp.ABP_F64, offs, md, st, traj=traj, traj_offsets=offs,
                               traj_step_stride=A, forces=F, force_offsets=offs, force_step_stride=A,
                               mode=abp.ABP_FORCES_ACCUMULATE, step0=t, nsteps=n)
            else:
                abp.abp_md_run(ctx.handle, ws, x, abp.ABP_F64, offs, md, st, step0=t, nsteps=n)

        def stopped():
            try:
                abp.abp_sync(ctx.handle)
            except abp.AbpError as e:
                return str(e)
            return ""

        call(1, 1)  # (caches the walker table)
        count = [stopped()]
        if captured:
            s = torch.cuda.Stream()
            torch.cuda.synchronize()
            ctx.set_stream(s.cuda_stream)
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                call(2, T)
            g.replay()
            torch.cuda.synchronize()
            ctx.set_stream(torch.cuda.current_stream().cuda_stream)
        else:
            call(2, T)
        count.append(stopped())
        if not record:
            abp.abp_forces(ctx.handle, ws, F[0], abp.ABP_F64, offs, abp.ABP_FORCES_OVERWRITE)
        torch.cuda.synchronize()
        return ([v.cpu().numpy() for v in (x, F) + ((traj,) if record else ())] + [ctx.bias(w) for w in ws],
                [ctx.readout(w) for w in ws], count)
    finally:
        torch.cuda.synchronize()
        ctx.close()


@pytest.mark.parametrize("record", [False, True])
def test_blocks_of_steps_equal_one_launch(record):
    from paper_1609_09833_gb300 import abp

    a, b = _md(abp, False, record), _md(abp, True, record)
    for u, v in zip(a[0], b[0]):
        assert np.array_equal(u, v, equal_nan=True)
    for u, v in zip(a[1], b[1]):
        assert u["flags"] == v["flags"] and u["status"] == v["status"]
        assert u["V"] == v["V"] and np.array_equal(u["s"], v["s"]) and np.array_equal(u["dV"], v["dV"])
    assert a[2] == b[2] and "1 walker steps" in a[2][0] and "2 walker steps" in a[2][1]
    assert [i for i, u in enumerate(a[1]) if u["flags"] & 8] == [3, 7]
