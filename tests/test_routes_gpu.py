"""Which kernels a call takes on both sides of the lines between the forms, and
that both sides give the same bits."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


def _call(abp, spec, nw, T, knob=0, fp64=False, md=False):
    """Kernel names of one call of T steps over nw walkers; its outputs."""
    ctx = abp.Context(0)
    try:
        if knob:
            abp.abp_ctx_tune(ctx.handle, abp.ABP_TUNE_GROUP_THREADS, knob)
        ws = ctx.make_walkers([spec] * nw, precision=abp.ABP_PREC_FP64 if fp64 else abp.ABP_PREC_FP32_COMP)
        n = spec["natoms"] * nw
        x = np.random.default_rng(T).random((1 if md else T, n, 3)) * 1.2
        rec = abp.to_records(x if fp64 else x.astype(np.float32)).cuda()
        F = torch.zeros(T, n, 4, dtype=rec.dtype, device="cuda")
        offs = torch.tensor(synth.offsets_of([spec] * nw), dtype=torch.int64, device="cuda")
        dt = abp.ABP_F64 if fp64 else abp.ABP_F32
        abp.abp_ctx_tune(ctx.handle, abp.ABP_TUNE_TIMING, 1)
        if md:
            abp.abp_md_run(ctx.handle, ws, rec[0], dt, offs, synth.md_double_well(seed=3),
                           np.zeros(nw, dtype=np.uint32), forces=F, force_offsets=offs, force_step_stride=n, nsteps=T)
        else:
            abp.abp_run(ctx.handle, ws, rec, dt, offs, n, F, offs, n, abp.ABP_FORCES_OVERWRITE, 0, T)
        torch.cuda.synchronize()
        names = set(abp.abp_kernel_times(ctx.handle))
        abp.abp_ctx_tune(ctx.handle, abp.ABP_TUNE_TIMING, 0)
        return names, [rec.cpu().numpy(), F.cpu().numpy(), ctx.bias(ws[0]), ctx.bias(ws[-1])]
    finally:
        torch.cuda.synchronize()
        ctx.close()


def _same(a, b):
    assert all(np.array_equal(u, v) for u, v in zip(a, b)) and a[1].any()


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


GROUP, ONE, SPLIT = {"k_run"}, {"k_sp_one"}, {"k_sp_cn", "k_sp_chain", "k_sp_cnf"}


@pytest.mark.parametrize("nl,npk,n,T,want", [
    (5, 20, "2s", 1, ONE), (5, 20, "2s+1", 1, GROUP), (40, 400, "2s+1", 1, GROUP), (41, 400, "2s+1", 1, SPLIT),
    (5, 20, 1, 2, GROUP), (40, 399, 3, 2, GROUP), (40, 400, 3, 2, SPLIT), (40, 49, "2s+1", 2, GROUP),
    (40, 50, "2s+1", 2, SPLIT), (5, 20, 16, 3, SPLIT), (5, 20, "2s", 3, GROUP), (5, 20, "2s+1", 3, SPLIT),
    (5, 20, 1, 4, SPLIT)])
def test_few_steps_of_coordination_numbers(nl, npk, n, T, want):
    from paper_1609_09833_gb300 import abp

    nw = {"2s": 2 * _sms(), "2s+1": 2 * _sms() + 1}.get(n, n)
    hi = 1.05 * nl * npk
    sp = {"natoms": nl + npk,
          "cvs": [{"type": "coord", "a": np.arange(nl), "b": np.arange(nl, nl + npk), "r0": 0.4, "n": 6, "m": 12}],
          "grid": synth.grid((0.0,), (hi,), (64,), (False,)), "hill": synth.hill(0.5, [hi / 20], 1, 15.0)}
    names, out = _call(abp, sp, nw, T)
    assert names == want
    group, ref = _call(abp, sp, nw, T, knob=128)
    assert group == GROUP
    _same(out, ref)


@pytest.mark.parametrize("natoms,T,line", [(16, 1, False), (99, 1, False), (100, 1, True), (49, 2, False),
                                           (50, 2, True), (16, 3, True)])
def test_few_steps_of_an_fp64_closed_loop(natoms, T, line):
    from paper_1609_09833_gb300 import abp

    sp = {"natoms": natoms, "cvs": [{"type": "com_dist", "a": np.arange(natoms // 2), "b": np.arange(natoms // 2, natoms)}],
          "grid": synth.grid((-2.0,), (4.0,), (512,), (False,)), "hill": synth.hill(0.8, (0.05,), 1, 8.0)}
    names, out = _call(abp, sp, 3, T, fp64=True, md=True)
    assert names == ({"k_md_noise", "k_md_line"} if line else {"k_md"})
    many, ref = _call(abp, sp, _sms() + 1, T, fp64=True, md=True)  # (more than one walker an SM: k_md)
    assert many == {"k_md"}
    n = 1 * natoms  # every walker has its own atoms but the first ones are drawn alike
    assert np.array_equal(out[0][:, :n], ref[0][:, :n]) and np.array_equal(out[1][:, :n], ref[1][:, :n])
    assert out[1].any() and np.array_equal(out[2], ref[2])


@pytest.mark.parametrize("natoms,d,stride,n,T,split", [
    (40, 2, 20, 3, 79, False), (40, 2, 20, 3, 80, True), (40, 2, 100, "s+1", 33, True), (200, 2, 20, 3, 64, True),
    (40, 1, 100, 3, 175, False), (40, 1, 100, 3, 176, True), (40, 1, 20, 3, 600, False), (40, 1, 1, 3, 300, False),
    (40, 1, 1 << 40, 3, 141, True), (200, 1, 20, 3, 64, True), (40, 1, 20, "s+1", 33, True)])
def test_long_calls_of_windowed_walkers(natoms, d, stride, n, T, split):
    from paper_1609_09833_gb300 import abp

    cvs = [{"type": "com_dist", "a": np.arange(natoms // 2), "b": np.arange(natoms // 2, natoms)},
           {"type": "dihedral", "a": np.arange(4)}][:d]
    g = synth.grid((0.0, -np.pi)[:d], (3.0, np.pi)[:d], (64, 64)[:d], (False, True)[:d])
    sp = {"natoms": natoms, "cvs": cvs, "grid": g,
          "hill": synth.hill(0.5, [synth.bins(g, k, 2.0) for k in range(d)], stride, 12.0)}
    nw = _sms() + 1 if n == "s+1" else n
    names, out = _call(abp, sp, nw, T)
    assert names == ({"k_sp_cv", "k_sp_chain", "k_sp_force"} if split else {"k_win"})
    group, ref = _call(abp, sp, nw, T, knob=256)
    assert group == {"k_win"}
    _same(out, ref)
