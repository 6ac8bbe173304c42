"""The split form of abp_run (its parts in launches of their own, over step
records) against the forms with a group per walker: the same bits, for every
kind of walker it takes, over deposits, non-finite steps, accumulated and
overlapping force records, blocks of steps and odd list sizes."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


def _pocket(nw, nl, npk, pbc, dims, stride=7, **hill):
    """Walkers with a coordination number on grids of 1 to 3 CVs."""
    lig, poc = np.arange(nl), np.arange(nl, nl + npk)[::-1].copy()
    box = (3.1, 3.3, 2.9)
    cn = {"type": "coord", "a": lig, "b": poc, "r0": 0.4, "n": 6, "m": 12, "pbc": pbc, "box": box}
    dist = {"type": "com_dist", "a": lig, "b": poc, "pbc": pbc, "box": box}
    dih = {"type": "dihedral", "a": np.array([0, 2, 1, 3])}
    hi = 0.03 * nl * npk + 2.0
    specs = []
    for i in range(nw):
        d = dims[i % len(dims)]
        axes = {1: [cn], 2: [dist, cn], 3: [dist, dih, cn]}[d]
        g = synth.grid((0.0,) + ((-np.pi,) if d == 3 else ()) + ((0.0,) if d > 1 else ()),
                       (hi,) if d == 1 else (2.0, hi) if d == 2 else (2.0, np.pi, hi),
                       (61,) if d == 1 else (45, 51) if d == 2 else (24, 26, 25),
                       (False,) if d == 1 else (False, False) if d == 2 else (False, True, False))
        sig = [synth.bins(g, k, 2.0) for k in range(d)]
        h = synth.hill(0.5, sig, stride, 12.0)
        if hill:
            h = synth.mabp_hill([synth.bins(g, k, 4.3) for k in range(d)], 4, 0.9, 0.05, stride=stride)
        specs.append({"natoms": nl + npk, "cvs": axes, "grid": g, "hill": h})
    return specs


def _frames(specs, T, seed):
    r = np.random.default_rng(seed)
    t = np.concatenate([r.uniform(0.5, 2.5, size=(s["natoms"], 3)) for s in specs])
    return (t[None] + 0.05 * r.normal(size=(T,) + t.shape)).astype(np.float32)


def _run(abp, specs, frames, mode, chunks, knob=None, stride_zero=False):
    ctx = abp.Context(0)
    try:
        if knob:
            abp.abp_ctx_tune(ctx.handle, *knob)
        ws = ctx.make_walkers(specs)
        rec = abp.to_records(frames).cuda()
        A, T = rec.shape[1], rec.shape[0]
        offs = torch.tensor(synth.offsets_of(specs), dtype=torch.int64, device="cuda")
        F = torch.full((A, 4) if stride_zero else tuple(rec.shape), 0.25, device="cuda")
        t = 0
        for n in chunks:
            abp.abp_run(ctx.handle, ws, rec[t:], abp.ABP_F32, offs, A, F if stride_zero else F[t:], offs,
                        0 if stride_zero else A, mode, t, n)
            t += n
        assert t == T
        torch.cuda.synchronize()
        state = [ctx.readout(w) for w in ws]
        return F.cpu().numpy(), [ctx.bias(w) for w in ws], state
    finally:
        torch.cuda.synchronize()
        ctx.close()


def _same(a, b):
    assert np.array_equal(a[0], b[0], equal_nan=True)
    for x, y in zip(a[1], b[1]):
        assert np.array_equal(x, y)
    for x, y in zip(a[2], b[2]):
        assert x["status"] == y["status"] and x["flags"] == y["flags"]
        if not x["flags"] & 8:
            assert x["V"] == y["V"] and np.array_equal(x["s"], y["s"]) and np.array_equal(x["dV"], y["dV"])


def _specs(kind):
    if kind == "sweep":
        return synth.mb64_specs(nw=5, n=(40, 36), stride=9, sigma=(0.08, 0.25))
    if kind == "sweep_wide":  # a deposit's box of one round
        return synth.mb64_specs(nw=3, n=(64, 64), stride=11, sigma=(0.03, 0.1))
    if kind == "rmsd":
        return synth.paper_rmsd_specs(nw=3, n=60, lo=0.0, hi=3.0, a_bins=5.0, stride=2)
    if kind == "mabp3":
        sp = {"natoms": 40, "cvs": [{"type": "com_dist", "a": np.arange(16), "b": np.arange(16, 32)},
                                    {"type": "dihedral", "a": np.arange(32, 36)},
                                    {"type": "com_dist", "a": np.arange(36, 38), "b": np.arange(38, 40)}],
              "grid": synth.grid((0.0, -np.pi, 0.0), (2.0, np.pi, 2.0), (23, 20, 21), (False, True, False))}
        sp["hill"] = synth.mabp_hill([synth.bins(sp["grid"], k, 3.0) for k in range(3)], 5, 0.9, 0.1)
        return [sp, dict(sp)]
    if kind == "mabp1":
        sp = {"natoms": 4, "cvs": [{"type": "dihedral", "a": np.arange(4)}],
              "grid": synth.grid((-np.pi,), (np.pi,), (37,), (True,))}
        sp["hill"] = synth.mabp_hill([synth.bins(sp["grid"], 0, 6.0)], 20, 0.9, 0.1, stride=3)
        return [sp]
    return {"pocket": _pocket(6, 40, 400, False, (1, 2, 3)), "pocket_odd": _pocket(3, 53, 307, True, (2, 3, 1)),
            "pocket_tiny": _pocket(3, 5, 7, False, (1, 2)), "pocket_big": _pocket(1, 7, 700, True, (2,)),
            "pocket_mabp": _pocket(2, 9, 50, False, (2, 3), mabp=True)}[kind]


KINDS = ["sweep", "sweep_wide", "rmsd", "mabp3", "mabp1", "pocket", "pocket_odd", "pocket_tiny", "pocket_big",
         "pocket_mabp"]


@pytest.mark.parametrize("kind", KINDS)
def test_split_form_gives_the_group_forms_bits(kind):
    """One long call (split) equals one-step calls (a group per walker), a
    call with the grid-tile knob set (which keeps the group forms) and calls
    of uneven lengths; overwritten and accumulated forces; a non-finite atom
    in one step."""
    from paper_1609_09833_gb300 import abp

    specs = _specs(kind)
    T = 101 if not kind.startswith("pocket") else 37
    frames = _frames(specs, T, 5)
    frames[17, specs[0]["natoms"] - 1, 1] = np.inf
    for mode in (abp.ABP_FORCES_OVERWRITE, abp.ABP_FORCES_ACCUMULATE):
        one = _run(abp, specs, frames, mode, [T])
        _same(one, _run(abp, specs, frames, mode, [1] * T))
        _same(one, _run(abp, specs, frames, mode, [T], knob=(abp.ABP_TUNE_TILE, 1)))
        _same(one, _run(abp, specs, frames, mode, [5, T - 30, 25]))


@pytest.mark.parametrize("kind", ["sweep", "pocket"])
def test_split_form_adds_overlapping_records_in_step_order(kind):
    """force_step_stride = 0: every step's force added to one record set, in
    the order of the steps (the same bits as one call per step)."""
    from paper_1609_09833_gb300 import abp

    specs = _specs(kind)
    T = 70
    frames = _frames(specs, T, 6)
    for mode in (abp.ABP_FORCES_OVERWRITE, abp.ABP_FORCES_ACCUMULATE):
        a = _run(abp, specs, frames, mode, [T], stride_zero=True)
        _same(a, _run(abp, specs, frames, mode, [1] * T, stride_zero=True))


@pytest.mark.parametrize("nw", [1, 3, 700])
def test_many_walkers_give_the_bits_of_one(nw):
    """A batch that fills the chip takes one step a warp, a small one a step
    a CTA: a walker's forces and grid do not depend on which."""
    from paper_1609_09833_gb300 import abp

    specs = _pocket(nw, 11, 90, False, (1, 2, 3))
    frames = _frames(specs, 9, 8)
    F, G, _ = _run(abp, specs, frames, abp.ABP_FORCES_OVERWRITE, [9])
    offs = synth.offsets_of(specs)
    for i in {0, nw // 2, nw - 1}:
        na = specs[i]["natoms"]
        f, g, _ = _run(abp, [specs[i]], frames[:, offs[i]:offs[i] + na], abp.ABP_FORCES_OVERWRITE, [9])
        assert np.array_equal(f, F[:, offs[i]:offs[i] + na]) and np.array_equal(g[0], G[i])


@pytest.mark.parametrize("form", ["sweep", "pocket", "double_well"])
def test_captured_calls_take_forms_without_scratch(form):
    """A long abp_run and an FP64 abp_md_run captured in a CUDA graph give the
    bits of the direct calls, and the graph can be cloned (one with memory
    nodes cannot)."""
    import ctypes

    from paper_1609_09833_gb300 import abp

    T, runs = 70, []
    md = form == "double_well"
    well = {"natoms": 16, "cvs": [{"type": "com_dist", "a": np.arange(8), "b": np.arange(8, 16)}],
            "grid": synth.grid((-2.0,), (4.0,), (512,), (False,)), "hill": synth.hill(0.8, (0.05,), 10, 8.0)}
    specs = [well] if md else _specs(form)
    x0 = np.random.default_rng(4).uniform(0.0, 1.5, size=(1, specs[0]["natoms"], 3))
    frames = x0 if md else _frames(specs, 2 * T, 7)
    for captured in (False, True):
        ctx = abp.Context(0)
        try:
            ws = ctx.make_walkers(specs, precision=abp.ABP_PREC_FP64 if md else abp.ABP_PREC_FP32_COMP)
            x = (torch.as_tensor(np.concatenate([frames, np.ones_like(frames[..., :1])], 2)) if md
                 else abp.to_records(frames)).cuda()
            A = x.shape[1]
            F = torch.zeros_like(x)
            offs = torch.tensor(synth.offsets_of(specs), dtype=torch.int64, device="cuda")

            def call(t):
                if md:
                    abp.abp_md_run(ctx.handle, ws, x[0], abp.ABP_F64, offs, synth.md_double_well(seed=3),
                                   np.zeros(1, dtype=np.uint32), step0=t, nsteps=T)
                else:
                    abp.abp_run(ctx.handle, ws, x[t:], abp.ABP_F32, offs, A, F[t:], offs, A,
                                abp.ABP_FORCES_OVERWRITE, t, T)

            call(0)  # (caches the walker table)
            if captured:
                s = torch.cuda.Stream()
                torch.cuda.synchronize()
                ctx.set_stream(s.cuda_stream)
                g = torch.cuda.CUDAGraph(keep_graph=True)
                with torch.cuda.graph(g, stream=s):
                    call(T)
                rt, copy = ctypes.CDLL("libcudart.so.13"), ctypes.c_void_p()
                assert rt.cudaGraphClone(ctypes.byref(copy), ctypes.c_void_p(g.raw_cuda_graph())) == 0
                assert rt.cudaGraphDestroy(copy) == 0
                g.instantiate()
                g.replay()
                torch.cuda.synchronize()
                ctx.set_stream(torch.cuda.current_stream().cuda_stream)
            else:
                call(T)
            torch.cuda.synchronize()
            runs.append((x.cpu().numpy(), F.cpu().numpy(), [ctx.bias(w) for w in ws]))
        finally:
            torch.cuda.synchronize()
            ctx.close()
    assert np.array_equal(runs[0][0], runs[1][0]) and np.array_equal(runs[0][1], runs[1][1])
    for a, b in zip(runs[0][2], runs[1][2]):
        assert np.array_equal(a, b)
