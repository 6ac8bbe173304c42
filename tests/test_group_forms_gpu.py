"""Calls in the split form and the short form against the forms with a group
per walker at their default width (128 threads with a coordination number, 256
in windows; the width knob keeps a call in those forms): the same bits, also
for calls whose records need several blocks of steps or of walkers."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth
from tests.test_split_gpu import KINDS, _frames, _run, _same, _specs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", KINDS)
def test_split_and_short_calls_give_the_bits_of_a_group_per_walker(kind):
    from paper_1609_09833_gb300 import abp

    specs, T = _specs(kind), 67
    frames = _frames(specs, T, 11)
    frames[5, specs[0]["natoms"] - 1, 2] = np.nan
    for mode in (abp.ABP_FORCES_OVERWRITE, abp.ABP_FORCES_ACCUMULATE):
        group = _run(abp, specs, frames, mode, [T],
                     knob=(abp.ABP_TUNE_GROUP_THREADS, 128 if kind.startswith("pocket") else 256))
        _same(group, _run(abp, specs, frames, mode, [T]))
        _same(group, _run(abp, specs, frames, mode, [1] * T))


def _three_cn(na, nb, stride):
    """A walker with three coordination numbers over the same lists."""
    cvs = [{"type": "coord", "a": np.arange(na), "b": np.arange(na, na + nb), "r0": r, "n": 6, "m": 12}
           for r in (0.3, 0.4, 0.5)]
    g = synth.grid((0.0,) * 3, (1.05 * na * nb,) * 3, (14, 15, 16), (False,) * 3)
    return {"natoms": na + nb, "cvs": cvs, "grid": g,
            "hill": synth.hill(0.5, [synth.bins(g, k, 1.0) for k in range(3)], stride, 12.0)}


def _blocks(abp, specs, x, calls, knob=0):
    """Forces and grids of calls [(first walker, walkers, first step, steps)]."""
    ctx = abp.Context(0)
    try:
        if knob:
            abp.abp_ctx_tune(ctx.handle, abp.ABP_TUNE_GROUP_THREADS, knob)
        ws = ctx.make_walkers(specs)
        offs = torch.tensor(synth.offsets_of(specs), dtype=torch.int64, device="cuda")
        F = torch.full_like(x, 0.25)
        A = x.shape[1]
        for w, nw, t, n in calls:
            abp.abp_run(ctx.handle, ws[w:w + nw], x[t:], abp.ABP_F32, offs[w:], A, F[t:], offs[w:], A,
                        abp.ABP_FORCES_OVERWRITE, t, n)
        torch.cuda.synchronize()
        try:
            abp.abp_sync(ctx.handle)
            stopped = ""
        except abp.AbpError as e:
            stopped = str(e)
        return F, [ctx.bias(w) for w in ws], [ctx.readout(w) for w in ws], stopped
    finally:
        torch.cuda.synchronize()
        ctx.close()


def _equal(a, b):
    assert torch.equal(a[0], b[0]) and bool(a[0].any())
    assert all(np.array_equal(u, v) for u, v in zip(a[1], b[1]))
    for u, v in zip(a[2], b[2]):
        assert u["V"] == v["V"] and u["flags"] == v["flags"] and np.array_equal(u["s"], v["s"])
        assert np.array_equal(u["dV"], v["dV"])
    assert a[3] == b[3] and "2 walker steps" in a[3]


def _records(T, A, seed, spread):
    """Records that drift slowly over `spread` nm."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.zeros(T, A, 4, device="cuda")
    base = torch.rand(A, 3, generator=g, device="cuda")
    t = torch.linspace(0.0, 1.0, T, device="cuda")[:, None]
    for q in range(3):
        x[:, :, q] = base[:, q] * (0.6 + spread * t) + 0.01 * torch.randn(T, A, generator=g, device="cuda")
    return x


@pytest.mark.parametrize("kind", ["windows", "mabp", "cn"])
def test_several_blocks_of_steps(kind):
    """Blocks of at most 200,000 steps (one walker), and of what fits 240 MB of
    records (45,000 steps of 4 walkers with 3 x 60 gradient records); a last
    block that is shorter; non-finite steps in the first and second block."""
    from paper_1609_09833_gb300 import abp

    if kind == "cn":
        specs, T, cut = [_three_cn(20, 40, 500)] * 4, 45000, 19000
    else:
        sp = {"natoms": 6, "cvs": [{"type": "dihedral", "a": np.array([0, 1, 2, 3])},
                                   {"type": "com_dist", "a": np.arange(3), "b": np.arange(3, 6)}],
              "grid": synth.grid((-np.pi, 0.0), (np.pi, 2.0), (40, 30), (True, False))}
        sp["hill"] = synth.hill(0.5, [synth.bins(sp["grid"], k, 2.0) for k in range(2)], 500, 12.0) \
            if kind == "windows" else synth.mabp_hill([synth.bins(sp["grid"], k, 4.0) for k in range(2)], 4, 0.9, 0.05,
                                                      stride=50)
        specs, T, cut = [sp], 450001, 199990
    A = sum(s["natoms"] for s in specs)
    x = _records(T, A, 5, 0.3)
    x[100, 2, 0] = float("nan")
    x[cut + 400, A - 1, 1] = float("inf")
    n = len(specs)
    whole = _blocks(abp, specs, x, [(0, n, 0, T)])
    _equal(whole, _blocks(abp, specs, x, [(0, n, t, min(9000, T - t)) for t in range(0, T, 9000)]))
    _equal(whole, _blocks(abp, specs, x, [(0, n, 0, T)], knob=128 if kind == "cn" else 256))


def test_several_blocks_of_walkers():
    """1700 walkers with 3 x 1500 gradient records each: more than 240 MB in a
    single step, so blocks of walkers, each with its atoms' terms."""
    from paper_1609_09833_gb300 import abp

    specs, T = [_three_cn(20, 1480, 2), _three_cn(30, 1470, 3)] * 850, 2
    x = _records(T, 1700 * 1500, 6, 0.3)
    x[0, 1234, 0] = float("nan")
    x[1, 1650 * 1500, 0] = float("nan")
    whole = _blocks(abp, specs, x, [(0, 1700, 0, T)])
    _equal(whole, _blocks(abp, specs, x, [(w, 340, 0, T) for w in range(0, 1700, 340)]))
    _equal(whole, _blocks(abp, specs, x, [(0, 1700, 0, T)], knob=128))
