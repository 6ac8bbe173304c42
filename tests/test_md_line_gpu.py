"""The closed loop of FP64 walkers of one COM distance with their coordinates
spread over warps (few walkers) against the general form (more walkers than
multiprocessors): the same bits, for odd atom counts, groups larger than a
half-warp, overlapping groups, periodic axes and boxes, potentials, recorded
trajectories and forces, and walkers that meet non-finite coordinates."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


def _spec(na, nb, extra, n, periodic, pbc, overlap, stride):
    a, b = np.arange(na), np.arange(na - overlap, na - overlap + nb)
    cv = {"type": "com_dist", "a": a, "b": b, "ma": 1.0 + 0.1 * np.arange(na), "pbc": pbc, "box": (2.9, 3.2, 3.5)}
    g = synth.grid((0.3,) if periodic else (-0.2,), (2.2,) if periodic else (1.5,), (n,), (periodic,))
    return {"natoms": na - overlap + nb + extra, "cvs": [cv], "grid": g, "hill": synth.hill(0.8, (0.05,), stride, 8.0)}


CASES = {"plain": (8, 8, 0, 512, False, False, 0, 10), "odd": (5, 23, 2, 97, False, False, 0, 7),
         "large": (40, 33, 1, 211, False, True, 0, 9), "overlap": (6, 7, 0, 128, False, False, 3, 5),
         "periodic": (3, 4, 1, 75, True, False, 0, 6), "single": (1, 1, 0, 60, False, True, 0, 4)}


@pytest.mark.parametrize("kind", CASES)
def test_few_walkers_move_as_many_do(kind):
    from paper_1609_09833_gb300 import abp

    spec = _spec(*CASES[kind])
    many, T = torch.cuda.get_device_properties(0).multi_processor_count + 3, 41
    r = np.random.default_rng(5)
    na = spec["natoms"]
    x0 = r.uniform(0.0, 1.5, size=(many, na, 4))
    x0[..., 3] = 7.0
    x0[2, na - 1, 1] = np.nan
    md = synth.md_double_well(seed=9) if kind != "odd" else synth.md_params(seed=9, mu=0.5)

    def run(idx):
        ctx = abp.Context(0)
        try:
            ws = ctx.make_walkers([spec] * len(idx), precision=abp.ABP_PREC_FP64)
            x = torch.as_tensor(x0[idx]).cuda().reshape(-1, 4).contiguous()
            offs = torch.arange(len(idx), dtype=torch.int64, device="cuda") * na
            A = len(idx) * na
            F = torch.full((T, A, 4), 0.5, dtype=torch.float64, device="cuda")
            tr = torch.zeros(T, A, 4, dtype=torch.float64, device="cuda")
            for t, n in ((0, 17), (17, 1), (18, T - 18)):
                abp.abp_md_run(ctx.handle, ws, x, abp.ABP_F64, offs, md, np.array(idx, dtype=np.uint32), traj=tr[t:],
                               traj_offsets=offs, traj_step_stride=A, forces=F[t:], force_offsets=offs,
                               force_step_stride=A, mode=abp.ABP_FORCES_ACCUMULATE, step0=t, nsteps=n)
            last = torch.zeros(A, 4, dtype=torch.float64, device="cuda")
            abp.abp_forces(ctx.handle, ws, last, abp.ABP_F64, offs, abp.ABP_FORCES_OVERWRITE)
            torch.cuda.synchronize()
            sh = (T, len(idx), na, 4)
            return (x.cpu().numpy().reshape(sh[1:]), F.cpu().numpy().reshape(sh), tr.cpu().numpy().reshape(sh),
                    last.cpu().numpy().reshape(sh[1:]), [ctx.bias(w) for w in ws], [ctx.readout(w) for w in ws])
        finally:
            torch.cuda.synchronize()
            ctx.close()

    big = run(list(range(many)))
    few = run([0, 1, 2, many - 1])
    for q, i in enumerate([0, 1, 2, many - 1]):
        assert np.array_equal(few[0][q], big[0][i], equal_nan=True)
        assert np.array_equal(few[1][:, q], big[1][:, i], equal_nan=True)
        assert np.array_equal(few[2][:, q], big[2][:, i], equal_nan=True)
        assert np.array_equal(few[4][q], big[4][i])
        assert few[5][q]["flags"] == big[5][i]["flags"]
        if i != 2:
            assert np.array_equal(few[3][q], big[3][i])
            assert few[5][q]["V"] == big[5][i]["V"] and np.array_equal(few[5][q]["dV"], big[5][i]["dV"])
