"""Walkers the library refuses for their size, at the first size past each limit."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


def _cn_spec(na, nb, shared=None):
    hi = 1.1 * na * nb
    sp = {"natoms": na + nb,
          "cvs": [{"type": "coord", "a": np.arange(na), "b": np.arange(na, na + nb), "r0": 0.4, "n": 6, "m": 12}],
          "grid": synth.grid((0.0,), (hi,), (64,), (False,)), "hill": synth.hill(0.5, [hi / 30], 7, 15.0)}
    if shared is not None:
        sp["shared"] = shared
    return sp


def test_phased_coordination_numbers_take_1828_a_atoms():
    from paper_1609_09833_gb300 import abp

    ctx = abp.Context(0)
    try:
        ctx.make_walkers([_cn_spec(1828, 40, shared="g")])
        with pytest.raises(abp.AbpError) as e:
            ctx.make_walkers([_cn_spec(1829, 40, shared="h")])
        assert e.value.code == abp.ABP_ERR_UNSUPPORTED
    finally:
        ctx.close()


@pytest.mark.parametrize("na", [1500, 1000])
def test_walkers_past_one_groups_shared_memory_are_refused_in_every_form(na):
    """Fused walkers with a coordination number: 2500 atoms fit one SM at one
    warp a group; at the default four warps' A sums 1500 A atoms do not."""
    from paper_1609_09833_gb300 import abp

    ctx = abp.Context(0)
    try:
        sp = _cn_spec(na, 2500 - na)
        ws = ctx.make_walkers([sp])
        x = abp.to_records(np.random.default_rng(1).random((25, 2500, 3)).astype(np.float32)).cuda()
        F, offs = torch.zeros_like(x), torch.zeros(1, dtype=torch.int64, device="cuda")
        for T in (1, 25):
            def call():
                abp.abp_run(ctx.handle, ws, x, abp.ABP_F32, offs, 2500, F, offs, 2500, abp.ABP_FORCES_OVERWRITE, 0, T)
            if na == 1500:
                with pytest.raises(abp.AbpError) as e:
                    call()
                assert e.value.code == abp.ABP_ERR_UNSUPPORTED
            else:
                call()
        torch.cuda.synchronize()
        assert bool(F.any()) == (na == 1000)
    finally:
        torch.cuda.synchronize()
        ctx.close()
