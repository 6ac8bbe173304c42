"""The memory of a phased-form walker counts against the context's budget,
its coordination number's partial sums included."""
import numpy as np
import pytest

from paper_1609_09833_gb300 import synth

pytestmark = pytest.mark.gpu


def test_a_phased_walkers_partial_sums_are_counted():
    from paper_1609_09833_gb300 import abp

    na, nb = 1500, 60000
    hi = 0.1 * na * nb
    sp = {"natoms": na + nb, "shared": "g",
          "cvs": [{"type": "coord", "a": np.arange(na), "b": np.arange(na, na + nb), "r0": 0.4, "n": 6, "m": 12}],
          "grid": synth.grid((0.0,), (hi,), (64,), (False,)), "hill": synth.hill(0.5, [hi / 30], 7, 15.0)}
    ctx = abp.Context(0)
    try:
        ctx.make_grid(sp["grid"], shared=True)
        grid = abp.abp_ctx_bytes(ctx.handle)[0]
    finally:
        ctx.close()
    ctx = abp.Context(0)
    try:
        ctx.make_walkers([sp])
        used = abp.abp_ctx_bytes(ctx.handle)[0]
    finally:
        ctx.close()
    # per atom its force record and six term codes, per list entry its index
    # and gradient record, per chunk of 384 B entries three sums an A atom
    atoms, chunks = na + nb, -(-nb // 384)
    assert used - grid >= atoms * (16 + 24) + atoms * (4 + 16) + chunks * na * 12
    for budget, fits in ((used, True), (used - 1, False)):
        ctx = abp.Context(0, budget=budget)
        try:
            if fits:
                ctx.make_walkers([sp])
                assert abp.abp_ctx_bytes(ctx.handle)[0] == used
            else:
                with pytest.raises(abp.AbpError) as e:
                    ctx.make_walkers([sp])
                assert e.value.code == abp.ABP_ERR_ADMISSION
                assert abp.abp_ctx_bytes(ctx.handle)[0] == grid  # nothing of the walker stays
        finally:
            ctx.close()
