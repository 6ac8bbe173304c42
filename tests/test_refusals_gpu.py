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
