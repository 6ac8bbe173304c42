"""mABP windows in the form of one group per walker: hill by hill (hills far
apart, a union larger than their stencils) and node by node (a slow path) give
the bits of one-step calls, windows that change between the two included."""
import numpy as np
import pytest
import torch

from paper_1609_09833_gb300 import synth
from tests.test_split_gpu import _run, _same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [2, 3])
@pytest.mark.parametrize("stride", [1, 2])
def test_scattered_and_close_hills(d, stride):
    from paper_1609_09833_gb300 import abp

    cvs = [{"type": "com_dist", "a": np.arange(20), "b": np.arange(20, 40)},
           {"type": "dihedral", "a": np.arange(4)},
           {"type": "com_dist", "a": np.arange(2), "b": np.arange(2, 4)}][:d]
    g = synth.grid((0.0, -np.pi, 0.0)[:d], (3.0, np.pi, 2.0)[:d], (64, 64, 32)[:d], (False, True, False)[:d])
    h = synth.mabp_hill([synth.bins(g, k, 4.3) for k in range(d)], 4, 0.9, 0.05, stride=stride)
    specs = [{"natoms": 40, "cvs": cvs, "grid": g, "hill": h}] * 2
    r = np.random.default_rng(17)
    T = 96
    far = r.random((T, 80, 3))  # every step elsewhere
    near = r.random((1, 80, 3)) + 0.01 * r.random((T, 80, 3))
    x = np.where((np.arange(T) // 16 % 2 == 0)[:, None, None], far, near).astype(np.float32)
    one = _run(abp, specs, x, abp.ABP_FORCES_OVERWRITE, [1] * T)
    group = (abp.ABP_TUNE_GROUP_THREADS, 256)
    _same(one, _run(abp, specs, x, abp.ABP_FORCES_OVERWRITE, [T], knob=group))
    _same(one, _run(abp, specs, x, abp.ABP_FORCES_OVERWRITE, [8] * (T // 8)))
    _same(one, _run(abp, specs, x, abp.ABP_FORCES_OVERWRITE, [T]))
