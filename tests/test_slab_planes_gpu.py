"""Slab boxes without guard planes (steps below a voxel: a sample that rounding puts across its slab's end is moved onto
it) and with them (longer steps), in the projector and the matched adjoint; adjoint tiles that take deeper slabs than
the configured depth; views along the axes and the diagonals, near and far sources. Against the FP64 oracle to the
suite's tolerance, with no sample outside its box and no slab that does not fit."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("step", [None, 0.11, 0.499, 0.5, 0.8, 1.7])
@pytest.mark.parametrize("shape,det,du,views,sid", [
    ((40, 64, 72), (40, 66), 0.9, 8, 750.0), ((33, 50, 52), (48, 70), 0.4, 5, 60.0), ((72, 24, 28), (90, 40), 0.7, 4, 200.0)])
def test_slab_ends(shape, det, du, views, sid, step):
    args = (shape, (0.5,) * 3, det, (du, du), views, 2 * math.pi, sid, 1.6 * sid)
    g, og = ops.Geometry.cone_circular(*args), oracle.cone_circular(*args)
    if step is not None:
        g.step = step
        og.dt = step
    x, y = inputs.uniform(shape, seed=1), inputs.gaussian((views,) + det, seed=2)
    p = ops.forward_project(torch.from_numpy(x).cuda(), g).cpu().numpy()
    a = ops.adjoint(torch.from_numpy(y).cuda(), g).cpu().numpy()
    assert rel_l2(p, oracle.fp(og, x)) <= 1e-5
    assert rel_l2(a, oracle.adjoint(og, y)) <= 1e-5
    flags = g.read_flags()
    assert flags[:4] == [0, 0, 0, 0]
    auto = g.adjoint_config()["depth"]
    g.set_tuning(ops.TUNE_ADJ_DEPTH, 5)   # every tile at one depth
    b = ops.adjoint(torch.from_numpy(y).cuda(), g).cpu().numpy()
    assert rel_l2(b, a) <= 2e-5   # each within 1e-5 of the oracle
    g.set_tuning(ops.TUNE_ADJ_DEPTH, 0)
    flat = g.read_flags()
    if auto >= 5:
        assert flat[4] + flat[5] >= flags[4] + flags[5]   # slabs: deeper ones are fewer
