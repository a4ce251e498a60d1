"""The 2D projector with many consecutive views per CTA (closely spaced views on several bin tiles), view counts that are not
a multiple of them, and the adjoint of the same scans. FP32 tolerance of the suite."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,nu,views", [("parallel", 330, 509), ("fan", 321, 1023), ("fan", 97, 1201)])
def test_many_views(kind, nu, views):
    shape, sp = (50, 61), (1.0, 0.9)
    if kind == "parallel":
        args = (shape, sp, nu, 0.3, views, math.pi)
        g, og = ops.Geometry.parallel2d(*args), oracle.parallel2d(*args)
    else:
        args = (shape, sp, nu, 0.5, views, 2 * math.pi, 300.0, 450.0)
        g, og = ops.Geometry.fan2d(*args), oracle.fan_circular(*args)
    x = torch.from_numpy(inputs.uniform(shape, seed=8))
    p = ops.forward_project(x.cuda(), g)
    assert rel_l2(p.cpu().numpy(), oracle.fp(og, x.numpy().reshape(og.vol_shape)).reshape(p.shape)) <= 1e-5
    y = inputs.gaussian((views, nu), seed=9)
    a = ops.adjoint(torch.from_numpy(np.ascontiguousarray(y)).cuda().float(), g)
    assert rel_l2(a.cpu().numpy(), oracle.adjoint(og, y.reshape(og.sino_shape)).reshape(a.shape)) <= 1e-5
    assert g.read_flags()[:4] == [0, 0, 0, 0]
