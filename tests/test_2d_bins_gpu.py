"""The 2D projector and adjoint at bin counts around the projector's tile of 32 bins and views around the sixteen a CTA may
take. Against the FP64 oracle to the suite's FP32 tolerance; a batch gives bit for bit what its images give."""
import math

import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu", [31, 32, 33, 63, 64, 65])
@pytest.mark.parametrize("views,arc", [(1, math.pi), (17, 0.02), (600, math.pi)])
def test_bins_around_a_tile(nu, views, arc):
    shape = (44, 39)
    args = (shape, (1.0, 0.9), nu, 70.0 / nu, views, arc)
    g, og = ops.Geometry.parallel2d(*args), oracle.parallel2d(*args)
    assert g.fp_config()["kernel"] == 6
    x = torch.from_numpy(inputs.uniform((3,) + shape, seed=91)).cuda()
    y = inputs.gaussian((views, nu), seed=92)
    p = ops.forward_project(x, g)
    for i in range(3):
        assert rel_l2(p[i].cpu().numpy(), oracle.fp(og, x[i].cpu().numpy().reshape(og.vol_shape))) <= 1e-5
        assert torch.equal(p[i], ops.forward_project(x[i].clone(), g))
    assert rel_l2(ops.adjoint(torch.from_numpy(y).cuda(), g).cpu().numpy(), oracle.adjoint(og, y.reshape(og.sino_shape))) <= 1e-5
    assert g.read_flags()[:4] == [0, 0, 0, 0]
