"""2D kernels at bins much wider and much finer than pixels, which change how a CTA's warps share the work: boxes loaded by
further warps (projector), lanes on spread rays (adjoint). Against the FP64 oracle to the suite's tolerances; a batch of
projections gives bit for bit what its images give."""
import math

import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu
TOL = {torch.float32: 1e-5, torch.bfloat16: 4e-3, torch.float16: 5e-4}


@pytest.mark.parametrize("kind", ["parallel", "fan"])
@pytest.mark.parametrize("shape,nu,px,views,batch,dtype", [
    ((130, 127), 40, 5.0, 7, 1, torch.float32), ((130, 127), 33, 6.0, 5, 5, torch.bfloat16), ((96, 300), 64, 6.0, 3, 2, torch.float16),
    ((60, 62), 90, 1.2, 9, 4, torch.bfloat16), ((40, 36), 500, 0.12, 6, 1, torch.float32), ((70, 33), 640, 0.15, 5, 3, torch.float32),
    ((33, 31), 300, 0.19, 4, 2, torch.float16), ((33, 31), 300, 0.21, 4, 1, torch.float32)])
def test_spacings(kind, shape, nu, px, views, batch, dtype):
    if kind == "parallel":
        args = (shape, (1.0, 1.0), nu, px, views, math.pi)
        g, og = ops.Geometry.parallel2d(*args), oracle.parallel2d(*args)
    else:
        args = (shape, (1.0, 1.0), nu, 1.5 * px, views, 2 * math.pi, 600.0, 900.0)
        g, og = ops.Geometry.fan2d(*args), oracle.fan_circular(*args)
    x = torch.from_numpy(inputs.uniform((batch,) + shape, seed=81)).to("cuda", dtype)
    y = torch.from_numpy(inputs.gaussian((batch, views, nu), seed=82)).to("cuda", dtype)
    p, a = ops.forward_project(x, g), ops.adjoint(y, g)
    for i in range(batch):
        assert rel_l2(p[i].float().cpu().numpy(), oracle.fp(og, x[i].float().cpu().numpy().reshape(og.vol_shape))) <= TOL[dtype]
        assert rel_l2(a[i].float().cpu().numpy(), oracle.adjoint(og, y[i].float().cpu().numpy().reshape(og.sino_shape))) <= TOL[dtype]
        assert torch.equal(p[i], ops.forward_project(x[i].clone(), g))
    assert g.read_flags()[:4] == [0, 0, 0, 0]
