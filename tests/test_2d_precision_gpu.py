"""Accuracy of the 2D matched adjoint against the FP64 oracle beyond the suite's common tolerance: white noise, whose adjoint
shows every error of the sample positions, on bricks of 32^2 and 64^2 pixels."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu


def fan(shape, nu, views):
    args = (shape, (0.5, 0.5), nu, 1.0, views, 2 * math.pi, 1000.0, 1500.0)
    return ops.Geometry.fan2d(*args), oracle.fan_circular(*args)


@pytest.mark.parametrize("shape,nu,views", [((256, 256), 512, 360), ((96, 100), 200, 90)])
def test_adjoint_of_noise(shape, nu, views):
    """FP32 positions of up to 32 pixels from the brick's centre carry about 0.4e-6 pixel rms from their own rounding and as
    much from each of the ray's offset and direction, 0.7e-6 per axis; white noise turns a shift of d pixels along an axis
    into a relative error of sqrt(3) d (the hat's slope against the hat, in the mean square), so 1.7e-6 over two axes."""
    g, og = fan(shape, nu, views)
    y = inputs.gaussian((views, nu), seed=31)
    a = ops.adjoint(torch.from_numpy(y).cuda(), g).cpu().numpy()
    assert rel_l2(a, oracle.adjoint(og, y.reshape(og.sino_shape)).reshape(shape)) <= 1.7e-6
