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


@pytest.mark.parametrize("accum", [0, 1])
@pytest.mark.parametrize("big", [1.0e2, 1.0e4, 1.0e6])
@pytest.mark.parametrize("kind", ["bin", "band"])
@pytest.mark.parametrize("batch", [1, 3])
def test_adjoint_of_a_wide_range(batch, kind, big, accum):
    """A hot bin in some views, or a band of hot bins in all: the pixels it does not reach keep the accuracy that FP32 sums
    give them, the suite's 1e-5 relative to their own values (by themselves, and with accumulation in FP32 asked for)."""
    shape, nu, views = (128, 132), 200, 180
    args = (shape, (1.0, 1.0), nu, 1.0, views, math.pi)
    g, og = ops.Geometry.parallel2d(*args), oracle.parallel2d(*args)
    g.set_tuning(ops.TUNE_ADJ_ACCUM, accum)
    y = inputs.gaussian((batch, views, nu), seed=32)
    hot = np.zeros((views, nu), dtype=np.float32)
    if kind == "bin":
        hot[::7, nu // 2] = 1.0
    else:
        hot[:, 30:50] = 1.0
    y[-1] += np.float32(big) * hot
    free = oracle.adjoint(og, hot.reshape(og.sino_shape)).reshape(shape) < 1e-9
    assert free.sum() > 1000
    a = ops.adjoint(torch.from_numpy(y[0] if batch == 1 else y).cuda(), g).cpu().numpy().reshape((batch,) + shape)
    for b in range(batch):
        want = oracle.adjoint(og, y[b].reshape(og.sino_shape)).reshape(shape)
        assert rel_l2(a[b], want) <= 1e-5
        assert rel_l2(a[b][free], want[free]) <= 1e-5
