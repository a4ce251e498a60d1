"""3D volumes of one plane (a single slice of a cone-beam scan) in the brick kernels: results against the FP64 oracle, and a
back-projection that does not compute planes the volume does not have."""
import math

import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu


def pair(shape, det, views):
    args = (shape, (0.5,) * 3, det, (0.9, 0.9), views, 2 * math.pi, 300.0, 480.0)
    return ops.Geometry.cone_circular(*args), oracle.cone_circular(*args)


@pytest.mark.parametrize("brick", [0, 4, 16])
@pytest.mark.parametrize("weight", [0, 1])
@pytest.mark.parametrize("side", [31, 33])
def test_one_plane(side, weight, brick):
    g, og = pair((1, side, side), (4, 45), 13)
    g.set_variant(1, 2)
    g.set_variant(2, 2)
    g.set_tuning(ops.TUNE_BP_BRICK_Z, brick)
    y = inputs.gaussian((13, 4, 45), seed=41)
    t = torch.from_numpy(y).cuda()
    assert rel_l2(ops.back_project(t, g, weight).cpu().numpy(), oracle.bp(og, y, weight)) <= 1e-5
    assert rel_l2(ops.adjoint(t, g).cpu().numpy(), oracle.adjoint(og, y)) <= 1e-5


def milliseconds(f):
    for _ in range(3):
        f()
    a, b = torch.cuda.Event(True), torch.cuda.Event(True)
    a.record()
    for _ in range(10):
        f()
    b.record()
    b.synchronize()
    return a.elapsed_time(b)


def test_one_plane_costs_less_than_eight():
    """One thread per voxel takes about a third of the time of one thread per eight; computing eight planes either way
    takes all of it."""
    times = []
    for nz in (1, 8):
        g, _ = pair((nz, 512, 512), (4, 701), 180)
        g.set_variant(2, 2)
        y = torch.rand(g.sinogram_shape, device="cuda")
        times.append(min(milliseconds(lambda: ops.back_project(y, g)) for _ in range(3)))
    assert times[0] < 0.7 * times[1]
