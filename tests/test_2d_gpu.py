"""The 2D projector, adjoint and back-projector (kernels of their own, unlike the 3D tiles) at the edges of their tiles: bins
around a 128-bin tile, image sides around a brick, view counts around a group of views, batches around the
images per CTA, and values the fixed-point sums refuse. FP32 results hold rel-L2 1e-5 against the FP64 oracle
(the FP32 tolerance of every operator here), 16-bit storage the roundings of its type."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu
TOL = {torch.float32: 1e-5, torch.bfloat16: 4e-3, torch.float16: 5e-4}


def pair(kind, shape, nu, views, du=0.9):
    if kind == "parallel":
        return (ops.Geometry.parallel2d(shape, (1.0, 0.9), nu, du, views, math.pi),
                oracle.parallel2d(shape, (1.0, 0.9), nu, du, views, math.pi))
    return (ops.Geometry.fan2d(shape, (1.0, 0.9), nu, 1.5 * du, views, 2 * math.pi, 300.0, 450.0),
            oracle.fan_circular(shape, (1.0, 0.9), nu, 1.5 * du, views, 2 * math.pi, 300.0, 450.0))


def dev(a, dtype=torch.float32):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dtype)


def host(t):
    return t.float().cpu().numpy().astype(np.float64)


@pytest.mark.parametrize("kind", ["parallel", "fan"])
@pytest.mark.parametrize("shape,nu,views,batch,dtype", [
    ((1, 1), 1, 1, 1, torch.float32), ((31, 33), 127, 3, 2, torch.float32), ((32, 32), 128, 4, 3, torch.float32),
    ((63, 65), 129, 5, 4, torch.float32), ((64, 130), 257, 33, 5, torch.float32), ((70, 66), 96, 34, 1, torch.bfloat16),
    ((65, 40), 130, 7, 3, torch.float16), ((200, 190), 300, 301, 1, torch.float32)])
def test_tile_edges(kind, shape, nu, views, batch, dtype):
    g, og = pair(kind, shape, nu, views)
    assert g.fp_config(dtype)["kernel"] == 6
    x, y = inputs.uniform((batch,) + shape, seed=3), inputs.gaussian((batch, views, nu), seed=4)
    xd, yd = dev(x, dtype), dev(y, dtype)
    p, a = ops.forward_project(xd, g), ops.adjoint(yd, g)
    for i in range(batch):
        assert rel_l2(host(p[i]), oracle.fp(og, host(xd[i]).reshape(og.vol_shape))) <= TOL[dtype]
        assert rel_l2(host(a[i]), oracle.adjoint(og, host(yd[i]).reshape(og.sino_shape))) <= TOL[dtype]
        assert torch.equal(p[i], ops.forward_project(xd[i].clone(), g))
    assert g.read_flags()[:4] == [0, 0, 0, 0]


def test_sums_outside_fixed_point():
    """Rays so dense that one view's bound passes the fixed-point limit, values near the ends of the FP32 range,
    and a NaN (which reaches the pixels of its ray and no others)."""
    g, og = pair("parallel", (24, 24), 1500, 6, du=0.02)
    y = inputs.gaussian((6, 1500), seed=5)
    assert rel_l2(host(ops.adjoint(dev(y), g)), oracle.adjoint(og, y.reshape(og.sino_shape))) <= 1e-5
    g, og = pair("fan", (40, 36), 70, 9)
    y = inputs.gaussian((9, 70), seed=6)
    ref = oracle.adjoint(og, y.reshape(og.sino_shape)).reshape(40, 36)
    for f in (1e-35, 3e36):
        assert rel_l2(host(ops.adjoint(dev(y * np.float32(f)), g)) / f, ref) <= 1e-5
    y[4, 30] = np.nan
    one = np.zeros_like(y)
    one[4, 30] = 1.0
    hit = oracle.adjoint(og, one.reshape(og.sino_shape)).reshape(40, 36) > 0
    a = host(ops.adjoint(dev(y), g))
    assert np.isnan(a[hit]).all() and np.isfinite(a[~hit]).mean() > 0.95


@pytest.mark.parametrize("kind,weight", [("parallel", 0), ("fan", 0), ("fan", 1)])
@pytest.mark.parametrize("shape,nu,views,batch,dtype", [
    ((1, 1), 1, 1, 1, torch.float32), ((7, 9), 20, 3, 2, torch.float32), ((8, 8), 12, 257, 3, torch.float32),
    ((17, 33), 41, 255, 5, torch.bfloat16), ((384, 384), 70, 5, 1, torch.float32), ((385, 384), 600, 6, 4, torch.float32)])
def test_back_projector_edges(kind, weight, shape, nu, views, batch, dtype):
    """Images around a brick and around the size at which the brick changes, views around the 256 of a set-up."""
    g, og = pair(kind, shape, nu, views)
    y = dev(inputs.gaussian((batch, views, nu), seed=8), dtype)
    b = ops.back_project(y, g, weight)
    for i in range(batch):
        assert rel_l2(host(b[i]), oracle.bp(og, host(y[i]).reshape(og.sino_shape), weight)) <= TOL[dtype]
        assert torch.equal(b[i], ops.back_project(y[i].clone(), g, weight))
