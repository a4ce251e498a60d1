"""Both sides of the lines below which small calls take the simpler kernels: the Ram-Lak filter at rows of 32 pixels, the motion
blur at 65536 samples, and the tiled kernels' edges above them. To the tolerances of the suite."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from oracle import artifacts as A
from paper_2511_08427_gb300 import artifacts, inputs, operators as ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu,dtype,tol", [(31, torch.float32, 1e-5), (32, torch.float32, 1e-5), (33, torch.bfloat16, 4e-3),
                                          (47, torch.float32, 1e-5)])
def test_ram_lak(nu, dtype, tol):
    args = ((4, 6, 6), (0.5,) * 3, (9, nu), (0.3, 0.3), 3, 2 * math.pi, 300.0, 480.0)
    g, og = ops.Geometry.cone_circular(*args), oracle.cone_circular(*args)
    x = torch.from_numpy(inputs.uniform((3, 9, nu), seed=nu)).to("cuda", dtype)
    got = ops.fbp_filter(x, g)
    assert rel_l2(got.float().cpu().numpy(), oracle.fbp_filter(og, x.float().cpu().numpy(), 0)) <= tol
    assert torch.equal(ops.fbp_filter(x, g, out=x), got)


@pytest.mark.parametrize("det,views,length", [((16, 31), 40, 6), ((33, 65), 20, 1), ((33, 65), 32, 1), ((16, 32), 18, 7), ((16, 32), 19, 7),
                                              ((100, 15), 60, 5), ((100, 16), 60, 5)])
def test_motion_blur(det, views, length):
    g = ops.Geometry.cone_circular((8, 8, 8), (0.5,) * 3, det, (0.8, 0.8), views, 2 * math.pi, 300.0, 480.0)
    p = torch.from_numpy(inputs.uniform(g.sinogram_shape, seed=78)).cuda()
    angles = np.linspace(-1.9, 2.5, views).astype(np.float32)
    out = artifacts.motion_blur(p, g, angles, length)
    assert rel_l2(out.double().cpu().numpy(), A.motion_blur(p.double().cpu().numpy(), angles, length)) <= 1e-5
