"""Motion blur on tiles staged in shared memory and beyond (long lines), at ragged tile edges, on detectors of few rows and
in half precision, against the FP64 reference. Tolerance: FP32 positions of up to 512 pixels are off by 8.8e-6 rms on each
axis; uniform values have a slope of 0.41 rms and 0.58 rms themselves, so a single tap is off by 9e-6 of the result."""
import math

import numpy as np
import pytest
import torch

from cases import rel_l2
from oracle import artifacts as A
from paper_2511_08427_gb300 import artifacts, inputs, operators as ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("det,length,dtype,tol", [
    ((1, 300), 5, torch.float32, 1e-5), ((1, 257), 78, torch.float32, 1e-5), ((5, 259), 8, torch.float32, 1e-5),
    ((9, 31), 2, torch.float32, 1e-5), ((16, 31), 6, torch.float32, 1e-5), ((33, 65), 1, torch.float32, 1e-5), ((64, 32), 7, torch.float16, 5e-4),
    ((120, 130), 77, torch.float32, 1e-5), ((120, 130), 78, torch.float32, 1e-5), ((40, 24), 300, torch.float32, 1e-5)])
def test_motion_blur_tiles(det, length, dtype, tol):
    g = ops.Geometry.cone_circular((8, 8, 8), (0.5,) * 3, det, (0.8, 0.8), 5, 2 * math.pi, 300.0, 480.0)
    p = torch.from_numpy(inputs.uniform((2,) + g.sinogram_shape, seed=77)).to("cuda", dtype)
    angles = np.array([0.0, 0.3, math.pi / 2, 2.5, -1.9], np.float32)
    out = artifacts.motion_blur(p, g, angles, length)
    for i in range(2):
        ref = A.motion_blur(p[i].double().cpu().numpy(), angles, length)
        assert rel_l2(out[i].double().cpu().numpy(), ref) <= tol


def test_angle_that_is_not_finite():
    g = ops.Geometry.cone_circular((8, 8, 8), (0.5,) * 3, (40, 70), (0.8, 0.8), 3, 2 * math.pi, 300.0, 480.0)
    p = torch.ones(g.sinogram_shape, device="cuda")
    out = artifacts.motion_blur(p, g, [0.0, math.nan, 1.0], 9)
    assert out[1].isnan().all() and not out[0].isnan().any() and not out[2].isnan().any()
