"""Cosine weights of the filter on wide fans, where the squared source-pixel distance written as a polynomial from the row's
end cancels. A Ram-Lak row keeps 1 / 4 of an isolated value at its own column, so the weights can be read off directly."""
import math

import numpy as np
import pytest
import torch

from paper_2511_08427_gb300 import operators as ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nu,du,sdd,offset", [(512, 1.0, 1500.0, 0.0), (2047, 4.0, 400.0, 0.0), (4096, 4.0, 400.0, 0.0), (1500, 3.1, 410.0, 0.0), (1024, 2.0, 400.0, 900.0)])
def test_cosine_weights(nu, du, sdd, offset):
    """Relative to 64 bits. A pixel position of up to |x| from the vertex carries 2^-24 |x|, its square, the sum, the reciprocal
    root and the products a few times 2^-24: 8 x 2^-24 = 4.8e-7 covers them where the distance does not cancel."""
    g = ops.Geometry.fan2d((64, 64), (1.0, 1.0), nu, du, 9, 2 * math.pi, 0.6 * sdd, sdd, detector_offset=offset)
    cols = np.arange(0, nu, 7)
    x = torch.zeros((len(cols), 9, nu), device="cuda")
    x[torch.arange(len(cols)), 1, torch.from_numpy(cols)] = 1.0   # the view at 40 degrees
    got = ops.fbp_filter(x, g)[:, 1].cpu().numpy()[np.arange(len(cols)), cols].astype(np.float64)
    pos = (cols - 0.5 * (nu - 1)) * du + offset
    want = sdd / np.sqrt(sdd * sdd + pos * pos)
    scale = (got * want).sum() / (want * want).sum()   # the scan's constant, common to the row
    assert np.sqrt(np.mean((got / (scale * want) - 1.0) ** 2)) <= 4.8e-7
