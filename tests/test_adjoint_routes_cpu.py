"""Which adjoint a scan gets: few detector tiles with boxes too large for two CTAs per SM take the bricks."""
import math

import pytest

from paper_2511_08427_gb300 import operators as ops


def cone(shape, det, du, views):
    return ops.Geometry.cone_circular(shape, (0.5,) * 3, det, (du, du), views, 2 * math.pi, 750.0, 1200.0)


@pytest.mark.parametrize("views,kernel", [(1, 2), (12, 2), (30, 3)])
def test_wide_pixels(views, kernel):
    g = cone((64, 64, 64), (13, 17), 4.4, views)   # one 32 x 32 tile
    assert g.adjoint_config()["kernel"] == kernel
    g.set_variant(1, 3)
    assert g.adjoint_config()["kernel"] == 3
