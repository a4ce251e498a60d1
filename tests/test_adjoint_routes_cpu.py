"""Which adjoint and which slab depth a scan gets: few detector tiles with boxes too large for two CTAs per SM take the bricks,
and per-tile deeper slabs (a box beyond the common depth's need) come only with enough CTAs."""
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


@pytest.mark.parametrize("views,deeper", [(8, False), (17, False), (18, True), (60, True)])
def test_deeper_slabs(views, deeper):
    g = cone((65, 80, 80), (89, 408), 0.25, views)   # 3 x 13 tiles
    c = g.adjoint_config()
    assert c["kernel"] == 3 and c["depth"] == 8
    g.set_tuning(ops.TUNE_ADJ_DEPTH, 12)
    whole = g.adjoint_config()["box_floats"]
    assert (c["box_floats"] >= whole) == deeper
