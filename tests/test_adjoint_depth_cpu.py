"""A slab depth set by hand that is the automatic one gives the automatic configuration (per-tile deeper slabs included), so
that the autotuner's depths hold the default; any other depth is the depth of every tile."""
import math

import pytest

from paper_2511_08427_gb300 import operators as ops


@pytest.mark.parametrize("side,det,du", [(48, 72, 0.8), (96, 144, 0.8), (160, 256, 0.6)])
def test_automatic_depth_by_hand(side, det, du):
    g = ops.Geometry.cone_circular((side,) * 3, (0.5,) * 3, (det, det), (du, du), 12, 2 * math.pi, 750.0, 1200.0)
    auto = g.adjoint_config()
    assert auto["kernel"] == 3
    g.set_tuning(ops.TUNE_ADJ_DEPTH, auto["depth"])
    assert g.adjoint_config() == auto
    for depth in (3, 4, 5, 6, 8):
        g.set_tuning(ops.TUNE_ADJ_DEPTH, depth)
        c = g.adjoint_config()
        assert c["depth"] == depth
        if depth != auto["depth"]:
            assert c["box_floats"] != auto["box_floats"]
    g.set_tuning(ops.TUNE_ADJ_DEPTH, 0)
    assert g.adjoint_config() == auto
