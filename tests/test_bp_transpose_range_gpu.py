"""The transposed back-projector on volumes of a wide range: single voxels or a block far above the rest. The pixels that they do
not reach keep the accuracy that FP32 sums give them, the suite's 1e-5 relative to their own values, by themselves and
with accumulation in FP32 asked for."""
import numpy as np
import pytest
import torch

from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops
from test_bp_transpose_gpu import geometry, transpose64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("accum", [0, 1])
@pytest.mark.parametrize("big", [1.0e2, 1.0e4, 1.0e6])
@pytest.mark.parametrize("kind", ["voxel", "block"])
def test_wide_range(kind, big, accum):
    shape, det, views, du, sid, sdd = (36, 34, 33), (40, 60), 40, 0.8, 200.0, 320.0
    g = geometry(shape, det, views, du, sid, sdd)
    g.set_tuning(ops.TUNE_ADJ_ACCUM, accum)
    x = inputs.gaussian(shape, seed=71)
    hot = np.zeros(shape, dtype=np.float32)
    if kind == "voxel":
        hot[5::16, 3::16, 9::16] = 1.0
    else:
        hot[10:14, 12:18, 10:15] = 1.0
    x += np.float32(big) * hot
    free = transpose64(shape, det, views, du, sid, sdd, 0.0, hot, 1) < 1e-9
    assert free.sum() > 1000
    want = transpose64(shape, det, views, du, sid, sdd, 0.0, x.astype(np.float64), 1)
    got = ops.back_project_transpose(torch.from_numpy(x).cuda(), g, ops.BP_INV_W2).cpu().numpy()
    assert rel_l2(got, want) <= 1e-5
    assert rel_l2(got[free], want[free]) <= 1e-5
