"""The brick kernel of the transposed back-projector with views enough to be taken (fewer updates go to the direct kernel), at the
edges of its bricks, and the two sides of that line. Whole results against the definition in plain FP64, to the
tolerances that every operator of this suite holds against FP64."""
import numpy as np
import pytest
import torch

from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops
from test_bp_transpose_gpu import TOL, geometry, transpose64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weight", [0, 1])
@pytest.mark.parametrize("shape,det,views,du,sid,pitch,batch,dtype", [
    ((33, 17, 15), (60, 70), 94, 0.8, 200.0, 0.0, 2, torch.float32),
    ((31, 15, 33), (19, 21), 103, 1.1, 200.0, 9.0, 1, torch.float32),       # overhangs the detector
    ((8, 40, 36), (30, 50), 137, 0.4, 200.0, 0.0, 1, torch.float32),        # flat, pixels finer than voxels
    ((34, 20, 18), (40, 44), 65, 0.8, 200.0, 0.0, 2, torch.bfloat16),
    ((64, 18, 20), (70, 44), 69, 0.8, 200.0, 0.0, 1, torch.float16),
    ((32, 32, 32), (40, 44), 47, 0.8, 200.0, 0.0, 1, torch.float32),        # 1.54e6 updates: the direct kernel
    ((32, 32, 32), (40, 44), 48, 0.8, 200.0, 0.0, 1, torch.float32)])       # 1.57e6: bricks
def test_bricks_match_definition(shape, det, views, du, sid, pitch, batch, dtype, weight):
    sdd = 320.0
    g = geometry(shape, det, views, du, sid, sdd, pitch)
    f = 1.0 if dtype != torch.float16 else 1e-2   # (sdd / sid)^2 sums stay within half precision
    x = (inputs.gaussian((batch,) + shape, seed=13) * f).astype(np.float32)
    xd = torch.from_numpy(x).to("cuda", dtype)
    got = ops.back_project_transpose(xd, g, ops.BP_INV_W2 if weight else ops.BP_PLAIN).float().cpu().numpy().astype(np.float64)
    xr = xd.float().cpu().numpy().astype(np.float64)
    for i in range(batch):
        assert rel_l2(got[i], transpose64(shape, det, views, du, sid, sdd, pitch, xr[i], weight)) <= TOL[dtype]


def test_source_inside_the_volume():
    """Bricks beside the source go voxel by voxel into global memory."""
    shape, det, views = (36, 48, 48), (50, 60), 19
    g = geometry(shape, det, views, 1.2, 9.0, 320.0)
    x = inputs.gaussian(shape, seed=13)
    got = ops.back_project_transpose(torch.from_numpy(x).cuda(), g, ops.BP_PLAIN).cpu().numpy()
    assert rel_l2(got, transpose64(shape, det, views, 1.2, 9.0, 320.0, 0.0, x.astype(np.float64), 0)) <= 1e-5
