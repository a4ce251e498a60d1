"""The slab projector on volumes whose y-fastest copy would have unaligned rows (x-march boxes from the volume itself): edges of
tiles and slabs, storage types, batches, every arithmetic mode with the same bits, and a plan. Against the FP64 oracle to
the suite's tolerances."""
import math

import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu
TOL = {torch.float32: 1e-5, torch.bfloat16: 4e-3, torch.float16: 5e-4}


@pytest.mark.parametrize("shape,det,batch,dtype", [
    ((20, 33, 36), (17, 33), 1, torch.float32), ((31, 45, 40), (33, 50), 2, torch.bfloat16),
    ((9, 13, 16), (16, 16), 3, torch.float16), ((40, 70, 72), (48, 90), 1, torch.float32)])
def test_plain_staging(shape, det, batch, dtype):
    args = (shape, (0.5,) * 3, det, (0.8, 0.8), 9, 2 * math.pi, 300.0, 480.0)
    g, og = ops.Geometry.cone_circular(*args), oracle.cone_circular(*args)
    assert g.fp_config(dtype)["kernel"] == 3 and not g.fp_config(dtype)["y_fastest_x_march"]
    x = torch.from_numpy(inputs.uniform((batch,) + shape, seed=6)).to("cuda", dtype)
    p = ops.forward_project(x, g)
    for i in range(batch):
        assert rel_l2(p[i].float().cpu().numpy(), oracle.fp(og, x[i].float().cpu().numpy())) <= TOL[dtype]
    out = torch.empty_like(p[0])
    plan = ops.Plan([g], dtype)
    plan.forward_project([x[0]], [out])
    assert torch.equal(out, p[0])
    for mode in (1, 2):
        g.set_tuning(ops.TUNE_FP_PACKED, mode)
        assert torch.equal(ops.forward_project(x, g), p)
    assert g.read_flags()[:4] == [0, 0, 0, 0]
