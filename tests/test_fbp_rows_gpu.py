"""The Ram-Lak filter kernel (half the products: taps of even offset are zero) at the edges of its blocks: rows from
one pixel to the longest accepted, row counts around the eight of a CTA, rows of several views in one CTA, storage
types, in place, and values that are not finite, which spoil their own row and no other. Against the FP64 oracle
to the suite's tolerances."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu
TOL = {torch.float32: 1e-5, torch.bfloat16: 4e-3, torch.float16: 5e-4}


@pytest.mark.parametrize("nu,nv,views,batch,dtype", [
    (1, 1, 1, 1, torch.float32), (2, 3, 2, 1, torch.float32), (15, 7, 3, 2, torch.float32), (16, 8, 3, 1, torch.float32),
    (17, 9, 2, 1, torch.bfloat16), (127, 5, 5, 1, torch.float32), (511, 3, 3, 1, torch.float16),
    (513, 1, 700, 1, torch.float32), (2049, 4, 2, 1, torch.float32), (4096, 3, 2, 1, torch.float32)])
def test_row_edges(nu, nv, views, batch, dtype):
    args = ((4, 6, 6), (0.5,) * 3, (nv, nu), (0.3, 0.3), views, 2 * math.pi, 300.0, 480.0)
    g, og = ops.Geometry.cone_circular(*args), oracle.cone_circular(*args)
    x = torch.from_numpy(inputs.uniform((batch, views, nv, nu), seed=nu)).to("cuda", dtype)
    got = ops.fbp_filter(x, g)
    for i in range(batch):
        ref = oracle.fbp_filter(og, x[i].float().cpu().numpy(), 0)
        assert rel_l2(got[i].float().cpu().numpy(), ref) <= TOL[dtype]
    assert torch.equal(ops.fbp_filter(x, g, out=x), got)


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_values_that_are_not_finite(bad):
    g = ops.Geometry.parallel2d((8, 8), (1.0, 1.0), 40, 1.0, 24, math.pi)
    x = torch.from_numpy(inputs.uniform((24, 40), seed=1)).cuda()
    want = ops.fbp_filter(x, g)
    x[5, 11] = bad
    got = ops.fbp_filter(x, g)
    rest = [i for i in range(24) if i != 5]
    assert torch.equal(got[rest], want[rest])
    assert not torch.isfinite(got[5]).any()
    if math.isnan(bad):
        assert torch.isnan(got[5]).all()
