"""Projection of volumes whose rows are not a multiple of 16 bytes, from padded copies: odd sizes around the alignment,
storage types, batches, with and without the y-fastest copy, first calls inside a stream capture (no buffer yet:
the thread-staged kernel), and volumes in a plan. Against the FP64 oracle to the suite's tolerances."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu
TOL = {torch.float32: 1e-5, torch.bfloat16: 4e-3, torch.float16: 5e-4}


def pair(shape, views=7):
    args = (shape, (0.5,) * 3, (33, 50), (0.8, 0.8), views, 2 * math.pi, 300.0, 480.0)
    return ops.Geometry.cone_circular(*args), oracle.cone_circular(*args)


@pytest.mark.parametrize("transpose", [0, 1])
@pytest.mark.parametrize("shape,batch,dtype", [
    ((32, 32, 33), 1, torch.float32), ((33, 35, 34), 2, torch.float32), ((30, 40, 35), 1, torch.float32),
    ((36, 31, 36), 3, torch.bfloat16), ((35, 33, 43), 1, torch.float16), ((64, 9, 61), 1, torch.float32)])
def test_padded_copies(shape, batch, dtype, transpose):
    g, og = pair(shape)
    g.set_tuning(ops.TUNE_FP_TRANSPOSE, transpose)
    assert g.fp_config(dtype)["kernel"] == 7 and g.fp_config(dtype)["y_fastest_x_march"] == (transpose == 0)
    x = torch.from_numpy(inputs.uniform((batch,) + shape, seed=4)).to("cuda", dtype)
    p = ops.forward_project(x, g)
    for i in range(batch):
        assert rel_l2(p[i].float().cpu().numpy(), oracle.fp(og, x[i].float().cpu().numpy())) <= TOL[dtype]
        assert torch.equal(p[i], ops.forward_project(x[i].clone(), g))
    assert g.read_flags()[:4] == [0, 0, 0, 0]


def test_capture_without_a_buffer_and_plan():
    shape = (33, 35, 34)
    g, og = pair(shape)
    y = torch.zeros((1,) + g.sinogram_shape, device="cuda")
    ops.adjoint(y[0], g)   # uploads the tables; the projection's buffer is still missing
    x = torch.from_numpy(inputs.uniform(shape, seed=5)).cuda()
    out = torch.empty(g.sinogram_shape, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ops.forward_project(x, g, out)
    graph.replay()
    torch.cuda.synchronize()
    want = oracle.fp(og, x.cpu().numpy())
    assert rel_l2(out.cpu().numpy(), want) <= 1e-5
    h, _ = pair((40, 32, 32))
    plan = ops.Plan([g, h])
    xs = [x, torch.rand(h.volume_shape, device="cuda")]
    ps = [torch.empty(k.sinogram_shape, device="cuda") for k in (g, h)]
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        plan.forward_project(xs, ps)
    graph.replay()
    torch.cuda.synchronize()
    assert rel_l2(ps[0].cpu().numpy(), want) <= 1e-5
