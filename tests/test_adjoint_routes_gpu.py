"""The autotuner on a scan whose automatic adjoint is the brick kernel because its detector tiles are few: the call is accepted, and
the adjoint stays the operator."""
import math

import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import autotune, inputs, operators as ops

pytestmark = pytest.mark.gpu


def test_tuning_few_tiles():
    args = ((64, 64, 64), (0.5,) * 3, (13, 17), (4.4, 4.4), 6, 2 * math.pi, 750.0, 1200.0)
    g, og = ops.Geometry.cone_circular(*args), oracle.cone_circular(*args)
    y = inputs.gaussian((6, 13, 17), seed=95)
    t = torch.from_numpy(y).cuda()
    assert g.adjoint_config()["kernel"] == 2
    want = oracle.adjoint(og, y)
    assert rel_l2(ops.adjoint(t, g).cpu().numpy(), want) <= 1e-5
    assert autotune.tune(g, "adjoint", use_cache=False)["candidates"] >= 1
    assert rel_l2(ops.adjoint(t, g).cpu().numpy(), want) <= 1e-5
    g.set_variant(1, 3)
    assert rel_l2(ops.adjoint(t, g).cpu().numpy(), want) <= 1e-5
