"""Host-buffer projection of 2D images, whose views go in chunks of whole groups (the views that share a CTA): 37 closely spaced
views of 2000 bins make groups of eight, so of the eight chunks some are empty and the last group is ragged. Bit for bit
the device-buffer projection."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2511_08427_gb300 import _lib, inputs, operators as ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("dtype,batch", [(torch.float32, 2), (torch.bfloat16, 3)])
@pytest.mark.parametrize("views,nu", [(37, 2000), (3, 65)])
def test_host_projection(views, nu, dtype, batch, pinned):
    g = ops.Geometry.parallel2d((64, 70), (1.0, 1.0), nu, 100.0 / nu, views, 0.005 * views)
    assert g.fp_config(dtype)["kernel"] == 6
    x = torch.from_numpy(np.stack([inputs.uniform((64, 70), seed=60 + b) for b in range(batch)])).to(dtype)
    want = ops.forward_project(x.cuda(), g).cpu()
    got = torch.full(tuple(want.shape), float("nan"), dtype=dtype)
    if pinned:
        x, got = x.pin_memory(), got.pin_memory()
    code = {torch.float32: _lib.F32, torch.bfloat16: _lib.BF16}[dtype]
    _lib.check(_lib.lib().pyronn_fp_host(g.handle, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(got.data_ptr()), code,
                                         batch, None))
    assert torch.equal(got, want)
