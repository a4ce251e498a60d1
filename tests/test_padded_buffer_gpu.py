"""The buffer of padded copies is allocated by the first projection of a volume with unaligned rows: that must not disturb a
capture under way elsewhere, and choosing a kernel that needs no copies gives the buffer back."""
import math
import threading

import pytest
import torch

from paper_2511_08427_gb300 import operators as ops

pytestmark = pytest.mark.gpu


def unaligned():
    return ops.Geometry.cone_circular((65, 67, 69), (0.5,) * 3, (40, 70), (0.8, 0.8), 30, 2 * math.pi, 300.0, 480.0)


def test_first_projection_beside_a_capture():
    g = unaligned()
    assert g.fp_config()["kernel"] == 7
    x, out = torch.rand(g.volume_shape, device="cuda"), torch.empty(g.sinogram_shape, device="cuda")
    ops.back_project(out.zero_(), g)   # uploads the tables; the buffer is still missing
    z, other = torch.zeros(8, device="cuda"), torch.cuda.Stream()
    torch.cuda.synchronize()

    def project():
        with torch.cuda.stream(other):
            ops.forward_project(x, g, out)

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):   # the global capture mode
        z += 1
        t = threading.Thread(target=project)
        t.start()
        t.join()
    graph.replay()
    torch.cuda.synchronize()
    assert float(z[0]) == 1.0
    assert torch.equal(out, ops.forward_project(x, g))


def test_buffer_is_given_back():
    g = ops.Geometry.cone_circular((255, 255, 255), (0.5,) * 3, (20, 30), (0.8, 0.8), 2, 2 * math.pi, 750.0, 1200.0)
    assert g.fp_config()["kernel"] == 7
    x, out = torch.zeros(g.volume_shape, device="cuda"), torch.empty(g.sinogram_shape, device="cuda")
    ops.back_project(out.zero_(), g)
    torch.cuda.synchronize()
    size = 2 * 255 * 255 * 256 * 4
    before = torch.cuda.mem_get_info()[0]
    ops.forward_project(x, g, out)
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] >= size
    g.set_variant(0, 2)   # the thread-staged kernel
    assert before - torch.cuda.mem_get_info()[0] < size // 8
    ops.forward_project(x, g, out)
    g.set_variant(0, 0)
    ops.forward_project(x, g, out)
    torch.cuda.synchronize()
