"""Projections of one geometry with unaligned rows from several streams and threads at once: they share the padded copies and
must not see one another's volume."""
import math
import threading

import pytest
import torch

from paper_2511_08427_gb300 import operators as ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [1, 4])
def test_streams_share_the_copies(threads):
    g = ops.Geometry.cone_circular((65, 67, 69), (0.5,) * 3, (40, 70), (0.8, 0.8), 30, 2 * math.pi, 300.0, 480.0)
    assert g.fp_config()["kernel"] == 7
    xs = [torch.rand(g.volume_shape, device="cuda") for _ in range(4)]
    want = [ops.forward_project(x, g) for x in xs]
    outs = [[torch.empty_like(w) for _ in range(5)] for w in want]
    streams = [torch.cuda.Stream() for _ in xs]
    torch.cuda.synchronize()

    def work(ids):
        for k in range(5):
            for i in ids:
                with torch.cuda.stream(streams[i]):
                    ops.forward_project(xs[i], g, outs[i][k])

    parts = [[0, 1, 2, 3]] if threads == 1 else [[i] for i in range(4)]
    ts = [threading.Thread(target=work, args=(ids,)) for ids in parts]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    torch.cuda.synchronize()
    for w, os_ in zip(want, outs):
        assert all(torch.equal(w, o) for o in os_)
