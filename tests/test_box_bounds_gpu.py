"""Shared-memory boxes on scans that see the volume from one side: rays that diverge away from the source make the last slab of
full depth the widest, wider than the cut one behind it, and no view from the other side bounds it. Every slab must fit its
box (flags: samples off the box, rays outside the march, slabs that overflow, copies lost)."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu


def one_sided(views=5):
    """Angles of views whose source stands on the low side of x."""
    return math.pi + np.linspace(-0.5, 0.5, views)


@pytest.mark.parametrize("side", [116, 117, 145])   # 29 planes per slab: the last one cut to 1, 2 and 1
def test_projector_2d(side):
    t = one_sided()
    sid, sdd, nu, du = 100.0, 200.0, 400, 0.8
    P = np.zeros((len(t), 2, 3))
    P[:, 1, 0], P[:, 1, 1], P[:, 1, 2] = -np.cos(t) / sdd, -np.sin(t) / sdd, sid / sdd
    P[:, 0] = 0.5 * (nu - 1) * P[:, 1]
    P[:, 0, 0] += -np.sin(t) / du
    P[:, 0, 1] += np.cos(t) / du
    g = ops.Geometry.from_matrices2d((side, side), (1.0, 1.0), nu, du, P)
    assert g.fp_config()["kernel"] == 6
    x = inputs.uniform((side, side), seed=51)
    p = ops.forward_project(torch.from_numpy(x).cuda(), g).cpu().numpy()
    assert g.read_flags()[:4] == [0, 0, 0, 0]
    full = ops.Geometry.fan2d((side, side), (1.0, 1.0), nu, du, 8, 2 * math.pi, sid, sdd)
    q = ops.forward_project(torch.from_numpy(x).cuda(), full).cpu().numpy()
    assert rel_l2(p[2], q[4]) <= 2e-5   # the view at pi of a full scan; both within 1e-5 of the operator


@pytest.mark.parametrize("side,depth,turn", [(49, 10, 0.0), (55, 8, 0.0), (61, 15, 0.2), (64, 16, 0.2), (55, 0, 0.0)])
def test_adjoint_3d(side, depth, turn):
    t = np.array([math.pi + turn])
    sid, sdd, det, du = 50.0, 150.0, (256, 320), 0.5
    c, s, zero = np.cos(t), np.sin(t), np.zeros(len(t))
    src = np.stack([sid * c, sid * s, zero], 1)
    cen = np.stack([-(sdd - sid) * c, -(sdd - sid) * s, zero], 1)
    eu, ev = np.stack([-s, c, zero], 1), np.tile([0.0, 0.0, 1.0], (len(t), 1))
    args = ((side,) * 3, (1.0,) * 3, det, (du, du), src, cen, eu, ev)
    g, og = ops.Geometry.cone_from_positions(*args), oracle.cone_from_positions(*args)
    g.set_variant(1, 3)
    g.set_tuning(ops.TUNE_ADJ_DEPTH, depth)
    y = inputs.gaussian((len(t),) + det, seed=52)
    a = ops.adjoint(torch.from_numpy(y).cuda(), g).cpu().numpy()
    assert g.read_flags()[:4] == [0, 0, 0, 0]
    assert rel_l2(a, oracle.adjoint(og, y)) <= 1e-5
