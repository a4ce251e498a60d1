"""The brick kernel of the transposed back-projector at the edges of its bricks (16 x 16 x 32) and of its use: volumes of
one voxel more and less than a brick, flat ones, views whose source stands inside the volume, detectors the
volume overhangs, dense and sparse detectors, storage types and batches. Whole results against the definition in
plain FP64, to the tolerances that every operator of this suite holds against FP64 (FP32 1e-5; 16-bit storage: its
rounding).
"""
import math

import numpy as np
import pytest
import torch

from cases import rel_l2
from paper_2511_08427_gb300 import inputs, operators as ops

pytestmark = pytest.mark.gpu
TOL = {torch.float32: 1e-5, torch.bfloat16: 4e-3, torch.float16: 5e-4}


def geometry(shape, det, views, du, sid=200.0, sdd=320.0, pitch=0.0):
    return ops.Geometry.cone_circular(shape, (0.5,) * 3, det, (du, du), views, 2 * math.pi, sid, sdd, helical_pitch=pitch)


def transpose64(shape, det, views, du, sid, sdd, pitch, x, weighted):
    """BP^T in plain FP64 from the geometry's definition (circular or helical orbit, detector centred on the axis)."""
    out = np.zeros((views,) + det)
    z, y, xx = np.meshgrid(*[(np.arange(n) - 0.5 * (n - 1)) * 0.5 for n in shape], indexing="ij")
    for n in range(views):
        t = n * 2 * math.pi / views
        zn = pitch * (n - 0.5 * (views - 1)) / views
        c, s = math.cos(t), math.sin(t)
        depth = sid - (xx * c + y * s)
        ok = depth > 0
        w = np.where(ok, depth, 1.0) / sdd
        u = (-xx * s + y * c) / w / du + 0.5 * (det[1] - 1)
        v = (z - zn) / w / du + 0.5 * (det[0] - 1)
        val = np.where(ok, x / w ** 2 if weighted else x, 0.0)
        iu, iv = np.floor(u).astype(np.int64), np.floor(v).astype(np.int64)
        for a in (0, 1):
            for b in (0, 1):
                wt = np.abs(1 - a - (v - iv)) * np.abs(1 - b - (u - iu)) * val
                k = (iv + a >= 0) & (iv + a < det[0]) & (iu + b >= 0) & (iu + b < det[1])
                np.add.at(out[n], (iv[k] + a, iu[k] + b), wt[k])
    return out


@pytest.mark.parametrize("weight", [0, 1])
@pytest.mark.parametrize("shape,det,views,du,sid,pitch,batch,dtype", [
    ((32, 16, 16), (24, 40), 5, 0.8, 200.0, 0.0, 1, torch.float32),
    ((33, 17, 15), (60, 70), 9, 0.8, 200.0, 0.0, 2, torch.float32),
    ((31, 15, 33), (19, 21), 33, 1.1, 200.0, 9.0, 1, torch.float32),       # overhangs the detector
    ((8, 40, 36), (30, 50), 12, 0.4, 200.0, 0.0, 1, torch.float32),        # flat, pixels finer than voxels
    ((7, 40, 36), (30, 50), 6, 0.8, 200.0, 0.0, 1, torch.float32),         # flatter: the direct kernel
    ((40, 40, 40), (12, 14), 6, 5.0, 200.0, 0.0, 1, torch.float32),        # voxels far finer than pixels
    ((36, 48, 48), (50, 60), 8, 1.2, 9.0, 0.0, 1, torch.float32),          # the source stands inside the volume
    ((34, 20, 18), (40, 44), 7, 0.8, 200.0, 0.0, 2, torch.bfloat16),
    ((64, 18, 20), (70, 44), 7, 0.8, 200.0, 0.0, 1, torch.float16)])
def test_transpose_matches_definition(shape, det, views, du, sid, pitch, batch, dtype, weight):
    sdd = 320.0
    g = geometry(shape, det, views, du, sid, sdd, pitch)
    w = ops.BP_INV_W2 if weight else ops.BP_PLAIN
    f = 1.0 if dtype != torch.float16 else 1e-2   # (sdd / sid)^2 sums stay within half precision
    x = (inputs.gaussian((batch,) + shape, seed=11) * f).astype(np.float32)
    xd = torch.from_numpy(x).to("cuda", dtype)
    got = ops.back_project_transpose(xd, g, w).float().cpu().numpy().astype(np.float64)
    xr = xd.float().cpu().numpy().astype(np.float64)
    for i in range(batch):
        assert rel_l2(got[i], transpose64(shape, det, views, du, sid, sdd, pitch, xr[i], weight)) <= TOL[dtype]


def test_values_the_fixed_point_sums_refuse():
    """A NaN reaches its voxel's four pixels of every view and no others; infinities pass as in FP32 sums."""
    shape, det = (32, 18, 20), (40, 44)
    g = geometry(shape, det, 4, 0.8)
    x = inputs.gaussian(shape, seed=12)
    one = np.zeros(shape, dtype=np.float32)
    one[9, 7, 5] = 1.0
    hit = transpose64(shape, det, 4, 0.8, 200.0, 320.0, 0.0, one, 0) > 1e-6
    x[9, 7, 5] = np.nan
    got = ops.back_project_transpose(torch.from_numpy(x).cuda(), g, 0).cpu().numpy()
    assert np.isnan(got[hit]).all() and np.isfinite(got[~hit]).mean() > 0.99
