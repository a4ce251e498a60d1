"""Plans whose volumes have slab tables of different lengths: the table lies after the largest box, and together they still
leave room for two CTAs per SM where each volume's own configuration does. Where one does not, the plan runs one."""
import math

import pytest
import torch

from paper_2511_08427_gb300 import operators as ops

pytestmark = pytest.mark.gpu


def scan(side, det, views, helix):
    pitch = 1.6 * side * 0.5 * math.sqrt(2.0) / (0.9 * det)
    return ops.Geometry.cone_circular((side,) * 3, (0.5,) * 3, (det, det), (round(pitch, 3),) * 2, views, 2 * math.pi, 750.0,
                                      1200.0, helical_pitch=0.25 * side * 0.5 if helix else 0.0)


# (volume side, detector side, views) of each volume, and the CTAs per SM
@pytest.mark.parametrize("parts,ctas", [
    ([(80, 128, 45), (88, 144, 60), (104, 160, 107), (128, 192, 153)], 2),   # a long table after another volume's filled box
    ([(96, 112, 47), (120, 160, 88), (144, 192, 128), (168, 240, 169)], 1),  # the first alone takes an SM for each CTA
    ([(64, 96, 48), (80, 128, 64), (96, 160, 90), (112, 192, 90), (136, 224, 111)], 2),
    ([(72, 96, 20), (24, 240, 5)], 2),
])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_ctas_per_sm(parts, ctas, dtype):
    geoms = [scan(*p, i % 2 == 1) for i, p in enumerate(parts)]
    assert all(g.adjoint_config()["kernel"] == 3 for g in geoms)
    plan = ops.Plan(geoms, dtype)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert plan.info()["grids"][1] == ctas * sms
    ys = [torch.randn(g.sinogram_shape, device="cuda", generator=torch.Generator("cuda").manual_seed(i)).to(dtype)
          for i, g in enumerate(geoms)]
    out = [torch.full(g.volume_shape, float("nan"), device="cuda", dtype=dtype) for g in geoms]
    plan.adjoint(ys, out)
    for g, y, x in zip(geoms, ys, out):
        ref = ops.adjoint(y, g).double()
        # FP32: the boxes' sums reach the volume in another order; BF16: one rounding of each side
        tol = 1e-5 if dtype == torch.float32 else 4e-3
        assert ((x.double() - ref).norm() / ref.norm()).item() <= tol
        assert g.read_flags()[:4] == [0, 0, 0, 0]
