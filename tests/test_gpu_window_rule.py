"""Which plans take the windowed lists: on either side of the lines for plans whose images do not share lists (patches,
detectors per pixel column, arc), and for the same sizes where images share them.  Whichever form is taken agrees with the
enumerating gather."""
import math

import pytest
import torch

from paper_2604_19176_gb300 import Geometry, PatPlan

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the stated FP32 parity bound of A and A^T
DEG = math.pi / 180.0


@pytest.mark.parametrize("geoms,windows", [
    ([Geometry(176, 292, 0.0, 200 * DEG, 352, 2.0, 352)], 0),            # 529 patches, no symmetry
    ([Geometry(196, 195, 0.0, 270 * DEG, 377, 2.0, 466)], 0),            # 625 patches, odd detectors
    ([Geometry(236, 100, 0.0, 260.75 * DEG, 451, 2.0, 472)], 0),         # 900 patches
    ([Geometry(128, 52, 0.0, 339.79 * DEG, 210, 2.0, 264)] * 3, 0),      # identical images, too little work to share
    ([Geometry(476, 391, 0.0, 309.41 * DEG, 652, 2.0, 923)], 0),         # 3600 patches
    ([Geometry(260, 185, 0.0, 270 * DEG, 300, 2.0, 421)], 0),            # 1089 patches, 0.71 detectors per column
    ([Geometry(196, 194, 0.0, 270 * DEG, 377, 2.0, 468)], 1),            # mirror images share lists
    ([Geometry(176, 292, 0.0, 197 * DEG, 352, 2.0, 352)], 1),            # the arc
    ([Geometry(260, 185, 0.0, 230 * DEG, 300, 2.0, 421)], 1),            # the arc, more patches
    ([Geometry(260, 181, 0.0, 270 * DEG, 300, 2.0, 421)], 1),            # the detectors, more patches
    ([Geometry(236, 93, 0.0, 260.75 * DEG, 451, 2.0, 472)], 1),          # the detectors
    ([Geometry(492, 391, 0.0, 309.41 * DEG, 652, 2.0, 923)], 1),         # 3844 patches
    ([Geometry(176, 292, 0.0, 200 * DEG, 352, 2.0, 352)] * 2, 1),        # two identical images
    ([Geometry(176, 292, 0.0, 200 * DEG, 352, 2.0, 352), Geometry(64, 8, 0.0, math.pi, 64, 2.0, 64)], 1),
])
def test_plans_without_shared_lists(cuda_dev, geoms, windows):
    plan = PatPlan(geoms, device=cuda_dev)
    assert plan.info()["adj_windows"] == windows
    d = torch.randn(plan.data_shape(), generator=torch.Generator(device=cuda_dev).manual_seed(2), device=cuda_dev)
    ref = PatPlan(geoms, device=cuda_dev, adj_mode=2).adjoint(d).double()
    assert float((plan.adjoint(d).double() - ref).norm()) <= TOL * float(ref.norm())
