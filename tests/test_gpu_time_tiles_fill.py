"""The large tiles of the separate time stages (64 detectors x 64 times or radii) where a third of their outputs is just not
padding, and the small ones just below: one row of tiles over a long time axis, every cluster split of the contraction."""
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_19176_gb300 import Geometry, PatPlan, inputs

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the stated FP32 parity bound of A and A^T


@pytest.mark.parametrize("split", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("n_det,n_t,auto_split", [
    (22, 2110, 8),   # 33 tiles of 64, 0.343 full: clusters of 8 (up to 3.5 CTAs of large tiles per SM)
    (21, 2110, 4),   # 0.328 full: 66 tiles of 32, clusters of 4 (up to 2 CTAs per SM)
])
def test_tiles_a_third_full(cuda_dev, n_det, n_t, auto_split, split):
    g = Geometry(16, n_det, 0.2, 1.3 * math.pi, n_t, 2.0, 16)
    og = O.Geometry(g.n, g.n_det, g.arc_start, g.arc_span, g.n_t, g.t_max, g.n_angles)
    plan = PatPlan(g, device=cuda_dev, abel_split=split, time_pair=1)
    info = plan.info()
    assert info["abel_split_fwd"] == info["abel_split_adj"] == (split or auto_split)   # (the tile size shows in the choice)
    f = inputs.random_image(16, seed=3).astype(np.float32)
    d = inputs.random_data(n_det, n_t, seed=4).astype(np.float32)
    rel = lambda a, b: np.linalg.norm(a.double().cpu().numpy() - b) / np.linalg.norm(b)  # noqa: E731
    assert rel(plan.forward(torch.tensor(f, device=cuda_dev)), O.forward(og, f.astype(np.float64))) <= TOL
    assert rel(plan.adjoint(torch.tensor(d, device=cuda_dev)), O.adjoint(og, d.astype(np.float64))) <= TOL
