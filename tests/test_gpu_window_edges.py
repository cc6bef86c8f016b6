"""The windowed adjoint on geometries with samples so close to the edge of a patch that the positions which neighbouring
patches stage for them lie on different sides of it: each such sample counts once.  (One sample too many or too few: 1.4e-5 to
8e-5 of the image's norm on these geometries; all other errors together: 4e-7 to 1.3e-6.)"""
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_19176_gb300 import Geometry, PatPlan, inputs

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the stated FP32 parity bound of A and A^T


@pytest.mark.parametrize("g", [
    Geometry(128, 445, 0.0, 2.2753451286971087, 453, 2.0, 1024),
    Geometry(256, 512, 0.0, 1.5 * math.pi, 2048, 2.0, 2048),                   # mirror images share lists
    Geometry(384, 440, 0.0, math.radians(185.31229848695062), 2048, 2.0, 1600),
    Geometry(128, 494, 0.0, math.radians(100.36926704147039), 256, 2.0, 2048),
    Geometry(256, 408, 0.0, 1.9492486455801319, 645, 2.0, 2048),
])
def test_samples_at_patch_edges_count_once(cuda_dev, g):
    plan = PatPlan(g, device=cuda_dev)
    assert plan.info()["adj_windows"] == 1
    d = inputs.random_data(g.n_det, g.n_t, seed=17).astype(np.float32)
    got = plan.adjoint(torch.tensor(d, device=cuda_dev)).double().cpu().numpy()
    ref = O.adjoint(O.Geometry(g.n, g.n_det, g.arc_start, g.arc_span, g.n_t, g.t_max, g.n_angles), d.astype(np.float64))
    assert np.linalg.norm(got - ref) <= TOL * np.linalg.norm(ref)
