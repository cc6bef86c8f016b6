"""The separate time stages on their large tiles (64 detectors x 64 times or
radii, from 32 tiles on) against the FP64 oracle: detector counts and time axes
at, below and past whole tiles, every cluster split of the contraction, and the
residual epilogue of the TV step."""
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_19176_gb300 import Geometry, PatPlan, inputs

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the stated FP32 parity bound of A and A^T


@pytest.mark.parametrize("split", [0, 1, 2, 4, 8])
@pytest.mark.parametrize("n_det,n_t", [(64, 2048), (65, 1055), (130, 700), (1, 2110), (257, 449)])
def test_large_tiles(cuda_dev, n_det, n_t, split):
    g = Geometry(16, n_det, 0.2, 1.3 * math.pi, n_t, 2.0, 16)
    og = O.Geometry(g.n, g.n_det, g.arc_start, g.arc_span, g.n_t, g.t_max, g.n_angles)
    plan = PatPlan(g, device=cuda_dev, abel_split=split, time_pair=1)
    f = inputs.random_image(16, seed=3).astype(np.float32)
    d = inputs.random_data(n_det, n_t, seed=4).astype(np.float32)
    ft, dt = torch.tensor(f, device=cuda_dev), torch.tensor(d, device=cuda_dev)
    ref_g, ref_f = O.forward(og, f.astype(np.float64)), O.adjoint(og, d.astype(np.float64))
    rel = lambda a, b: np.linalg.norm(a.double().cpu().numpy() - b) / np.linalg.norm(b)  # noqa: E731
    assert rel(plan.forward(ft), ref_g) <= TOL
    assert rel(plan.adjoint(dt), ref_f) <= TOL
    # r = A f - d through the step (no TV term, no projection): f - step = tau A^T r
    out, tau = torch.empty_like(ft), 1e-2
    plan.tv_step(ft, out, dt, tau, 0.0, 1e-3, nonneg=False)
    step = O.adjoint(og, ref_g - d.astype(np.float64)) * tau
    # (the difference of two FP32 images is off by their rounding, 2^-24 max|f| per pixel and image)
    slack = 2 * 2.0 ** -24 * np.abs(f).max() * 16 / np.linalg.norm(step)
    assert rel(ft.double() - out.double(), step) <= 2 * TOL + slack
