"""The list form that a windowed plan names is the one that the same plan takes without windows (codes of up to 31, of 32
and of more bits), and the one-sample codes of all 32 bits at the size that needs them."""
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_19176_gb300 import Geometry, PatPlan, inputs, workloads

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the stated FP32 parity bound of A and A^T


@pytest.mark.parametrize("g,mode", [
    (Geometry(256, 128, 0.0, math.pi, 512, 2.0, 512), 4),            # 9 + 7 + 10 bits: run pairs
    (Geometry(256, 257, 0.0, 1.0, 2050, 40.0, 2047), 1),             # 11 + 9 + 12 = 32: one sample per code
    (Geometry(256, 1025, 0.0, 1.0, 1030, 40.0, 1025), 3),            # 11 + 11 + 11 = 33: fractions
])
def test_mode_without_windows(cuda_dev, g, mode):
    plan, cells = PatPlan(g, device=cuda_dev), PatPlan(g, device=cuda_dev, adj_groups=2)
    assert plan.info()["adj_windows"] == 1 and cells.info()["adj_windows"] == 0
    assert plan.info()["adj_mode"] == cells.info()["adj_mode"] == mode


def test_codes_of_32_bits_at_full_size(cuda_dev):
    """8 x 1024^2, 512 detectors, 2048 times and angles, per-cell codes asked for: the adjoint of data on the first or
    last four detectors of two instances against the oracle on those detectors alone, zero elsewhere."""
    wl = workloads.vessel1024_b8()
    geoms = list(wl.geometries)
    g = geoms[0]
    plan = PatPlan(geoms, device=cuda_dev, adj_mode=1)
    assert plan.info()["adj_mode"] == 1 and plan.info()["adj_windows"] == 0
    data, rows = torch.zeros(plan.data_shape(), device=cuda_dev), {0: 0, 7: g.n_det - 4}
    for i, j0 in rows.items():
        data[i, j0:j0 + 4] = torch.tensor(inputs.random_data(4, g.n_t, seed=700 + i), dtype=torch.float32, device=cuda_dev)
    f = plan.adjoint(data)
    step = g.arc_span / g.n_det
    for i in range(len(geoms)):
        if i not in rows:
            assert not bool(f[i].any())
            continue
        og = O.Geometry(g.n, 4, g.arc_start + rows[i] * step, 4 * step, g.n_t, g.t_max, g.n_angles)
        ref = O.adjoint(og, data[i, rows[i]:rows[i] + 4].double().cpu().numpy())
        assert np.linalg.norm(f[i].double().cpu().numpy() - ref) <= TOL * np.linalg.norm(ref)
