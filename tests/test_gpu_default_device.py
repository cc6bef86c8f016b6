"""tv_reconstruct in a program whose default device is the GPU (torch.set_default_device, or torch.device as a context):
its host buffers stay on the host."""
import math

import pytest
import torch

from paper_2604_19176_gb300 import Geometry, PatPlan, inputs
from paper_2604_19176_gb300.recon import tv_reconstruct

pytestmark = pytest.mark.gpu


def test_tv_reconstruct_with_a_default_device(cuda_dev):
    g = Geometry(48, 20, 0.2, math.pi, 96, 2.0, 96)
    plan = PatPlan(g, device=cuda_dev)
    f = torch.tensor(inputs.gaussian_phantom(48, 4, seed=1), dtype=torch.float32, device=cuda_dev)
    data = plan.forward(f)
    want, changes = tv_reconstruct(plan, data, 1e-3, iters=5, tau=0.02)
    with torch.device(cuda_dev):
        got, again = tv_reconstruct(plan, data, 1e-3, iters=5, tau=0.02)
    assert torch.equal(got, want) and again == changes
