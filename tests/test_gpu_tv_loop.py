"""tv_reconstruct without a callback (the next iteration is enqueued before the stop rule of the last one is tested)
against the loop with a callback, which takes one iteration at a time."""
import math

import pytest
import torch

from paper_2604_19176_gb300 import Geometry, PatPlan, inputs
from paper_2604_19176_gb300.recon import tv_reconstruct

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 3])
@pytest.mark.parametrize("iters,stop_at", [(0, None), (1, None), (2, None), (7, None), (12, 6), (12, 7), (12, 11)])
def test_loops_agree(cuda_dev, batch, iters, stop_at):
    """Both run the same kernels on the same buffers in the same order: equal results, bit for bit, also when the
    stop rule holds (at an odd, an even and the last iteration) and an iteration behind it was enqueued already."""
    g = Geometry(48, 20, 0.2, math.pi, 96, 2.0, 96)
    plan = PatPlan([g] * batch, device=cuda_dev)
    f = torch.stack([torch.tensor(inputs.gaussian_phantom(48, 4, seed=i), dtype=torch.float32) for i in range(batch)])
    data = plan.forward(f.reshape(plan.image_shape()).to(cuda_dev))
    f0 = torch.full(plan.image_shape(), 0.1, device=cuda_dev)
    kept, kw = f0.clone(), dict(iters=iters, tau=0.02, f0=f0)
    tol = -1.0
    if stop_at is not None:   # the changes fall, so this tolerance is first met at stop_at
        changes = tv_reconstruct(plan, data, 1e-3, stop_tol=-1.0, callback=lambda *a: None, **kw)[1]
        tol = changes[stop_at]
        assert all(c > tol for c in changes[1:stop_at])
    seen = []
    a, ha = tv_reconstruct(plan, data, 1e-3, stop_tol=tol, callback=lambda k, x, r: seen.append((x.data_ptr(), r)), **kw)
    b, hb = tv_reconstruct(plan, data, 1e-3, stop_tol=tol, **kw)
    assert len(ha) == (iters if stop_at is None else stop_at + 1)
    assert ha == hb == [r for _, r in seen] and torch.equal(a, b) and torch.equal(f0, kept)
    assert all(p == a.data_ptr() for p, _ in seen)
