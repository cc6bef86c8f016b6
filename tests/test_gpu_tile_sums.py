"""The per-instance sums of tile partials (TV value, squared norms of the
descent and primal-dual steps): image sizes below, at and past one tile, one
512-thread pass over the tiles and several, instances of different size in
one plan."""
import math

import pytest
import torch

from paper_2604_19176_gb300 import Geometry, PatPlan

pytestmark = pytest.mark.gpu

# One sum's error: a 256-value tree (13 additions deep), tiles / 512 sequential
# additions (8 at 1024^2), a 5 + 16 deep tree, and a few roundings per term:
# below 48 ulp of positive terms.
TOL = 48 * 2.0 ** -24


@pytest.mark.parametrize("sizes", [(8,), (32,), (36,), (1024,), (1028,), (8, 260, 64, 1024, 100)])
def test_tile_sums(cuda_dev, sizes):
    plan = PatPlan([Geometry(n, 1, 0.0, math.pi, 4, 2.0, 4) for n in sizes], device=cuda_dev)
    gen = torch.Generator(device=cuda_dev).manual_seed(sum(sizes))
    f = torch.rand(plan.image_shape(), generator=gen, device=cuda_dev)
    adj = torch.randn(plan.image_shape(), generator=gen, device=cuda_dev)
    eps, tau = 1e-2, 0.1
    val = plan.tv_value(f, eps)
    new, delta = f.clone(), torch.empty(2 * len(sizes), device=cuda_dev)
    plan.descent_step(new, adj, None, tau, 0.0, delta=delta)
    offs = plan.layout()[0]
    for i, n in enumerate(sizes):
        a, b = offs[i], offs[i + 1]
        x, y = f.reshape(-1)[a:b].reshape(n, n).double(), new.reshape(-1)[a:b].double()
        dx, dy = torch.zeros_like(x), torch.zeros_like(x)
        dx[:, :-1], dy[:-1] = x[:, 1:] - x[:, :-1], x[1:] - x[:-1]
        want = [torch.sqrt(dx * dx + dy * dy + eps * eps).sum(), ((y - x.reshape(-1)) ** 2).sum(), (y * y).sum()]
        for got, ref in zip((val[i], delta[2 * i], delta[2 * i + 1]), want):
            # (the step's difference new - old is exact to one rounding of values up to 1)
            assert abs(float(got) - float(ref)) <= TOL * float(ref) + (1e-6 * float(ref) if ref is want[1] else 0.0)
