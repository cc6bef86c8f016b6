"""The windowed adjoint lists (the default gather) against the FP64 oracle at
the sizes where their staging can go wrong: images smaller than a patch and
one cell past whole patches, windows of more rays than a block stages, single
detectors, angles and times, long and short radius steps, plans of several
identical instances (processed two and four at a time) beside others, and the
radius step below which a plan keeps the per-cell lists."""
import math

import numpy as np
import pytest
import torch

import oracle as O
from paper_2604_19176_gb300 import Geometry, PatPlan, inputs

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the stated FP32 parity bound of A and A^T
# Plans of few patches and little work keep the per-cell lists: a large image with one detector brings a plan of small
# geometries above that line.
LARGE = Geometry(248, 1, 0.9, 1.0, 20, 2.0, 31)


def _adjoint_error(plan, geoms, dev, seed):
    data = [inputs.random_data(g.n_det, g.n_t, seed=seed + i).astype(np.float32) for i, g in enumerate(geoms)]
    d = torch.tensor(np.concatenate([x.ravel() for x in data]), device=dev).reshape(plan.data_shape())
    got = plan.adjoint(d).double().cpu().numpy().ravel()
    assert plan.sync_status() == 0
    offs, worst = plan.layout()[0], 0.0
    for i, g in enumerate(geoms):
        ref = O.adjoint(O.Geometry(g.n, g.n_det, g.arc_start, g.arc_span, g.n_t, g.t_max, g.n_angles),
                        data[i].astype(np.float64)).ravel()
        x = got[offs[i]:offs[i + 1]]
        worst = max(worst, np.linalg.norm(x - ref) / max(np.linalg.norm(ref), 1e-300))
        if not ref.any():
            assert not x.any()
    return worst


@pytest.mark.parametrize("g", [
    Geometry(8, 3, 0.1, 2.0, 6, 2.0, 16),                    # an image smaller than a patch
    Geometry(16, 5, 0.0, 2 * math.pi, 24, 2.0, 40),          # 17 cells: one past a patch
    Geometry(64, 1, 0.7, 0.5, 96, 2.0, 130),                 # one detector
    Geometry(32, 7, 0.3, math.pi, 1, 2.0, 33),               # one time
    Geometry(36, 6, 0.0, math.pi, 48, 2.0, 3),               # three angles
    Geometry(24, 4, 1.0, math.pi, 30, 2.0, 2500),            # windows of more than 256 rays
    Geometry(100, 9, 0.0, 2 * math.pi, 40, 7.5, 200),        # radii far beyond the image, steps of 9 pixels
    Geometry(64, 12, 0.2, 2 * math.pi, 2400, 2.0, 256),      # 40 radii per pixel: 900-slot windows
    Geometry(264, 40, -0.4, 1.6 * math.pi, 500, 1.7, 511),
    # symmetric geometries with enough detectors that their copies share lists, in pairs or fours
    Geometry(252, 90, -0.6, 1.2, 70, 2.0, 95),               # mirror images in the x axis (any angle count)
    Geometry(252, 90, 0.0, 0.5 * math.pi, 70, 2.0, 96),      # ... in the diagonal
    Geometry(252, 90, 0.0, math.pi, 70, 2.0, 94),            # ... in the y axis
    Geometry(252, 90, 0.0, math.pi, 70, 2.0, 95),            # (odd angle count: none)
    Geometry(252, 90, 0.0, 1.5 * math.pi, 70, 2.0, 96),      # ... in the other diagonal
    Geometry(252, 144, 0.3, 2 * math.pi, 70, 2.0, 96),       # quarter turns
    Geometry(252, 88, 0.3, 2 * math.pi, 70, 2.0, 96),        # half turns (quarter turns would leave warps idle)
    Geometry(252, 142, 0.3, 2 * math.pi, 70, 2.0, 98),       # half turns
    Geometry(252, 90, 0.25 * math.pi, 2 * math.pi, 70, 2.0, 98),
    Geometry(260, 96, 0.0, math.pi, 90, 2.0, 1400),          # windows of more than 192 rays, whole blocks of them
    Geometry(248, 90, 0.0, math.pi, 1400, 2.0, 96),          # 6 radii per pixel
])
def test_windowed_adjoint(cuda_dev, g):
    geoms = [g, LARGE] if g.n < 200 else [g]
    plan = PatPlan(geoms, device=cuda_dev)
    assert plan.info()["adj_windows"] == 1
    assert _adjoint_error(plan, geoms, cuda_dev, 5) <= TOL
    # and the transpose of the forward operator
    gen = torch.Generator(device=cuda_dev).manual_seed(6)
    f = torch.randn(plan.image_shape(), generator=gen, device=cuda_dev)
    d = torch.randn(plan.data_shape(), generator=gen, device=cuda_dev)
    Af, Ad = plan.forward(f).double(), plan.adjoint(d).double()
    lhs, rhs = float((Af * d).sum()), float((f * Ad).sum())
    assert abs(lhs - rhs) <= TOL * float(Af.norm() * d.double().norm())


@pytest.mark.parametrize("counts", [(2,), (3,), (4,), (5,), (7, 1, 2), (1, 4, 3), (0, 5, 0), (0, 0, 5), (0, 2, 1)])
def test_identical_instances_share_lists(cuda_dev, counts):
    a = Geometry(252, 73, 0.2, 1.4 * math.pi, 70, 2.0, 96)
    b = Geometry(196, 58, 0.0, math.pi, 61, 2.0, 76)       # two images per instance
    c = Geometry(180, 64, 2.0, 2 * math.pi, 33, 2.0, 60)   # four
    kinds = [x for x, n in zip((a, b, c), counts) for _ in range(n)]
    geoms = [kinds[(5 * i) % len(kinds)] for i in range(len(kinds))] if len(kinds) % 5 else kinds   # mixed order
    plan = PatPlan(geoms, device=cuda_dev)
    assert plan.info()["adj_windows"] == 1
    assert _adjoint_error(plan, geoms, cuda_dev, 20) <= TOL
    # the images of a group do not depend on one another
    d = torch.randn(plan.g_elems, generator=torch.Generator(device=cuda_dev).manual_seed(9), device=cuda_dev)
    ref = plan.adjoint(d.reshape(plan.data_shape())).reshape(-1).clone()
    fo, go = plan.layout()
    for i in range(0, len(geoms), 2):
        one = torch.zeros_like(d)
        one[go[i]:go[i + 1]] = d[go[i]:go[i + 1]]
        out = plan.adjoint(one.reshape(plan.data_shape())).reshape(-1)
        assert torch.equal(out[fo[i]:fo[i + 1]], ref[fo[i]:fo[i + 1]])
        assert not out[:fo[i]].any() and not out[fo[i + 1]:].any()


@pytest.mark.parametrize("geoms", [
    [Geometry(8, 3, 0.0, math.pi, 420, 2.0, 24), LARGE],   # 52 radii per pixel: more than a block stages
    [Geometry(64, 40, 0.0, math.pi, 128, 2.0, 128)],       # few patches, little work
])
def test_plans_that_keep_the_per_cell_lists(cuda_dev, geoms):
    plan = PatPlan(geoms, device=cuda_dev)
    assert plan.info()["adj_windows"] == 0 and plan.info()["adj_mode"] == 4
    assert _adjoint_error(plan, geoms, cuda_dev, 31) <= TOL


@pytest.mark.parametrize("g,count", [
    (Geometry(1024, 512, 0.4, 1.1 * math.pi, 2048, 2.0, 2048), 1),   # lists of one image
    (Geometry(1024, 512, 0.0, 1.5 * math.pi, 2048, 2.0, 2048), 1),   # ... of two (mirrored)
    (Geometry(768, 512, 0.0, math.pi, 1536, 2.0, 1536), 2),          # ... of four (two mirrored)
    (Geometry(768, 500, 0.0, 2 * math.pi, 1500, 2.0, 1536), 7),      # ... quarter turns, one instance per list
])
def test_queued_shares_of_large_plans(cuda_dev, g, count):
    """The last shares of a large plan are taken from a queue: the result does not depend on which warp takes which
    (equal bits on every call, on any stream, with the queue armed again after each), and agrees with the per-cell
    gather of the same plan within the parity bound."""
    plan = PatPlan([g] * count, device=cuda_dev)
    assert plan.info()["adj_windows"] == 1
    d = torch.randn(plan.data_shape(), generator=torch.Generator(device=cuda_dev).manual_seed(3), device=cuda_dev)
    first = plan.adjoint(d)
    side = torch.cuda.Stream(cuda_dev)
    side.wait_stream(torch.cuda.current_stream(cuda_dev))
    again = [plan.adjoint(d, stream=side) for _ in range(3)]
    side.synchronize()
    assert plan.sync_status() == 0 and all(torch.equal(first, x) for x in again)
    ref = PatPlan([g] * count, device=cuda_dev, adj_mode=2).adjoint(d).double().reshape(count, -1)
    err = (first.double().reshape(count, -1) - ref).norm(dim=1) / ref.norm(dim=1)
    assert float(err.max()) <= TOL
