"""The windowed lists inside the solver steps and in the debug build: symmetric plans (whose images the step epilogues turn
back pixel by pixel) against the separate calls and the FP64 oracle, and the gather's device-side bounds checks, clean and
with a planted entry, over groups of one, two and four images and with queued shares."""
import dataclasses
import math
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest
import torch

import oracle as O
from oracle import pdhg as OP
from paper_2604_19176_gb300 import Geometry, PatPlan, inputs

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOL = 1e-5   # the stated FP32 parity bound of A and A^T

SYMMETRIC = [
    Geometry(252, 90, -0.6, 1.2, 70, 2.0, 95),                # mirror image in the x axis
    Geometry(252, 90, 0.0, math.pi, 70, 2.0, 94),             # ... in the y axis
    Geometry(252, 90, 0.0, 0.5 * math.pi, 70, 2.0, 96),       # ... in the diagonal
    Geometry(252, 90, 0.0, 1.5 * math.pi, 70, 2.0, 96),       # ... in the other
    Geometry(252, 142, 0.3, 2 * math.pi, 70, 2.0, 98),        # half turns
    Geometry(252, 144, 0.3, 2 * math.pi, 70, 2.0, 96),        # quarter turns
]


@pytest.mark.parametrize("g", SYMMETRIC)
def test_tv_step_of_a_windowed_plan(cuda_dev, g):
    """With separate time-stage launches the step is the separate calls in fewer kernels: equal bits (where 1 / K is
    exact: the step's residual is one fused multiply-add)."""
    g = dataclasses.replace(g, n_angles=128)
    plan = PatPlan(g, device=cuda_dev, time_pair=1)
    assert plan.info()["adj_windows"] == 1
    f0 = torch.tensor(np.abs(inputs.random_image(g.n, seed=71)), dtype=torch.float32, device=cuda_dev)
    data = torch.tensor(inputs.random_data(g.n_det, g.n_t, seed=72), dtype=torch.float32, device=cuda_dev)
    tau, lam, eps = 0.05, 0.3, 1e-2
    want = f0.clone()
    adj = plan.adjoint(plan.residual(plan.forward(want), data))
    plan.descent_step(want, adj, plan.tv_grad(want, eps)[1], tau, lam, nonneg=True)
    got = torch.empty_like(f0)
    plan.tv_step(f0, got, data, tau, lam, eps, nonneg=True)
    assert torch.equal(got, want)


@pytest.mark.parametrize("g", SYMMETRIC)
def test_pdhg_step_of_a_windowed_plan(cuda_dev, g):
    plan = PatPlan(g, device=cuda_dev)
    assert plan.info()["adj_windows"] == 1
    og = O.Geometry(g.n, g.n_det, g.arc_start, g.arc_span, g.n_t, g.t_max, g.n_angles)
    data = O.forward(og, inputs.vessel_phantom(g.n, seed=6)).astype(np.float32)
    st = {k: torch.zeros(plan.data_shape() if k == "y" else plan.image_shape(), device=cuda_dev)
          for k in ("f", "fbar", "y", "px", "py")}
    ost, s, alpha = None, 0.2, 1e-3
    for k in range(3):
        plan.pdhg_step(st["f"], st["fbar"], st["y"], st["px"], st["py"], torch.tensor(data, device=cuda_dev), s, s, alpha)
        ost, _ = OP.pdhg(lambda f: O.forward(og, f), lambda y: O.adjoint(og, y), data.astype(np.float64), g.n, alpha, s, s, 1,
                         nonneg=True, state=ost)
        for name in ("f", "fbar", "y"):
            err = np.linalg.norm(st[name].double().cpu().numpy() - ost[name])
            assert err <= (k + 1) * TOL * np.linalg.norm(ost[name]), (k, name)


CHILD = textwrap.dedent(r"""
    import math, sys
    import numpy as np
    sys.path.insert(0, ROOT)
    from paper_2604_19176_gb300 import _lib, build
    lib = _lib.load(build.build(debug=True))       # before any plan: the operators use this build
    assert lib.pat_debug_build() == 1
    import torch
    import oracle as O
    from paper_2604_19176_gb300 import Geometry, PatPlan, inputs

    PAT_OK, PAT_ERR_BOUNDS = 0, 7
    dev = torch.device("cuda", 0)
    pi = math.pi
    for name, geoms in [
        ("one image", [Geometry(252, 73, 0.2, 1.4 * pi, 70, 2.0, 96)]),
        ("two images", [Geometry(252, 90, 0.0, pi, 70, 2.0, 94)]),
        ("four images", [Geometry(252, 144, 0.3, 2 * pi, 70, 2.0, 96)]),
        ("groups of four, two and one", [Geometry(252, 73, 0.2, 1.4 * pi, 70, 2.0, 96)] * 7),
        ("a sample staged on its own", [Geometry(128, 445, 0.0, 2.2753451286971087, 453, 2.0, 1024)]),
    ]:
        g = geoms[0]
        plan = PatPlan(geoms, device=dev)
        assert plan.info()["adj_windows"] == 1, name
        d = inputs.random_data(g.n_det, g.n_t, seed=52).astype(np.float32)
        ref = O.adjoint(O.Geometry(g.n, g.n_det, g.arc_start, g.arc_span, g.n_t, g.t_max, g.n_angles), d.astype(np.float64))
        data = torch.tensor(d, device=dev).expand(len(geoms), -1, -1).contiguous().reshape(plan.data_shape())
        def error():
            f = plan.adjoint(data).double().cpu().numpy().reshape(len(geoms), g.n, g.n)
            assert plan.sync_status() == PAT_OK, name
            return max(np.linalg.norm(x - ref) for x in f) / np.linalg.norm(ref)
        assert error() <= 1e-5, name
        plan.set_bounds_probe()
        plan.adjoint(data)                             # one entry is skipped: this result is undefined
        assert plan.sync_status() == PAT_ERR_BOUNDS, name
        assert plan.sync_status() == PAT_OK, name      # reported once, then cleared
        assert error() <= 1e-5, name                   # the probe disarmed itself
        plan.close()
        print(name, "ok", flush=True)

    # queued shares: clean, and the release arithmetic
    plan = PatPlan([Geometry(768, 512, 0.0, pi, 1536, 2.0, 1536)] * 2, device=dev)
    assert plan.info()["adj_windows"] == 1
    data = torch.randn(plan.data_shape(), generator=torch.Generator(device=dev).manual_seed(3), device=dev)
    f = plan.adjoint(data)
    assert plan.sync_status() == PAT_OK and bool(torch.isfinite(f).all())
    assert torch.equal(plan.adjoint(data), f) and plan.sync_status() == PAT_OK
    print("all ok", flush=True)
""")


def test_bounds_checks_of_the_windowed_gather():
    code = "ROOT = " + repr(ROOT) + "\n" + CHILD
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "all ok" in r.stdout
