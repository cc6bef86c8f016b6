"""A plan that has no room for the windowed lists is built over the per-cell ones: every device allocation of plan creation
fails in turn (host-side injection: nothing runs out on the GPU)."""
import math

import pytest
import torch

from paper_2604_19176_gb300 import Geometry, PatPlan, _lib

pytestmark = pytest.mark.gpu

TOL = 1e-5   # the stated FP32 parity bound of A and A^T


@pytest.mark.parametrize("geoms", [
    [Geometry(252, 90, 0.0, math.pi, 70, 2.0, 96)],                              # two images share each list
    [Geometry(248, 40, 0.2, 1.4 * math.pi, 61, 2.0, 76)] * 3 + [Geometry(64, 9, 0.0, 1.0, 24, 2.0, 40)],
])
def test_allocation_failures_of_a_windowed_plan(cuda_dev, geoms):
    lib = _lib.load()
    plan = PatPlan(geoms, device=cuda_dev)
    assert plan.info()["adj_windows"] == 1
    d = torch.randn(plan.data_shape(), generator=torch.Generator(device=cuda_dev).manual_seed(4), device=cuda_dev)
    ref = plan.adjoint(d).double()
    error = lambda p: float((p.adjoint(d).double() - ref).norm()) / float(ref.norm())  # noqa: E731
    assert error(plan) == 0.0
    plan.close()
    PatPlan(geoms, device=cuda_dev, adj_mode=4).close()   # (loads the kernels that building either form uses)
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    refused, windows = 0, []
    try:
        for k in range(16):
            assert lib.pat_debug_fail_alloc(k) == 0
            try:
                plan = PatPlan(geoms, device=cuda_dev)
            except _lib.PatError as e:
                assert e.status == 3                       # PAT_ERR_OOM: tables and workspace, which every form needs
                refused += 1
            else:
                lib.pat_debug_fail_alloc(-1)               # (where k was past the last allocation)
                windows.append(plan.info()["adj_windows"])
                assert error(plan) <= TOL and plan.sync_status() == 0
                plan.close()
            torch.cuda.synchronize()
            assert free0 - torch.cuda.mem_get_info()[0] < (1 << 20), k   # nothing leaked
            if windows and windows[-1]:
                break
    finally:
        lib.pat_debug_fail_alloc(-1)
    # two refusals, then each allocation of the windowed lists in turn, then none left to fail
    assert refused == 2 and windows == [0] * (len(windows) - 1) + [1] and len(windows) >= 5
