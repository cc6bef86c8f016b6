"""The autotuner times the launches that the plan's calls make: csrc/tune.cpp compiled for the host with the kernels'
launchers, plan building and the CUDA runtime replaced by stand-ins that write down what is launched."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "kernels.h"
#include "plan.h"

static int g_chunks = 0;
#define LOG(...) (std::printf(__VA_ARGS__), cudaSuccess)

namespace patgpu {
pat_status_t build_plan(Plan& P, const pat_geometry_t*, int, const pat_options_t& opt, cudaStream_t)
{
    std::printf("build mode=%d split=%d\n", (int)opt.adj_mode, (int)opt.abel_split);
    P.opt = opt;
    P.dp.time_chunks = g_chunks;
    P.info.adj_windows = opt.adj_mode == 0 && opt.adj_groups == 0 && opt.adj_jblock == 0;
    return PAT_OK;
}
void free_plan_memory(Plan&) {}
cudaError_t dev_malloc(void** p, size_t)
{
    *p = reinterpret_cast<void*>(16);
    return cudaSuccess;
}
cudaError_t launch_circmean(const DevPlan&, const void*, cudaStream_t, bool msum) { return LOG("circmean msum=%d\n", (int)msum); }
cudaError_t launch_abel_fwd(const DevPlan&, float*, cudaStream_t, const float*) { return LOG("abel_fwd\n"); }
cudaError_t launch_abel_adj(const DevPlan&, const float*, cudaStream_t) { return LOG("abel_adj\n"); }
cudaError_t launch_time_fwd(const DevPlan&, float*, cudaStream_t) { return LOG("time_fwd\n"); }
cudaError_t launch_adjoint_gather(const DevPlan&, void*, cudaStream_t) { return LOG("gather\n"); }
}   // namespace patgpu

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 1 << 20; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaFree(void*) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = nullptr; return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
}

int main(int, char** a)
{
    using namespace patgpu;
    g_chunks = atoi(a[1]);
    pat_geometry_t g{64, 16, 0.0, 3.0, 64, 2.0, 64};
    pat_options_t opt{};
    opt.tune = 1;
    for (int i = 2; a[i]; ++i) {
        opt.adj_groups = atoi(a[i]);
        std::printf("call groups=%d\n", (int)opt.adj_groups);
        Plan* p = nullptr;
        if (autotune_plan(&p, &g, 1, opt, nullptr) != PAT_OK || !p) return 1;
        std::printf("plan windows=%d\n", (int)p->info.adj_windows);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if not os.path.exists("/usr/local/cuda/include/cuda_runtime.h"):
        pytest.skip("no CUDA headers")
    d = tmp_path_factory.mktemp("tune")
    src, exe = d / "tune_main.cpp", d / "tune_main"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2604_19176_gb300", "csrc")
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", csrc, "-I", os.path.join(ROOT, "include"), "-I",
                    "/usr/local/cuda/include", str(src), os.path.join(csrc, "tune.cpp"), "-o", str(exe)], check=True)
    return str(exe)


def _run(program, *args):
    return subprocess.run([program, *map(str, args)], check=True, capture_output=True, text=True).stdout.splitlines()


@pytest.mark.parametrize("chunks,forward,split", [
    (2, ["circmean msum=0", "time_fwd"], ["abel_adj"]),                  # fused time stage, as pat_forward runs it
    (0, ["circmean msum=1", "abel_fwd"], ["abel_fwd", "abel_adj"]),      # separate
])
def test_timed_launches(program, chunks, forward, split):
    plans, launches = [], None
    for x in _run(program, chunks, 0)[1:-1]:
        if x.startswith("build"):
            launches = []
            plans.append((x, launches))
        else:
            launches.append(x)
    def timed(which):
        return [run for name, run in plans if which(name) and run]
    fwd = timed(lambda s: s == "build mode=2 split=0")
    splits = timed(lambda s: s.startswith("build mode=2") and not s.endswith("split=0"))
    adjoint = timed(lambda s: s.startswith("build mode=0"))
    assert len(fwd) >= 3 and all(r == forward * 7 for r in fwd)          # 2 warm and 5 timed calls
    assert len(splits) == 4 and all(r == split * 7 for r in splits)
    assert adjoint and all(r == ["abel_adj", "gather"] * 7 for r in adjoint)


@pytest.mark.parametrize("calls", [(0, 4, 0), (4, 0, 4)])
def test_list_parts_asked_for_are_not_answered_from_the_cache(program, calls):
    """A request for a number of list parts never takes the windowed lists, also when an automatic plan of the same
    geometry was tuned before, and the other way round."""
    lines = [x for x in _run(program, 2, *calls) if x.startswith(("call", "plan"))]
    # (the stand-in's candidates all take the same time: an automatic plan keeps its first, the windowed one)
    assert lines == [x for c in calls for x in (f"call groups={c}", f"plan windows={int(c == 0)}")]
