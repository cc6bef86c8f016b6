"""Every sample of the windowed adjoint lists has one owner: the fixed-point positions of csrc/win_position.h, compiled for
the host, over the samples of whole geometries that lie next to grid lines, where the positions that neighbouring patches
stage for one sample can fall on different sides of the line."""
import json
import math
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include "win_position.h"
using namespace patgpu;

int main(int, char** a)
{
    const int n = atoi(a[1]), n_det = atoi(a[2]), n_t = atoi(a[5]), K = atoi(a[7]), j0 = atoi(a[8]), j1 = atoi(a[9]);
    const double start = atof(a[3]), span = atof(a[4]), t_max = atof(a[6]), delta = t_max * n / (2.0 * n_t);
    const int n_r = n_t + 2, c0 = n / 2, px = (n + 8) / 8;
    int m_pitch = 2;
    while (m_pitch < n_r + 1) m_pitch *= 2;
    long near = 0, staged_twice = 0, staged_never = 0, owners_wrong = 0, outside = 0, position_wrong = 0, own = 0;
    const uint32_t T = 4096;   // 1e-6 pixel, more than the two forms of a position can differ by
    for (int j = j0; j < j1; ++j) {
        const double th = start + (j + 0.5) * span / n_det;
        const double U = std::cos(th) * (n / 2.0) - 0.5, V = std::sin(th) * (n / 2.0) - 0.5;
        const int64_t ud = win_detector(U), vd = win_detector(V);
        for (int q = 0; q < K; ++q) {
            const double ph = 2.0 * 3.14159265358979323846 * q / K;
            const double dx = delta * std::cos(ph), dy = delta * std::sin(ph);
            const Fixed x = fixed_of(dx), y = fixed_of(dy);
            const uint32_t xh = x.frac >> 32, yh = y.frac >> 32;
            auto u_of = [&](int m) { return win_position(ud, x.whole, xh, (uint32_t)x.frac, m); };
            auto v_of = [&](int m) { return win_position(vd, y.whole, yh, (uint32_t)y.frac, m); };
            for (int m = 0; m < n_r; ++m) {
                const int64_t u = u_of(m), v = v_of(m);
                if ((uint32_t)u + T >= 2 * T && (uint32_t)v + T >= 2 * T) continue;
                const int cx = win_cell(u), cy = win_cell(v);
                if (cx < -1 - c0 || cx >= n - c0 || cy < -1 - c0 || cy >= n - c0) continue;
                ++near;
                // the sample's own position against the real one
                const long double eu = (long double)U + (long double)m * dx, ev = (long double)V + (long double)m * dy;
                const long double unit = 1.0L / 4294967296.0L;
                if (fabsl((long double)u * unit - eu) > 3 * unit || fabsl((long double)v * unit - ev) > 3 * unit)
                    ++position_wrong;
                // the patches of the cells around it (patch (0, 0) begins at cell (-1, -1) of the image)
                int owners = 0, staged_in = 0;
                const int pxl = std::max(0, (cx - 1 + c0 + 1) / 8), pxh = std::min(px - 1, (cx + 1 + c0 + 1) / 8);
                const int pyl = std::max(0, (cy - 1 + c0 + 1) / 8), pyh = std::min(px - 1, (cy + 1 + c0 + 1) / 8);
                for (int py = pyl; py <= pyh; ++py)
                    for (int p = pxl; p <= pxh; ++p) {
                        const int x0 = p * 8 - 1, y0 = py * 8 - 1, x1 = std::min(x0 + 8, n), y1 = std::min(y0 + 8, n);
                        auto in = [&](int c, int d) { return c + c0 >= x0 && c + c0 < x1 && d + c0 >= y0 && d + c0 < y1; };
                        const WinRange r = win_range((double)ud / 4294967296.0, (double)vd / 4294967296.0, x0 - c0,
                                                     y0 - c0, x1 - c0, y1 - c0, K, n_r, m_pitch, delta);
                        const bool inside = r.nq > 0 && ((q - r.q0) % K + K) % K < r.nq && m >= r.m0 && m < r.m0 + r.nm;
                        const int mc = win_anchor(r.m0, r.nm);
                        const int64_t su = win_staged(u_of(mc), win_step(x.whole, xh), m, mc);
                        const int64_t sv = win_staged(v_of(mc), win_step(y.whole, yh), m, mc);
                        if (inside && in(win_cell(su), win_cell(sv))) ++staged_in;
                        if (!in(cx, cy)) continue;
                        if (!inside) {
                            ++outside;
                            continue;
                        }
                        ++owners;
                        if (win_cell(su) == cx && win_cell(sv) == cy) {
                            const long double bound = unit * (2 * std::abs(m - mc) + 3);
                            if (fabsl((long double)su * unit - eu) > bound || fabsl((long double)sv * unit - ev) > bound)
                                ++position_wrong;
                        } else {   // anchored at its own radius
                            ++own;
                            if (win_staged(u, win_step(x.whole, xh), m, m) != u) ++position_wrong;
                        }
                    }
                owners_wrong += owners != 1;
                staged_twice += staged_in > 1;
                staged_never += staged_in < 1;
            }
        }
    }
    printf("{\"near\": %ld, \"owners_wrong\": %ld, \"outside\": %ld, \"position_wrong\": %ld, \"own\": %ld, "
           "\"staged_twice\": %ld, \"staged_never\": %ld}\n",
           near, owners_wrong, outside, position_wrong, own, staged_twice, staged_never);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("owner")
    src, exe = d / "owner.cpp", d / "owner"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2604_19176_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("geometry,detectors,wrong_without", [
    # (n, detectors, arc start, arc span, times, t_max, angles)
    ((128, 445, 0.0, 2.2753451286971087, 453, 2.0, 1024), (0, 445), ("staged_twice", "staged_never", "own")),
    ((256, 512, 0.0, 1.5 * math.pi, 2048, 2.0, 2048), (240, 245), ("staged_twice",)),
    ((64, 12, 0.2, 2 * math.pi, 2400, 2.0, 2048), (0, 12), ()),    # 40 radii per pixel
    ((100, 9, 0.0, 2 * math.pi, 40, 7.5, 65536), (0, 9), ()),      # radius steps of 9 pixels
    ((36, 7, -0.125, 0.25, 36, 2.0, 6000), (0, 7), ()),            # detector 3 at angle 0: samples on grid lines
    ((8, 64, 0.1, 2.0, 6, 2.0, 65536), (0, 64), ()),               # an image smaller than a patch
])
def test_every_sample_has_one_owner(program, geometry, detectors, wrong_without):
    out = subprocess.run([program, *[repr(x) for x in geometry], *map(str, detectors)], check=True, capture_output=True,
                         text=True).stdout
    r = json.loads(out)
    assert r["near"] > 0
    assert r["owners_wrong"] == 0 and r["outside"] == 0 and r["position_wrong"] == 0, r
    # cells taken from the staged position alone: a sample in two patches, or in none
    assert all(r[k] > 0 for k in wrong_without), r
