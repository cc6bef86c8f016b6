// win_position.h — sample positions of the windowed adjoint lists in fixed
// point, and which patch lists a sample (windows.cu).  Host and device code.
//
// A position along one axis is held in units of 2^-32 pixel, integer part
// included.  Two forms of it matter:
//   win_position: detector + radius x direction, a function of the sample
//     (j, m, q) alone.  Its integer part is the sample's cell: the one cell,
//     of the one patch, that lists the sample.
//   win_staged: what k_adj_win forms from the ray that it staged for a patch's
//     window: win_position at the window's anchor radius, then steps rounded
//     to 2^-30 pixel.  Anchors differ from patch to patch, so the staged
//     positions of a sample differ too, by up to 2^-31 pixel per radius from
//     the anchor and a few 2^-32.
// Where the two fall on different sides of a grid line, the staged fraction
// would be one of another cell (and were the staged cell taken for the sample's,
// two patches could list it, or neither).  Such samples, some ten in 10^9,
// are staged once more in their cell's patch with their own radius for the
// anchor, where both forms are equal.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define PAT_HD __host__ __device__ __forceinline__
#else
#define PAT_HD inline
#endif

namespace patgpu {

// x as whole + frac / 2^64
struct Fixed {
    int32_t whole;
    uint64_t frac;
};
inline Fixed fixed_of(double x)
{
    double w = std::floor(x), f = x - w;
    if (f >= 1.0) {   // (x a rounding error below a whole number)
        w += 1.0;
        f = 0.0;
    }
    return {(int32_t)w, (uint64_t)(f * 18446744073709551616.0)};
}
// a detector coordinate: 32 fraction bits, rounded (a carry goes to the integer part)
inline int64_t win_detector(double x)
{
    const Fixed f = fixed_of(x);
    return (int64_t)f.whole * 4294967296ll + (int64_t)((f.frac >> 32) + ((f.frac >> 31) & 1u));
}

PAT_HD uint32_t win_mulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }

// Position of radius m from the detector's `at`, for a direction (pixels per
// radius) of integer part `whole` and fraction hi : lo.
PAT_HD int64_t win_position(int64_t at, int32_t whole, uint32_t hi, uint32_t lo, int m)
{
    return at + (int64_t)m * ((int64_t)whole * 4294967296ll + (int64_t)hi) + (int64_t)win_mulhi((uint32_t)m, lo);
}
// The staged step per radius: four times the step per byte that k_adj_win holds.
PAT_HD int64_t win_step(int32_t whole, uint32_t hi)
{
    return (int64_t)whole * 4294967296ll + (int64_t)(((uint64_t)hi + 2ull) & ~3ull);
}
// Staged position of radius m in a window anchored at radius mc, where the
// position is `at_mc`.
PAT_HD int64_t win_staged(int64_t at_mc, int64_t step, int m, int mc) { return at_mc + (int64_t)(m - mc) * step; }

PAT_HD int win_cell(int64_t position) { return (int)(position >> 32); }

// The rays q0 .. q0 + nq - 1 (mod K) and radii m0 .. m0 + nm - 1 of a detector
// that can reach a patch, and the rays through the patch's nearest cell.  None:
// nq = nm = 0.
struct WinRange {
    int q0, nq, m0, nm, near;
};
PAT_HD int win_anchor(int m0, int nm) { return m0 + nm / 2; }

// Every sample of the detector at (U, V) that lands in the cells [x0, x1) x
// [y0, y1) (centred coordinates) is in the range.  The patch is widened by
// 0.02 pixel (the positions' error is below 1e-3), its distance range gives
// the radii and its corners' angles the rays; a detector within half a pixel
// sees the whole circle.
PAT_HD WinRange win_range(double U, double V, int x0, int y0, int x1, int y1, int K, int n_r, int m_pitch, double delta)
{
    const double eps = 0.02;
    const double ax = x0 - eps - U, bx = x1 + eps - U, ay = y0 - eps - V, by = y1 + eps - V;
    const double nx = fmax(0.0, fmax(ax, -bx)), ny = fmax(0.0, fmax(ay, -by));
    const double fx = fmax(fabs(ax), fabs(bx)), fy = fmax(fabs(ay), fabs(by));
    const double rmin = sqrt(nx * nx + ny * ny), rmax = sqrt(fx * fx + fy * fy);
    int m0 = (int)fmin(1e6, ceil(rmin / delta - 1e-6));
    const int m1 = (int)fmin((double)(n_r - 1), floor(rmax / delta + 1e-6));
    if (m0 > m1) return {0, 0, 0, 0, 0};
    int q0 = 0, nq = K;
    if (rmin > 0.5) {
        const double cx = 0.5 * (ax + bx), cy = 0.5 * (ay + by);
        double lo = 0.0, hi = 0.0;
        const double px[4] = {ax, bx, ax, bx}, py[4] = {ay, ay, by, by};
        for (int i = 0; i < 4; ++i) {
            const double a = atan2(cx * py[i] - cy * px[i], cx * px[i] + cy * py[i]);
            lo = fmin(lo, a);
            hi = fmax(hi, a);
        }
        const double per = K / 6.283185307179586476925, pc = atan2(cy, cx);
        const int qa = (int)ceil((pc + lo) * per - 1e-3), qb = (int)floor((pc + hi) * per + 1e-3);
        nq = qb - qa + 1 < K ? qb - qa + 1 : K;
        q0 = nq == K ? 0 : ((qa % K) + K) % K;
    }
    if (nq <= 0) return {0, 0, 0, 0, 0};
    m0 &= ~3;   // (16-byte reads of Mbar)
    const int nmp = (m1 - m0 + 1 + 7) / 8 * 8;
    if (m0 + nmp > m_pitch) m0 = m_pitch > nmp ? m_pitch - nmp : 0;   // (padded radii stay inside the row)
    const double near = fmin(32767.0, ceil(1.3 * K / (6.283185307179586476925 * fmax(rmin, 0.7))));
    return {q0, nq, m0, m1 - m0 + 1, (int)near};
}

} // namespace patgpu
