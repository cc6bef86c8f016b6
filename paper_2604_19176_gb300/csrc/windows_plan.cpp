// windows_plan.cpp — builds the windowed adjoint lists of a plan (windows.cu):
// detector windows and blocks per patch, code lists, and the cut of all
// blocks into equal-cost shares, one per resident warp.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <tuple>
#include <vector>

#include <cuda_runtime.h>

#include "kernels.h"
#include "plan.h"

namespace patgpu {

namespace {

// Device memory that is given back when it goes out of scope.
struct DevBuf {
    void* p = nullptr;
    cudaStream_t st;
    explicit DevBuf(cudaStream_t s) : st(s) {}
    ~DevBuf()
    {
        if (!p) return;
        cudaStreamSynchronize(st);
        cudaFree(p);
    }
    bool alloc(size_t bytes)
    {
        if (dev_malloc(&p, std::max<size_t>(bytes, 1)) == cudaSuccess) return true;
        p = nullptr;
        cudaGetLastError();
        return false;
    }
};

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

int patches_of(int n) { return (n + 1 + kWinCells - 1) / kWinCells; }

// Cost of a block for a group of nb instances, in instructions: its pair and
// single entries and the staging of its rays and radii.
double block_cost(const WinBlock& b, int nb)
{
    const double pair = nb == 4 ? 40.0 : nb == 2 ? 31.0 : 26.0, one = nb == 4 ? 27.0 : nb == 2 ? 20.0 : 16.0;
    double c = 100.0 + b.n_rays * (26.0 / 32.0) + b.n_slots * ((6.0 + 3.0 * nb) / 32.0);
    for (const uint2& h : b.half) c += 2.0 * (pair * (double)(h.y & 0xffffu) + one * (double)(h.y >> 16)) + 20.0;
    return c;
}
// Warps differ in what an instruction costs them (bank conflicts go by the
// directions of their rays), so on plans with this many instructions per warp
// the last quarter of the work is cut into small shares that the warps take
// from a queue as they run out.  Gather without and with it: 5343 and 4775 us
// for 8 x 1024^2, 1983 and 1761 us for 64 uneven instances, 1437 and 1379 us
// for one 1024^2 image with single-image lists.  Below, a share that takes
// some 8000 cycles to begin and to end is no longer small: 139 and 165 us at
// 512^2, 341 and 356 us at 760^2.  Shares of 0.15 of a warp's mean instead of
// 0.05: 4918 us for 8 x 1024^2; a tail of 0.15 or 0.4 of the work: 5044, 4810.
constexpr double kTailFrom = 1e5, kTailPart = 0.25, kTailShare = 0.05;
constexpr double kFlushCost = 100.0;   // end of a patch, per instance

// Samples with a position of their own that the first pass has room for (5 x
// 10^8 samples at 8 radii per pixel have some ten).
constexpr uint32_t kOwnFirst = 1 << 12;
constexpr double kPatchRays = 11.0;   // rays of a detector that an 8 x 8 patch sees, about
constexpr int kMinRays = 96;

// Whether angle a (radians) is a multiple of pi / 4 to rounding, and which.
bool eighth_turns(double a, int& k)
{
    const double x = a / (6.283185307179586476925 / 8.0);
    if (!(std::fabs(x) < 1e6)) return false;
    k = (int)std::lround(x);
    return std::fabs(x - k) < 1e-10;
}

// The largest symmetry (of those in WinSym, of at most the given order) of a
// geometry.  The detectors sit
// at theta0 + (j + 1/2) Phi / n_det: an arc is its own mirror image in its
// bisector, a ring also turns into itself by a quarter (half) when n_det is a
// multiple of 4 (2).  The map must be one of the square's, and take the angles
// 2 pi q / K to one another.
int32_t win_symmetry(const pat_geometry_t& g, int max_order)
{
    if (max_order < 2) return kSymNone;
    const bool ring = std::fabs(g.arc_span - 6.283185307179586476925) < 1e-12;
    if (max_order >= 4 && ring && g.n_det % 4 == 0 && g.n_angles % 4 == 0) return kSymQuarter;
    if (g.n_det % 2 != 0) return kSymNone;
    int k = 0;
    if (eighth_turns(g.arc_start + 0.5 * g.arc_span, k)) {
        k = ((k % 4) + 4) % 4;   // the bisector as an axis, in eighths of a turn
        if (k == 0) return kSymMirrorY;
        if (k == 2 && g.n_angles % 2 == 0) return kSymMirrorX;
        if (k % 2 == 1 && g.n_angles % 4 == 0) return k == 1 ? kSymDiag : kSymAnti;
    }
    return ring && g.n_angles % 2 == 0 ? kSymHalf : kSymNone;
}

// Images that share lists are fewer, longer pieces of work: as many together
// as leave every resident warp two blocks of 64 rays (adjoint at 128^2, 64
// detectors: 19 us single, 21.5 us in pairs; at 256^2, 128 detectors: 42 us
// single, 36 us in pairs).
int images_together(const pat_geometry_t* geoms, int n_inst, double warps)
{
    double rays = 0.0;
    for (int i = 0; i < n_inst; ++i) rays += kPatchRays * patches_of(geoms[i].n) * patches_of(geoms[i].n) * geoms[i].n_det;
    int nb = 4;
    while (nb > 1 && rays / nb < 2.0 * 64.0 * warps) nb /= 2;
    return nb;
}

bool same_geometry(const pat_geometry_t& a, const pat_geometry_t& b)
{
    return a.n == b.n && a.n_det == b.n_det && a.arc_start == b.arc_start && a.arc_span == b.arc_span &&
           a.n_t == b.n_t && a.t_max == b.t_max && a.n_angles == b.n_angles;
}

// Whether any two images of a plan share lists: those of one symmetric
// geometry or of two equal ones.
bool share_lists(const pat_geometry_t* geoms, int n_inst, int nb_max)
{
    if (nb_max < 2) return false;
    for (int i = 0; i < n_inst; ++i) {
        if (win_symmetry(geoms[i], nb_max) != kSymNone) return true;
        for (int k = 0; k < i; ++k)
            if (same_geometry(geoms[i], geoms[k])) return true;
    }
    return false;
}

} // namespace

bool windows_fit(const pat_geometry_t* geoms, int n_inst, int num_sms)
{
    double windows = 0.0, patches = 0.0, samples = 0.0;   // (about 41 % of a full circle's samples fall on the image)
    for (int i = 0; i < n_inst; ++i) {
        const pat_geometry_t& g = geoms[i];
        // radii across a patch's diagonal (11.31 pixels and the widening), with both ends, the alignment and the padding
        const double delta = g.t_max * g.n / (2.0 * g.n_t);
        if (11.5 / delta + 7.0 > win_slots(4) - 8) return false;
        windows += (double)patches_of(g.n) * patches_of(g.n) * g.n_det;
        patches += (double)patches_of(g.n) * patches_of(g.n);
        samples += 0.41 * g.n_det * std::min(g.n_t + 2.0, 2.2 * g.n_t / g.t_max + 2.0) * g.n_angles;
    }
    // Few patches and little work: a patch is split over many warps, each of
    // which spends more on beginning and ending than on its entries, and the
    // per-cell lists are as fast or faster (adjoint over them / over windows:
    // 18.7 / 20.1 us for 100^2 with 110 detectors, 24.2 / 26.4 for 160^2 with
    // 100, 26.9 / 32.6 for 128^2 with 256).  From 600 patches (36 / 29 us for
    // 4 x 140^2 with 48 detectors) or 12 M samples on (48.6 / 41.8 us for 160^2
    // with 320 detectors, 70.6 / 47.3 for 128^2 with 512) the windows win.
    const double warps = 20.0 * num_sms;
    if (patches < warps / 5.0 && samples < 4000.0 * warps) return false;
    // Lists that serve one image each cost twice as much per sample as shared
    // ones.  Where, besides, the detectors lie all around the image, the cells'
    // lists are about equally long (the per-cell form's weakness is the crowd of
    // a short arc), and with many detectors and not too many patches the
    // per-cell lists are faster.  Measured over 400 drawn geometries on arcs of
    // 185 degrees and more, per-cell / windows: 0.79 to 1.02, mostly 0.85 to
    // 0.95, below 1064 patches from 0.4 detectors per pixel column on (46 / 52
    // us for 176^2 with 292 detectors on 200 degrees), and 0.82 to 1.05 below
    // 3800 from 0.7 on (216 / 249 us for 476^2 with 391 on 309 degrees).
    // Outside: 1.04 to 1.35 at 3800 to 4500 patches (418 / 491 us for 512^2
    // with 511 on a ring over windows / per cell), 1.0 to 1.3 with few
    // detectors, 1.2 to 1.9 on half a ring and less.
    // (Both forms are far inside the 1e-5 bound: 2e-7 to 6e-7 of the image per
    // cell, whose sums are one chain, 1.3e-7 to 1.7e-7 over windows, for bipolar
    // pulses with 1 % noise.)
    if (patches < 1.25 * warps && !share_lists(geoms, n_inst, images_together(geoms, n_inst, warps))) {
        const double half_turn = 3.14159265358979323846;
        const bool few = patches < 0.35 * warps;
        bool around = true;
        for (int i = 0; i < n_inst; ++i)
            around = around && geoms[i].arc_span > (few ? 1.1 : 1.3) * half_turn &&
                     geoms[i].n_det > (few ? 0.4 : 0.7) * geoms[i].n;
        if (around) return false;
    }
    return windows * sizeof(int4) <= 4e9;   // (build-time table)
}

pat_status_t build_windows(Plan& P, std::vector<InstDev>& inst, const std::vector<int>& inst_tmpl, int n_tmpl,
                           InstDev* d_inst, int64_t* bytes, int* parts_max, cudaStream_t st)
{
    DevPlan& dp = P.dp;
    const int n_inst = (int)inst.size();
    const int64_t warps = (int64_t)std::max(1, adj_win_blocks_per_sm(1)) * P.num_sms * (kWinThreads / kWarp);
    std::vector<int> rep(n_tmpl, -1);
    for (int i = 0; i < n_inst; ++i) {
        if (rep[inst_tmpl[i]] < 0) rep[inst_tmpl[i]] = i;
        inst[i].win_px = patches_of(inst[i].n);
    }
    const int nb_max = images_together(P.geoms.data(), n_inst, (double)warps);
    for (int i = 0; i < n_inst; ++i) {
        inst[i].win_sym = win_symmetry(P.geoms[i], nb_max);
        inst[i].win_ndet = inst[i].n_det / win_sym_order(inst[i].win_sym);
    }
    if (cudaMemcpyAsync(d_inst, inst.data(), sizeof(InstDev) * inst.size(), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return PAT_ERR_CUDA;

    // blocks of templates with several instances hold fewer radii (their weights
    // take more room each)
    std::vector<int> mult(n_tmpl, 0), slots_of(n_tmpl);
    int rays_max = 0, longest_max = 0;
    for (int i = 0; i < n_inst; ++i) ++mult[inst_tmpl[i]];
    {
        double grouped = 0.0;
        for (int t = 0; t < n_tmpl; ++t) {
            const int images = mult[t] * win_sym_order(inst[rep[t]].win_sym);
            grouped += (double)((images + nb_max - 1) / nb_max) * inst[rep[t]].win_px * inst[rep[t]].win_px *
                       inst[rep[t]].win_ndet * kPatchRays;
        }
        // Rays of a block: as many as fit, or fewer where the plan has too few
        // blocks of that size to give every resident warp two.  A small plan
        // takes as long as its longest single block, so its blocks next to
        // detectors are cut shorter (adjoint at 64^2, 64 detectors: 15.5 us
        // with 48 entries, 13.2 us with 32; at 256^2, 128 detectors, 47 us
        // with 24, 40 us with 48, 37 us with 64).
        const double rays = grouped / (2.0 * (double)warps);
        rays_max = std::max(kMinRays, std::min(win_rays(1), (int)(rays / 16.0) * 16));
        longest_max = rays >= 80.0 ? 64 : 32;
        for (int t = 0; t < n_tmpl; ++t) {
            const int images = nb_max == 1 ? 1 : mult[t] * win_sym_order(inst[rep[t]].win_sym);
            slots_of[t] = images == 1 ? 768 : win_slots(4);   // (records of a block fit a warp's registers)
        }
    }

    // ---- windows, and the blocks of every patch (counts) -------------------
    std::vector<int64_t> win_off(n_tmpl + 1, 0), patch_off(n_tmpl + 1, 0);
    for (int t = 0; t < n_tmpl; ++t) {
        const int64_t np = (int64_t)inst[rep[t]].win_px * inst[rep[t]].win_px;
        patch_off[t + 1] = patch_off[t] + np;
        win_off[t + 1] = win_off[t] + np * inst[rep[t]].win_ndet;
    }
    DevBuf tmp(st);
    const size_t o_cnt = align256(sizeof(int4) * win_off[n_tmpl]);
    const size_t o_own = o_cnt + align256(sizeof(int4) * patch_off[n_tmpl]);
    const size_t o_misc = o_own + align256(sizeof(WinOwn) * kOwnFirst);
    if (!tmp.alloc(o_misc + 256)) return PAT_ERR_OOM;
    unsigned char* tb = static_cast<unsigned char*>(tmp.p);
    int4* d_win = reinterpret_cast<int4*>(tb);
    int4* d_cnt = reinterpret_cast<int4*>(tb + o_cnt);
    int32_t* d_err = reinterpret_cast<int32_t*>(tb + o_misc);
    if (cudaMemsetAsync(d_err, 0, sizeof(int32_t), st) != cudaSuccess) return PAT_ERR_CUDA;
    if (patch_off[n_tmpl] > INT32_MAX) return PAT_ERR_UNSUPPORTED;
    for (int t = 0; t < n_tmpl; ++t) {
        const int i = rep[t], np = (int)(patch_off[t + 1] - patch_off[t]);
        const double delta = P.geoms[i].t_max * P.geoms[i].n / (2.0 * P.geoms[i].n_t);
        if (launch_win_windows(dp, i, inst[i].win_ndet, delta, np, d_win + win_off[t], st) != cudaSuccess)
            return PAT_ERR_CUDA;
    }
    // the samples that need a position of their own, by patch of all templates (a second
    // pass where there are more of them than the first has room for)
    std::vector<WinOwn> own;
    std::vector<int> own_off(n_tmpl + 1, 0);
    DevBuf own_buf(st);
    WinOwn* d_own = reinterpret_cast<WinOwn*>(tb + o_own);
    for (uint32_t cap = kOwnFirst, n = 0;; cap = n) {
        uint32_t* d_count = reinterpret_cast<uint32_t*>(d_err) + 1;
        if (cudaMemsetAsync(d_count, 0, sizeof(uint32_t), st) != cudaSuccess) return PAT_ERR_CUDA;
        for (int t = 0; t < n_tmpl; ++t)
            if (launch_win_own(dp, rep[t], inst[rep[t]].win_ndet, (int)(patch_off[t + 1] - patch_off[t]),
                               (int)patch_off[t], d_win + win_off[t], d_own, cap, d_count, st) != cudaSuccess)
                return PAT_ERR_CUDA;
        if (cudaMemcpyAsync(&n, d_count, sizeof(n), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return PAT_ERR_CUDA;
        if (n > (uint32_t)INT32_MAX) return PAT_ERR_UNSUPPORTED;
        if (n <= cap) {
            own.resize(n);
            break;
        }
        if (!own_buf.alloc(sizeof(WinOwn) * n)) return PAT_ERR_OOM;
        d_own = static_cast<WinOwn*>(own_buf.p);
    }
    if (!own.empty() &&
        (cudaMemcpyAsync(own.data(), d_own, sizeof(WinOwn) * own.size(), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
         cudaStreamSynchronize(st) != cudaSuccess))
        return PAT_ERR_CUDA;
    std::sort(own.begin(), own.end(), [](const WinOwn& a, const WinOwn& b) {
        return std::tie(a.patch, a.j, a.q, a.m) < std::tie(b.patch, b.j, b.q, b.m);
    });
    for (int t = 0, k = 0; t < n_tmpl; ++t) {
        for (; k < (int)own.size() && own[k].patch < patch_off[t + 1]; ++k) own[k].patch -= (int32_t)patch_off[t];
        own_off[t + 1] = k;
    }
    if (!own.empty() &&
        cudaMemcpyAsync(d_own, own.data(), sizeof(WinOwn) * own.size(), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return PAT_ERR_CUDA;
    auto part = [&](int t, WinBlock* blocks, WinSub* subs) {
        return launch_win_part(dp, rep[t], (int)(patch_off[t + 1] - patch_off[t]), rays_max, slots_of[t], longest_max,
                               d_win + win_off[t], d_own + own_off[t], own_off[t + 1] - own_off[t], d_cnt + patch_off[t],
                               blocks, subs, d_err, st);
    };
    for (int t = 0; t < n_tmpl; ++t)
        if (part(t, nullptr, nullptr) != cudaSuccess) return PAT_ERR_CUDA;
    std::vector<int4> cnt(patch_off[n_tmpl]);
    int32_t err = 0;
    if (cudaMemcpyAsync(cnt.data(), d_cnt, sizeof(int4) * cnt.size(), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemcpyAsync(&err, d_err, sizeof(err), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return PAT_ERR_CUDA;
    if (err) return PAT_ERR_UNSUPPORTED;

    // ---- offsets -------------------------------------------------------------
    std::vector<int64_t> blk_off(n_tmpl + 1, 0);
    int64_t n_blocks = 0, n_subs = 0, n_rayrec = 0, n_slotrec = 0;
    for (int t = 0; t < n_tmpl; ++t) {
        blk_off[t] = n_blocks;
        for (int64_t p = patch_off[t]; p < patch_off[t + 1]; ++p) {
            const int4 c = cnt[p];
            cnt[p] = make_int4((int)n_blocks, (int)n_subs, (int)n_rayrec, (int)n_slotrec);
            n_blocks += c.x;
            n_subs += c.y;
            n_rayrec += c.z;
            n_slotrec += c.w;
        }
        if (std::max(std::max(n_blocks, n_subs), std::max(n_rayrec, n_slotrec)) > INT32_MAX) return PAT_ERR_UNSUPPORTED;
    }
    blk_off[n_tmpl] = n_blocks;
    // block heads | staging records (each with the spares that the kernel reads ahead), and the blocks and
    // sub-windows (building only)
    const size_t o_rays = align256(sizeof(uint4) * (n_blocks + 1));
    const size_t o_slots = o_rays + align256(sizeof(uint2) * (n_rayrec + 64));
    const size_t lists_bytes = o_slots + align256(sizeof(uint32_t) * (n_slotrec + 96));
    const size_t o_subs = align256(sizeof(WinBlock) * (n_blocks + 1));
    DevBuf subs(st);
    if (!subs.alloc(o_subs + sizeof(WinSub) * n_subs)) return PAT_ERR_OOM;
    if (dev_malloc(&P.d_lists, lists_bytes) != cudaSuccess) {
        P.d_lists = nullptr;
        cudaGetLastError();
        return PAT_ERR_OOM;
    }
    unsigned char* lb = static_cast<unsigned char*>(P.d_lists);
    uint4* d_heads = reinterpret_cast<uint4*>(lb);
    WinBlock* d_blocks = static_cast<WinBlock*>(subs.p);
    uint2* d_rays = reinterpret_cast<uint2*>(lb + o_rays);
    uint32_t* d_slots = reinterpret_cast<uint32_t*>(lb + o_slots);
    WinSub* d_subs = reinterpret_cast<WinSub*>(static_cast<unsigned char*>(subs.p) + o_subs);
    if (cudaMemsetAsync(lb, 0, lists_bytes, st) != cudaSuccess ||
        cudaMemcpyAsync(d_cnt, cnt.data(), sizeof(int4) * cnt.size(), cudaMemcpyHostToDevice, st) != cudaSuccess)
        return PAT_ERR_CUDA;
    for (int t = 0; t < n_tmpl; ++t) {
        const int i = rep[t], nb = (int)(blk_off[t + 1] - blk_off[t]);
        WinBlock* tb0 = d_blocks + blk_off[t];
        if (part(t, d_blocks, d_subs) != cudaSuccess ||
            launch_win_recs(dp, i, nb, tb0, d_subs, d_rays, d_slots, st) != cudaSuccess ||
            launch_win_lists(dp, i, nb, tb0, d_subs, nullptr, st) != cudaSuccess)
            return PAT_ERR_CUDA;
    }
    std::vector<WinBlock> blocks(n_blocks);
    if (cudaMemcpyAsync(blocks.data(), d_blocks, sizeof(WinBlock) * blocks.size(), cudaMemcpyDeviceToHost, st) !=
            cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return PAT_ERR_CUDA;

    // ---- code offsets ----------------------------------------------------------
    int64_t n_vecs = 0;
    std::vector<uint4> heads;
    heads.reserve(blocks.size());
    for (WinBlock& b : blocks) {
        heads.push_back(make_uint4((uint32_t)b.patch, (uint32_t)b.n_rays | (uint32_t)b.n_slots << 16, b.half[0].y,
                                   b.half[1].y));
        for (uint2& h : b.half) {
            h.x = (uint32_t)n_vecs;
            n_vecs += (h.y & 0xffffu) + (h.y >> 16);
        }
        if (n_vecs > (int64_t)UINT32_MAX) return PAT_ERR_UNSUPPORTED;
    }

    // ---- groups of four, two and one images, and their warp shares -----------
    std::vector<std::vector<int>> members(n_tmpl);
    for (int i = 0; i < n_inst; ++i) members[inst_tmpl[i]].push_back(i);
    std::vector<WinGroup> groups;
    std::vector<WinShare> shares;
    std::vector<int2> zinfo;
    int64_t n_tiles = 0;
    *parts_max = 1;
    for (int cls = 0; cls < 3; ++cls) {
        const int nb = cls == 0 ? 4 : cls == 1 ? 2 : 1;
        const int g0 = (int)groups.size();
        for (int t = 0; t < n_tmpl; ++t) {
            // groups of nb_max while they last; three images left over also share one group of four
            const InstDev& d = inst[rep[t]];
            const int order = win_sym_order(d.win_sym), per = std::max(1, nb / order);   // instances per group
            const int m = (int)members[t].size(), images = m * order, left = images % nb_max;
            const int first = nb == nb_max ? 0 : images / nb_max * nb_max / order;
            const int n_groups = nb > nb_max    ? 0
                                 : nb == nb_max ? images / nb_max + (left == 3 ? 1 : 0)
                                                : left == nb ? 1 : 0;
            for (int k = 0; k < n_groups; ++k) {
                WinGroup g;
                std::memset(&g, 0, sizeof(g));
                const int n_members = std::min(per, m - first - k * per);
                g.n_img = n_members * order;
                g.zinfo_off = (int32_t)zinfo.size();
                g.m_mask = d.m_pitch - 1;
                for (int c = 0; c < 4; ++c) {
                    const int cc = std::min(c, g.n_img - 1), s = cc % order;
                    const int i = members[t][first + k * per + cc / order];
                    g.mbar_off[c] = inst[i].mbar_off;
                    if (s > 0 && (d.win_sym == kSymHalf || d.win_sym == kSymQuarter)) {
                        g.mbar_off[c] += (int64_t)s * d.win_ndet * d.m_pitch;
                    } else if (s > 0) {
                        g.mbar_off[c] += (int64_t)(d.n_det - 1) * d.m_pitch;
                        g.flip |= 1 << c;
                    }
                    if (c < g.n_img && s == 0) {
                        inst[i].win_img = c;
                        inst[i].win_nimg = g.n_img;
                        inst[i].win_tile0 = (int32_t)n_tiles;
                    }
                }
                g.block0 = blk_off[t];
                g.n_blocks = (int32_t)(blk_off[t + 1] - blk_off[t]);
                if (g.n_blocks > 0) {
                    const WinBlock& b0 = blocks[g.block0];
                    g.ray_rec0 = b0.ray_rec;
                    g.slot_rec0 = b0.slot_rec;
                    g.code0 = b0.half[0].x;
                }
                g.det_off = inst[rep[t]].det_off;
                g.ray_off = inst[rep[t]].win_ray_off;
                g.tile0 = (int32_t)n_tiles;
                n_tiles += (patch_off[t + 1] - patch_off[t]) * g.n_img;
                zinfo.resize(zinfo.size() + (patch_off[t + 1] - patch_off[t]), make_int2(0, 0));
                if (g.n_blocks > 0) groups.push_back(g);
            }
        }
        const int g1 = (int)groups.size();
        if (n_tiles > INT32_MAX) return PAT_ERR_UNSUPPORTED;
        dp.win_n_warps[cls] = dp.win_n_tail[cls] = 0;
        if (g0 == g1) continue;
        const int bps = adj_win_blocks_per_sm(nb);
        if (bps < 1) return PAT_ERR_UNSUPPORTED;
        double total = 0.0;
        int64_t seq = 0;
        auto cost_of = [&](const WinGroup& g, int b) {
            const WinBlock* x = &blocks[g.block0 + b];
            const bool end = b + 1 == g.n_blocks || x[1].patch != x[0].patch;
            return block_cost(*x, nb) + (end ? kFlushCost * g.n_img : 0.0);
        };
        for (int g = g0; g < g1; ++g)
            for (int b = 0; b < groups[g].n_blocks; ++b, ++seq) total += cost_of(groups[g], b);
        const int64_t n = std::min<int64_t>((int64_t)bps * P.num_sms * (kWinThreads / kWarp), seq);
        const double tail_part = total / (double)n >= kTailFrom ? kTailPart : 0.0;
        const double share = (1.0 - tail_part) * total / (double)n, tail_share = kTailShare * total / (double)n;
        auto begin_at = [&](int64_t k) {   // cost before share k
            return k <= n ? share * (double)k : share * (double)n + tail_share * (double)(k - n);
        };
        double done = 0.0;
        int64_t k = 0;   // shares begun
        int last_patch = -1, last_group = -1;
        for (int g = g0; g < g1; ++g)
            for (int b = 0; b < groups[g].n_blocks; ++b) {
                const double c = cost_of(groups[g], b);
                // a block belongs to the share that its middle falls into
                const bool begin = k == 0 || ((k < n || tail_part > 0.0) && done + 0.5 * c >= begin_at(k));
                const int patch = blocks[groups[g].block0 + b].patch;
                int2& z = zinfo[groups[g].zinfo_off + patch];
                const bool fresh = g != last_group || patch != last_patch;
                if (fresh) z = make_int2((int)n_tiles, 0);
                if (fresh || begin) {
                    if (begin) {
                        const WinBlock& b0 = blocks[groups[g].block0 + b];
                        shares.push_back({g, b, 0, z.y, b0.ray_rec, b0.slot_rec, b0.half[0].x, 0});
                    }
                    ++z.y;
                    n_tiles += groups[g].n_img;   // (a patch that stays whole leaves its part's tile unused)
                    *parts_max = std::max(*parts_max, z.y);
                }
                if (begin) {
                    ++(k < n ? dp.win_n_warps : dp.win_n_tail)[cls];
                    ++k;
                }
                ++shares.back().count;
                done += c;
                last_group = g;
                last_patch = patch;
            }
    }
    if (n_tiles > INT32_MAX) return PAT_ERR_UNSUPPORTED;

    // ---- codes, tables and pixel sums -----------------------------------------
    const size_t b_codes = align256(256 * (size_t)(n_vecs + 64));
    const size_t o_groups = b_codes, o_shares = o_groups + align256(sizeof(WinGroup) * (groups.size() + 1));
    const size_t o_zinfo = o_shares + align256(sizeof(WinShare) * (shares.size() + 1));
    const size_t o_arr = o_zinfo + align256(sizeof(int2) * (zinfo.size() + 1));
    const size_t o_z = o_arr + align256(sizeof(int32_t) * (zinfo.size() + 1));
    const size_t codes_bytes = o_z + sizeof(float) * kWinTile * (size_t)n_tiles;
    if (dev_malloc(&P.d_codes, codes_bytes) != cudaSuccess) {
        P.d_codes = nullptr;
        cudaGetLastError();
        return PAT_ERR_OOM;
    }
    unsigned char* cb = static_cast<unsigned char*>(P.d_codes);
    uint2* d_codes = reinterpret_cast<uint2*>(cb);
    auto up = [&](void* dst, const void* src, size_t b) {
        return b == 0 || cudaMemcpyAsync(dst, src, b, cudaMemcpyHostToDevice, st) == cudaSuccess;
    };
    // (patches without samples keep their zero sums; no part has arrived)
    if (cudaMemsetAsync(cb + o_arr, 0, codes_bytes - o_arr, st) != cudaSuccess) return PAT_ERR_CUDA;
    if (!up(d_blocks, blocks.data(), sizeof(WinBlock) * blocks.size()) ||
        !up(d_heads, heads.data(), sizeof(uint4) * heads.size()) ||
        !up(cb + o_groups, groups.data(), sizeof(WinGroup) * groups.size()) ||
        !up(cb + o_shares, shares.data(), sizeof(WinShare) * shares.size()) ||
        !up(cb + o_zinfo, zinfo.data(), sizeof(int2) * zinfo.size()) ||
        !up(d_inst, inst.data(), sizeof(InstDev) * inst.size()))
        return PAT_ERR_CUDA;
    for (int t = 0; t < n_tmpl; ++t)
        if (launch_win_lists(dp, rep[t], (int)(blk_off[t + 1] - blk_off[t]), d_blocks + blk_off[t], d_subs, d_codes, st) != cudaSuccess)
            return PAT_ERR_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return PAT_ERR_CUDA;
    dp.win_heads = d_heads;
    dp.win_rays = d_rays;
    dp.win_slots = d_slots;
    dp.win_codes = d_codes;
    dp.win_groups = reinterpret_cast<const WinGroup*>(cb + o_groups);
    dp.win_shares = reinterpret_cast<const WinShare*>(cb + o_shares);
    dp.win_zinfo = reinterpret_cast<const int2*>(cb + o_zinfo);
    dp.win_arrived = reinterpret_cast<int32_t*>(cb + o_arr);
    dp.win_z = reinterpret_cast<float*>(cb + o_z);
    dp.n_win_vecs = n_vecs + 1;   // (> 0: in use)
    *bytes = (int64_t)(lists_bytes + codes_bytes);
    return PAT_OK;
}

} // namespace patgpu
