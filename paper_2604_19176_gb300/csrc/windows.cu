// windows.cu — adjoint circular means f = C^T Mbar over windowed run-pair lists
// (the default gather; gather.cu holds the other list forms).
//
// As in gather.cu, work happens per cell and every output is summed by the
// lane that owns it, in a fixed order.  What differs is where an entry finds
// its detector, ray and weight.  The per-cell lists of gather.cu read three
// tables through L1 at addresses that differ from lane to lane, and the L1
// data path bounds them (82 % of its peak).  Here a warp owns an 8 x 8 patch
// of cells and walks its detectors block by block: the few rays and radii of
// those detectors that can reach the patch (its windows) are staged in shared
// memory, and a list entry is just two shared-memory offsets.
//
// Sample position.  A staged ray holds its position modulo one pixel in 32-bit
// fixed point, extrapolated to offset 0 of the staged radii, and its step per
// byte of that offset, so an entry's fraction is one multiply-add:
//     u = X + offset * D  (mod 2^32),   a = u / 2^32 .
// The cell is known (it is the lane's), so the integer part is never needed.
// X is formed at the centre radius of the window from 64-bit tables; the step
// is rounded to 2^-30 pixel, so u is within 2^-31 x (radii from the centre) +
// 2^-32 of the exact position: 6e-9 pixel at two radii per pixel (13 from the
// centre), 1.3e-7 at the finest radii that a patch's window may have (some 48
// per pixel, 275 from the centre); the FP32 split form is within 3 x 2^-25 =
// 9e-8.  Which cell of which patch lists a sample is decided by its position
// formed at its own radius, the same in every patch; the few samples whose
// staged position lies in another cell get a staged ray of their own
// (win_position.h).  The fraction is read as the 23-bit mantissa of 1 + a,
// centred in its truncation interval.
//
// Lists.  Two samples of one ray at consecutive radii in one cell make a pair
// entry; others are single.  Half a patch (8 x 4 cells, lane = cell) has, per
// block, P pair vectors, then S single vectors (two entries per lane and
// vector, the 32 cells interleaved), padded with null entries (a staged weight
// of zero).  P and S are chosen for the least cost: a cell with more pairs
// than P lists the rest as singles.
//
// Schedule.  Warps work alone: each has its own staged tables and nothing but
// warp barriers, because the lists of the cells near a detector are many times
// longer than the others' (one CTA per 16 x 16 patch, its eight warps meeting
// at a barrier per block, left the warps waiting for the longest list more
// than half of the time: 61 us at 256^2).  The blocks of all patches and
// instances form one sequence, cut into equal-cost shares, one per resident
// warp, so a patch is split over a few warps where there are few patches; on
// large plans (TAIL) the end of the sequence makes smaller shares, which the
// warps take from a queue as they run out (kTailFrom in windows_plan.cpp).  A
// warp adds its cells' corner sums into 9 x 9 pixel sums and writes those (81
// values instead of 256), which the combining kernels add (adj_pixel).
//
// Images that share lists.  Most geometries have a symmetry (WinSym): every
// arc is its own mirror image in its bisector, and where that is an axis or a
// diagonal of the grid the second half of the detectors is the mirror image
// of the first; a ring also repeats by quarter turns.  The lists then hold the
// first half (quarter) of the detectors, and the copies' weights are gathered
// with the same entries into further images, which adj_pixel turns back.
// Instances with the same geometry share lists in the same way.  Up to four
// images are processed together (NB): the code, the staged ray and the
// fractions serve all, and their weights sit side by side in shared memory.
//
// Bound by the L1 data path, which shared memory shares: about 10 wavefronts
// per 32 real samples for one image, most of them the 16-byte ray of every
// entry, 6 for two images and 4.5 for four; issue slots are half used.  At
// 512^2 (256 detectors on a half ring, pairs of images) ncu counts 27 M shared
// wavefronts and 79 M warp instructions, 70 % of the L1 data path's peak.
// Gather and combine, per-cell run-pair lists -> windowed lists: 49 -> 32 us
// at 256^2 (128 detectors, half ring), 328 -> 139 us at 512^2, 595 -> 330 us
// at 760^2 (256 detectors, 270 degrees), 3.53 -> 1.75 ms for 64 uneven
// instances, 13.4 -> 4.8 ms for 8 x 1024^2 (90 % of the L1 data path's peak
// in the uneven batch; two fifths of the wavefronts are bank conflicts).
#include <algorithm>

#include "device_common.cuh"
#include "kernels.h"
#include "win_position.h"

namespace patgpu {

namespace {

// 1 + (u / 2^32 cut to 23 bits): the mantissa is that of 0x7f : u >> 9.
// Adding kFracBias, exactly, leaves the cut fraction + 2^-24.
constexpr float kFracBias = -0.99999994f;
__device__ __forceinline__ float frac_bits(uint32_t u)
{
    return __uint_as_float(__funnelshift_r(u, 0x7fu, 9));
}

// Staged ray: position at offset 0 and step per offset byte, both modulo one
// pixel in 2^-32 pixel units.
__device__ __forceinline__ uint4 staged_ray(uint2 uv, uint4 r, uint32_t mb, uint32_t mob)
{
    const uint32_t dx = (r.x + 2u) >> 2, dy = (r.y + 2u) >> 2;
    const uint32_t x = uv.x + mb * r.x + __umulhi(mb, r.z);
    const uint32_t y = uv.y + mb * r.y + __umulhi(mb, r.w);
    return make_uint4(x - mob * dx, y - mob * dy, dx, dy);
}

// Two samples' values in one f32x2 register pair: a pair entry's, or two single
// entries'.
using F2 = unsigned long long;

// Moments of one image, sum w, sum w a, sum w b, sum w a b, the two halves of
// every register pair for the two samples that an instruction handles.
struct Sums {
    F2 s0, sa, sb, sab;
    __device__ __forceinline__ void clear() { s0 = sa = sb = sab = 0ull; }
    __device__ __forceinline__ void add(F2 w, F2 a, F2 b, F2 ab)
    {
        s0 = f2_add(s0, w);
        sa = f2_fma(a, w, sa);
        sb = f2_fma(b, w, sb);
        sab = f2_fma(ab, w, sab);
    }
    __device__ __forceinline__ void add_to(float4& t) const
    {
        auto both = [](F2 v) {
            const float2 h = f2_unpack(v);
            return h.x + h.y;
        };
        t.x += both(s0);
        t.y += both(sa);
        t.z += both(sb);
        t.w += both(sab);
    }
};

} // namespace

// Codes are read once by one warp: past L1, which the staging loads need.
__device__ __forceinline__ uint2 load_code(const uint2* p)
{
    uint2 v;
    asm volatile("ld.global.nc.L1::no_allocate.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ void prefetch_l2_line(const void* p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Cell of lane `lane` in half h of a patch.  Shared memory serves 16-byte reads
// eight lanes at a time: eight lanes hold 4 x 2 cells rather than a row of
// eight, so that they meet fewer different rays.
__device__ __forceinline__ int cell_x(int lane) { return (lane & 3) + ((lane >> 1) & 4); }
__device__ __forceinline__ int cell_y(int h, int lane) { return 4 * h + ((lane >> 2) & 1) + ((lane >> 3) & 2); }

// Shared memory of a warp: rays, then the images' radii (slots 0 .. 7 zero).  It
// starts on a multiple of kWinAlign, so that the address of a staged ray is
// the entry's offset bits or'ed into the warp's base.
constexpr uint32_t kWinAlign = 4096;
__host__ __device__ constexpr int win_warp_bytes(int nb)
{
    return win_rays(nb) * 16 + win_slots(nb) * 4 * nb;
}
static_assert(win_warp_bytes(1) % kWinAlign == 0 && win_warp_bytes(2) % kWinAlign == 0 &&
                  win_warp_bytes(4) % kWinAlign == 0 && win_rays(1) * 16 <= (int)kWinAlign &&
                  win_slots(1) * 4 <= 0x1400 && win_slots(2) * 4 <= 0x1400 && win_slots(4) * 4 <= 0x1400,
              "staged tables of a warp");

__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
template <int OFF>
__device__ __forceinline__ float lds32(uint32_t addr)
{
    float v;
    asm volatile("ld.shared.f32 %0, [%1 + %2];" : "=f"(v) : "r"(addr), "n"(OFF));
    return v;
}

// 20 warps per SM (96 registers; 16 for four images): 24 warps at 80 registers
// took 150 instead of 144 us at 512^2, and left L1 too little room.
template <int NB, bool TAIL>
__global__ void __launch_bounds__(kWinThreads, NB == 4 ? 4 : 5)
    k_adj_win(DevPlan dp, int share0, int n_warps, int n_tail)
{
    extern __shared__ __align__(16) unsigned char win_smem[];
    const int lane = threadIdx.x & 31;
    const int wid = blockIdx.x * (kWinThreads / kWarp) + (threadIdx.x >> 5);
    // (dynamic shared memory starts past a reserved part of it: align by hand)
    unsigned char* rays_b = win_smem + ((kWinAlign - smem_u32(win_smem) % kWinAlign) % kWinAlign) +
                            (threadIdx.x >> 5) * win_warp_bytes(NB);
    unsigned char* m_b = rays_b + win_rays(NB) * 16;
    uint4* s_rays = reinterpret_cast<uint4*>(rays_b);
    float* s_m = reinterpret_cast<float*>(m_b);
    const uint32_t rays_a = smem_u32(rays_b), m_a = smem_u32(m_b);
    if (wid >= n_warps) {
        pdl_wait();
        return;
    }
    WinShare sh = dp.win_shares[share0 + wid];
    int gi = sh.group, bi = sh.block, part = sh.part;
    for (int i = lane; i < 8 * NB; i += kWarp) s_m[(i >> 3) * win_slots(NB) + (i & 7)] = 0.f;

    // A block's head, staging records and codes follow the previous block's, so
    // the next block's can be requested before its head is here: heads, records
    // and codes are read one block (two vectors) ahead, past the end of the
    // share into what follows (the arrays end with spares).
    const uint4* heads = nullptr;           // the next block's head
    const uint2* ray_recs = nullptr;        // the current block's records
    const uint32_t* slot_recs = nullptr;
    const uint2* cp = nullptr;              // codes: c0, c1 the next two vectors, cp the one after
    uint4 head;                             // (patch, rays | radii << 16, lengths of the halves' lists)
    uint2 rrec[2], c0, c1;
    uint32_t srec[3];
    auto load_recs = [&]() {                // lane l holds records l, l + 32, ...
        rrec[0] = __ldg(ray_recs + lane);
        rrec[1] = __ldg(ray_recs + lane + 32);
#pragma unroll
        for (int i = 0; i < 3; ++i) srec[i] = __ldg(slot_recs + lane + 32 * i);
    };
    auto start = [&](int block, uint32_t ray_rec, uint32_t slot_rec, uint32_t code) {
        heads = dp.win_heads + dp.win_groups[gi].block0 + block;
        ray_recs = dp.win_rays + ray_rec;
        slot_recs = dp.win_slots + slot_rec;
        head = __ldg(heads++);
        load_recs();
        cp = dp.win_codes + (size_t)code * 32 + lane;
        c0 = load_code(cp);
        c1 = load_code(cp + 32);
        cp += 64;
    };
    start(bi, sh.ray_rec, sh.slot_rec, sh.code);
    int32_t* const queue = dp.work_counters + kQueueStride;
    float4 tot[2][NB];   // moments of the two halves' cells over the blocks
    auto clear_totals = [&]() {
#pragma unroll
        for (int c = 0; c < NB; ++c) tot[0][c] = tot[1][c] = make_float4(0.f, 0.f, 0.f, 0.f);
    };
    clear_totals();
#ifdef PAT_DEBUG
    bool plant = dp.bounds_probe != 0 && share0 == 0 && threadIdx.x == 0;   // (in every CTA: some warps have no entries)
#endif
    int ticket = wid;
    for (int k = 0; k < sh.count; ++k) {
        const WinGroup* G = dp.win_groups + gi;
        const int patch = (int)head.x;
        const int n_rays = (int)(head.y & 0xffffu), n_slots = (int)(head.y >> 16);
        const uint32_t len0 = head.z, len1 = head.w;   // pair vectors | single vectors << 16
        // ---- stage the block's radii and rays -------------------------------
        auto stage_weights = [&]() {
            // (four radii per lane; a flipped image's rows run backwards from its first)
#pragma unroll
            for (int t = 0; t < (NB == 1 ? 6 : 5); ++t) {   // (768 or 576 radii at most)
                const uint32_t idx = __shfl_sync(0xffffffffu, srec[t >> 1], (t & 1) * 16 + (lane >> 1)) + (uint32_t)(lane & 1) * 4u;
                const int s = (t * kWarp + lane) * 4;
                // (of the images of an instance only the second can be flipped)
                const int odd = NB > 1 && G->flip ? 2 * (int)(idx & (uint32_t)G->m_mask) - (int)idx : (int)idx;
                if (s < n_slots)
#pragma unroll
                    for (int c = 0; c < NB; ++c)
                        cp_async16_l1(s_m + c * win_slots(NB) + 8 + s, dp.mbar + G->mbar_off[c] + ((c & 1) ? odd : (int)idx));
            }
            cp_async_commit();
        };
        if (k > 0) stage_weights();
        const int4* det = dp.win_det + G->det_off;
        const uint4* dirs = dp.win_dirs + G->ray_off + (lane & 3);
#pragma unroll
        for (int g = 0; g < 2; ++g) {   // 96 rays at a time, their loads in flight together
            if (g * 3 * kWarp >= n_rays) break;
            uint2 rc[3], uv[3];
            uint4 rd[3];
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int t = 3 * g + i;   // (records past the end are the next block's: read, not used)
                rc[i].x = __shfl_sync(0xffffffffu, rrec[t >> 2].x, (t & 3) * 8 + (lane >> 2));
                rc[i].y = __shfl_sync(0xffffffffu, rrec[t >> 2].y, (t & 3) * 8 + (lane >> 2));
                uv[i] = __ldg(reinterpret_cast<const uint2*>(det + (rc[i].x & 0x3fffu)));
                rd[i] = __ldg(dirs + (rc[i].y & 0xffffu));
            }
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const int s = (3 * g + i) * kWarp + lane;
                if (s < n_rays) s_rays[s] = staged_ray(uv[i], rd[i], rc[i].x >> 14, m_a + (rc[i].y >> 16) * 4u);
            }
        }
        if (k == 0) {   // Mbar comes from the previous kernel, the rays from plan tables
            if (!TAIL || ticket == wid) pdl_wait();
            stage_weights();
            if (TAIL && lane == 0) ticket = n_warps + atomicAdd(queue, 1);
        }
        // ---- the next block's head and records, in flight while this one is processed
        const bool more = k + 1 < sh.count;
        const bool same = bi + 1 < G->n_blocks;   // (else the next block is another group's first)
        {   // and the codes after this block's on their way to L2, 64 lines of 128 bytes
            const int nv = (int)((len0 & 0xffffu) + (len0 >> 16) + (len1 & 0xffffu) + (len1 >> 16));
            const char* next = reinterpret_cast<const char*>(cp - 64 - lane + nv * 32) + lane * 128;
            if (more) {
                prefetch_l2_line(next);
                prefetch_l2_line(next + 4096);
            }
        }
        if (more && same) {
            ray_recs += n_rays >> 2;
            slot_recs += n_slots >> 3;
            head = __ldg(heads++);
            load_recs();
        }
        cp_async_wait_group<0>();
        __syncwarp();
        // ---- the entries of the two halves -----------------------------------
        // the staged ray and weights of an entry, and its position
        // (the staged positions are extrapolated to shared-memory address 0 of the radii)
        auto locate = [&](uint32_t c, bool pair, uint4& ray, uint32_t& ma, uint32_t& u, uint32_t& v) {
            uint32_t mo = c >> 16, ro = c & (kWinAlign - 16u);
#ifdef PAT_DEBUG
            if (plant) {
                mo += 0x1400u;   // past the radii of any form, inside the CTA's shared memory
                plant = false;
            }
            // (an entry out of bounds is given the null entry's place)
            if (!dbg_ok(dp, ro < (uint32_t)n_rays * 16u + 16u && mo + (pair ? 4u : 0u) < (uint32_t)win_slots(NB) * 4u,
                        kSiteListEntry))
                mo = ro = 0u;
#endif
            ray = lds128(ro | rays_a);
            ma = mo + m_a;
            u = ray.x + ma * ray.z;
            v = ray.y + ma * ray.w;
        };
        const F2 bias = f2_pack(kFracBias, kFracBias);
        auto pair_entry = [&](Sums(&acc)[NB], uint32_t c) {
            uint4 ray;
            uint32_t ma, u, v;
            locate(c, true, ray, ma, u, v);
            const F2 a = f2_add(f2_pack(frac_bits(u), frac_bits(u + 4u * ray.z)), bias);
            const F2 b = f2_add(f2_pack(frac_bits(v), frac_bits(v + 4u * ray.w)), bias);
            const F2 ab = f2_mul(a, b);
            constexpr int kImg = win_slots(NB) * 4;   // bytes of an image's radii
            acc[0].add(f2_pack(lds32<0>(ma), lds32<4>(ma)), a, b, ab);
            if constexpr (NB > 1) acc[1].add(f2_pack(lds32<kImg>(ma), lds32<kImg + 4>(ma)), a, b, ab);
            if constexpr (NB > 2) {
                acc[2].add(f2_pack(lds32<2 * kImg>(ma), lds32<2 * kImg + 4>(ma)), a, b, ab);
                acc[3].add(f2_pack(lds32<3 * kImg>(ma), lds32<3 * kImg + 4>(ma)), a, b, ab);
            }
        };
        auto two_singles = [&](Sums(&acc)[NB], uint2 c) {
            uint4 r0, r1;
            uint32_t m0, m1, u0, v0, u1, v1;
            locate(c.x, false, r0, m0, u0, v0);
            locate(c.y, false, r1, m1, u1, v1);
            const F2 a = f2_add(f2_pack(frac_bits(u0), frac_bits(u1)), bias);
            const F2 b = f2_add(f2_pack(frac_bits(v0), frac_bits(v1)), bias);
            const F2 ab = f2_mul(a, b);
            constexpr int kImg = win_slots(NB) * 4;
            acc[0].add(f2_pack(lds32<0>(m0), lds32<0>(m1)), a, b, ab);
            if constexpr (NB > 1) acc[1].add(f2_pack(lds32<kImg>(m0), lds32<kImg>(m1)), a, b, ab);
            if constexpr (NB > 2) {
                acc[2].add(f2_pack(lds32<2 * kImg>(m0), lds32<2 * kImg>(m1)), a, b, ab);
                acc[3].add(f2_pack(lds32<3 * kImg>(m0), lds32<3 * kImg>(m1)), a, b, ab);
            }
        };
        // (the codes of both halves and of the following blocks are one stream)
        if (dbg_ok(dp, n_rays <= win_rays(NB) && n_slots + 8 <= win_slots(NB) && cp <= dp.win_codes + dp.n_win_vecs * 32 + 96,
                   kSiteListItem)) {
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const uint32_t len = h ? len1 : len0;
                const int np = (int)(len & 0xffffu), ns = (int)(len >> 16);
                Sums acc[NB];
#pragma unroll
                for (int c = 0; c < NB; ++c) acc[c].clear();
                auto step = [&]() {   // the current vector; the one after next starts loading
                    const uint2 c = c0;
                    c0 = c1;
                    c1 = load_code(cp);
                    cp += 32;
                    return c;
                };
#pragma unroll 2
                for (int i = 0; i < np; ++i) {
                    const uint2 c = step();
                    pair_entry(acc, c.x);
                    pair_entry(acc, c.y);
                }
#pragma unroll 2
                for (int i = 0; i < ns; ++i) two_singles(acc, step());
#pragma unroll
                for (int c = 0; c < NB; ++c) {
                    if (h == 0) acc[c].add_to(tot[0][c]);
                    else acc[c].add_to(tot[1][c]);
                }
            }
        }
        __syncwarp();   // the staged tables are free

        // ---- end of the patch (or of this warp's share of it) -----------------
        if (!more || !same || (int)head.x != patch) {
            const int zi = G->zinfo_off + patch, n_img = G->n_img;
            const int2 z = __ldg(dp.win_zinfo + zi);   // first tile of the parts, parts
            float* sum_out = dp.win_z + (size_t)(G->tile0 + patch * n_img) * kWinTile;
            float* part_out = z.y > 1 ? dp.win_z + (size_t)(z.x + part * n_img) * kWinTile : sum_out;
            float* ex = reinterpret_cast<float*>(rays_b);   // corner sums of the 8 x 8 cells, over the staged rays
#pragma unroll
            for (int c = 0; c < NB; ++c) {
                if (c >= n_img) break;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float4 t = tot[h][c];   // sum w, sum w a, sum w b, sum w a b
                    const float z10 = t.y - t.w, z01 = t.z - t.w;
                    const int lc = cell_y(h, lane) * 8 + cell_x(lane);
                    ex[lc] = t.x - t.y - z01;
                    ex[64 + lc] = z10;
                    ex[128 + lc] = z01;
                    ex[192 + lc] = t.w;
                }
                __syncwarp();
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    const int o = t * 32 + lane;
                    if (o >= kWinPixels) break;
                    // core pixels, then the right column (9 values), then the top row
                    const int x = o < 64 ? o & 7 : o < 73 ? 8 : o - 73;
                    const int y = o < 64 ? o >> 3 : o < 73 ? o - 64 : 8;
                    float s = 0.f;
                    if (x < 8 && y < 8) s += ex[y * 8 + x];
                    if (x > 0 && y < 8) s += ex[64 + y * 8 + x - 1];
                    if (x < 8 && y > 0) s += ex[128 + (y - 1) * 8 + x];
                    if (x > 0 && y > 0) s += ex[192 + (y - 1) * 8 + x - 1];
                    part_out[c * kWinTile + o] = s;
                }
                __syncwarp();
            }
            if (z.y > 1) {   // the last warp to finish a part adds them all, in part order
                __threadfence();
                __syncwarp();
                int arrived = 0;
                if (lane == 0) arrived = atomicAdd(dp.win_arrived + zi, 1);
                if (__shfl_sync(0xffffffffu, arrived, 0) == z.y - 1) {
                    __threadfence();
                    // (eight parts' loads in flight: a patch next to detectors has dozens)
                    const float4* src = reinterpret_cast<const float4*>(dp.win_z + (size_t)z.x * kWinTile);
                    const int n4 = n_img * (kWinTile / 4);
                    for (int o = lane; o < n4; o += kWarp) {
                        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
                        for (int g = 0; g < z.y; g += 8) {
                            float4 v[8];
#pragma unroll
                            for (int u = 0; u < 8; ++u)
                                v[u] = g + u < z.y ? __ldcg(src + (size_t)(g + u) * n4 + o)
                                                   : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                            for (int u = 0; u < 8; ++u) {
                                s.x += v[u].x;
                                s.y += v[u].y;
                                s.z += v[u].z;
                                s.w += v[u].w;
                            }
                        }
                        reinterpret_cast<float4*>(sum_out)[o] = s;
                    }
                    if (lane == 0) dp.win_arrived[zi] = 0;   // for the next launch
                }
            }
            clear_totals();
            part = 0;
        }
        ++bi;
        if (more && !same) {
            bi = 0;
            const WinGroup* N = dp.win_groups + ++gi;
            start(0, N->ray_rec0, N->slot_rec0, N->code0);
        }
        if constexpr (TAIL) {   // the next share from the queue
            if (k + 1 < sh.count) continue;
            ticket = __shfl_sync(0xffffffffu, ticket, 0);
            if (ticket >= n_warps + n_tail) break;
            sh = dp.win_shares[share0 + ticket];
            gi = sh.group;
            bi = sh.block;
            part = sh.part;
            start(bi, sh.ray_rec, sh.slot_rec, sh.code);
            k = -1;
        }
    }
    // the last warp to run out of shares re-arms the queue for the next launch
    if (TAIL && lane == 0 && atomicAdd(queue + 1, 1) == n_warps - 1) queue[0] = queue[1] = 0;
}

// ---------------------------------------------------------------------------
// List building (plan creation)
// ---------------------------------------------------------------------------
namespace {

__device__ __forceinline__ int pad_to(int v, int m) { return (v + m - 1) / m * m; }

// Cells [x0, x1) x [y0, y1) of patch p of an instance (absolute indices).
__device__ __forceinline__ void patch_cells(const InstDev& in, int p, int& x0, int& y0, int& x1, int& y1)
{
    x0 = (p % in.win_px) * kWinCells - 1;
    y0 = (p / in.win_px) * kWinCells - 1;
    x1 = min(x0 + kWinCells, in.n);
    y1 = min(y0 + kWinCells, in.n);
}

} // namespace

// win[j * patches + p] = (q0, nq, m0, nm | near << 16): the range of detector j
// and patch p (win_range).
__global__ void k_win_windows(DevPlan dp, int inst_idx, double delta, int patches, int4* __restrict__ win)
{
    const InstDev in = dp.inst[inst_idx];
    const int p = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (p >= patches) return;
    int x0, y0, x1, y1;
    patch_cells(in, p, x0, y0, x1, y1);
    for (int jj = j; jj < in.win_ndet; jj += gridDim.y) {
        const int4 d = dp.win_det[in.det_off + jj];
        const double U = (double)d.z + (double)(uint32_t)d.x * (1.0 / 4294967296.0);
        const double V = (double)d.w + (double)(uint32_t)d.y * (1.0 / 4294967296.0);
        const WinRange r =
            win_range(U, V, x0 - in.c0, y0 - in.c0, x1 - in.c0, y1 - in.c0, in.K, in.n_r, in.m_pitch, delta);
        win[(size_t)jj * patches + p] = make_int4(r.q0, r.nq, r.m0, r.nm | r.near << 16);
    }
}

namespace {

// Fixed-point detector and direction of a sample's ray.
struct RayFixed {
    int4 det;
    uint4 dir;
    int2 whole;
    __device__ __forceinline__ int64_t u(int m) const
    {
        return win_position((int64_t)det.z * 4294967296ll + (int64_t)(uint32_t)det.x, whole.x, dir.x, dir.z, m);
    }
    __device__ __forceinline__ int64_t v(int m) const
    {
        return win_position((int64_t)det.w * 4294967296ll + (int64_t)(uint32_t)det.y, whole.y, dir.y, dir.w, m);
    }
};
__device__ __forceinline__ RayFixed ray_fixed(const DevPlan& dp, const InstDev& in, int j, int q)
{
    return {__ldg(dp.win_det + in.det_off + j), __ldg(dp.win_dirs + in.win_ray_off + q),
            __ldg(dp.win_dirs_int + in.win_ray_off + q)};
}

} // namespace

// The samples of every window that land in its patch but whose staged position
// lands in another cell: (patch0 + patch, j, q, m) into own[], the first `cap`
// of them in no order; *count counts all.  A warp per window, lane = ray.
__global__ void __launch_bounds__(256) k_win_own(DevPlan dp, int inst_idx, int patches, int patch0,
                                                 const int4* __restrict__ win, WinOwn* __restrict__ own, uint32_t cap,
                                                 uint32_t* __restrict__ count)
{
    const InstDev in = dp.inst[inst_idx];
    const int lane = threadIdx.x & 31;
    const int64_t n_win = (int64_t)patches * in.win_ndet;
    for (int64_t w = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); w < n_win; w += (int64_t)gridDim.x * 8) {
        const int4 wv = win[w];
        const int nm = wv.w & 0xffff, m0 = wv.z;
        if (wv.y <= 0 || nm <= 0) continue;
        const int j = (int)(w / patches), p = (int)(w % patches), mc = win_anchor(m0, nm);
        int x0, y0, x1, y1;
        patch_cells(in, p, x0, y0, x1, y1);
        for (int i = lane; i < wv.y; i += kWarp) {
            int q = wv.x + i;
            if (q >= in.K) q -= in.K;
            const RayFixed r = ray_fixed(dp, in, j, q);
            const int64_t uc = r.u(mc), vc = r.v(mc);
            const int64_t su = win_step(r.whole.x, r.dir.x), sv = win_step(r.whole.y, r.dir.y);
            for (int m = m0; m < m0 + nm; ++m) {
                const int cx = win_cell(r.u(m)), cy = win_cell(r.v(m));
                if (win_cell(win_staged(uc, su, m, mc)) == cx && win_cell(win_staged(vc, sv, m, mc)) == cy) continue;
                if (cx + in.c0 < x0 || cx + in.c0 >= x1 || cy + in.c0 < y0 || cy + in.c0 >= y1) continue;
                const uint32_t at = atomicAdd(count, 1u);
                if (at < cap) own[at] = {patch0 + p, j, q, m};
            }
        }
    }
}

// Cuts the detectors of every patch into blocks whose windows fit the staged
// tables (max_rays rays, max_slots radii) and whose longest list stays near
// max_longest entries (the warps are the unit of scheduling, and the cells
// next to a detector see every one of its rays); a window of more rays becomes
// several.  The patch's samples of own[] (n_own, ascending) follow, one
// sub-window each.  With blocks == nullptr counts (blocks, sub-windows, ray and slot
// groups) per patch into cnt; else writes them from the offsets in cnt.
__global__ void k_win_part(DevPlan dp, int inst_idx, int patches, int max_rays, int max_slots, int max_longest,
                           const int4* __restrict__ win, const WinOwn* __restrict__ own, int n_own,
                           int4* __restrict__ cnt, WinBlock* __restrict__ blocks, WinSub* __restrict__ subs,
                           int32_t* __restrict__ err)
{
    const InstDev in = dp.inst[inst_idx];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= patches) return;
    const int4 base = blocks ? cnt[p] : make_int4(0, 0, 0, 0);
    int nb = 0, ns = 0, rg = 0, sg = 0, sub_first = 0;
    int rays = 0, slots = 8, longest = 0;
    bool open = false;
    auto close = [&]() {
        if (!open) return;
        if (blocks) {
            WinBlock b{};
            b.patch = p;
            b.n_rays = (uint16_t)rays;
            b.n_slots = (uint16_t)(slots - 8);
            b.ray_rec = (uint32_t)(base.z + rg);
            b.slot_rec = (uint32_t)(base.w + sg);
            b.sub0 = (uint32_t)(base.y + sub_first);
            b.n_sub = (uint32_t)(ns - sub_first);
            blocks[base.x + nb] = b;
        }
        ++nb;
        rg += rays / 4;
        sg += (slots - 8) / 8;
        open = false;
    };
    // rays q0 .. q0 + n - 1 and radii m0 .. m0 + nm - 1 of detector j, anchored at mc; len: their part of the longest list
    // (an odd number of fours: the next window's rays then start in the other half of the eight
    // 16-byte bank groups; shared-memory conflicts of the gather, 144 -> 138 us at 512^2)
    auto add = [&](int j, int q0, int n, int m0, int nm, int mc, int len, int own_sample) {
        const int n4 = min(pad_to(n, 4) | 4, max_rays), nmp = pad_to(nm, 8);
        if (open && (rays + n4 > max_rays || slots + nmp > max_slots || longest + len > max_longest)) close();
        if (!open) {
            open = true;
            rays = longest = 0;
            slots = 8;
            sub_first = ns;
        }
        if (subs)
            subs[base.y + ns] = {j, q0, (uint16_t)n, (uint16_t)nm, (uint16_t)m0, (uint16_t)mc, (uint16_t)rays, (uint16_t)slots,
                                 own_sample};
        rays += n4;
        slots += nmp;
        longest += len;
        ++ns;
    };
    for (int j = 0; j < in.win_ndet; ++j) {
        const int4 wv = win[(size_t)j * patches + p];
        const int nm = wv.w & 0xffff, near = wv.w >> 16;
        if (wv.y <= 0 || nm <= 0) continue;
        if (8 + pad_to(nm, 8) > max_slots) {
            if (!blocks) atomicExch(err, 1);
            return;
        }
        const int chunk = near > max_longest ? min(max_rays, max_longest) : max_rays;
        for (int qd = 0; qd < wv.y; qd += chunk) {
            const int n = min(chunk, wv.y - qd);
            add(j, (wv.x + qd) % in.K, n, wv.z, nm, win_anchor(wv.z, nm), min(n, near), 0);
        }
    }
    int o = 0;   // the patch's first
    for (int hi = n_own; o < hi;) {
        const int mid = (o + hi) / 2;
        if (own[mid].patch < p) o = mid + 1;
        else hi = mid;
    }
    for (; o < n_own && own[o].patch == p; ++o) {
        const int m = own[o].m, m0 = max(0, min(m & ~3, in.m_pitch - 8));   // (eight radii, 16-byte reads)
        add(own[o].j, own[o].q, 1, m0, m - m0 + 1, m, 1, 1);
    }
    close();
    if (!blocks) cnt[p] = make_int4(nb, ns, rg, sg);
}

// The staging records of every block: one per four rays (detector and centre
// radius; first ray and the centre radius's slot) and one per eight radii
// (index of the first in the instance's Mbar).
__global__ void k_win_recs(DevPlan dp, int inst_idx, const WinBlock* __restrict__ blocks,
                           const WinSub* __restrict__ subs, uint2* __restrict__ rayrec, uint32_t* __restrict__ slotrec)
{
    const InstDev in = dp.inst[inst_idx];
    const WinBlock b = blocks[blockIdx.x];
    for (uint32_t i = 0; i < b.n_sub; ++i) {
        const WinSub s = subs[b.sub0 + i];
        for (int g = threadIdx.x; 4 * g < s.nq; g += blockDim.x)
            rayrec[b.ray_rec + s.ray0 / 4 + g] =
                make_uint2((uint32_t)s.j | (uint32_t)s.mc << 14,
                           (uint32_t)((s.q0 + 4 * g) % in.K) | (uint32_t)(s.slot0 + s.mc - s.m0) << 16);
        for (int g = threadIdx.x; 8 * g < s.nm; g += blockDim.x)
            slotrec[b.slot_rec + (s.slot0 - 8) / 8 + g] = (uint32_t)s.j * (uint32_t)in.m_pitch + (uint32_t)(s.m0 + 8 * g);
    }
}

namespace {

// Candidate search margins, as in gather.cu: half cell diagonal plus rounding,
// slab widening (pixels), angle (radians).
constexpr float kWinRcell = 0.70710678f + 0.004f, kWinSlabEps = 0.01f, kWinAngMargin = 1.0e-5f;

// Calls hit(rel, m) for the samples of sub-window s (ray q0 + rel, radius m)
// that land in centred cell (cxi, cyi) and whose staged position, the one whose
// fraction k_adj_win uses, lands there too, rays ascending from the cell's
// first, radii ascending.
template <typename Hit>
__device__ __forceinline__ void enumerate_window(const DevPlan& dp, const InstDev& in, const WinSub& s, int cxi,
                                                 int cyi, Hit&& hit)
{
    if (s.own) {
        const RayFixed r = ray_fixed(dp, in, s.j, s.q0);
        if (win_cell(r.u(s.mc)) == cxi && win_cell(r.v(s.mc)) == cyi) hit(0, s.mc);
        return;
    }
    const float cxf = (float)cxi, cyf = (float)cyi;
    const float4 d = __ldg(dp.det + in.det_off + s.j);
    const float U = d.x + d.z, V = d.y + d.w;
    const float du = cxf + 0.5f - U, dv = cyf + 0.5f - V;
    const float rc = sqrtf(fmaf(du, du, dv * dv));
    const int mlo = max(0, (int)ceilf((rc - kWinRcell) * in.inv_delta));
    const int mhi = min(in.n_r - 1, (int)floorf((rc + kWinRcell) * in.inv_delta));
    if (mlo > mhi) return;
    const int K = in.K;
    int qlo = 0, qn = K;
    if (rc > 1.25f * kWinRcell) {
        const float phic = atan2_approx(dv, du);
        const float alpha = asin_upper(__fdividef(kWinRcell, rc)) + kWinAngMargin;
        qlo = (int)ceilf((phic - alpha) * in.inv_dphi);
        qn = min((int)floorf((phic + alpha) * in.inv_dphi) - qlo + 1, K);
        if (qlo < 0) qlo += K;
    }
    const float ax0 = (cxf - kWinSlabEps) - U, ax1 = (cxf + 1.f + kWinSlabEps) - U;
    const float ay0 = (cyf - kWinSlabEps) - V, ay1 = (cyf + 1.f + kWinSlabEps) - V;
    const float2* rtrig = dp.rtrig + in.ray_off;
    for (int i = 0; i < qn; ++i) {
        int q = qlo + i;
        if (q >= K) q -= K;
        int rel = q - s.q0;
        if (rel < 0) rel += K;
        if (rel >= s.nq) continue;
        const float2 ri = __ldg(rtrig + q);
        const float tx0 = ax0 * ri.x, tx1 = ax1 * ri.x;
        const float ty0 = ay0 * ri.y, ty1 = ay1 * ri.y;
        const float lo = fmaxf(fminf(tx0, tx1), fminf(ty0, ty1));
        const float hi = fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1));
        const int m0 = max(max(mlo, (int)ceilf(lo)), s.m0), m1 = min(min(mhi, (int)floorf(hi)), s.m0 + s.nm - 1);
        if (m0 > m1) continue;
        const RayFixed r = ray_fixed(dp, in, s.j, q);
        const int64_t uc = r.u(s.mc), vc = r.v(s.mc);
        const int64_t su = win_step(r.whole.x, r.dir.x), sv = win_step(r.whole.y, r.dir.y);
        for (int m = m0; m <= m1; ++m)
            if (win_cell(win_staged(uc, su, m, s.mc)) == cxi && win_cell(win_staged(vc, sv, m, s.mc)) == cyi &&
                win_cell(r.u(m)) == cxi && win_cell(r.v(m)) == cyi)
                hit(rel, m);
    }
}

} // namespace

// One CTA of two warps per block, warp = half a patch, lane = cell.  FILL
// false: the counts of pair and single vectors of both (WinBlock::half[].y);
// FILL true: the codes.
template <bool FILL>
__global__ void __launch_bounds__(64) k_win_lists(DevPlan dp, int inst_idx, WinBlock* __restrict__ blocks,
                                                           const WinSub* __restrict__ subs, uint2* __restrict__ codes)
{
    const InstDev in = dp.inst[inst_idx];
    WinBlock* B = blocks + blockIdx.x;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x0, y0, x1, y1;
    patch_cells(in, B->patch, x0, y0, x1, y1);
    const int cx = x0 + cell_x(lane), cy = y0 + cell_y(w, lane);
    const bool valid = cx < x1 && cy < y1;
    const uint2 wc = FILL ? B->half[w] : make_uint2(0u, 0u);
    const int P = 2 * (int)(wc.y & 0xffffu), S = 2 * (int)(wc.y >> 16);
    uint32_t* out = reinterpret_cast<uint32_t*>(codes + (size_t)wc.x * 32 + lane);
    int p = 0, s = 0;
    auto put = [&](int pos, uint32_t code) { out[(size_t)(pos >> 1) * 64 + (pos & 1)] = code; };
    if (valid) {
        for (uint32_t i = 0; i < B->n_sub; ++i) {
            const WinSub sub = subs[B->sub0 + i];
            int pr = -1, pm = 0;   // pending hit that may start a pair
            auto code_of = [&](int rel, int m) {
                return (uint32_t)(sub.slot0 + m - sub.m0) << 18 | (uint32_t)(sub.ray0 + rel) << 4;
            };
            auto single = [&](int rel, int m) {
                if (FILL && s < S) put(P + s, code_of(rel, m));
                ++s;
            };
            auto pair = [&](int rel, int m) {
                if (FILL && p >= P) {   // more pairs than the warp's vectors hold: two singles
                    single(rel, m);
                    single(rel, m + 1);
                    return;
                }
                if (FILL) put(p, code_of(rel, m));
                ++p;
            };
            enumerate_window(dp, in, sub, cx - in.c0, cy - in.c0, [&](int rel, int m) {
                if (pr == rel && pm + 1 == m) {
                    pair(rel, pm);
                    pr = -1;
                } else {
                    if (pr >= 0) single(pr, pm);
                    pr = rel;
                    pm = m;
                }
            });
            if (pr >= 0) single(pr, pm);
        }
    }
    if (FILL) {
        // Null entries (radius slot 0 holds zero) up to P and S, and each lane's
        // entries moved apart so that they stand where their ray stands among
        // the block's rays: lanes then read rays and radii of the same
        // detectors at the same time (fewer bank conflicts: 11.7 -> 10.0
        // shared-memory wavefronts per pair step in a count of the lists)
        auto spread = [&](int at, int n, int room) {
            for (int k = n; k < room; ++k) put(at + k, 0u);
            int next = room;
            for (int k = n - 1; k >= 0; --k) {
                const uint32_t c = out[(size_t)((at + k) >> 1) * 64 + ((at + k) & 1)];
                const int t = max(k, min(next - 1, (int)((c & 0xffffu) >> 4) * room / (int)B->n_rays));
                if (t != k) {
                    put(at + t, c);
                    put(at + k, 0u);
                }
                next = t;
            }
        };
        spread(0, p, P);
        spread(P, min(s, S), S);
        return;
    }
    // the number of pair vectors with the least cost over the warp (a pair
    // entry costs about 25 instructions, a single one 17)
    auto warp_max = [](int v) {
        for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
        return v;
    };
    const int pmax = (warp_max(p) + 1) & ~1;
    int best = 1 << 30, bp = 0, bs = 0;
    for (int d = 0; d <= 16; d += 2) {
        const int Pd = max(0, pmax - d);
        const int Sd = (warp_max(s + 2 * max(0, p - Pd)) + 1) & ~1;
        if (25 * Pd + 17 * Sd < best) {
            best = 25 * Pd + 17 * Sd;
            bp = Pd;
            bs = Sd;
        }
    }
    if (lane == 0) B->half[w] = make_uint2(0u, (uint32_t)(bp / 2) | (uint32_t)(bs / 2) << 16);
}

// ---------------------------------------------------------------------------
namespace {
const void* win_fn(int nb)
{
    return nb == 4   ? reinterpret_cast<const void*>(k_adj_win<4, false>)
           : nb == 2 ? reinterpret_cast<const void*>(k_adj_win<2, false>)
                     : reinterpret_cast<const void*>(k_adj_win<1, false>);
}
int win_smem_bytes(int nb) { return (kWinThreads / kWarp) * win_warp_bytes(nb) + (int)kWinAlign - 16; }
} // namespace

int adj_win_blocks_per_sm(int nb)
{
    if (cudaFuncSetAttribute(win_fn(nb), cudaFuncAttributeMaxDynamicSharedMemorySize, win_smem_bytes(nb)) !=
        cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, win_fn(nb), kWinThreads, win_smem_bytes(nb)) !=
        cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_adj_win(const DevPlan& dp, cudaStream_t st)
{
    int share0 = 0;
    for (int c = 0; c < 3; ++c) {   // groups of 4, 2 and 1 images
        const int n = dp.win_n_warps[c], tail = dp.win_n_tail[c], nb = c == 0 ? 4 : c == 1 ? 2 : 1;
        if (n == 0) continue;
        const int warps = kWinThreads / kWarp;
        const size_t smem = (size_t)win_smem_bytes(nb);
        auto* fn = c == 0   ? (tail ? k_adj_win<4, true> : k_adj_win<4, false>)
                   : c == 1 ? (tail ? k_adj_win<2, true> : k_adj_win<2, false>)
                            : (tail ? k_adj_win<1, true> : k_adj_win<1, false>);
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = launch_pdl(fn, dim3((n + warps - 1) / warps), dim3(kWinThreads), smem, st, 1, dp, share0, n,
                           tail);
        if (e != cudaSuccess) return e;
        share0 += n + tail;
    }
    return cudaSuccess;
}

cudaError_t launch_win_windows(const DevPlan& dp, int inst_idx, int n_det, double delta, int patches, int4* win,
                               cudaStream_t st)
{
    k_win_windows<<<dim3((unsigned)((patches + 127) / 128), (unsigned)(n_det < 32768 ? n_det : 32768)), 128, 0, st>>>(
        dp, inst_idx, delta, patches, win);
    return cudaGetLastError();
}

cudaError_t launch_win_own(const DevPlan& dp, int inst_idx, int n_det, int patches, int patch0, const int4* win,
                           WinOwn* own, uint32_t cap, uint32_t* count, cudaStream_t st)
{
    const int64_t blocks = ((int64_t)n_det * patches + 7) / 8;
    k_win_own<<<(unsigned)std::min<int64_t>(blocks, 1 << 20), 256, 0, st>>>(dp, inst_idx, patches, patch0, win, own, cap, count);
    return cudaGetLastError();
}

cudaError_t launch_win_part(const DevPlan& dp, int inst_idx, int patches, int max_rays, int max_slots, int max_longest,
                            const int4* win, const WinOwn* own, int n_own, int4* cnt, WinBlock* blocks, WinSub* subs,
                            int32_t* err, cudaStream_t st)
{
    k_win_part<<<(patches + 63) / 64, 64, 0, st>>>(dp, inst_idx, patches, max_rays, max_slots, max_longest, win, own,
                                                   n_own, cnt, blocks, subs, err);
    return cudaGetLastError();
}

cudaError_t launch_win_recs(const DevPlan& dp, int inst_idx, int n_blocks, const WinBlock* blocks, const WinSub* subs,
                            uint2* rayrec, uint32_t* slotrec, cudaStream_t st)
{
    if (n_blocks == 0) return cudaSuccess;
    k_win_recs<<<n_blocks, 64, 0, st>>>(dp, inst_idx, blocks, subs, rayrec, slotrec);
    return cudaGetLastError();
}

cudaError_t launch_win_lists(const DevPlan& dp, int inst_idx, int n_blocks, WinBlock* blocks, const WinSub* subs,
                             uint2* codes, cudaStream_t st)
{
    if (n_blocks == 0) return cudaSuccess;
    if (codes) k_win_lists<true><<<n_blocks, 64, 0, st>>>(dp, inst_idx, blocks, subs, codes);
    else k_win_lists<false><<<n_blocks, 64, 0, st>>>(dp, inst_idx, blocks, subs, codes);
    return cudaGetLastError();
}

} // namespace patgpu
