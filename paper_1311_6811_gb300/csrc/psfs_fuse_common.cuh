// psfs_fuse_common.cuh -- pieces shared by the two fusion kernels (direct
// gathers and shared-memory staged gathers): the voxel coordinates a thread
// owns in a tile, and the tile epilogue (posterior, strict threshold,
// compaction of the occupied voxels).
#pragma once

#include "psfs_internal.cuh"

namespace psfs {

// Voxel coordinates of a thread in tile `tc`: lane % LX along x, lane / LX
// and the warp index along y, TZ consecutive voxels along z.  Lanes past the
// grid edge (ragged tiles) project the nearest voxel of the grid instead, so
// that the host's per-tile proofs cover them; their results are discarded by
// the epilogue.
template <int LX, int WY, int TZ>
struct TileCoords {
    int i, j, k0;
    float fi, fj;
    float fk[TZ];

    // `part` of `parts`: the thread block takes the part-th TZ planes of a tile
    // of parts * TZ planes.
    __device__ __forceinline__ void init(const FuseArgs &a, uint64_t tc, int lane, int wy, int parts = 1, int part = 0)
    {
        constexpr int LY = 32 / LX;
        const int tx = (int)(tc & 0x1FFFFFu);
        const int ty = (int)((tc >> 21) & 0x1FFFFFu);
        const int tz = (int)(tc >> 42);
        i = tx * LX + (lane % LX);
        j = ty * (LY * WY) + wy * LY + lane / LX;
        k0 = (tz * parts + part) * TZ;
        fi = (float)min(i, a.nx - 1) - a.ci;
        fj = (float)min(j, a.ny - 1) - a.cj;
#pragma unroll
        for (int t = 0; t < TZ; ++t) fk[t] = (float)min(k0 + t, a.nz - 1) - a.ck;
    }
};

// Parts that the tiles of a plan are cut into along z, a CTA each (log2): a
// grid of few tiles would leave most of the GPU idle while each thread walks
// its whole column of voxels.  Cut until there are three CTAs per SM or four
// planes per part; a tile's camera flags hold for its parts.  64^3 x 4 cameras,
// 128 tiles of 16 planes: the adjoint's voxel pass 14.3 -> 8.2 us, a batch of 16
// such rigs 78 -> 67 (one frame per call is bound by its launches either way).
inline int tile_parts_log2(int n_tiles, int tz)
{
    int s = 0;
    while ((tz >> s) > 4 && ((int64_t)n_tiles << s) < 3 * (int64_t)device_sm_count()) ++s;
    return s;
}

// Posterior 1 / (1 + e^-L) (written to the occupancy grid), strict
// threshold L > logit(threshold), and compaction: a ballot per z step in warps
// that hold an occupied voxel, one atomicAdd per CTA on the global count, then
// these warps write their indices at their prefix offsets.  Contains two
// __syncthreads.
template <int WY, int TZ>
__device__ __forceinline__ void tile_epilogue_to(const FuseArgs &a, float *occ, uint32_t *list, uint32_t *count,
                                                 int i, int j, int k0, const float *L, int lane, int wy,
                                                 uint32_t *s_warp_off, uint32_t *s_base)
{
    const bool in_xy = (i < a.nx) && (j < a.ny);
    float top = -INFINITY;   // the largest log-odds of the thread's voxels
#pragma unroll
    for (int t = 0; t < TZ; ++t) {
        const int k = k0 + t;
        if (in_xy && (k < a.nz)) {
            const float lo = L[t] + a.logit_prior;
            const uint32_t lin = (uint32_t)i + (uint32_t)a.nx * ((uint32_t)j + (uint32_t)a.ny * (uint32_t)k);
            __stcs(occ + lin, posterior_of_logodds(lo));
            top = fmaxf(top, lo);
        }
    }
    // few warps hold an occupied voxel (1-3 % of the voxels are): only they
    // form ballots, for the count and again for the list
    uint32_t warp_count = 0;
    auto ballot = [&](int t) {
        return __ballot_sync(0xFFFFFFFFu, in_xy && (k0 + t < a.nz) && (L[t] + a.logit_prior > a.logit_tau));
    };
    if (__any_sync(0xFFFFFFFFu, top > a.logit_tau)) {
#pragma unroll
        for (int t = 0; t < TZ; ++t) warp_count += __popc(ballot(t));
    }
    if (lane == 0) s_warp_off[wy] = warp_count;
    __syncthreads();
    if (wy == 0 && lane == 0) {
        uint32_t total = 0;
#pragma unroll
        for (int w = 0; w < WY; ++w) {
            const uint32_t cnt = s_warp_off[w];
            s_warp_off[w] = total;
            total += cnt;
        }
        uint32_t base = 0;
        if (total) {
            base = atomicAdd(count, total);
            if ((uint64_t)base + total > (uint64_t)a.capacity) atomicOr(a.status, kStatusCapacity);
        }
        *s_base = base;
    }
    __syncthreads();
    if (!warp_count) return;
    uint32_t pos = *s_base + s_warp_off[wy];
    const uint32_t lt_mask = (1u << lane) - 1u;
#pragma unroll
    for (int t = 0; t < TZ; ++t) {
        const uint32_t b = ballot(t);
        if ((b >> lane) & 1u) {
            const uint32_t p = pos + __popc(b & lt_mask);
            if (p < a.capacity) {
                const int k = k0 + t;
                list[p] = (uint32_t)i + (uint32_t)a.nx * ((uint32_t)j + (uint32_t)a.ny * (uint32_t)k);
            }
        }
        pos += __popc(b);
    }
}

// The epilogue into the frame's own outputs a.occ, a.list, a.count.
template <int WY, int TZ>
__device__ __forceinline__ void tile_epilogue(const FuseArgs &a, int i, int j, int k0, const float *L, int lane,
                                              int wy, uint32_t *s_warp_off, uint32_t *s_base)
{
    tile_epilogue_to<WY, TZ>(a, a.occ, a.list, a.count, i, j, k0, L, lane, wy, s_warp_off, s_base);
}

// Two voxels (fi, fj, f0), (fi, fj, f1) of a column projected at once, the
// bits of project_biased for each: every fma but none of the reciprocals takes
// both lanes of a packed instruction.  Only fuse_kernel's two-camera loop
// gains by it (256^3 x 16 cameras, 16-bit maps: 190 against 194 us a frame);
// in the one-camera loops of gather_global the register pairs it needs cost as
// much as it saves (the adjoint's voxel pass: 28.4 against 26.9 us).
struct ProjPair {
    Proj a, b;
};

__device__ __forceinline__ ProjPair project_pair(const float *m, float bu, float bv, float bw, float f0, float f1)
{
    const float2 f = make_float2(f0, f1);
    const float2 u = __ffma2_rn(make_float2(m[2], m[2]), f, make_float2(bu, bu));
    const float2 v = __ffma2_rn(make_float2(m[6], m[6]), f, make_float2(bv, bv));
    const float2 w = __ffma2_rn(make_float2(m[10], m[10]), f, make_float2(bw, bw));
    const float2 rw = make_float2(rcp_approx(w.x), rcp_approx(w.y));
    const float2 magic = make_float2(kFloorMagic, kFloorMagic);
    const float2 x = __ffma2_rd(u, rw, magic), y = __ffma2_rd(v, rw, magic);
    ProjPair p;
    p.a = {w.x, __float_as_uint(x.x), __float_as_uint(y.x)};
    p.b = {w.y, __float_as_uint(x.y), __float_as_uint(y.y)};
    return p;
}

// A map value as it is stored, loaded read-only, or (kCoherent) through the
// coherent path for maps written by other CTAs of the same kernel.
template <typename MapT>
struct MapRaw {
    using T = unsigned short;
};
template <>
struct MapRaw<float> {
    using T = float;
};

template <typename MapT, bool kCoherent = false>
__device__ __forceinline__ typename MapRaw<MapT>::T load_raw(const MapT *p)
{
    const auto *q = reinterpret_cast<const typename MapRaw<MapT>::T *>(p);
    return kCoherent ? *q : __ldg(q);
}

// L0 += g0, L1 += g1: one packed add, or one mixed-precision add each (the
// 16-bit value is widened exactly and added with one rounding, so the sum is
// that of converting first).
template <typename MapT>
__device__ __forceinline__ void add_raw(typename MapRaw<MapT>::T g0, typename MapRaw<MapT>::T g1, float &L0, float &L1);
template <>
__device__ __forceinline__ void add_raw<float>(float g0, float g1, float &L0, float &L1)
{
    const float2 s = __fadd2_rn(make_float2(L0, L1), make_float2(g0, g1));
    L0 = s.x;
    L1 = s.y;
}
template <>
__device__ __forceinline__ void add_raw<__half>(unsigned short g0, unsigned short g1, float &L0, float &L1)
{
    asm("add.rn.f32.f16 %0, %1, %0;" : "+f"(L0) : "h"(g0));
    asm("add.rn.f32.f16 %0, %1, %0;" : "+f"(L1) : "h"(g1));
}
template <>
__device__ __forceinline__ void add_raw<__nv_bfloat16>(unsigned short g0, unsigned short g1, float &L0, float &L1)
{
    asm("add.rn.f32.bf16 %0, %1, %0;" : "+f"(L0) : "h"(g0));
    asm("add.rn.f32.bf16 %0, %1, %0;" : "+f"(L1) : "h"(g1));
}

// The planner's claim for a tile and camera marked inside: the voxel's pixel
// lies in the image (tested in the bounds-checked build only).
__device__ __forceinline__ bool proved_inside(const Proj &p, uint32_t W, uint32_t H)
{
    return (p.bx - kFloorBias) < W && (p.by - kFloorBias) < H;
}

// The gathers of two voxels whose pixels the host proved inside the image
// (0 in the bounds-checked build where the proof fails); min() only guards the
// buffer.
template <typename MapT, bool kCoherent>
__device__ __forceinline__ void gather_inside(const Proj &pa, const Proj &pb, const MapT *map, uint32_t W, uint32_t H,
                                              typename MapRaw<MapT>::T &g0, typename MapRaw<MapT>::T &g1,
                                              uint32_t *status)
{
    (void)status;
    (void)H;
    const uint32_t last_pix = W * H - 1u;
    // (by - B) W + (bx - B) = by W + bx + bias_off (mod 2^32)
    const uint32_t bias_off = 0u - (kFloorBias * W + kFloorBias);
    g0 = g1 = 0;
    if (PSFS_IN_BOUNDS(proved_inside(pa, W, H), status))
        g0 = load_raw<MapT, kCoherent>(map + min(pa.by * W + pa.bx + bias_off, last_pix));
    if (PSFS_IN_BOUNDS(proved_inside(pb, W, H), status))
        g1 = load_raw<MapT, kCoherent>(map + min(pb.by * W + pb.bx + bias_off, last_pix));
}

// One camera's contribution to the TZ voxels of a thread, gathering from
// global memory.  `inside`: the host proved every voxel centre of the tile is
// in front of the camera and inside the image, so no test is made.
// kCoherent: load the maps through the coherent path (maps written by other
// CTAs of the same kernel).
template <typename MapT, int TZ, bool kCoherent = false>
__device__ __forceinline__ void gather_global(const float *m, float bu, float bv, float bw, const float *fk,
                                              const MapT *map, uint32_t W, uint32_t H, bool inside, float *L,
                                              uint32_t *status = nullptr)
{
    static_assert(TZ % 2 == 0, "voxels go in pairs");
    if (inside) {
#pragma unroll
        for (int t = 0; t < TZ; t += 2) {
            typename MapRaw<MapT>::T g0, g1;
            gather_inside<MapT, kCoherent>(project_biased(m, bu, bv, bw, fk[t]),
                                           project_biased(m, bu, bv, bw, fk[t + 1]), map, W, H, g0, g1, status);
            add_raw<MapT>(g0, g1, L[t], L[t + 1]);
        }
    } else {
#pragma unroll
        for (int t = 0; t < TZ; t += 2) {
            const Proj pa = project_biased(m, bu, bv, bw, fk[t]), pb = project_biased(m, bu, bv, bw, fk[t + 1]);
            typename MapRaw<MapT>::T g0 = 0, g1 = 0;   // a voxel that is not seen adds +0: L is never -0
            int pix;
            if (proj_pixel(pa, W, H, &pix)) g0 = load_raw<MapT, kCoherent>(map + pix);
            if (proj_pixel(pb, W, H, &pix)) g1 = load_raw<MapT, kCoherent>(map + pix);
            add_raw<MapT>(g0, g1, L[t], L[t + 1]);
        }
    }
}

}  // namespace psfs
