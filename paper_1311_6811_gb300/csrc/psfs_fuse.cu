// psfs_fuse.cu -- per-voxel stage of the reconstruction: projection of every
// voxel centre into every camera (Eq. 3), gather of the per-pixel log ratio,
// sum over cameras (log form of the product of Eq. 4), posterior, strict
// threshold and compaction of the occupied voxels.
//
// Work decomposition.  A CTA owns a tile of LX (x) x (32/LX) WY (y) x TZ (z)
// voxels: each warp is an LX x 32/LX patch of one z-slice and each thread
// walks TZ voxels along z, sharing the x/y part of the projection.  With the
// cameras on a ring around the grid, a z-slice maps to a band of a few image
// rows, so a square-ish patch (LX = 8) gathers from a handful of 32-byte
// sectors per warp where a 32-voxel row along x spans over a hundred pixels.
// Occupancy stores stay whole sectors (LX consecutive floats per row).  CTAs
// are issued in Morton order of their tiles, so that neighbouring CTAs gather
// from neighbouring parts of the (L2-resident) maps.
//
// Gather.  The instruction stream per voxel and camera is kept minimal:
// three fma for (u, v, w), one approximate reciprocal, two fma with
// round-down that floor u / w and v / w into biased integers, one integer
// multiply-add for the pixel offset, one load, one add.  The host proves per
// (tile, camera) when every voxel centre is in front of the camera and inside
// the image; only the other tiles pay for the visibility test, and cameras
// that see nothing of a tile are skipped.
//
// Compaction: per warp a ballot per z step, per CTA one atomicAdd on the
// global count, then each warp writes its indices at its prefix offset.
#include "psfs_fuse_common.cuh"

namespace psfs {

namespace {

// Beside other frames' kernels (kBeside: a batch's graph) FP32 maps with 16
// planes per thread are held to 64 registers (8 CTAs per SM instead of 6): the
// occupancy is then worth more than the 8 bytes of spills (batches of 16 rigs
// 614.7 us, 619.0 without the bound; of other rigs 481 and 503).  Alone they keep
// the compiler's own 72 (a 128^3 x 8 frame 28.9 us, 31.3 with the bound; 256^3 x
// 16 214 and 224; 20 frames one by one beside their likelihoods 620 and 660), and
// so do 16-bit maps (256^3 x 16: the fusion 114 us with 72, 124 with 64, 133 with
// more than 72).
template <typename MapT, int LX, int WY, int TZ, bool kBeside>
__global__ void __launch_bounds__(32 * WY, kBeside && sizeof(MapT) == 4 && TZ == 16 ? 8 : 0)
    fuse_kernel(const __grid_constant__ FuseArgs a, int parts_log2)
{
    __shared__ int s_flags[PSFS_MAX_CAMS];
    __shared__ uint32_t s_warp_off[WY];
    __shared__ uint32_t s_base;

    const int lane = threadIdx.x;
    const int wy = threadIdx.y;
    const int tid = wy * 32 + lane;
    const uint32_t tile = blockIdx.x >> parts_log2;
    if (tid < a.n_cams) s_flags[tid] = __ldg(&a.tilecam[(int64_t)tile * a.n_cams + tid].w) >> 16;

    TileCoords<LX, WY, TZ> tc;
    tc.init(a, a.tiles[tile], lane, wy, 1 << parts_log2, (int)(blockIdx.x - (tile << parts_log2)));
    const uint32_t W = (uint32_t)a.W, H = (uint32_t)a.H;
    float L[TZ];
#pragma unroll
    for (int t = 0; t < TZ; ++t) L[t] = 0.0f;
    __syncthreads();

    const MapT *maps = reinterpret_cast<const MapT *>(a.maps);
    int c = 0;
    while (c < a.n_cams) {
        const int flags = s_flags[c];
        const int flags1 = c + 1 < a.n_cams ? s_flags[c + 1] : kTcSkip;
        if ((flags & kTcInside) && (flags1 & kTcInside)) {
            // two proven cameras at once: all 2 TZ gathers in flight before
            // any add; the adds keep the camera order of the sequential sum
            float m0[12], m1[12];
#pragma unroll
            for (int q = 0; q < 12; ++q) {
                m0[q] = a.cam[c].m[q];
                m1[q] = a.cam[c + 1].m[q];
            }
            float bu0, bv0, bw0, bu1, bv1, bw1;
            project_base(m0, tc.fi, tc.fj, &bu0, &bv0, &bw0);
            project_base(m1, tc.fi, tc.fj, &bu1, &bv1, &bw1);
            const MapT *map0 = maps + (int64_t)c * a.map_stride, *map1 = map0 + a.map_stride;
            typename MapRaw<MapT>::T g0[TZ], g1[TZ];
#pragma unroll
            for (int t = 0; t < TZ; t += 2) {
                const ProjPair p = project_pair(m0, bu0, bv0, bw0, tc.fk[t], tc.fk[t + 1]);
                const ProjPair q = project_pair(m1, bu1, bv1, bw1, tc.fk[t], tc.fk[t + 1]);
                gather_inside<MapT, false>(p.a, p.b, map0, W, H, g0[t], g0[t + 1], a.status);
                gather_inside<MapT, false>(q.a, q.b, map1, W, H, g1[t], g1[t + 1], a.status);
            }
#pragma unroll
            for (int t = 0; t < TZ; t += 2) {
                add_raw<MapT>(g0[t], g0[t + 1], L[t], L[t + 1]);
                add_raw<MapT>(g1[t], g1[t + 1], L[t], L[t + 1]);
            }
            c += 2;
            continue;
        }
        if (!(flags & kTcSkip)) {
            float m[12];
#pragma unroll
            for (int q = 0; q < 12; ++q) m[q] = a.cam[c].m[q];
            float bu, bv, bw;
            project_base(m, tc.fi, tc.fj, &bu, &bv, &bw);
            gather_global<MapT, TZ>(m, bu, bv, bw, tc.fk, maps + (int64_t)c * a.map_stride, W, H,
                                    (flags & kTcInside) != 0, L, a.status);
        }
        ++c;
    }
    tile_epilogue<WY, TZ>(a, tc.i, tc.j, tc.k0, L, lane, wy, s_warp_off, &s_base);
}

}  // namespace

namespace {

template <typename MapT, int LX, int TZ>
cudaError_t launch_typed(const FuseArgs &a, int parts_log2, bool beside, cudaStream_t s)
{
    const dim3 grid((unsigned)a.n_tiles << parts_log2), block(32, 4);
    if (beside && sizeof(MapT) == 4 && TZ == 16)
        fuse_kernel<MapT, LX, 4, TZ, true><<<grid, block, 0, s>>>(a, parts_log2);
    else
        fuse_kernel<MapT, LX, 4, TZ, false><<<grid, block, 0, s>>>(a, parts_log2);
    return cudaGetLastError();
}

template <typename MapT, int LX>
cudaError_t launch_lx(const FuseArgs &a, int tz, bool beside, cudaStream_t s)
{
    const int p = tile_parts_log2(a.n_tiles, tz);
    switch (tz >> p) {
    case 2: return launch_typed<MapT, LX, 2>(a, p, beside, s);
    case 4: return launch_typed<MapT, LX, 4>(a, p, beside, s);
    case 8: return launch_typed<MapT, LX, 8>(a, p, beside, s);
    case 16: return launch_typed<MapT, LX, 16>(a, p, beside, s);
    default: return cudaErrorInvalidValue;
    }
}

template <typename MapT>
cudaError_t launch_shape(const FuseArgs &a, const FuseShape &sh, bool beside, cudaStream_t s)
{
    if (sh.wy != 4) return cudaErrorInvalidValue;
    if (sh.lx == 8) return launch_lx<MapT, 8>(a, sh.tz, beside, s);
    if (sh.lx == 16) return launch_lx<MapT, 16>(a, sh.tz, beside, s);
    if (sh.lx == 32) return launch_lx<MapT, 32>(a, sh.tz, beside, s);
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_fuse(const FuseArgs &a, const FuseShape &shape, int map_dtype, cudaStream_t s, bool beside)
{
    if (a.n_tiles <= 0) return cudaSuccess;
    if (shape.staged) return launch_fuse_staged(a, shape, map_dtype, s);
    if (map_dtype == PSFS_MAP_F16) return launch_shape<__half>(a, shape, beside, s);
    if (map_dtype == PSFS_MAP_BF16) return launch_shape<__nv_bfloat16>(a, shape, beside, s);
    return launch_shape<float>(a, shape, beside, s);
}

}  // namespace psfs
