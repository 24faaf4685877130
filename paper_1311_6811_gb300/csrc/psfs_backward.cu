// psfs_backward.cu -- adjoint of the reconstruction (no counterpart in the
// paper, which only runs the forward; this is the gradient of a loss on the
// posterior of Eq. 3-4 with respect to the maps of Eq. 2 and the background
// model of Eq. 1).
//
// Loss gradient d_occ per voxel in, gradients per pixel out:
//   dLoss/dL_v   = d_occ_v occ_v (1 - occ_v)                     (voxel pass)
//   dLoss/dg_kp  = sum over voxels v whose centre projects to pixel p of
//                  camera k of dLoss/dL_v                         (pixel pass)
//   dLoss/ds     = dLoss/dg ((2 P_D - 1) / a - (2 q - 1) / b)
//   dLoss/dr     = dLoss/ds s (1 - s),  s = sigmoid(r), r = log U - log N
//   dLoss/dmu_c  = dLoss/dr (-(I_c - mu_c) / var_c)
//   dLoss/dvar_c = dLoss/dr (1 / (2 var_c) - (I_c - mu_c)^2 / (2 var_c^2))
//
// The forward is recomputed (maps, then the log-odds of every voxel), not
// stored.  This file holds the voxel pass; the pixel pass, which sums each
// pixel's owners in a fixed order from per-handle owner lists, is in
// psfs_owners.cu.
#include "psfs_fuse_common.cuh"

namespace psfs {

namespace {

template <typename MapT, int LX, int WY, int TZ>
__global__ void __launch_bounds__(32 * WY) backward_voxel_kernel(const __grid_constant__ BackwardArgs b,
                                                                 int parts_log2)
{
    const FuseArgs &a = b.f;
    __shared__ int s_flags[PSFS_MAX_CAMS];
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
    for (int c = 0; c < a.n_cams; ++c) {
        const int flags = s_flags[c];
        if (flags & kTcSkip) continue;
        float m[12];
#pragma unroll
        for (int q = 0; q < 12; ++q) m[q] = a.cam[c].m[q];
        float bu, bv, bw;
        project_base(m, tc.fi, tc.fj, &bu, &bv, &bw);
        gather_global<MapT, TZ>(m, bu, bv, bw, tc.fk, maps + (int64_t)c * a.map_stride, W, H,
                                (flags & kTcInside) != 0, L, a.status);
    }
    if (tc.i >= a.nx || tc.j >= a.ny) return;
#pragma unroll
    for (int t = 0; t < TZ; ++t) {
        const int k = tc.k0 + t;
        if (k >= a.nz) break;
        const uint32_t lin = (uint32_t)tc.i + (uint32_t)a.nx * ((uint32_t)tc.j + (uint32_t)a.ny * (uint32_t)k);
        const float occ = posterior_of_logodds(L[t] + a.logit_prior);
        b.dl[(size_t)lin * b.dl_stride] = __ldg(b.d_occ + lin) * occ * (1.0f - occ);
    }
}

template <typename MapT, int LX, int TZ>
cudaError_t launch_voxel_typed(const BackwardArgs &b, int parts_log2, cudaStream_t s)
{
    backward_voxel_kernel<MapT, LX, 4, TZ><<<(unsigned)b.f.n_tiles << parts_log2, dim3(32, 4), 0, s>>>(b, parts_log2);
    return cudaGetLastError();
}

template <typename MapT, int LX>
cudaError_t launch_voxel_lx(const BackwardArgs &b, int tz, cudaStream_t s)
{
    const int p = tile_parts_log2(b.f.n_tiles, tz);
    switch (tz >> p) {
    case 2: return launch_voxel_typed<MapT, LX, 2>(b, p, s);
    case 4: return launch_voxel_typed<MapT, LX, 4>(b, p, s);
    case 8: return launch_voxel_typed<MapT, LX, 8>(b, p, s);
    case 16: return launch_voxel_typed<MapT, LX, 16>(b, p, s);
    default: return cudaErrorInvalidValue;
    }
}

template <typename MapT>
cudaError_t launch_voxel_shape(const BackwardArgs &b, const FuseShape &sh, cudaStream_t s)
{
    if (sh.wy != 4) return cudaErrorInvalidValue;
    if (sh.lx == 8) return launch_voxel_lx<MapT, 8>(b, sh.tz, s);
    if (sh.lx == 16) return launch_voxel_lx<MapT, 16>(b, sh.tz, s);
    if (sh.lx == 32) return launch_voxel_lx<MapT, 32>(b, sh.tz, s);
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_backward_voxel(const BackwardArgs &b, const FuseShape &shape, int map_dtype, cudaStream_t s)
{
    if (b.f.n_tiles <= 0) return cudaSuccess;
    if (map_dtype == PSFS_MAP_F16) return launch_voxel_shape<__half>(b, shape, s);
    if (map_dtype == PSFS_MAP_BF16) return launch_voxel_shape<__nv_bfloat16>(b, shape, s);
    return launch_voxel_shape<float>(b, shape, s);
}

}  // namespace psfs
