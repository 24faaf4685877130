// psfs_smooth.cu -- smoothing of the voxel probabilities before the threshold
// (end of Section 2.2.2: the probabilities are filtered, then thresholded;
// step (d) of Section 3.3.3 merges the smoothing with the voxel generation).
// The paper does not give the filter; this is the 3 x 3 x 3 box mean over
// the neighbours inside the grid (a voxel's 27-neighbourhood clipped to the
// grid, divided by the number of voxels in it), then the strict threshold
// smoothed > tau and the compaction of the voxels above it.
//
// One CTA owns 32 (x) x 16 (y) columns over up to 32 planes (z) of one frame; a
// thread owns the columns (x, y) and (x, y + 8).  The planes, each with its
// one-voxel halo (34 x 18, zeros outside the grid), stream through two
// shared-memory buffers in z order with one barrier per plane: the 3-sums
// along x of plane p are formed while plane p + 1 is stored and plane p + 2
// is loaded; after the barrier each thread forms its 3-sums along y, and the
// 3-sums along z come from the y-sums of the last three planes kept in
// registers: ((x-sums) y-sums) z-sums, the same order for every voxel.  The
// scaling by the FP32 reciprocal of the clipped count (one rounding more than
// a division), the optional store of the smoothed value, the threshold and
// the warp-aggregated compaction (one atomicAdd per CTA) follow in the same
// pass, so the frame's probabilities are read once and the smoothed grid is
// written at most once.
//
// When the rows are 16-byte multiples (nx % 4 == 0) smooth_tma_kernel does
// the same sums with far fewer instructions; see there.
#include <algorithm>
#include <climits>

#include "psfs_internal.cuh"

namespace psfs {

namespace {

constexpr int kSX = 32, kSY = 16, kSZ = 32;   // outputs per CTA: 32 x 16 columns, at most 32 planes
// resident per SM: the compiler's own 48 registers; held to 40, for six, the
// kernel is 5 to 10 % slower (20 frames of 190^3 355 against 338 us, 9 of 93 x 110
// x 77 27.0 against 24.9)
constexpr int kSCtas = 5;
constexpr int kHX = kSX + 2, kHY = kSY + 2;    // one plane with its halo: 34 x 18
constexpr int kPlane = kHX * kHY;              // 612 floats
constexpr int kThreads = 256;                  // 8 warps, rows y and y + 8
constexpr int kPerThread = (kPlane + kThreads - 1) / kThreads;   // 3
constexpr int kSums = kHY * kSX;               // 576 x-sums per plane
constexpr int kSumsPerThread = (kSums + kThreads - 1) / kThreads;   // 3

__global__ void __launch_bounds__(kThreads) smooth_kernel(const SmoothArgs a, int tiles_z, int planes)
{
    __shared__ float v[2][kPlane];
    __shared__ float sx[2][kSums];                // [kHY][kSX] x-sums per buffer
    __shared__ uint32_t s_bal[kSZ][2][8];   // ballot per output plane, row half and warp
    __shared__ uint32_t s_off[2][8];
    __shared__ uint32_t s_base;

    const int tid = threadIdx.x;
    const int lx = tid & 31, ly = tid >> 5;
    const int f = blockIdx.z / tiles_z;
    const int x0 = blockIdx.x * kSX, y0 = blockIdx.y * kSY, z0 = (blockIdx.z - f * tiles_z) * planes;
    const int n_in = min(planes, a.nz - z0) + 2;   // z0 - 1 .. the plane after the last
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    // per-frame indices fit 32 bits (the handle's voxel count does)
    const uint32_t nxy = (uint32_t)nx * (uint32_t)ny, n_vox = nxy * (uint32_t)nz;
    const float *prob = a.prob + (size_t)f * n_vox;
    float *out = a.smoothed ? a.smoothed + (size_t)f * n_vox : nullptr;

    // this thread's halo elements e = tid + k * 256 of every plane (row e / 34,
    // column e % 34): in-plane offset and in-grid test, the same for all planes
    uint32_t off[kPerThread];
    bool ok[kPerThread];
#pragma unroll
    for (int k = 0; k < kPerThread; ++k) {
        const int e = tid + k * kThreads;
        const int y = e / kHX, x = e - y * kHX;
        const int ex = x0 - 1 + x, ey = y0 - 1 + y;
        ok[k] = e < kPlane && ex >= 0 && ey >= 0 && ex < nx && ey < ny;
        off[k] = ok[k] ? (uint32_t)ex + (uint32_t)nx * (uint32_t)ey : 0u;
    }
    // this thread's x-sums e = tid + k * 256 (row e / 32, column e % 32): the
    // sum's index in sx is e, its first term's index in v is e + 2 (e / 32)
    int vsrc[kSumsPerThread];
#pragma unroll
    for (int k = 0; k < kSumsPerThread; ++k) {
        const int e = tid + k * kThreads;
        vsrc[k] = e + 2 * (e >> 5);
    }
    auto load_plane = [&](int gz, float (&r)[kPerThread]) {
        const bool okz = gz >= 0 && gz < nz;
        const uint32_t zoff = okz ? (uint32_t)gz * nxy : 0u;
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) r[k] = (okz && ok[k]) ? __ldg(prob + (zoff + off[k])) : 0.0f;
    };
    auto store_plane = [&](int buf, const float (&r)[kPerThread]) {
#pragma unroll
        for (int k = 0; k < kPerThread; ++k)
            if (k * kThreads + kThreads <= kPlane || tid + k * kThreads < kPlane) v[buf][tid + k * kThreads] = r[k];
    };

    // the two columns: clipped neighbourhood counts and output offsets
    const int gx = x0 + lx;
    int gy[2] = {y0 + ly, y0 + ly + 8};
    bool in_xy[2];
    float inv1[2], inv2[2], inv3[2];
    uint32_t col[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        in_xy[h] = gx < nx && gy[h] < ny;
        const int cxy = (1 + (gx > 0) + (gx + 1 < nx)) * (1 + (gy[h] > 0) + (gy[h] + 1 < ny));
        inv1[h] = 1.0f / (float)cxy;
        inv2[h] = 1.0f / (float)(2 * cxy);
        inv3[h] = 1.0f / (float)(3 * cxy);
        col[h] = (uint32_t)gx + (uint32_t)nx * (uint32_t)gy[h];
    }

    // prologue: plane z0 - 1 in buffer 0, plane z0 in registers
    float cur[kPerThread], nxt[kPerThread];
    load_plane(z0 - 1, nxt);
    store_plane(0, nxt);
    load_plane(z0, cur);
    __syncthreads();

    float ya[2] = {0.0f, 0.0f}, yb[2] = {0.0f, 0.0f};   // y-sums of planes p - 2, p - 1
    uint32_t warp_count[2] = {0u, 0u};
    // unrolled by two, so that the buffer of each copy (q & 1) is a
    // compile-time constant
#pragma unroll 2
    for (int q = 0; q < n_in; ++q) {
        const int buf = q & 1;
        // x-sums of plane p = z0 - 1 + q (in v[buf]) into sx[buf]
#pragma unroll
        for (int k = 0; k < kSumsPerThread; ++k) {
            if (k * kThreads + kThreads <= kSums || tid + k * kThreads < kSums) {
                const float *vp = &v[buf][vsrc[k]];
                sx[buf][tid + k * kThreads] = (vp[0] + vp[1]) + vp[2];
            }
        }
        // plane p + 1 into the other buffer, plane p + 2 in flight
        if (q + 1 < n_in) store_plane(buf ^ 1, cur);
        if (q + 2 < n_in) load_plane(z0 + 1 + q, nxt);
        __syncthreads();
        // y-sums of this thread's two columns; z-sums of plane p - 1
        const int t = q - 2, gz = z0 + t;
        const int cz = 1 + (gz > 0) + (gz + 1 < nz);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float *sp = &sx[buf][tid + 256 * h];
            const float yc = (sp[0] + sp[kSX]) + sp[2 * kSX];
            if (q >= 2) {
                const bool valid = in_xy[h] && gz < nz;
                const float sum = (ya[h] + yb[h]) + yc;
                const float sm = sum * (cz == 3 ? inv3[h] : cz == 2 ? inv2[h] : inv1[h]);
                if (valid && out) __stcs(out + (col[h] + (uint32_t)gz * nxy), sm);
                const uint32_t b = __ballot_sync(0xFFFFFFFFu, valid && sm > a.threshold);
                if (lx == 0) s_bal[t][h][ly] = b;
                warp_count[h] += __popc(b);
            }
            ya[h] = yb[h];
            yb[h] = yc;
        }
#pragma unroll
        for (int k = 0; k < kPerThread; ++k) cur[k] = nxt[k];
    }

    // compaction of the CTA's voxels above the threshold: one atomicAdd
    if (lx == 0) {
        s_off[0][ly] = warp_count[0];
        s_off[1][ly] = warp_count[1];
    }
    __syncthreads();
    if (tid == 0) {
        uint32_t total = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                const uint32_t c = s_off[h][w];
                s_off[h][w] = total;
                total += c;
            }
        uint32_t base = 0;
        if (total) {
            base = atomicAdd(a.counts + f, total);
            if ((uint64_t)base + total > (uint64_t)a.capacity) atomicOr(a.status, kStatusCapacity);
        }
        s_base = base;
    }
    __syncthreads();
    uint32_t *list = a.lists + (size_t)f * a.capacity;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (!warp_count[h]) continue;
        uint32_t pos = s_base + s_off[h][ly];
#pragma unroll 4
        for (int t = 0; t < n_in - 2; ++t) {
            const uint32_t b = s_bal[t][h][ly];
            if ((b >> lx) & 1u) {
                const uint32_t pp = pos + __popc(b & ((1u << lx) - 1u));
                if (pp < a.capacity)
                    list[pp] = (uint32_t)gx + (uint32_t)nx * ((uint32_t)gy[h] + (uint32_t)ny * (uint32_t)(z0 + t));
            }
            pos += __popc(b);
        }
    }
}

// ---------------------------------------------------------------------------
// Tensor-box variant (rows of 16-byte multiples)
// ---------------------------------------------------------------------------
constexpr int kTX = 128, kTRows = 4, kTWarps = 4;   // columns per CTA, rows per warp, computing warps
constexpr int kTY = kTRows * kTWarps, kTZ = 32;     // rows per CTA, most planes per CTA
constexpr int kBoxX = kTX + 8, kBoxY = kTY + 2;     // plane box: columns x0 - 4 .. x0 + 131, rows y0 - 1 .. y0 + 16
constexpr int kBoxFloats = kBoxX * kBoxY;           // 2448
constexpr int kBoxStride = (kBoxFloats + 31) / 32 * 32;   // floats per stage, a multiple of 128 bytes
constexpr int kTStages = 4;                         // 38 KB per CTA, four CTAs per SM: 154 KB in flight
constexpr int kTThreads = 32 * (kTWarps + 1);       // and one warp that issues the boxes

// One box of a 4-D tensor map (x, y, z, frame), global -> shared, completion
// counted on `bar`; x a multiple of 4 floats, elements outside the tensor
// read as zero.
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *tmap, int x, int y, int z, int w,
                                            uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];\n" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
        : "memory");
}

// A CTA owns 128 (x) x 16 (y) columns over `tz` planes (z) of one frame; warp
// w < 4 the rows y0 + 4 w .. + 3, lane l the columns x0 + 4 l .. + 3, so a
// thread holds 4 x 4 outputs per plane.  Each plane with its halo (columns x0
// - 4 .. x0 + 131, rows y0 - 1 .. y0 + 16; zeros outside the grid) arrives as
// one tensor box (TMA) through a 4-stage ring of full / empty mbarriers: warp
// 4 issues, the computing warps wait for a stage, read their six rows of it
// and release it, and never wait for each other.
//
// Per row one 16-byte shared-memory read gives four columns and two shuffles
// their neighbours; six rows of x-sums serve four rows of y-sums (two adds of
// column pairs per instruction); the z-sum comes from the running sum of the
// last two planes' y-sums: ((x-sums) y-sums) z-sums and the scaling by the
// FP32 reciprocal of the clipped count, as in smooth_kernel, so the same
// bits.  Few voxels lie above the threshold (1-3 % of a grid), so a warp only
// looks for them (ballots into s_bal) in the planes whose largest value is
// above it, and the compaction (one atomicAdd per warp) visits these planes.
//
// 100 frames of 128^3 (8.4 MB in, 8.4 MB out each) take 312 us with the list,
// 5.4 TB/s, 79 % of the copy rate.  Fewer frames reach less of it: 32 (1024 CTAs,
// 1.7 waves of the 608 that are resident) 3.9 TB/s, DRAM at 46 %, 28 % of the issue
// slots and 22 % of the warps active (ncu): the last wave, and the loads that each
// thread waits for.  Before (one row of four columns per thread, three rows of
// x-sums per output row, a CTA barrier per plane, every plane's ballots kept and
// walked again): 479 us, 82 % of the issue slots.
__global__ void __launch_bounds__(kTThreads, 4) smooth_tma_kernel(const __grid_constant__ SmoothArgs a, int tiles_x,
                                                                  int tiles_y, int tz)
{
    __shared__ __align__(128) float box[kTStages][kBoxStride];   // stages start 128-byte aligned
    __shared__ uint32_t s_bal[kTZ][kTY][4];   // ballot per output plane, row and quad position
    __shared__ __align__(8) uint64_t full[kTStages], empty[kTStages];

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int f = blockIdx.y;
    const int t = blockIdx.x;
    const int tx = t % tiles_x, ty = (t / tiles_x) % tiles_y, tzi = t / (tiles_x * tiles_y);
    const int x0 = tx * kTX, y0 = ty * kTY, z0 = tzi * tz;
    const int nx = a.nx, ny = a.ny, nz = a.nz;
    const int n_planes = min(tz, nz - z0) + 2;                               // z0 - 1 .. the plane after the last
    const int n_warps = min(kTWarps, (ny - y0 + kTRows - 1) / kTRows);       // warps with rows in the grid
    if (threadIdx.x == 0) {
        for (int s = 0; s < kTStages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], (uint32_t)n_warps);
        }
        mbar_fence_init();
    }
    __syncthreads();
    if (w == kTWarps) {
        if (lane == 0) {
            for (int q = 0; q < n_planes; ++q) {
                const int s = q % kTStages;
                if (q >= kTStages && !mbar_wait_bounded(&empty[s], (uint32_t)((q / kTStages - 1) & 1), a.status)) break;
                mbar_arrive_expect_tx(&full[s], (uint32_t)(kBoxFloats * 4));
                tma_load_4d(box[s], &a.tmap, x0 - 4, y0 - 1, z0 - 1 + q, f, &full[s]);
            }
        }
        return;   // every box that was issued is waited for by the computing warps
    }
    if (w >= n_warps) return;

    const uint32_t nxy = (uint32_t)nx * (uint32_t)ny, n_vox = nxy * (uint32_t)nz;
    float *out = a.smoothed ? a.smoothed + (size_t)f * n_vox : nullptr;
    const bool vec_out = (reinterpret_cast<uintptr_t>(a.smoothed) & 15u) == 0;
    const int x = x0 + 4 * lane, y = y0 + kTRows * w;
    const bool in_x = x < nx;   // nx % 4 == 0: then all four columns are
    const bool rows_inner = y > 0 && y + kTRows < ny;
    // clipped counts along x and the reciprocals of the whole counts where y and z are not clipped
    int cx[4];
    float2 inv[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) cx[k] = 1 + (x + k > 0) + (x + k + 1 < nx);
    inv[0] = make_float2(1.0f / (float)(9 * cx[0]), 1.0f / (float)(9 * cx[1]));
    inv[1] = make_float2(1.0f / (float)(9 * cx[2]), 1.0f / (float)(9 * cx[3]));
    // the halo column of the first and the last lane: box columns 3 and 132
    const int edge_off = lane == 0 ? 3 : kTX + 4;
    const bool edge_lane = lane == 0 || lane == 31;

    float2 yp[kTRows][2], s2[kTRows][2];   // y-sums of plane p - 1; their sum with those of plane p - 2
#pragma unroll
    for (int r = 0; r < kTRows; ++r)
#pragma unroll
        for (int h = 0; h < 2; ++h) yp[r][h] = s2[r][h] = make_float2(0.0f, 0.0f);
    uint32_t warp_count = 0, hit_planes = 0;
    bool arriving = true;   // false after a timed-out wait: the status word marks the result invalid
#pragma unroll 1
    for (int q = 0; q < n_planes; ++q) {
        const int s = q % kTStages;
        if (arriving) arriving = mbar_wait_bounded(&full[s], (uint32_t)((q / kTStages) & 1), a.status);
        const float *rows = box[s] + kTRows * w * kBoxX;
        float2 xs[kTRows + 2][2];   // x-sums of rows y - 1 .. y + 4 of plane p = z0 - 1 + q
#pragma unroll
        for (int r = 0; r < kTRows + 2; ++r) {
            const float4 v = *reinterpret_cast<const float4 *>(rows + r * kBoxX + 4 + 4 * lane);
            float left = __shfl_up_sync(0xFFFFFFFFu, v.w, 1), right = __shfl_down_sync(0xFFFFFFFFu, v.x, 1);
            if (edge_lane) {
                const float e = rows[r * kBoxX + edge_off];
                left = lane == 0 ? e : left;
                right = lane == 0 ? right : e;
            }
            xs[r][0] = make_float2((left + v.x) + v.y, (v.x + v.y) + v.z);
            xs[r][1] = make_float2((v.y + v.z) + v.w, (v.z + v.w) + right);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
        const int tq = q - 2, gz = z0 + tq;   // the output plane p - 1
        float2 sm[kTRows][2];
#pragma unroll
        for (int r = 0; r < kTRows; ++r)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 yc = __fadd2_rn(__fadd2_rn(xs[r][h], xs[r + 1][h]), xs[r + 2][h]);
                sm[r][h] = __fadd2_rn(s2[r][h], yc);
                s2[r][h] = __fadd2_rn(yp[r][h], yc);
                yp[r][h] = yc;
            }
        if (q < 2) continue;
        if (rows_inner && gz > 0 && gz + 1 < nz) {
#pragma unroll
            for (int r = 0; r < kTRows; ++r)
#pragma unroll
                for (int h = 0; h < 2; ++h) sm[r][h] = __fmul2_rn(sm[r][h], inv[h]);
        } else {
            const int cz = 1 + (gz > 0) + (gz + 1 < nz);
#pragma unroll
            for (int r = 0; r < kTRows; ++r) {
                const int cyz = cz * (1 + (y + r > 0) + (y + r + 1 < ny));
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    sm[r][h] = __fmul2_rn(sm[r][h], make_float2(1.0f / (float)(cx[2 * h] * cyz),
                                                                1.0f / (float)(cx[2 * h + 1] * cyz)));
            }
        }
        if (out && in_x) {
            float *o = out + ((uint32_t)gz * nxy + (uint32_t)y * (uint32_t)nx + (uint32_t)x);
#pragma unroll
            for (int r = 0; r < kTRows; ++r) {
                if (y + r >= ny) break;
                if (vec_out) {
                    __stcs(reinterpret_cast<float4 *>(o), make_float4(sm[r][0].x, sm[r][0].y, sm[r][1].x, sm[r][1].y));
                } else {
                    __stcs(o, sm[r][0].x);
                    __stcs(o + 1, sm[r][0].y);
                    __stcs(o + 2, sm[r][1].x);
                    __stcs(o + 3, sm[r][1].y);
                }
                o += nx;
            }
        }
        float top = -INFINITY;
#pragma unroll
        for (int r = 0; r < kTRows; ++r)
#pragma unroll
            for (int h = 0; h < 2; ++h) top = fmaxf(top, fmaxf(sm[r][h].x, sm[r][h].y));
        if (__any_sync(0xFFFFFFFFu, top > a.threshold)) {
            hit_planes |= 1u << tq;
#pragma unroll
            for (int r = 0; r < kTRows; ++r) {
                const bool ok = in_x && y + r < ny;
                uint32_t b[4];
                b[0] = __ballot_sync(0xFFFFFFFFu, ok && sm[r][0].x > a.threshold);
                b[1] = __ballot_sync(0xFFFFFFFFu, ok && sm[r][0].y > a.threshold);
                b[2] = __ballot_sync(0xFFFFFFFFu, ok && sm[r][1].x > a.threshold);
                b[3] = __ballot_sync(0xFFFFFFFFu, ok && sm[r][1].y > a.threshold);
                warp_count += __popc(b[0]) + __popc(b[1]) + __popc(b[2]) + __popc(b[3]);
                if (lane < 4)
                    s_bal[tq][kTRows * w + r][lane] = lane == 0 ? b[0] : lane == 1 ? b[1] : lane == 2 ? b[2] : b[3];
            }
        }
    }

    // compaction of the warp's voxels above the threshold: one atomicAdd
    if (!warp_count) return;
    uint32_t pos = 0;
    if (lane == 0) {
        pos = atomicAdd(a.counts + f, warp_count);
        if ((uint64_t)pos + warp_count > (uint64_t)a.capacity) atomicOr(a.status, kStatusCapacity);
    }
    pos = __shfl_sync(0xFFFFFFFFu, pos, 0);   // also orders s_bal's writes before the reads below
    __syncwarp();
    uint32_t *list = a.lists + (size_t)f * a.capacity;
    const uint32_t lt_mask = (1u << lane) - 1u;
    for (; hit_planes; hit_planes &= hit_planes - 1u) {
        const int tq = __ffs(hit_planes) - 1;
        for (int r = 0; r < kTRows; ++r) {
            const uint32_t lin = (uint32_t)x + (uint32_t)nx * ((uint32_t)(y + r) + (uint32_t)ny * (uint32_t)(z0 + tq));
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t b = s_bal[tq][kTRows * w + r][k];
                if ((b >> lane) & 1u) {
                    const uint32_t pp = pos + __popc(b & lt_mask);
                    if (pp < a.capacity) list[pp] = lin + (uint32_t)k;
                }
                pos += __popc(b);
            }
        }
    }
}

}  // namespace

// Planes per CTA of smooth_kernel, 8 to 32: a CTA walks its planes one after
// the other, so a call of at most a few waves takes about waves x (planes +
// 2) steps; the count that makes that least (32 for larger calls, where the
// two extra planes per CTA are what counts): 9 frames of 93 x 110 x 77, 20
// planes instead of 32, 33.2 -> 24.9 us.
static int best_planes(int nz, int64_t columns, int64_t slots)
{
    int best = kSZ;
    int64_t best_cost = INT64_MAX;
    for (int p = kSZ; p >= 8; --p) {
        const int64_t ctas = columns * ((nz + p - 1) / p), waves = (ctas + slots - 1) / slots;
        if (p == kSZ && waves > 4) return kSZ;
        if (waves * (p + 2) < best_cost) {
            best_cost = waves * (p + 2);
            best = p;
        }
    }
    return best;
}

cudaError_t launch_smooth(const SmoothArgs &a_in, int n_frames, cudaStream_t s)
{
    if (n_frames <= 0) return cudaSuccess;
    cudaError_t e = cudaMemsetAsync(a_in.counts, 0, (size_t)n_frames * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    // rows of 16-byte multiples: the tensor-box kernel
    SmoothArgs a = a_in;
    // planes per CTA: the most that still give four CTAs per SM (a few frames
    // of a small grid would leave SMs idle; each halving re-reads two planes
    // per tile more)
    const int64_t ttx = (a.nx + kTX - 1) / kTX, tty = (a.ny + kTY - 1) / kTY;
    int planes = kTZ;
    while (planes > 8 && ttx * tty * ((a.nz + planes - 1) / planes) * n_frames < 4 * (int64_t)device_sm_count()) planes /= 2;
    const int64_t ttz = (a.nz + planes - 1) / planes;
    if (n_frames <= 65535 && ttx * tty * ttz <= INT_MAX &&
        encode_grid_tensor(a.prob, a.nx, a.ny, a.nz, n_frames, kBoxX, kBoxY, &a.tmap)) {
        smooth_tma_kernel<<<dim3((unsigned)(ttx * tty * ttz), (unsigned)n_frames), kTThreads, 0, s>>>(
            a, (int)ttx, (int)tty, planes);
        return cudaGetLastError();
    }
    const int tx = (a.nx + kSX - 1) / kSX, ty = (a.ny + kSY - 1) / kSY;
    if ((int64_t)((a.nz + kSZ - 1) / kSZ) * n_frames > 65535) return cudaErrorInvalidValue;
    int p = best_planes(a.nz, (int64_t)tx * ty * n_frames, kSCtas * (int64_t)std::max(device_sm_count(), 1));
    if ((int64_t)((a.nz + p - 1) / p) * n_frames > 65535) p = kSZ;   // grid.z
    const int tz = (a.nz + p - 1) / p;
    smooth_kernel<<<dim3(tx, ty, tz * n_frames), kThreads, 0, s>>>(a, tz, p);
    return cudaGetLastError();
}

}  // namespace psfs
