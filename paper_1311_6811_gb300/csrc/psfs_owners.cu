// psfs_owners.cu -- owner lists and the pixel pass of the adjoint.
//
// The adjoint of the fusion (Eq. 3-4 summed in log space) sends dLoss/dL of
// every voxel back to the one pixel per camera that the voxel's centre
// projects into (Eq. 3):  dLoss/dg_kp = sum over voxels v with pix_k(v) = p
// of dLoss/dL_v.  Which voxels a pixel owns depends on the grid and the rig
// only, so it is worked out once per handle, with the forward's own float32
// projection (project_voxel, the same helper and the same arithmetic as the
// fusion kernels, so the ownership is the forward's bit for bit):
//
//   count  one thread per voxel, per camera the pixel it falls in, an integer
//          atomicAdd on that pixel's count;
//   scan   exclusive prefix sum of the counts: the offsets of each pixel's
//          segment (a two-level block scan);
//   fill   the same projection again; each voxel claims a slot of its
//          pixel's segment (integer atomics, so the order is arbitrary);
//   sort   one warp per slice of 32 consecutive pixels sorts each pixel's
//          segment by voxel index and lays the slice out for the pixel pass
//          (see kSliceMax).
//
// The pixel pass of every frame then owns one pixel per thread and adds the
// dLoss/dL of its segment's voxels in ascending voxel order: no float
// atomics, the same order on every run and in every form (one frame per call
// or eight frames per pass), so the gradients are deterministic and the
// batched pass is bit-identical to one frame per call.  The work is one load
// per (voxel, camera) pair, instead of a walk along each pixel's ray.
#include <algorithm>

#include "psfs_fuse_common.cuh"

namespace psfs {

namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanChunk = kScanThreads * kScanItems;   // entries per block of the first level
constexpr int kScanTopItems = 64;                       // second level: one block, 64 sums per thread

// Voxel v's centre in the centred index coordinates of the fusion kernels.
__device__ __forceinline__ void voxel_coords(const FuseArgs &a, uint64_t v, float &fi, float &fj, float &fk)
{
    const uint64_t nxy = (uint64_t)a.nx * (uint64_t)a.ny;
    const uint32_t k = (uint32_t)(v / nxy);
    const uint32_t r = (uint32_t)(v - (uint64_t)k * nxy);
    const uint32_t j = r / (uint32_t)a.nx;
    const uint32_t i = r - j * (uint32_t)a.nx;
    fi = (float)i - a.ci;
    fj = (float)j - a.cj;
    fk = (float)k - a.ck;
}

__global__ void __launch_bounds__(256) owner_count_kernel(const __grid_constant__ FuseArgs a, uint32_t *cnt)
{
    const uint64_t n_vox = (uint64_t)a.nx * a.ny * a.nz;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_vox; v += stride) {
        float fi, fj, fk;
        voxel_coords(a, v, fi, fj, fk);
        for (int c = 0; c < a.n_cams; ++c) {
            int pix;
            if (project_voxel(a.cam[c].m, fi, fj, fk, (uint32_t)a.W, (uint32_t)a.H, &pix))
                atomicAdd(cnt + (int64_t)c * a.map_stride + pix, 1u);
        }
    }
}

__global__ void __launch_bounds__(256) owner_fill_kernel(const __grid_constant__ FuseArgs a, const uint32_t *off,
                                                         uint32_t *cursor, uint32_t *vox)
{
    const uint64_t n_vox = (uint64_t)a.nx * a.ny * a.nz;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t v = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_vox; v += stride) {
        float fi, fj, fk;
        voxel_coords(a, v, fi, fj, fk);
        for (int c = 0; c < a.n_cams; ++c) {
            int pix;
            if (project_voxel(a.cam[c].m, fi, fj, fk, (uint32_t)a.W, (uint32_t)a.H, &pix)) {
                const int64_t p = (int64_t)c * a.map_stride + pix;
                const uint32_t e = off[p] + atomicAdd(cursor + p, 1u);
                if (e < off[p + 1]) vox[e] = (uint32_t)v;   // the count pass made room: e is always inside
            }
        }
    }
}

// Layout of the lists.  A slice is 32 consecutive pixels, one lane of a warp
// each; its entries lie at vox[off[32 s] .. off[32 s + 32)).  In a slice of at
// most kSliceMax entries they are jagged rows: first the first voxel of every
// pixel that has one, in lane order, then the second voxels, and so on.  The
// lanes of a warp that walk their lists together then read consecutive
// entries: one or two lines per step, where a pixel's entries side by side
// spread a step over eleven lines (11 voxels per pixel on average), which
// took as many L1 wavefronts as the gathers they serve.  Nothing is padded.
// Larger slices (more than 128 voxels per pixel: images much coarser than the
// grid) keep each pixel's entries side by side at vox[off[p] .. off[p + 1]).
constexpr uint32_t kSliceMax = 4096;
constexpr uint32_t kSortBytes = 32768;   // shared memory of a sorting CTA
constexpr uint32_t kLaneSortMax = 16;    // longest segment that one lane sorts

// Sorts the n <= 32 K distinct entries at seg in place, one warp: every entry's
// rank is the number of smaller ones.
template <int K>
__device__ __forceinline__ void rank_sort(uint32_t *seg, uint32_t n, int lane)
{
    uint32_t v[K], r[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t i = 32 * k + lane;
        v[k] = i < n ? seg[i] : 0u;
        r[k] = 0;
    }
#pragma unroll 4
    for (uint32_t q = 0; q < n; ++q) {
        const uint32_t x = seg[q];
#pragma unroll
        for (int k = 0; k < K; ++k) r[k] += x < v[k] ? 1u : 0u;
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (32u * k + lane < n) seg[r[k]] = v[k];
    __syncwarp();
}

// Sorts the n entries at seg in place with a bitonic network, a warp or (kCta)
// the whole CTA.  All comparators point upwards (each merge starts with mirrored
// pairs), so that n need not be a power of two: entries past the end would be
// the largest and never move.
template <bool kCta>
__device__ __forceinline__ void bitonic_sort(uint32_t *seg, uint32_t n)
{
    const uint32_t first = kCta ? threadIdx.x : threadIdx.x & 31, threads = kCta ? blockDim.x : 32;
    for (uint32_t k = 2; (k >> 1) < n; k <<= 1) {
        for (uint32_t s = k >> 1; s; s >>= 1) {
            const bool mirror = s == k >> 1;
            const uint32_t pairs = (n + 2 * s - 1) / (2 * s) * s;
            for (uint32_t t = first; t < pairs; t += threads) {
                const uint32_t i = 2 * (t & ~(s - 1)) + (t & (s - 1));
                const uint32_t j = mirror ? (i | (s - 1)) + s - (t & (s - 1)) : i + s;
                if (j < n) {
                    const uint32_t x = seg[i], y = seg[j];
                    if (x > y) {
                        seg[i] = y;
                        seg[j] = x;
                    }
                }
            }
            if (kCta)
                __syncthreads();
            else
                __syncwarp();
        }
    }
}

// Sorts the n distinct entries at seg in place, one warp.
__device__ void warp_sort(uint32_t *seg, uint32_t n, int lane)
{
    if (n <= 32)
        rank_sort<1>(seg, n, lane);
    else if (n <= 64)
        rank_sort<2>(seg, n, lane);
    else if (n <= 128)
        rank_sort<4>(seg, n, lane);
    else
        bitonic_sort<false>(seg, n);
}

// Sorts each pixel's segment by voxel index and writes the jagged layout, one
// warp per slice of kMin + 1 to kMax entries (small buffers, and many warps per
// SM, for the usual slices); once per handle.  Short segments are sorted by
// their lane (insertion), longer ones by the whole warp.  With insertion alone,
// n^2 / 4 dependent steps, the first adjoint call for 128^3 voxels and 8 cameras
// of 160 x 120 (109 voxels per pixel) took 10.8 ms, of 80 x 60 116 ms; 1.1 and
// 1.6 ms with this (of 640 x 480 0.92 and 0.72).
template <uint32_t kMin, uint32_t kMax>
__global__ void __launch_bounds__(kSortBytes / kMax * 8) owner_sort_kernel(const uint32_t *off, uint32_t *vox,
                                                                           int64_t n_pix)
{
    constexpr int kWarps = kSortBytes / (4 * kMax);
    __shared__ uint32_t s_seg[kWarps][kMax];
    const int lane = threadIdx.x & 31;
    uint32_t *buf = s_seg[threadIdx.x >> 5];
    const int64_t n_slices = (n_pix + 31) / 32, stride = (int64_t)gridDim.x * kWarps;
    const uint32_t lt_mask = (1u << lane) - 1u;
    for (int64_t sl = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5); sl < n_slices; sl += stride) {
        const uint32_t e0 = off[min(32 * sl + lane, n_pix)], e1 = off[min(32 * sl + lane + 1, n_pix)];
        const uint32_t base = __shfl_sync(0xFFFFFFFFu, e0, 0), end = __shfl_sync(0xFFFFFFFFu, e1, 31);
        const uint32_t b0 = e0 - base, n = e1 - e0;
        if (end - base > kMin && end - base <= kMax) {
            for (uint32_t e = lane; e < end - base; e += 32) buf[e] = vox[base + e];
            __syncwarp();
            for (uint32_t e = b0 + 1; n <= kLaneSortMax && e < b0 + n; ++e) {
                const uint32_t x = buf[e];
                uint32_t q = e;
                while (q > b0 && buf[q - 1] > x) {
                    buf[q] = buf[q - 1];
                    --q;
                }
                buf[q] = x;
            }
            __syncwarp();
            for (uint32_t todo = __ballot_sync(0xFFFFFFFFu, n > kLaneSortMax); todo; todo &= todo - 1u) {
                const int l = __ffs(todo) - 1;
                warp_sort(buf + __shfl_sync(0xFFFFFFFFu, b0, l), __shfl_sync(0xFFFFFFFFu, n, l), lane);
            }
            uint32_t pos = base;
            for (uint32_t j = 0; __any_sync(0xFFFFFFFFu, j < n); ++j) {
                const uint32_t has = __ballot_sync(0xFFFFFFFFu, j < n);
                if (j < n) vox[pos + __popc(has & lt_mask)] = buf[b0 + j];
                pos += __popc(has);
            }
            __syncwarp();   // the buffer is reused by the next slice
        }
    }
}

// The segments of slices of more than kSliceMax entries, a CTA per slice: its
// warps a pixel each, those that do not fit a warp's buffer by the whole CTA, and
// in place those that do not fit the CTA's.  A CTA looks at 256 slices at a time, one per thread: few images have any.
constexpr int kLongThreads = 256;

__global__ void __launch_bounds__(kLongThreads) owner_sort_long_kernel(const uint32_t *off, uint32_t *vox, int64_t n_pix)
{
    constexpr uint32_t kWarps = kLongThreads / 32, kMax = kSortBytes / (4 * kWarps);
    __shared__ uint32_t s_seg[kWarps * kMax];
    __shared__ uint32_t s_long[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *buf = s_seg + warp * kMax;
    const int64_t n_slices = (n_pix + 31) / 32;
    for (int64_t sl0 = blockIdx.x; sl0 < n_slices; sl0 += (int64_t)kLongThreads * gridDim.x) {
        const int64_t first = 32 * (sl0 + (int64_t)threadIdx.x * gridDim.x);
        const uint32_t lanes =
            __ballot_sync(0xFFFFFFFFu, first < n_pix && off[min(first + 32, n_pix)] - off[min(first, n_pix)] > kSliceMax);
        if (lane == 0) s_long[warp] = lanes;
        __syncthreads();
        for (uint32_t w = 0; w < kWarps; ++w) {
            for (uint32_t todo = s_long[w]; todo; todo &= todo - 1u) {
                const int64_t p0 = 32 * (sl0 + (int64_t)(32 * w + __ffs(todo) - 1) * gridDim.x);
                for (int64_t p = p0 + warp; p < min(p0 + 32, n_pix); p += kWarps) {
                    uint32_t *seg = vox + off[p];
                    const uint32_t n = off[p + 1] - off[p];
                    if (n > kMax) continue;
                    for (uint32_t e = lane; e < n; e += 32) buf[e] = seg[e];
                    __syncwarp();
                    warp_sort(buf, n, lane);
                    for (uint32_t e = lane; e < n; e += 32) seg[e] = buf[e];
                    __syncwarp();
                }
                for (int64_t p = p0; p < min(p0 + 32, n_pix); ++p) {
                    uint32_t *seg = vox + off[p];
                    const uint32_t n = off[p + 1] - off[p];
                    if (n <= kMax) continue;
                    uint32_t *at = n <= kWarps * kMax ? s_seg : seg;
                    __syncthreads();   // the warps' buffers, or the last pixel's, are done with
                    for (uint32_t e = threadIdx.x; at != seg && e < n; e += kLongThreads) at[e] = seg[e];
                    __syncthreads();
                    bitonic_sort<true>(at, n);
                    for (uint32_t e = threadIdx.x; at != seg && e < n; e += kLongThreads) seg[e] = at[e];
                }
                __syncthreads();
            }
        }
        __syncthreads();
    }
}

// One lane's walk along its pixel's list, K voxels per step, in ascending
// voxel order; every lane of the warp walks with it (step needs them all).
template <int K>
struct OwnerWalk {
    const uint32_t *next;   // jagged: the warp's next row; otherwise the lane's next entry
    uint32_t left;          // entries of the lane not yet fetched
    bool jagged;
#ifdef PSFS_BOUNDS_CHECK
    const uint32_t *lists;   // and the slice's entries of them
    uint32_t slice0, slice1;
    uint32_t *status;
#endif

    // The segment e0 .. e1 - 1 of this lane's pixel; `total` entries in all
    // lists.  `left` is then the segment's length (0 in the bounds-checked build
    // where it does not lie in the lists).
    __device__ __forceinline__ void init(const uint32_t *vox, uint32_t e0, uint32_t e1, const uint32_t *total,
                                         uint32_t *status_word)
    {
        const uint32_t base = __shfl_sync(0xFFFFFFFFu, e0, 0), end = __shfl_sync(0xFFFFFFFFu, e1, 31);
        jagged = end - base <= kSliceMax;
        next = vox + (jagged ? base : e0);
        left = e1 - e0;
        (void)total;
        (void)status_word;
#ifdef PSFS_BOUNDS_CHECK
        lists = vox;
        slice0 = base;
        slice1 = end;
        status = status_word;
        if (!PSFS_IN_BOUNDS(owner_segment_ok(e0, e1, base, end, __ldg(total)), status)) left = 0;
#endif
    }
    // Whether entry q may be read.
    __device__ __forceinline__ bool readable(const uint32_t *q) const
    {
        (void)q;
        return PSFS_IN_BOUNDS(owner_entry_ok(q, lists, slice0, slice1), status);
    }
    // The next K voxels: v[k] for the first min(K, left) of them.
    __device__ __forceinline__ void step(uint32_t (&v)[K])
    {
        const uint32_t lt_mask = (1u << (threadIdx.x & 31)) - 1u;
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const bool has = (uint32_t)k < left;
            const uint32_t lanes = __ballot_sync(0xFFFFFFFFu, has);
            const uint32_t *q = next + (jagged ? __popc(lanes & lt_mask) : 0);
            v[k] = has && readable(q) ? __ldg(q) : 0u;
            next += jagged ? __popc(lanes) : 1;
        }
        left = left > (uint32_t)K ? left - (uint32_t)K : 0u;
    }
};

// Exclusive scan of one block's kScanThreads values in registers.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t *s_warp, uint32_t *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, d);
        if (lane >= d) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        const uint32_t w = lane < (kScanThreads / 32) ? s_warp[lane] : 0u;
        uint32_t winc = w;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, winc, d);
            if (lane >= d) winc += y;
        }
        s_warp[lane] = winc - w;   // exclusive prefix of each warp
        if (lane == 31) *total = winc;
    }
    __syncthreads();
    return s_warp[warp] + inc - x;
}

// First level: out[i] = sum of in[chunk start .. i) for i < n_in, in[i >= n_in]
// read as 0; the chunk's total goes to sums[blockIdx.x].  n_out entries.
__global__ void __launch_bounds__(kScanThreads) scan_chunks_kernel(const uint32_t *in, int64_t n_in, uint32_t *out,
                                                                   int64_t n_out, uint32_t *sums)
{
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_total;
    const int64_t base = (int64_t)blockIdx.x * kScanChunk + (int64_t)threadIdx.x * kScanItems;
    uint32_t v[kScanItems];
    uint32_t t = 0;
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        v[q] = base + q < n_in ? in[base + q] : 0u;
        t += v[q];
    }
    uint32_t run = block_exclusive_scan(t, s_warp, &s_total);
#pragma unroll
    for (int q = 0; q < kScanItems; ++q) {
        if (base + q < n_out) out[base + q] = run;
        run += v[q];
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = s_total;
}

// Second level, one block: exclusive scan of the chunk totals in place.
__global__ void __launch_bounds__(kScanThreads) scan_top_kernel(uint32_t *sums, int64_t n)
{
    __shared__ uint32_t s_warp[32];
    __shared__ uint32_t s_total;
    const int64_t base = (int64_t)threadIdx.x * kScanTopItems;
    uint32_t t = 0;
    for (int q = 0; q < kScanTopItems; ++q)
        if (base + q < n) t += sums[base + q];
    uint32_t run = block_exclusive_scan(t, s_warp, &s_total);
    for (int q = 0; q < kScanTopItems; ++q)
        if (base + q < n) {
            const uint32_t x = sums[base + q];
            sums[base + q] = run;
            run += x;
        }
}

__global__ void __launch_bounds__(256) scan_add_kernel(uint32_t *out, int64_t n, const uint32_t *sums)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
        out[i] += sums[i / kScanChunk];
}

// Chain rule of one frame from the pixel's background loaded once (mu, h =
// 1 / (2 var), base = c0 - log(h0 h1 h2) / 2 = pixel_log_base, so that r =
// base + pixel_quad is pixel_log_odds bit for bit):
//   s = sigmoid(r) (the bits of sigmoid_fast), from u = e^-|r|;
//   dLoss/ds = acc (da / a(s) - db / b(s))            (Eq. 5-9, a, b linear in s)
//   dLoss/dr = dLoss/ds s (1 - s), with s (1 - s) = u / (1 + u)^2 (no cancellation)
//   dLoss/dmu_c, dLoss/dvar_c from dLoss/dr (Eq. 1).
__device__ __forceinline__ void chain_rule_pre(const BackwardArgs &b, const float (&im)[3], const float (&mu)[3],
                                               const float (&hh)[3], float base, float acc, float &dslm,
                                               float (&dm)[3], float (&dv)[3])
{
    dslm = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) dm[c] = dv[c] = 0.0f;
    if (acc != 0.0f) {
        float dd[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) dd[c] = im[c] - mu[c];
        const float r = base + pixel_quad(im[0], im[1], im[2], mu[0], mu[1], mu[2], hh[0], hh[1], hh[2]);
        const float u = exp_fast(-fabsf(r));
        const float inv = rcp_approx(1.0f + u);
        const float s_val = r > 0.0f ? inv : u * inv;
        const float av = fmaf(b.da, s_val, b.one_minus_pd), bv = fmaf(b.db, s_val, b.one_minus_q);
        dslm = acc * (div_fast(b.da, av) - div_fast(b.db, bv));
        const float dr = dslm * (u * inv * inv);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            dm[c] = -2.0f * dr * dd[c] * hh[c];
            dv[c] = dr * hh[c] * (1.0f - 2.0f * dd[c] * dd[c] * hh[c]);
        }
    }
}

// dLoss/dSLM of pixel p from a caller-supplied SLM (psfs_backward_slm).
__device__ __forceinline__ float chain_rule_slm(const BackwardArgs &b, int64_t p, float acc)
{
    if (acc == 0.0f) return 0.0f;
    const float s_val = __ldg(b.slm + p);
    const float av = fmaf(b.da, s_val, b.one_minus_pd), bv = fmaf(b.db, s_val, b.one_minus_q);
    return acc * (div_fast(b.da, av) - div_fast(b.db, bv));
}

// An owner's index names a voxel of the grid (tested in the bounds-checked
// build only).
__device__ __forceinline__ bool owner_in_grid(const BackwardArgs &b, uint32_t v)
{
    (void)b;
    (void)v;
    return PSFS_IN_BOUNDS(v < (uint64_t)b.f.nx * b.f.ny * b.f.nz, b.f.status);
}

// The warps of the one-frame pixel pass take the slices of eight rows column
// by column (about W / 32 slices make a row): the eight warps of a CTA then
// work on eight rows of the same 32 columns, whose owners lie close together,
// so that more of the 32-byte sectors their dL share (eight voxels along x)
// are still in L1: 63.6 -> 59.6 us per 128^3 x 8 frame.  A permutation of the
// slices, padded to whole groups of eight rows.  The group pass reads whole
// 32-byte records, which no two owners share, and is faster in plain order
// (218 against 238 us per 16 frames).
__device__ __forceinline__ uint32_t slice_of(uint32_t i, uint32_t per_row)
{
    const uint32_t rows = i / (8u * per_row), in = i - rows * (8u * per_row);
    return (rows * 8u + (in & 7u)) * per_row + (in >> 3);
}

// One frame: pixel p sums b.dl over its list in ascending voxel order, one
// warp per slice.  Four owners' dL are in flight while the next four indices
// load; the adds stay in ascending order.  Its warps wait for the scattered dL
// reads, a 32-byte sector for most owners (ncu: long scoreboard; L1 59 %, issue
// 55 %, DRAM 40 %, 79 % of the warps active): 59.6 us per 128^3 x 8 x 640 x 480 frame
// (16.0 M owners), 67.8 before with each pixel's indices side by side.  Of few
// owners per pixel it is the slices themselves that count: 32-bit arithmetic for
// their order took the whole call on 96^3 voxels (2.9 per pixel) from 52.7 to
// 50.6 us, 49.0 before there were slices.
__global__ void __launch_bounds__(256) owner_pixel_kernel(const __grid_constant__ BackwardArgs b, const uint32_t *off,
                                                          const uint32_t *vox)
{
    // slices fit 32 bits: the offset scan takes at most 2^28 pixels
    const uint32_t per_row = (uint32_t)max(b.f.W / 32, 1), n_slices = (uint32_t)((b.n_pix + 31) / 32);
    const uint32_t n_padded = (n_slices + 8u * per_row - 1u) / (8u * per_row) * (8u * per_row);
    const uint32_t stride = gridDim.x * (blockDim.x / 32);
    for (uint32_t i = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; i < n_padded; i += stride) {
        const uint32_t sl = slice_of(i, per_row);
        if (sl >= n_slices) continue;
        const int64_t p = 32 * (int64_t)sl + (threadIdx.x & 31);
        const uint32_t e0 = __ldg(off + min(p, b.n_pix)), e1 = __ldg(off + min(p + 1, b.n_pix));
        float acc = 0.0f;
        OwnerWalk<4> walk;
        walk.init(vox, e0, e1, off + b.n_pix, b.f.status);
        const uint32_t cnt = walk.left;
        const uint32_t longest = __reduce_max_sync(0xFFFFFFFFu, cnt);
        uint32_t v[4];
        walk.step(v);
        for (uint32_t j = 0; j < longest; j += 4) {
            float d[4];
#pragma unroll
            for (int k = 0; k < 4; ++k)
                d[k] = j + k < cnt && owner_in_grid(b, v[k]) ? __ldg(b.dl + v[k]) : 0.0f;
            walk.step(v);
            // a lane past its list adds +0, which leaves its sum (never -0) as it is
#pragma unroll
            for (int k = 0; k < 4; ++k) acc += d[k];
        }
        if (p >= b.n_pix) continue;
        float dslm, dm[3], dv[3];
        if (b.img) {
            float mu[3] = {0.0f, 0.0f, 0.0f}, hh[3] = {0.0f, 0.0f, 0.0f}, im[3] = {0.0f, 0.0f, 0.0f}, base = 0.0f;
            if (acc != 0.0f) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    im[c] = (float)__ldg(b.img + 3 * p + c);
                    mu[c] = __ldg(b.mean + 3 * p + c);
                    hh[c] = __ldg(b.hinv + 3 * p + c);
                }
                base = pixel_log_base(hh[0], hh[1], hh[2], b.c0);
            }
            chain_rule_pre(b, im, mu, hh, base, acc, dslm, dm, dv);
        } else {
            dslm = chain_rule_slm(b, p, acc);
#pragma unroll
            for (int c = 0; c < 3; ++c) dm[c] = dv[c] = 0.0f;
        }
        if (b.d_slm) b.d_slm[p] = dslm;
        if (b.d_mean)
            for (int c = 0; c < 3; ++c) b.d_mean[3 * p + c] = dm[c];
        if (b.d_var)
            for (int c = 0; c < 3; ++c) b.d_var[3 * p + c] = dv[c];
    }
}

// One voxel's 32-byte record of dLoss/dL (kBwRecord frames) with one 256-bit
// read-only load; zeros, and no load, unless `on`.
__device__ __forceinline__ void load_record(const float *rec, bool on, uint32_t (&w)[8])
{
#pragma unroll
    for (int q = 0; q < 8; ++q) w[q] = 0u;
    asm("{\n .reg .pred p;\n setp.ne.u32 p, %9, 0;\n"
        " @p ld.global.nc.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n}\n"
        : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]), "+r"(w[4]), "+r"(w[5]), "+r"(w[6]), "+r"(w[7])
        : "l"(rec), "r"((uint32_t)on));
}

// Up to R * kBwRecord frames: b.dl holds R planes of records of kBwRecord
// floats per voxel (frame r * kBwRecord + f of voxel v at b.dl[r * n_vox *
// kBwRecord + v * kBwRecord + f]); one 32-byte load per owned voxel and
// plane serves its frames, so the owner list, the background and d_mean /
// d_var are read once per R * kBwRecord frames.  Per frame the sum (same
// voxels, same order) and the chain rule are those of owner_pixel_kernel, so
// d_slm (frame f at b.d_slm + f n_pix) is bit-identical to one frame per
// call; d_mean and d_var receive the frames' gradients added in frame order
// to 0 (or, with `accumulate`, to what they hold).
// Issue slots (66 %) and the record reads (1.0 GB of sectors per 16 frames of
// 128^3 x 8; L2 48 %, 45 % of the warps active) hold it: 214-218 us per 16 frames;
// 305 when each frame's colours were byte loads in that frame's branch, a memory
// latency each.  Four CTAs per SM: 64 registers.
template <int R>
__global__ void __launch_bounds__(256, 4) owner_pixel_group_kernel(const __grid_constant__ BackwardArgs b,
                                                                const uint32_t *off, const uint32_t *vox,
                                                                int n_frames, int64_t img_fstride, int accumulate)
{
    constexpr int kF = R * kBwRecord;
    constexpr int K = 4 / R;   // owners per step: four records in flight
    const size_t plane = (size_t)b.f.nx * b.f.ny * b.f.nz * kBwRecord;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    const int64_t n_lanes = (b.n_pix + 31) / 32 * 32;   // whole warps: a warp walks its slice together
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n_lanes; p += stride) {
        const uint32_t e0 = __ldg(off + min(p, b.n_pix)), e1 = __ldg(off + min(p + 1, b.n_pix));
        OwnerWalk<K> walk;
        walk.init(vox, e0, e1, off + b.n_pix, b.f.status);
        float acc[kF];
#pragma unroll
        for (int f = 0; f < kF; ++f) acc[f] = 0.0f;
        uint32_t v[K];
        const uint32_t cnt = walk.left;
        const uint32_t longest = __reduce_max_sync(0xFFFFFFFFu, cnt);
        walk.step(v);
        for (uint32_t j = 0; j < longest; j += K) {
            uint32_t w[K][R][8];
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const bool on = j + k < cnt && owner_in_grid(b, v[k]);
#pragma unroll
                for (int r = 0; r < R; ++r) load_record(b.dl + r * plane + (size_t)v[k] * kBwRecord, on, w[k][r]);
            }
            walk.step(v);
            // owners in ascending order per frame; a lane past its list adds
            // +0, which leaves its sums (never -0) as they are
#pragma unroll
            for (int k = 0; k < K; ++k)
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int f = 0; f < kBwRecord; ++f) acc[r * kBwRecord + f] += __uint_as_float(w[k][r][f]);
        }
        const bool in_img = p < b.n_pix;
        bool any = false;
#pragma unroll
        for (int f = 0; f < kF; ++f) any |= (f < n_frames) & (acc[f] != 0.0f);
        // every frame's colours of the warp's 32 pixels (96 consecutive bytes,
        // one 4-byte word per lane) and the background in flight together;
        // byte loads inside each frame's branch waited for memory frame by frame
        const bool any_lane = __any_sync(0xFFFFFFFFu, any);
        const int lane = threadIdx.x & 31;
        const int64_t word = (p - lane) * 3 / 4 + lane;
        const bool load_word = any_lane && lane < 24 && 4 * word < 3 * b.n_pix;
        uint32_t iw[kF];
#pragma unroll
        for (int f = 0; f < kF; ++f)
            iw[f] = f < n_frames && load_word
                        ? __ldg(reinterpret_cast<const uint32_t *>(b.img + f * img_fstride) + word) : 0u;
        float mu[3] = {0.0f, 0.0f, 0.0f}, hh[3] = {0.0f, 0.0f, 0.0f}, base = 0.0f;
        if (any) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                mu[c] = __ldg(b.mean + 3 * p + c);
                hh[c] = __ldg(b.hinv + 3 * p + c);
            }
            base = pixel_log_base(hh[0], hh[1], hh[2], b.c0);
        }
        float tm[3] = {0.0f, 0.0f, 0.0f}, tv[3] = {0.0f, 0.0f, 0.0f};
        if (accumulate && in_img) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                if (b.d_mean) tm[c] = b.d_mean[3 * p + c];
                if (b.d_var) tv[c] = b.d_var[3 * p + c];
            }
        }
        const int w0 = 3 * lane / 4, shift = 8 * (3 * lane % 4);
#pragma unroll
        for (int f = 0; f < kF; ++f) {
            if (f < n_frames) {
                float dslm, dm[3], dv[3];
                const uint32_t px = __funnelshift_r(__shfl_sync(0xFFFFFFFFu, iw[f], w0),
                                                    __shfl_sync(0xFFFFFFFFu, iw[f], w0 + 1), shift);
                const float im[3] = {(float)(px & 255u), (float)((px >> 8) & 255u), (float)((px >> 16) & 255u)};
                chain_rule_pre(b, im, mu, hh, base, acc[f], dslm, dm, dv);
                if (b.d_slm && in_img) b.d_slm[f * b.n_pix + p] = dslm;
                // separate round-to-nearest adds: the compiler may not fuse
                // them with the products above, so the sums are those of the
                // per-frame gradients as psfs_backward stores them
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    tm[c] = __fadd_rn(tm[c], dm[c]);
                    tv[c] = __fadd_rn(tv[c], dv[c]);
                }
            }
        }
        if (!in_img) continue;
        if (b.d_mean)
            for (int c = 0; c < 3; ++c) b.d_mean[3 * p + c] = tm[c];
        if (b.d_var)
            for (int c = 0; c < 3; ++c) b.d_var[3 * p + c] = tv[c];
    }
}

// dLoss/dL = d_occ occ (1 - occ) from the forward's own occupancy (the
// expression of the voxel passes, so the same bits as their recomputation):
// n_frames frames of n_vox voxels, frame f's value into slot f of each
// voxel's 8-slot record (slots n_frames .. 7 set to 0; the whole 32-byte
// record in one vector store), or densely (dl_stride 1, one frame).
__global__ void __launch_bounds__(256) dl_from_occ_kernel(const float *occ, const float *d_occ, float *dl,
                                                          int64_t n_vox, int n_frames, int dl_stride)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n_vox; v += stride) {
        if (dl_stride == kBwRecord) {
            float r[kBwRecord];
#pragma unroll
            for (int f = 0; f < kBwRecord; ++f) {
                r[f] = 0.0f;
                if (f < n_frames) {
                    const float o = __ldg(occ + f * n_vox + v);
                    r[f] = __ldg(d_occ + f * n_vox + v) * o * (1.0f - o);
                }
            }
            float4 *rec = reinterpret_cast<float4 *>(dl + v * kBwRecord);
            rec[0] = make_float4(r[0], r[1], r[2], r[3]);
            rec[1] = make_float4(r[4], r[5], r[6], r[7]);
        } else {
            for (int f = 0; f < n_frames; ++f) {
                const float o = __ldg(occ + f * n_vox + v);
                dl[v * dl_stride + f] = __ldg(d_occ + f * n_vox + v) * o * (1.0f - o);
            }
        }
    }
}

int64_t grid_for(int64_t n, int per_sm = 8)
{
    int64_t blocks = (n + 255) / 256;
    const int64_t cap = (int64_t)per_sm * device_sm_count();
    if (blocks > cap) blocks = cap;
    return blocks < 1 ? 1 : blocks;
}

}  // namespace

bool owner_lists_supported(const FuseArgs &a, int64_t n_pix)
{
    const uint64_t pairs = (uint64_t)a.nx * a.ny * a.nz * (uint64_t)a.n_cams;
    const int64_t n_chunks = (n_pix + 1 + kScanChunk - 1) / kScanChunk;
    return pairs < (1ull << 32) && n_chunks <= (int64_t)kScanThreads * kScanTopItems;
}

cudaError_t launch_build_owners(const FuseArgs &a, int64_t n_pix, uint32_t *cnt, uint32_t *sums, uint32_t *off,
                                uint32_t *vox, cudaStream_t s)
{
    if (!owner_lists_supported(a, n_pix)) return cudaErrorInvalidValue;
    const uint64_t n_vox = (uint64_t)a.nx * a.ny * a.nz;
    const int64_t vox_blocks = grid_for((int64_t)n_vox, 16);
    cudaError_t e = cudaMemsetAsync(cnt, 0, (size_t)n_pix * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    owner_count_kernel<<<(int)vox_blocks, 256, 0, s>>>(a, cnt);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // offsets: n_pix + 1 entries, the last one the total
    const int64_t n_chunks = (n_pix + 1 + kScanChunk - 1) / kScanChunk;
    scan_chunks_kernel<<<(int)n_chunks, kScanThreads, 0, s>>>(cnt, n_pix, off, n_pix + 1, sums);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    scan_top_kernel<<<1, kScanThreads, 0, s>>>(sums, n_chunks);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    scan_add_kernel<<<(int)grid_for(n_pix + 1), 256, 0, s>>>(off, n_pix + 1, sums);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    e = cudaMemsetAsync(cnt, 0, (size_t)n_pix * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    owner_fill_kernel<<<(int)vox_blocks, 256, 0, s>>>(a, off, cnt, vox);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int64_t n_slices = (n_pix + 31) / 32, most = 64 * (int64_t)device_sm_count();
    owner_sort_kernel<0, 1024><<<(int)std::min(most, (n_slices + 7) / 8), 256, 0, s>>>(off, vox, n_pix);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    owner_sort_kernel<1024, kSliceMax><<<(int)std::min(most, (n_slices + 1) / 2), 64, 0, s>>>(off, vox, n_pix);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    owner_sort_long_kernel<<<(int)std::min(4 * (int64_t)device_sm_count(), n_slices), kLongThreads, 0, s>>>(off, vox,
                                                                                                            n_pix);
    return cudaGetLastError();
}

cudaError_t launch_dl_from_occ(const float *occ, const float *d_occ, float *dl, int64_t n_vox, int n_frames,
                               int dl_stride, cudaStream_t s)
{
    if (n_frames < 1 || n_frames > dl_stride) return cudaErrorInvalidValue;
    if (dl_stride == kBwRecord && ((uintptr_t)dl & 31u)) return cudaErrorMisalignedAddress;
    dl_from_occ_kernel<<<(int)grid_for(n_vox), 256, 0, s>>>(occ, d_occ, dl, n_vox, n_frames, dl_stride);
    return cudaGetLastError();
}

cudaError_t launch_owner_pixel(const BackwardArgs &b, const uint32_t *off, const uint32_t *vox, cudaStream_t s)
{
    owner_pixel_kernel<<<(int)grid_for(b.n_pix), 256, 0, s>>>(b, off, vox);
    return cudaGetLastError();
}

cudaError_t launch_owner_pixel_group(const BackwardArgs &b, const uint32_t *off, const uint32_t *vox, int n_frames,
                                     int64_t img_fstride, bool accumulate, cudaStream_t s)
{
    // whole 4-byte words of whole frames (the entry points ask for 16 bytes of both)
    if (n_frames < 1 || n_frames > 2 * kBwRecord || !b.img || ((uintptr_t)b.dl & 31u) ||
        (((uintptr_t)b.img | (uintptr_t)img_fstride) & 3u) || (3 * b.n_pix) % 4 != 0)
        return cudaErrorInvalidValue;
    if (n_frames > kBwRecord)
        owner_pixel_group_kernel<2><<<(int)grid_for(b.n_pix), 256, 0, s>>>(b, off, vox, n_frames, img_fstride,
                                                                             accumulate ? 1 : 0);
    else
        owner_pixel_group_kernel<1><<<(int)grid_for(b.n_pix), 256, 0, s>>>(b, off, vox, n_frames, img_fstride,
                                                                             accumulate ? 1 : 0);
    return cudaGetLastError();
}

}  // namespace psfs
