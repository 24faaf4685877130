// psfs_reproject.cu -- silhouettes of the reconstructed voxels in every camera
// (Section 2.3: the projection of the voxels is the tracker's prior knowledge,
// matched against the particles' projected body models; Section 3.3.3,
// "Voxel Projection").  Pixel (x, y) of camera c is set iff the ray from the
// camera centre through the pixel centre meets, in front of the camera, the
// cube of a listed voxel.
//
// A CTA holds one camera's silhouette as a bitmask in shared memory (one bit
// per pixel: 38 KB for 640 x 480), so every voxel of the frame's list sets its
// pixels there, and the finished mask is written out once, as whole bytes,
// zeros included: no memset before and no read-modify-write of the mask.
// Images of more than kRpBandPixels take several CTAs, each a range of pixels;
// when frames x cameras are fewer than the SMs, a cluster of CTAs shares one
// mask, each with every S-th chunk of the list, and each writes one share of
// the OR of the S bitmasks, read through distributed shared memory.  Where that
// still leaves SMs idle, a list that is long (only the GPU knows) is taken by a
// second kernel instead, in as many parts as CTAs are resident: each part's
// pixels are OR-ed into the mask, which the first kernel's clusters then only
// fill with zeros, beside the second kernel's projections (see
// reproject_split).
//
// One thread per listed voxel, with the forward kernels' matrices.  When
// all eight cube corners lie in front of the camera, a centre ray meets the
// cube iff the pixel centre lies in the cube's projection: a convex polygon
// whose vertices are the projections of the cube's silhouette loop (the
// corners between faces turned towards the camera and faces turned away).
// Which corners form that loop, and in which cyclic order, depends only on
// where the camera centre lies relative to the cube's three slabs (below,
// within or above each: 26 cases outside the cube), so a table made once on
// the host gives the 4 or 6 corners to project.  A row of pixel centres
// meets the polygon in one interval whose ends are the row's crossings with
// its edges; the interval's bits are OR-ed into the words that lack them
// (neighbouring surface voxels cover a pixel several times, so most words
// need no atomic).  Cubes not wholly in front of the camera, and projections
// too large for float32 rows, take a float32 slab test of the centre ray of
// every pixel whose centre can fall inside the projection's bounding box; cubes
// wholly behind it are passed over.
// Run on the surface list, the work is proportional to the body's surface;
// the silhouette of a solid equals that of its surface voxels.
#include <algorithm>
#include <climits>
#include <cmath>

#include "psfs_internal.cuh"

namespace psfs {

namespace {

constexpr int kRpSmThreads = 1024;   // of an SM, 64 registers each: one CTA, or two of half, ...
constexpr int kRpMaxCluster = 8;

// Silhouette loops of a unit cube by camera region: entry (rx + 1) + 3 (ry +
// 1) + 9 (rz + 1), r = -1 / 0 / +1 for a camera centre below / within /
// above the slab of that axis; bits 0-3 the corner count n (4 or 6; 0 for
// the cube's interior), then n corners of 3 bits each (corner q = bx + 2 by +
// 4 bz) in cyclic order.
struct SilTable {
    uint32_t e[27];
};

// Projects the unit cube's corners from a point of each region (along each
// axis 3 cube sizes below the lower face, at the centre, or 3 above the
// upper face) along the view towards the cube's centre and keeps the convex
// hull of the projections (Andrew's monotone chain), in order.
SilTable make_sil_table()
{
    SilTable t{};
    const double pos[3] = {-3.0, 0.5, 4.0};
    for (int code = 0; code < 27; ++code) {
        const int r[3] = {code % 3, (code / 3) % 3, code / 9};
        if (r[0] == 1 && r[1] == 1 && r[2] == 1) continue;   // inside the cube
        const double P[3] = {pos[r[0]], pos[r[1]], pos[r[2]]};
        double d[3] = {0.5 - P[0], 0.5 - P[1], 0.5 - P[2]};
        const double dn = std::sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
        for (double &x : d) x /= dn;
        // a basis (e1, e2) of the image plane: e1 = unit(d x a) with a the axis least aligned with d
        int ax = 0;
        for (int k = 1; k < 3; ++k)
            if (std::fabs(d[k]) < std::fabs(d[ax])) ax = k;
        double a[3] = {0.0, 0.0, 0.0};
        a[ax] = 1.0;
        double e1[3] = {d[1] * a[2] - d[2] * a[1], d[2] * a[0] - d[0] * a[2], d[0] * a[1] - d[1] * a[0]};
        const double n1 = std::sqrt(e1[0] * e1[0] + e1[1] * e1[1] + e1[2] * e1[2]);
        for (double &x : e1) x /= n1;
        const double e2[3] = {d[1] * e1[2] - d[2] * e1[1], d[2] * e1[0] - d[0] * e1[2], d[0] * e1[1] - d[1] * e1[0]};
        double px[8], py[8];
        int idx[8];
        for (int q = 0; q < 8; ++q) {
            const double X[3] = {(double)(q & 1) - P[0], (double)((q >> 1) & 1) - P[1], (double)((q >> 2) & 1) - P[2]};
            const double z = X[0] * d[0] + X[1] * d[1] + X[2] * d[2];
            px[q] = (X[0] * e1[0] + X[1] * e1[1] + X[2] * e1[2]) / z;
            py[q] = (X[0] * e2[0] + X[1] * e2[1] + X[2] * e2[2]) / z;
            idx[q] = q;
        }
        std::sort(idx, idx + 8, [&](int i, int j) { return px[i] < px[j] || (px[i] == px[j] && py[i] < py[j]); });
        auto cross = [&](int o, int i, int j) {
            return (px[i] - px[o]) * (py[j] - py[o]) - (py[i] - py[o]) * (px[j] - px[o]);
        };
        int hull[16], k = 0;
        for (int i = 0; i < 8; ++i) {   // lower chain
            while (k >= 2 && cross(hull[k - 2], hull[k - 1], idx[i]) <= 1e-12) --k;
            hull[k++] = idx[i];
        }
        for (int i = 6, lo = k + 1; i >= 0; --i) {   // upper chain
            while (k >= lo && cross(hull[k - 2], hull[k - 1], idx[i]) <= 1e-12) --k;
            hull[k++] = idx[i];
        }
        const int n = k - 1;   // the last point repeats the first
        uint32_t ent = (uint32_t)n;
        for (int i = 0; i < n && i < 6; ++i) ent |= (uint32_t)hull[i] << (4 + 3 * i);
        t.e[code] = n <= 6 ? ent : 0u;
    }
    return t;
}

// ORs m into a word of a bitmask.  A word that already holds it is only read:
// bits are never cleared, so a stale read costs an atomic, not a bit.
__device__ __forceinline__ void or_word(uint32_t *word, uint32_t m)
{
    if (m & ~*reinterpret_cast<volatile uint32_t *>(word)) atomicOr(word, m);
}

// Sets the bits lo .. hi (lo <= hi).  Nearly every run of a voxel's pixels lies
// in one word, and the others' code is kept out of its way: with one loop over
// the words 100 frames of 8.4 K voxels, 8 cameras, took 239 us, with this 204.
__device__ __forceinline__ void set_bits(uint32_t *bits, int lo, int hi)
{
    uint32_t *w = bits + (lo >> 5), *const last = bits + (hi >> 5);
    const uint32_t first_m = 0xFFFFFFFFu << (lo & 31), last_m = 0xFFFFFFFFu >> (31 - (hi & 31));
    if (w == last) {
        or_word(w, first_m & last_m);
        return;
    }
    or_word(w, first_m);
    for (++w; w < last; ++w) or_word(w, 0xFFFFFFFFu);
    or_word(last, last_m);
}

// The projection of one listed voxel's cube in camera c: the silhouette
// polygon (n >= 3 corners, a 4-corner loop padded with its first corner, so
// that zero-length edges cross no row), the du/dv of its edges and the
// range of pixel rows and columns whose centres it can hold; n = 0 when a
// corner is not in front of the camera or the projection is too large for
// float32 rows (the caller then takes the slab test).  Cubes wholly behind the
// camera have no columns.
struct CubeProj {
    float pu[6], pv[6], sl[6];
    int n;
    int xa, xb, ya, yb;   // candidate pixels, none if xa > xb (the slab test's box when n = 0)
    float o1[3];          // the cube's lower faces minus the camera centre (index coordinates)
};

// `corners`: the silhouette table as corner offsets (see kernel).
__device__ __forceinline__ void project_cube(const ReprojectArgs &a, const float4 *corners, const DivAny &by_nxy,
                                             const DivAny &by_nx, int c, uint32_t v, CubeProj &P)
{
    uint32_t r, ix;
    const uint32_t kz = div_any(v, by_nxy, r), jy = div_any(r, by_nx, ix);
    const int W = a.W, H = a.H;
    float m[12];
#pragma unroll
    for (int q = 0; q < 12; ++q) m[q] = a.cam[c].m[q];
    // centred index coordinates of the cube's centre
    const float x0 = (float)ix - a.ci, y0 = (float)jy - a.cj, z0 = (float)kz - a.ck;
    // all corners in front: depth of the centre beyond half the cube's extent
    // in depth, with a margin far above the float32 rounding of a corner's
    // depth; only cubes near the camera plane test their eight corners
    const float w0 = fmaf(m[8], x0, fmaf(m[9], y0, fmaf(m[10], z0, m[11])));
    const float ext = 0.5f * (fabsf(m[8]) + fabsf(m[9]) + fabsf(m[10]));
    const float mag = fabsf(m[8] * x0) + fabsf(m[9] * y0) + fabsf(m[10] * z0) + fabsf(m[11]);
    bool behind = false;
    P.xa = 0;
    P.xb = -1;
    if (!(w0 > 1.0001f * ext + 1e-5f * mag)) {
        // the same margin behind the camera: no ray meets the cube in front of it
        if (w0 < -(1.0001f * ext + 1e-5f * mag)) return;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const float X = x0 + ((q & 1) ? 0.5f : -0.5f), Y = y0 + ((q & 2) ? 0.5f : -0.5f),
                        Z = z0 + ((q & 4) ? 0.5f : -0.5f);
            behind |= !(fmaf(m[8], X, fmaf(m[9], Y, fmaf(m[10], Z, m[11]))) > 0.0f);
        }
    }
    P.o1[0] = (float)ix - 0.5f - a.inv[c].qc[0];
    P.o1[1] = (float)jy - 0.5f - a.inv[c].qc[1];
    P.o1[2] = (float)kz - 0.5f - a.inv[c].qc[2];
    P.n = 0;
    P.xb = W - 1;
    P.ya = 0;
    P.yb = H - 1;
    if (behind) return;   // the whole image: the per-pixel test decides
    int code = 0;
#pragma unroll
    for (int ax = 2; ax >= 0; --ax)
        code = 3 * code + (P.o1[ax] > 0.0f ? 0 : (P.o1[ax] + 1.0f < 0.0f ? 2 : 1));
    const float4 *loop = corners + 6 * code;
    const int n = (int)loop[0].w;
    float umin = INFINITY, umax = -INFINITY, vmin = INFINITY, vmax = -INFINITY;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const float4 q = loop[k];
        const float X = x0 + q.x, Y = y0 + q.y, Z = z0 + q.z;
        const float u = fmaf(m[0], X, fmaf(m[1], Y, fmaf(m[2], Z, m[3])));
        const float vv = fmaf(m[4], X, fmaf(m[5], Y, fmaf(m[6], Z, m[7])));
        // hardware reciprocal (about 1 ulp): the corners move by ~1e-7 of their
        // distance from the principal point, far below the 2e-3 voxel the
        // silhouettes are checked against
        const float iw = rcp_approx(fmaf(m[8], X, fmaf(m[9], Y, fmaf(m[10], Z, m[11]))));
        P.pu[k] = u * iw;
        P.pv[k] = vv * iw;
        umin = fminf(umin, P.pu[k]);
        umax = fmaxf(umax, P.pu[k]);
        vmin = fminf(vmin, P.pv[k]);
        vmax = fmaxf(vmax, P.pv[k]);
    }
    if (n >= 3 && fmaxf(fmaxf(fabsf(umin), fabsf(umax)), fmaxf(fabsf(vmin), fabsf(vmax))) < 1e5f) {
        P.n = n;
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const int j = (k + 1) % 6;
            const float dv = P.pv[j] - P.pv[k];
            P.sl[k] = dv != 0.0f ? div_fast(P.pu[j] - P.pu[k], dv) : 0.0f;
        }
        P.xa = max((int)ceilf(umin - 0.5f), 0);
        P.xb = min((int)floorf(umax - 0.5f), W - 1);
        P.ya = max((int)ceilf(vmin - 0.5f), 0);
        P.yb = min((int)floorf(vmax - 0.5f), H - 1);
        return;
    }
    // the slab test's candidates: centres within the box, widened by 0.01 px
    // plus a relative float32 margin
    const float du = 0.01f + 1e-5f * fmaxf(fabsf(umin), fabsf(umax));
    const float dv = 0.01f + 1e-5f * fmaxf(fabsf(vmin), fabsf(vmax));
    P.xa = max(0, (int)fmaxf(ceilf(umin - 0.5f - du), -1.0f));
    P.xb = min(W - 1, (int)fminf(floorf(umax - 0.5f + du), (float)W));
    P.ya = max(0, (int)fmaxf(ceilf(vmin - 0.5f - dv), -1.0f));
    P.yb = min(H - 1, (int)fminf(floorf(vmax - 0.5f + dv), (float)H));
}

// Row y of the silhouette polygon: the columns [xs, xe] whose centres it
// holds (xs > xe: none), kept within the polygon's column range [xa, xb] (a
// rounded crossing may fall just outside its corners' extent).
__device__ __forceinline__ void polygon_row(const CubeProj &P, int y, int &xs, int &xe)
{
    const float yc = (float)y + 0.5f;
    float lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int j = (k + 1) % 6;
        if ((P.pv[k] <= yc) != (P.pv[j] <= yc)) {
            const float x = fmaf(yc - P.pv[k], P.sl[k], P.pu[k]);
            lo = fminf(lo, x);
            hi = fmaxf(hi, x);
        }
    }
    xs = 1;
    xe = 0;
    if (lo <= hi) {
        xs = max((int)ceilf(lo - 0.5f), P.xa);
        xe = min((int)floorf(hi - 0.5f), P.xb);
    }
}

// Slab test of the centre ray through pixel (px, py) (coordinates of its
// centre), with `mi` from the camera's pixels to directions and the cube's
// faces o1, o1 + 1 from the camera's centre.  Hardware reciprocals (about 1
// ulp; 1/0 = inf as with the division): the slab distances move by far less
// than the 2e-3 voxel the silhouettes are checked against.
__device__ __forceinline__ bool slab_test(const float (&mi)[9], const float (&o1)[3], float px, float py)
{
    float t_in = 0.0f, t_out = INFINITY;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const float id = rcp_approx(fmaf(mi[3 * ax], px, fmaf(mi[3 * ax + 1], py, mi[3 * ax + 2])));
        const float t1 = o1[ax] * id, t2 = (o1[ax] + 1.0f) * id;
        t_in = fmaxf(t_in, fminf(t1, t2));
        t_out = fminf(t_out, fmaxf(t1, t2));
    }
    return t_in <= t_out;
}

// Slab test of a box's pixels (cubes not wholly in front of the camera, or
// projections too large for float32 rows) within the pixels p0 .. p1 - 1 of
// the band, by one thread.
__device__ void slab_test_pixels(const ReprojectArgs &a, int c, const CubeProj &P, uint32_t *bits, int p0, int p1)
{
    float mi[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) mi[q] = a.inv[c].minv[q];
    const int yb = min(P.yb, (p1 - 1) / a.W);
    for (int y = max(P.ya, p0 / a.W); y <= yb; ++y) {
        const int xb = min(P.xb, p1 - 1 - y * a.W);
        for (int x = max(P.xa, p0 - y * a.W); x <= xb; ++x)
            if (slab_test(mi, P.o1, (float)x + 0.5f, (float)y + 0.5f)) set_bits(bits, y * a.W + x - p0, y * a.W + x - p0);
    }
}

// The same for `n` queued voxels by the whole CTA: a row of a cube's pixels per
// warp, 32 pixels that share a word of the bitmask at a time, words whose
// pixels are all set passed over.  A cube at the camera plane may cover the
// whole image: 3000 voxels around a camera at 320 x 240 take 0.37 ms, 5.4 with
// one thread per cube.
__device__ __forceinline__ void slab_test_queue(const ReprojectArgs &a, const float4 *corners, const DivAny by_nxy,
                                             const DivAny by_nx, int c, const uint32_t *queue, uint32_t n,
                                             uint32_t *bits, int p0, int p1)
{
    const int lane = threadIdx.x & 31, W = a.W;
    float mi[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) mi[q] = a.inv[c].minv[q];
    for (uint32_t q = 0; q < n; ++q) {
        CubeProj P;
        project_cube(a, corners, by_nxy, by_nx, c, queue[q], P);
        const int yb = min(P.yb, (p1 - 1) / W);
        for (int y = max(P.ya, p0 / W) + (int)(threadIdx.x >> 5); y <= yb; y += (int)(blockDim.x >> 5)) {
            const int lo = max(y * W + P.xa, p0) - p0, hi = min(y * W + P.xb, p1 - 1) - p0;
            for (int b0 = lo & ~31; b0 <= hi; b0 += 32) {
                const int b = b0 + lane;
                const uint32_t word = *reinterpret_cast<volatile uint32_t *>(bits + (b0 >> 5));
                const bool need = b >= lo && b <= hi && !((word >> lane) & 1u);
                if (!__any_sync(0xFFFFFFFFu, need)) continue;
                const bool hit = need && slab_test(mi, P.o1, (float)(p0 + b - y * W) + 0.5f, (float)y + 0.5f);
                const uint32_t m = __ballot_sync(0xFFFFFFFFu, hit);
                if (lane == 0 && m) atomicOr(bits + (b0 >> 5), m);
            }
        }
    }
}

// ---- the cluster's other bitmasks (distributed shared memory) ----
__device__ __forceinline__ uint32_t load_peer(const uint32_t *p, uint32_t rank)
{
    uint32_t a, v;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}

// The low four bits of v as four bytes of 0 or 1.
__device__ __forceinline__ uint32_t spread4(uint32_t v) { return ((v & 15u) * 0x00204081u) & 0x01010101u; }

// Stores the pixels q0 .. q1 - 1 of a band that starts at pixel p0 as bytes
// (kZero: zeros): single bytes up to the first and after the last whole
// aligned 16 bytes.
template <bool kZero>
__device__ __forceinline__ void store_bits(const uint32_t *bits, uint8_t *mask, int p0, int q0, int q1)
{
    if (q0 >= q1) return;
    const int tid = threadIdx.x;
    const int head = min(q1 - q0, (int)((16u - (uint32_t)(reinterpret_cast<uintptr_t>(mask + q0) & 15u)) & 15u));
    const int n16 = (q1 - q0 - head) / 16, tail0 = q0 + head + 16 * n16;
    for (int u = tid; u < n16; u += (int)blockDim.x) {
        const int b = q0 + head + 16 * u - p0, w = b >> 5, sh = b & 31;
        const uint32_t v = kZero ? 0u : __funnelshift_r(bits[w], sh > 16 ? bits[w + 1] : 0u, sh);
        *reinterpret_cast<uint4 *>(mask + p0 + b) =
            make_uint4(spread4(v), spread4(v >> 4), spread4(v >> 8), spread4(v >> 12));
    }
    if (tid < 32) {
        const int p = tid < 16 ? q0 + tid : tail0 + tid - 16;
        if (tid < 16 ? tid < head : p < q1)
            mask[p] = kZero ? (uint8_t)0 : (uint8_t)((bits[(p - p0) >> 5] >> ((p - p0) & 31)) & 1u);
    }
}

// ORs the words wa .. wb of a band's bitmask (`words` words in all, the last
// one zero) into the band's `n` bytes at dst.  A warp takes 32 words at a time
// and of these only the groups of four with a set pixel, so that it passes
// quickly over what its voxels left empty; a lane then has four pixels of a
// group: one atomic per aligned 4 bytes with a set pixel, next to those of the
// other lanes, or single bytes where these 4 reach beyond the band.
__device__ __forceinline__ void or_words(const uint32_t *bits, int wa, int wb, int words, uint8_t *dst, int n)
{
    const int lane = threadIdx.x & 31, off = (int)(reinterpret_cast<uintptr_t>(dst) & 3u);
    // window w: the 32 pixels from pixel 32 w - off on, whose bytes start aligned
    wb = min(wb + (off ? 1 : 0), words - 1);
    for (int w0 = wa + (int)(threadIdx.x & ~31u); w0 <= wb; w0 += (int)blockDim.x) {
        const int w = w0 + lane;
        const uint32_t hi = w <= wb ? bits[w] : 0u, lo = w <= wb && w > 0 ? bits[w - 1] : 0u;
        const uint32_t v = __funnelshift_l(lo, hi, off);
        uint32_t any = __ballot_sync(0xFFFFFFFFu, v != 0u);
        while (any) {
            const int g = (__ffs(any) - 1) & ~3;   // words w0 + g .. w0 + g + 3
            any &= ~(15u << g);
            const uint32_t q = (__shfl_sync(0xFFFFFFFFu, v, g + (lane >> 3)) >> (4 * (lane & 7))) & 15u;
            if (!q) continue;
            const int b = 32 * (w0 + g) + 4 * lane - off;
            if (b >= 0 && b + 4 <= n) {
                atomicOr(reinterpret_cast<unsigned int *>(dst + b), spread4(q));
            } else {
                for (int k = 0; k < 4; ++k)
                    if ((q >> k) & 1u) dst[b + k] = 1;
            }
        }
    }
}

// Programmatic dependent launch: lets the next kernel's CTAs start beside this
// one's, and in these waits until this one has finished.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void wait_dependency() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// What a CTA of reproject_kernel works on.
struct RpPlace {
    int c, f, p0, p1;      // camera, frame, pixels p0 .. p1 - 1
    int S, rank;           // CTAs that share the entries, and this one among them
    uint32_t entries;      // of the frame's list
    uint64_t e0, e1;       // the entries e0 .. e1 - 1 that these CTAs take
};

template <bool kParts>
__device__ __forceinline__ RpPlace locate(const ReprojectArgs &a, int bands, int band_pix, int n)
{
    RpPlace l;
    l.S = kParts ? 1 : n;
    l.rank = l.S == 1 ? 0 : (int)cluster_rank();
    const int K = a.n_cams, part = kParts ? (int)blockIdx.x / (K * bands) : 0;
    const int cb = kParts ? (int)blockIdx.x - part * (K * bands) : (int)blockIdx.x / n;
    l.c = cb / bands;
    l.f = blockIdx.y;
    l.p0 = (cb - l.c * bands) * band_pix;
    l.p1 = min(a.W * a.H, l.p0 + band_pix);
    l.entries = min(__ldg(a.counts + l.f), a.list_stride);
    // parts: equal ranges of whole warps (listed neighbours lie close together,
    // so that a part's pixels overlap)
    const uint32_t per = kParts ? max((l.entries / (uint32_t)n + 32u) & ~31u, 128u) : l.entries;
    l.e0 = (uint64_t)part * per;
    l.e1 = min(l.e0 + per, (uint64_t)l.entries);
    return l;
}

// The slab tests of the voxels that the threads of a CTA left pending (bit i:
// mine[i * step]), one of each thread at a time.
__device__ __forceinline__ void slab_phase(const ReprojectArgs &a, const float4 *corners, const DivAny by_nxy,
                                        const DivAny by_nx, int c, const uint32_t *mine, uint64_t step,
                                        uint32_t pending, uint32_t *bits, int p0, int p1)
{
    __shared__ uint32_t queue[kRpSmThreads], queued;
    do {
        if (threadIdx.x == 0) queued = 0;
        __syncthreads();
        if (pending) {
            queue[atomicAdd(&queued, 1u)] = __ldg(mine + (uint64_t)(__ffs(pending) - 1) * step);
            pending &= pending - 1u;
        }
        __syncthreads();
        slab_test_queue(a, corners, by_nxy, by_nx, c, queue, queued, bits, p0, p1);
    } while (__syncthreads_or(pending != 0));
}

// blockIdx.y = frame.  The pixels of a camera are numbered row by row; band b
// holds b * band_pix .. min(W H, (b + 1) band_pix) - 1.
//   kParts false: blockIdx.x = (camera * bands + band) * n + rank; the n CTAs
// of a cluster take one mask band and store all its bytes.  Of a frame with
// more than `most` entries they store zeros; the second kernel takes it.
//   kParts true: blockIdx.x = (part * n_cams + camera) * bands + band; of a
// frame with more than `most` entries a CTA takes the part-th of n ranges and
// ORs its pixels into the zeros of the first kernel, beside which it starts.
// (Parts outermost: those that a shorter list leaves empty come last.)
//
// 100 frames of 4.7 K surface voxels, 8 cameras of 640 x 480, take 142 us, most
// of it the six edge tests of each voxel's pixel rows.  Before (chunks of 256
// voxels staged as bytes over their common box, OR-ed into a zeroed mask word
// by word): 275 us; with eight corner depths, corner offsets from selects and
// integer divisions per voxel instead of the depth bound, the offset table and
// div_any: 175 us; with a loop over the words of each run in set_bits: 164 us.
template <bool kParts>
__global__ void __launch_bounds__(kRpSmThreads, 1) reproject_kernel(const __grid_constant__ ReprojectArgs a,
                                                                  const __grid_constant__ SilTable sil,
                                                                  DivAny by_nxy, DivAny by_nx, int bands,
                                                                  int band_pix, int n, uint32_t most)
{
    extern __shared__ __align__(16) uint32_t bits[];   // band_words(band_pix) words, the last of them zero
    __shared__ int s_rows[2];                          // kParts: -first, last row with pixels that may be set
    // per camera region the corners of the silhouette loop as offsets from the
    // cube's centre (.w: their number; a 4-corner loop padded with its first)
    __shared__ float4 s_corners[27 * 6];
    const int tid = threadIdx.x;
    const RpPlace l = locate<kParts>(a, bands, band_pix, n);
    const int S = l.S, W = a.W, p0 = l.p0, p1 = l.p1;
    const int threads = blockDim.x;
    if (kParts) {
        if (l.entries <= most || l.e0 >= l.e1) {
            if ((blockIdx.x | blockIdx.y) == 0) wait_dependency();   // this grid ends after the first kernel's
            return;
        }
        if (tid < 2) s_rows[tid] = INT_MIN;
    } else {
        launch_dependents();
    }
    uint8_t *mask = a.masks + ((size_t)l.f * a.n_cams + l.c) * (a.W * a.H);
    // the CTA's share of the band in whole words
    const int share = ((p1 - p0 + S - 1) / S + 31) & ~31;
    const int q0 = p0 + l.rank * share, q1 = min(p1, q0 + share);
    if (!kParts && l.entries > most) {
        store_bits<true>(nullptr, mask, p0, q0, q1);
        return;
    }
    if (tid < 27 * 6) {
        const uint32_t ent = sil.e[tid / 6], len = ent & 15u, k = tid % 6;
        const uint32_t q = (ent >> (4 + 3 * (k < len ? k : 0))) & 7u;
        s_corners[tid] = make_float4((q & 1) ? 0.5f : -0.5f, (q & 2) ? 0.5f : -0.5f, (q & 4) ? 0.5f : -0.5f, (float)len);
    }
    const uint32_t *list = a.lists + (size_t)l.f * a.list_stride;
    const uint64_t e1 = l.e1, step = (uint64_t)S * threads;
    uint64_t e = l.e0 + (uint64_t)l.rank * threads + tid;
    uint32_t next = e < e1 ? __ldg(list + e) : 0u;   // in flight while the bitmask is zeroed
    const int n_words = (p1 - p0 + 31) / 32 + 1;
    for (int w = tid; w < (n_words + 3) / 4; w += threads) reinterpret_cast<uint4 *>(bits)[w] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();

    const int y_lo = p0 / W, y_hi = (p1 - 1) / W;
    int ya = INT_MAX, yb = -1;   // rows of this thread's candidate pixels
    const uint32_t *mine = list + e;
    // of this thread's first 32 entries, those that take the slab test: done by
    // the whole CTA after the others (a queue filled from inside the loop let
    // lanes with fewer rows run on apart from the others, 1.5 times the time
    // for images of several bands)
    uint32_t pending = 0, bit = 1;
    for (; e < e1; e += step, bit <<= 1) {
        const uint32_t v = next;
        if (e + step < e1) next = __ldg(list + e + step);
        if (v >= a.n_vox) continue;
        CubeProj P;
        project_cube(a, s_corners, by_nxy, by_nx, l.c, v, P);
        if (P.xa > P.xb) continue;
        if (kParts) {
            ya = min(ya, P.ya);
            yb = max(yb, P.yb);
        }
        if (P.n >= 3) {
            const int ye = min(P.yb, y_hi);
            for (int y = max(P.ya, y_lo); y <= ye; ++y) {
                int xs, xe;
                polygon_row(P, y, xs, xe);
                if (xs > xe || !PSFS_IN_BOUNDS(y >= 0 && y < a.H && xs >= 0 && xe < W, a.status)) continue;
                const int lo = max(y * W + xs, p0), hi = min(y * W + xe, p1 - 1);
                if (lo <= hi) set_bits(bits, lo - p0, hi - p0);
            }
        } else if (bit) {
            pending |= bit;
        } else {
            slab_test_pixels(a, l.c, P, bits, p0, p1);
        }
    }
    if (__syncthreads_or(pending != 0))
        slab_phase(a, s_corners, by_nxy, by_nx, l.c, mine, step, pending, bits, p0, p1);
    if (kParts) {
        ya = __reduce_max_sync(0xFFFFFFFFu, -ya);
        yb = __reduce_max_sync(0xFFFFFFFFu, yb);
        if ((tid & 31) == 0) {
            atomicMax(&s_rows[0], ya);
            atomicMax(&s_rows[1], yb);
        }
        __syncthreads();
        ya = max(-s_rows[0], y_lo);
        yb = min(s_rows[1], y_hi);
        wait_dependency();
        if (ya <= yb)
            or_words(bits, max(ya * W - p0, 0) >> 5, (min((yb + 1) * W, p1) - 1 - p0) >> 5, n_words, mask + p0, p1 - p0);
        return;
    }
    if (S == 1)
        __syncthreads();
    else
        cluster_sync();

    // this CTA's share of the band: whole words, so that it can OR the peers'
    // into its own (they read other words of it), then bits as bytes
    if (S > 1) {
        for (int w = (q0 - p0) / 32 + tid; w < (q1 - p0 + 31) / 32; w += threads) {
            uint32_t v = 0;
#pragma unroll
            for (int r = 0; r < kRpMaxCluster; ++r)   // independent loads, in flight together
                if (r < S) v |= load_peer(bits + w, (uint32_t)r);
            bits[w] = v;
        }
        __syncthreads();
    }
    store_bits<false>(bits, mask, p0, q0, q1);
    if (S > 1) cluster_sync();   // the peers read this CTA's bitmask until here
}

}  // namespace

constexpr int kRpSmShared = 224 * 1024;   // shared memory of an SM's CTAs
constexpr int kRpStatic = 8192;           // of a CTA beside its bitmask, no less

// Shared memory words of a band's bitmask: its pixels, a zero word, whole 16 bytes.
static int band_words(int band_pix) { return (band_pix / 32 + 1 + 3) & ~3; }

// Bands: as few as hold kRpBandPixels each, because every band projects the
// whole list again and the body's rows are seldom shared out evenly; CTAs of
// 512 threads where two of them fit an SM, of 1024 otherwise.  36 masks, 43 K
// voxels: 1280 x 720 75 us in one band, 114 in two of 96 KB and 512 threads;
// 1920 x 1080 155 in two, 212 in three (105 and 154 with chunks staged over
// their common box and no bands); 32 x 8 masks of 3840 x 2160, 8.4 K: 622 in
// five, 706 in eleven.  (A test that passes over voxels above or below the band
// gains nothing: their warps wait for the others.)
//
// Cluster size: the one with the least time for the SM that gets most CTAs, if
// a CTA costs 1 / S of a mask's list and 1 / 8 for its bitmask, and CTAs beside
// each other on an SM 0.82 of that (fitted to 8 to 800 masks and lists of 2.7 K
// to 43 K voxels; 72 masks of 640 x 480, 8.4 K: 45.9, 29.7, 29.4 and 35.6 us
// with 1, 2, 4 and 8; 160 masks: 74.7, 65.7, 60.5, 71.0; 800 masks: 204 with 1;
// sizes that are not powers of two are sometimes placed badly, 24 masks with 6
// 64 us and with 4 56).
//
// Parts, for at most a third as many masks as SMs: four CTAs of 256 threads per
// SM in all (as shared memory allows).  us with parts / with a cluster per mask
// only (640 x 480): one mask, 43 K voxels 9.7 / 31.7, 562 K 27 / 290; 8 masks,
// 43 K 19.6 / 33; 16 masks, 8.4 K 15 / 19.6; 48 masks, 8.4 K 24 / 27.9; 56
// masks, 8.4 K: the cluster is faster.  Lists of up to 4096 entries, which a
// cluster of 8 takes in one round, are left to it (8 masks, 4000 voxels in any
// order 10.8, with parts 10.4 in the grid's order but 14.7 shuffled, as the
// smoothing leaves them: more atomics), but not where four CTAs per mask do not
// fit the SMs at once (45 masks, 2.7 K voxels 14.8 / 19.2).
ReprojectSplit reproject_split(int64_t n_pix, int64_t frame_cams, uint32_t list_stride, int sms)
{
    ReprojectSplit r;
    r.bands = (int)((n_pix + kRpBandPixels - 1) / kRpBandPixels);
    r.band_pix = (int)(((n_pix + r.bands - 1) / r.bands + 31) & ~(int64_t)31);
    r.cluster = 1;
    r.parts = r.part_threads = 0;
    r.most = UINT32_MAX;
    r.threads = 2 * (4 * band_words(r.band_pix) + kRpStatic) <= kRpSmShared ? kRpSmThreads / 2 : kRpSmThreads;
    const int64_t masks = frame_cams * r.bands;
    sms = std::max(sms, 1);
    double best = 1e300;
    for (int S = 1; S <= kRpMaxCluster; S *= 2) {
        const int64_t load = (masks * S + sms - 1) / sms;   // CTAs of the fullest SM
        const double cost = (load == 1 ? 1.0 : 0.82 * (double)load) * (1.0 / S + 0.125);
        if (cost < best) {
            best = cost;
            r.cluster = S;
        }
    }
    const uint32_t most = 4 * masks <= sms ? 4096u : 0u;
    if (3 * masks <= sms && list_stride > most) {
        const int per_sm = std::max(1, std::min(4, kRpSmShared / (4 * band_words(r.band_pix) + kRpStatic)));
        r.most = most;
        r.parts = (int)std::min<int64_t>(per_sm * (int64_t)sms / masks, ((int64_t)list_stride + 127) / 128);
        r.part_threads = (kRpSmThreads / per_sm) & ~31;
    }
    return r;
}

cudaError_t launch_reproject(const ReprojectArgs &a, int n_frames, cudaStream_t s)
{
    if (n_frames <= 0) return cudaSuccess;
    static const SilTable sil = make_sil_table();
    const int n_pix = a.W * a.H;
    const ReprojectSplit sp = reproject_split(n_pix, (int64_t)n_frames * a.n_cams, a.list_stride, device_sm_count());
    static bool configured[64] = {false};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!configured[dev]) {
        for (const auto k : {reproject_kernel<true>, reproject_kernel<false>}) {
            const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       4 * band_words(kRpBandPixels));
            if (e != cudaSuccess) return e;
        }
        configured[dev] = true;
    }
    const DivAny by_nxy = make_div_any((uint32_t)a.nx * (uint32_t)a.ny), by_nx = make_div_any((uint32_t)a.nx);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.n_cams * sp.bands * sp.cluster), (unsigned)n_frames);
    cfg.blockDim = dim3((unsigned)sp.threads);
    cfg.dynamicSmemBytes = (size_t)(4 * band_words(sp.band_pix));
    cfg.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)sp.cluster;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = sp.cluster > 1 ? 1 : 0;
    cudaError_t e = cudaLaunchKernelEx(&cfg, reproject_kernel<false>, a, sil, by_nxy, by_nx, sp.bands, sp.band_pix,
                                       sp.cluster, sp.most);
    if (e == cudaSuccess && sp.parts) {
        cfg.gridDim.x = (unsigned)(a.n_cams * sp.bands * sp.parts);
        cfg.blockDim = dim3((unsigned)sp.part_threads);
        attr = {};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, reproject_kernel<true>, a, sil, by_nxy, by_nx, sp.bands, sp.band_pix, sp.parts,
                               sp.most);
    }
    return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace psfs
