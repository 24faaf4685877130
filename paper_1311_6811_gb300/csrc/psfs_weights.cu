// psfs_weights.cu -- particle weights of the tracker (Section 2.3.2, Eq.
// 14-16; Section 3.3.3, "Compute Sum-squared Difference" steps b-d): how well
// each particle's projected body model matches the voxel silhouettes and
// their edges in every camera.
//
// A particle is n_cyl cylinders (a, b, r).  For a cylinder and a camera
// centre C, the outline seen from C runs along a + t (b - a) +- r n with n
// the unit vector across the axis and the line of sight, n = unit(u x (m - C))
// (u = b - a, m the midpoint).  Silhouette samples sit at t = (k + 1/2) / kt
// and w = (2 l + 1) / kw - 1 across (a + t u + w r n), edge samples at the
// same t on the two outline lines (w = -1, +1).  A sample's value is the
// silhouette (or edge) bit of the pixel its projection falls in, 0 behind the
// camera or outside the image; an edge pixel is a set pixel with a 4-neighbour
// inside the image that is not set.  Per camera S_r = misses / (n_cyl kt kw),
// S_e = misses / (2 n_cyl kt) (Eq. 14-15), weight = exp(-sum_c (S_e + S_r))
// (Eq. 16).
//
// A cluster of S CTAs takes one particle, CTA r the cameras r, r + S, ...: 200
// particles alone are 1.3 CTAs per SM, too few warps to cover the latency of
// the scattered mask reads (many particles: a CTA each).  What the samples share is formed once per CTA in
// shared memory: the t and w of the sample grid, the cylinders, and n per
// (camera, cylinder).  A warp takes 32 consecutive samples of one camera at a
// time, so the camera's matrix comes from the constant bank and the misses
// are counted with ballots; one shared-memory add per warp and camera block
// sends them to CTA 0 of the cluster (integers: exact in any order), where
// one thread forms the terms and the weight in camera order.
//
// Bound by latency (cylinders, then masks, through two cluster barriers; 38 % of
// the issue slots, 60 % of the warps active, most of them waiting for the masks'
// bytes or a barrier): 200 particles x 10 cylinders x 8 cameras x 48 samples take
// 12.3 us.  Before (one
// CTA of 256 threads per particle, each sample with its own normal, three
// run-time divisions and a shared-memory atomic per miss): 24.6 us; clusters of
// 8 CTAs of 256 threads: 14.3 us.
#include "psfs_internal.cuh"

namespace psfs {

namespace {

constexpr int kWMaxSamples = 64;   // largest kt, kw and n_cyl
constexpr int kWMaxCluster = 8;

__device__ __forceinline__ bool mask_at(const uint8_t *m, int W, int x, int y) { return __ldg(m + (size_t)y * W + x) != 0; }

// *p += v in the shared memory of the cluster's CTA 0.
__device__ __forceinline__ void add_to_first(int *p, int v)
{
    uint32_t addr;
    asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(addr) : "r"(smem_u32(p)));
    asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// kCluster false: S = 1, a particle per CTA, without cluster barriers.
template <int kThreads, bool kCluster>
__global__ void __launch_bounds__(kThreads, 1536 / kThreads) weights_kernel(const __grid_constant__ WeightArgs a, int S,
                                                                            DivSmall by_cyl, DivSmall by_kw)
{
    constexpr int kWarps = kThreads / 32;
    __shared__ int s_miss_r[PSFS_MAX_CAMS], s_miss_e[PSFS_MAX_CAMS];   // CTA 0's are the particle's
    __shared__ float s_t[kWMaxSamples], s_w[kWMaxSamples];
    __shared__ float s_cyl[kWMaxSamples][7];                           // a, u = b - a, r
    extern __shared__ float s_n[];                                     // n: [own cameras][n_cyl][3]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = kCluster ? (int)cluster_rank() : 0;
    const int p = kCluster ? (int)blockIdx.x / S : (int)blockIdx.x;
    const int K = a.n_cams, W = a.W, H = a.H, n_cyl = a.n_cyl;
    const int own = kCluster ? (K - rank + S - 1) / S : K;   // cameras rank, rank + S, ... < K
    if (tid < PSFS_MAX_CAMS) {
        s_miss_r[tid] = 0;
        s_miss_e[tid] = 0;
    }
    // CTA 0's counters are zero and it runs before any peer adds to them
    if (kCluster) cluster_arrive();
    for (int i = tid; i < a.kt; i += kThreads) s_t[i] = ((float)i + 0.5f) / (float)a.kt;
    for (int i = kThreads - 1 - tid; i < a.kw; i += kThreads) s_w[i] = (2.0f * (float)i + 1.0f) / (float)a.kw - 1.0f;
    const float *cyl0 = a.cyl + (size_t)p * n_cyl * 7;
    for (int it = tid; it < max(own, 1) * n_cyl; it += kThreads) {
        const int ci = it / n_cyl, q = it - ci * n_cyl;
        const int c = min(rank + ci * S, K - 1);
        const float *cy = cyl0 + q * 7;
        const float ax = cy[0], ay = cy[1], az = cy[2];
        const float ux = cy[3] - ax, uy = cy[4] - ay, uz = cy[5] - az, rad = cy[6];
        const float vx = ax + 0.5f * ux - a.C[c][0], vy = ay + 0.5f * uy - a.C[c][1], vz = az + 0.5f * uz - a.C[c][2];
        float nx = uy * vz - uz * vy, ny = uz * vx - ux * vz, nz = ux * vy - uy * vx;
        const float nn = sqrtf(nx * nx + ny * ny + nz * nz);
        const float in = nn > 0.0f ? 1.0f / nn : 0.0f;
        nx *= in;
        ny *= in;
        nz *= in;
        s_n[3 * it + 0] = nx;
        s_n[3 * it + 1] = ny;
        s_n[3 * it + 2] = nz;
        if (ci == 0) {
            s_cyl[q][0] = ax;
            s_cyl[q][1] = ay;
            s_cyl[q][2] = az;
            s_cyl[q][3] = ux;
            s_cyl[q][4] = uy;
            s_cyl[q][5] = uz;
            s_cyl[q][6] = rad;
        }
    }
    __syncthreads();
    if (kCluster) cluster_wait();

    const int n_sil = a.kt * a.kw, per_cam = n_cyl * (n_sil + 2 * a.kt);
    const int blocks = (per_cam + 31) / 32;   // warp blocks of 32 samples per camera
    for (int ci = 0; ci < own; ++ci) {
        const int c = kCluster ? rank + ci * S : ci;
        const float *P = a.P[c];
        const uint8_t *m = a.masks + (size_t)c * W * H;
        const float *nrm = s_n + 3 * n_cyl * ci;
        int miss_r = 0, miss_e = 0;
        // warps start at different blocks per camera, so that the blocks left over even out
        for (int blk = (warp + ci * (kWarps - blocks % kWarps)) % kWarps; blk < blocks; blk += kWarps) {
            const int r0 = blk * 32 + lane;
            bool miss = false, edge = false;
            if (r0 < per_cam) {
                const int q = (int)div_small((uint32_t)r0, by_cyl), smp = r0 - q * (int)by_cyl.d;
                float t, w;
                if (smp < n_sil) {   // silhouette sample (k, l)
                    const int k = (int)div_small((uint32_t)smp, by_kw), l = smp - k * a.kw;
                    t = s_t[k];
                    w = s_w[l];
                } else {             // edge sample (k, side)
                    const int e = smp - n_sil;
                    t = s_t[e >> 1];
                    w = (e & 1) ? 1.0f : -1.0f;
                    edge = true;
                }
                const float *cy = s_cyl[q];
                const float rad = cy[6], nx = nrm[3 * q], ny = nrm[3 * q + 1], nz = nrm[3 * q + 2];
                const float X = cy[0] + t * cy[3] + w * rad * nx, Y = cy[1] + t * cy[4] + w * rad * ny,
                            Z = cy[2] + t * cy[5] + w * rad * nz;
                const float pu = fmaf(P[0], X, fmaf(P[1], Y, fmaf(P[2], Z, P[3])));
                const float pv = fmaf(P[4], X, fmaf(P[5], Y, fmaf(P[6], Z, P[7])));
                const float pw = fmaf(P[8], X, fmaf(P[9], Y, fmaf(P[10], Z, P[11])));
                miss = true;
                if (pw > 0.0f) {
                    const float xf = pu / pw, yf = pv / pw;
                    if (xf >= 0.0f && xf < (float)W && yf >= 0.0f && yf < (float)H) {
                        const int x = min((int)xf, W - 1), y = min((int)yf, H - 1);
                        bool hit = mask_at(m, W, x, y);
                        if (edge) {
                            // all four neighbours in flight with the pixel itself (outside the image: the
                            // pixel, which counts as set whenever the result depends on it)
                            const bool l = mask_at(m, W, max(x - 1, 0), y), r = mask_at(m, W, min(x + 1, W - 1), y);
                            const bool u = mask_at(m, W, x, max(y - 1, 0)), d = mask_at(m, W, x, min(y + 1, H - 1));
                            hit = hit && !(l && r && u && d);
                        }
                        miss = !hit;
                    }
                }
            }
            miss_r += __popc(__ballot_sync(0xFFFFFFFFu, miss && !edge));
            miss_e += __popc(__ballot_sync(0xFFFFFFFFu, miss && edge));
        }
        if (lane == 0 && (miss_r | miss_e)) {
            if (kCluster) {
                add_to_first(&s_miss_r[c], miss_r);
                add_to_first(&s_miss_e[c], miss_e);
            } else {
                atomicAdd(&s_miss_r[c], miss_r);
                atomicAdd(&s_miss_e[c], miss_e);
            }
        }
    }
    if (kCluster)
        cluster_sync();
    else
        __syncthreads();
    if (rank == 0 && tid == 0) {
        const float inv_r = 1.0f / (float)(n_cyl * a.kt * a.kw), inv_e = 1.0f / (float)(2 * n_cyl * a.kt);
        float total = 0.0f;
        for (int c = 0; c < K; ++c) {
            const float se = (float)s_miss_e[c] * inv_e, sr = (float)s_miss_r[c] * inv_r;
            if (a.terms) {
                a.terms[((size_t)p * K + c) * 2 + 0] = se;
                a.terms[((size_t)p * K + c) * 2 + 1] = sr;
            }
            total += se + sr;
        }
        a.weights[p] = expf(-total);
    }
}

}  // namespace

// Cluster size: the largest of 1, 2, 4 and 8 whose CTAs of 512 threads all run
// at once (three per SM), no more than there are cameras.  More particles take
// a CTA each, of 512, 256 or 128 threads: no more than they have warp blocks
// for, and fewer as long as the SMs stay full, because a CTA's set-up costs more
// than its threads (5000 particles, one camera, 160 samples: 13 us with 128
// threads, 17 with 256, 29 with 512, 42 with clusters of one CTA of 512; 10000,
// eight cameras of 480: 230, 242, 275 and 312; 456, the same: 27, 19 and 19).
cudaError_t launch_weights(const WeightArgs &a, int n_particles, cudaStream_t s)
{
    if (n_particles <= 0) return cudaSuccess;
    const int64_t sms = device_sm_count();
    int S = 1, threads = 512;
    while (S < kWMaxCluster && 2 * S <= a.n_cams && (int64_t)n_particles * 2 * S <= 3 * sms) S *= 2;
    const int blocks = a.n_cams * ((a.n_cyl * a.kt * (a.kw + 2) + 31) / 32);
    while (S == 1 && threads > 128 && ((int64_t)n_particles * threads / 2 >= 1536 * sms || threads / 2 >= 32 * blocks))
        threads /= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_particles * (unsigned)S);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)((a.n_cams + S - 1) / S) * a.n_cyl * 3 * sizeof(float);
    cfg.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)S;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = S > 1 ? 1 : 0;
    const auto kernel = S > 1            ? weights_kernel<512, true>
                        : threads == 512 ? weights_kernel<512, false>
                        : threads == 256 ? weights_kernel<256, false>
                                         : weights_kernel<128, false>;
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, kernel, a, S, make_div_small((uint32_t)(a.kt * a.kw + 2 * a.kt)),
                           make_div_small((uint32_t)a.kw));
    return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace psfs
