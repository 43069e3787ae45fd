// boac_plain.cu -- the unfused operators: forward projection (Eq. 1-2), its
// exact adjoint, the launch-per-step MLEM loop used as the comparison
// baseline, and the float64 log-likelihood reduction (Eq. 5).
//
// Ray kernels run one thread per (candidate, view, bin) and walk the ray from
// the detector side (k = n-1) inwards, so the attenuation suffix sum of
// Eq. 1's inner integral is a running register sum; the images are in shared
// memory where they fit (ray_smem_kernel).  The back-projector is a
// per-pixel gather over the <= 3 x 3 ray samples whose bilinear footprint
// contains the pixel, with the weights recomputed exactly as the projector
// computes them (sample_uw + pixel_weight), so no atomics are needed and the
// result is deterministic.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>

#include "boac_device.cuh"
#include "boac_internal.h"
#include "boac_ops.h"
#include "boac_plain_kernels.cuh"

namespace cg = cooperative_groups;

namespace boac {

// The ray kernels below read images too large for shared memory through L1, a
// warp per CTA: where a view's rays run along the rows, a warp's loads touch 32
// lines each, and the CTAs of that view bound the call, so they have to lie on
// many SMs (one image of 256 x 256, us of boac_project with 128 / 64 / 32 threads
// per CTA: 60 views 181 / 119 / 107, 90 views 142 / 113 / 103; 32 images and 60
// views 999 / 1010 / 805).
constexpr int kRayGlobalThreads = 32;
static dim3 ray_global_grid(const boac_geom* g, int B) {
    return dim3((g->n + kRayGlobalThreads - 1) / kRayGlobalThreads, g->n_views, B);
}

// Walks a ray from the detector side (k = n - 1) inwards: use(k, load(k)) in
// order, the loads of DEPTH samples in flight at a time (a sample's four
// neighbours are an L1 or L2 latency away, and one thread's ray is serial).  Two
// where mu is integrated from global memory (one image of 256 x 256, table and
// back-projection with 1 / 2 / 4 / 8: 9 views 106 / 103 / 126 / 104 us, 60 views
// 166 / 164 / 188 / 166).
template <int DEPTH = 4, class Load, class Use>
__device__ __forceinline__ void walk_ray(int n, Load load, Use use) {
    int k = n - 1;
    for (; k >= DEPTH - 1; k -= DEPTH) {
        decltype(load(0)) v[DEPTH];
#pragma unroll
        for (int j = 0; j < DEPTH; ++j) v[j] = load(k - j);
#pragma unroll
        for (int j = 0; j < DEPTH; ++j) use(k - j, v[j]);
    }
    for (; k >= 0; --k) use(k, load(k));
}

__device__ __forceinline__ float ray_sample(const float* __restrict__ img, int n, int k, int b, float cs, float sn,
                                            float c) {
    float u, w;
    sample_uw(k, b, cs, sn, c, &u, &w);
    return bilerp_global(img, n, u, w);
}

// attenuation factor of every ray sample: tab[cand][v][k][b]
__global__ void attenuation_table_kernel(int n, int V, float dx, const float* __restrict__ mu,
                                         float* __restrict__ tab) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x, v = blockIdx.y, cand = blockIdx.z;
    const size_t nn = (size_t)n * n;
    const float* m_img = mu + cand * nn;
    float* t = tab + ((size_t)cand * V + v) * nn;
    float cs, sn;
    cta_view_cos_sin(v, V, &cs, &sn);
    if (b >= n) return;
    const float c = 0.5f * (float)(n - 1);
    float suffix = 0.0f;
    walk_ray<2>(
        n, [&](int k) { return ray_sample(m_img, n, k, b, cs, sn, c); },
        [&](int k, float m) {
            t[(size_t)k * n + b] = expf(-dx * (0.5f * m + suffix));
            suffix += m;
        });
}

// q[cand][v][b] = dx sum_k a_k F_k with the attenuation integrated on the fly
__global__ void project_otf_kernel(int n, int V, float dx, const float* __restrict__ mu,
                                   const float* __restrict__ F, float* __restrict__ q) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x, v = blockIdx.y, cand = blockIdx.z;
    const size_t nn = (size_t)n * n;
    const float* m_img = mu + cand * nn;
    const float* f_img = F + cand * nn;
    float cs, sn;
    cta_view_cos_sin(v, V, &cs, &sn);
    if (b >= n) return;
    const float c = 0.5f * (float)(n - 1);
    float suffix = 0.0f, acc = 0.0f;
    walk_ray<2>(
        n,
        [&](int k) {
            return make_float2(ray_sample(m_img, n, k, b, cs, sn, c), ray_sample(f_img, n, k, b, cs, sn, c));
        },
        [&](int, float2 s) {
            const float a = expf(-dx * (0.5f * s.x + suffix));
            suffix += s.x;
            acc = fmaf(a, s.y, acc);
        });
    q[((size_t)cand * V + v) * n + b] = dx * acc;
}

// The ray kernels above and below with their images in shared memory (padded by
// a ring of zeros, so a sample needs no test per neighbour), for the sides
// where they fit: blockDim.y views of one candidate per CTA, a thread per ray.
// Same operations and sums.  4 candidates of 100 x 100 and 75 views: a
// projection from the table took 52 us through L1, here 35.
// A warp's 32 samples are 32 steps along a line across the image, at any angle:
// at pitch P the cell (row w, column u) lies in bank P w + u, so a line along a
// short vector of the lattice P w + u = 0 (mod 32) falls on few banks.  Sides that
// are multiples of 32 would have P = n + 1 = 1 (mod 32) and the vector (1, -1): 20-odd
// lanes on a bank around 45 and 135 degrees.  ray_pitch takes the next pitch whose
// shortest vector is at least 5 cells long (us of boac_project, 64 images: 128 x
// 128 and 75 views 325 -> 248, 96 x 96 and 75 216 -> 142; one image of 128 x 128
// and 511 views 155 -> 69, 100 x 100, whose pitch was good, 54).
__device__ __forceinline__ const float* padded_image(float* smem, int slot, int n, int P,
                                                     const float* __restrict__ src) {
    const int size = P * (n + 2) + 1;
    float* img = smem + slot * size;
    const int tid = threadIdx.y * blockDim.x + threadIdx.x, nt = blockDim.x * blockDim.y;
    for (int i = tid; i < P; i += nt) img[i] = img[(n + 1) * P + i] = 0.0f;
    for (int i = tid; i <= n + 1; i += nt) {
        img[i * P] = 0.0f;
        if (P > n + 1) img[i * P + n + 1] = 0.0f;  // else the next row's left padding
    }
    if (tid == 0) img[size - 1] = 0.0f;
    const int j = threadIdx.x;  // blockDim.x >= n
#pragma unroll 8
    for (int r = threadIdx.y; r < n; r += blockDim.y)
        if (j < n) img[(r + 1) * P + j + 1] = __ldg(src + (size_t)r * n + j);
    return img;
}
__device__ __forceinline__ float ray_sample_padded(const float* img, int n, int P, int k, int b, float cs, float sn,
                                                   float c) {
    float u, w;
    sample_uw(k, b, cs, sn, c, &u, &w);
    return bilerp_padded(img, P, n, u, w);
}

constexpr int kRayViews = 8;  // most views of a CTA
enum class RayOp { kTable, kProjectTable, kProject };
template <RayOp OP>
__global__ void __launch_bounds__(1024) ray_smem_kernel(int n, int P, int V, float dx, const float* __restrict__ mu,
                                                       const float* __restrict__ F, const float* __restrict__ tab,
                                                       float* __restrict__ out) {
    extern __shared__ float smem[];
    const int b = threadIdx.x, v = blockIdx.x * blockDim.y + threadIdx.y, cand = blockIdx.y;
    const size_t nn = (size_t)n * n;
    const float* m_img = nullptr;
    const float* f_img = nullptr;
    int slots = 0;
    if (OP != RayOp::kProjectTable) m_img = padded_image(smem, slots++, n, P, mu + cand * nn);
    if (OP != RayOp::kTable) f_img = padded_image(smem, slots++, n, P, F + cand * nn);
    __shared__ float csn[kRayViews][2];  // one float64 sine and cosine per view, not per thread
    if (b == 0) view_cos_sin(v, V, &csn[threadIdx.y][0], &csn[threadIdx.y][1]);
    __syncthreads();
    if (b >= n || v >= V) return;
    const float cs = csn[threadIdx.y][0], sn = csn[threadIdx.y][1];
    const float c = 0.5f * (float)(n - 1);
    const size_t plane = ((size_t)cand * V + v) * nn;
    float suffix = 0.0f, acc = 0.0f;
    if constexpr (OP == RayOp::kTable) {
        walk_ray<8>(
            n, [&](int k) { return ray_sample_padded(m_img, n, P, k, b, cs, sn, c); },
            [&](int k, float m) {
                out[plane + (size_t)k * n + b] = expf(-dx * (0.5f * m + suffix));
                suffix += m;
            });
        return;
    } else if constexpr (OP == RayOp::kProjectTable) {
        walk_ray<8>(
            n,
            [&](int k) {
                return make_float2(__ldg(tab + plane + (size_t)k * n + b),
                                   ray_sample_padded(f_img, n, P, k, b, cs, sn, c));
            },
            [&](int, float2 s) { acc = fmaf(s.x, s.y, acc); });
    } else {
        walk_ray<4>(
            n,
            [&](int k) {
                return make_float2(ray_sample_padded(m_img, n, P, k, b, cs, sn, c),
                                   ray_sample_padded(f_img, n, P, k, b, cs, sn, c));
            },
            [&](int, float2 s) {
                const float a = expf(-dx * (0.5f * s.x + suffix));
                suffix += s.x;
                acc = fmaf(a, s.y, acc);
            });
    }
    out[((size_t)cand * V + v) * n + b] = dx * acc;
}

// The pitch of a padded image of side n (at least n + 1), `images` of which go
// into shared memory together: see padded_image.  n + 1 where a better one does
// not fit.
constexpr size_t kRaySmem = 226 * 1024;
static size_t ray_smem_bytes(int n, int P, int images) {
    return sizeof(float) * images * ((size_t)P * (n + 2) + 1);
}
static int ray_pitch(int n, int images) {
    // residues mod 32 with no lattice vector shorter than 5
    constexpr unsigned kSpread = 1u << 5 | 1u << 6 | 1u << 7 | 1u << 9 | 1u << 12 | 1u << 13 | 1u << 19 | 1u << 20 |
                                 1u << 23 | 1u << 25 | 1u << 26 | 1u << 27;
    int P = n + 1;
    while (!(kSpread >> (P % 32) & 1)) ++P;
    return ray_smem_bytes(n, P, images) <= kRaySmem ? P : n + 1;
}

// Launches it where `images` padded images fit an SM, with enough views per CTA
// to fill it; false: not launched (use the kernels that read global memory).
template <RayOp OP>
static bool ray_smem_launch(int n, int V, int B, float dx, const float* mu, const float* F, const float* tab, float* out,
                            cudaStream_t st) {
    constexpr int kDev = 64;
    static int allowed[kDev];
    const int images = OP == RayOp::kProject ? 2 : 1;
    const int P = ray_pitch(n, images);
    const size_t smem = ray_smem_bytes(n, P, images);
    if (smem > kRaySmem) return false;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDev) {
        cudaGetLastError();
        return false;
    }
    if (!allowed[dev]) {
        if (cudaFuncSetAttribute(ray_smem_kernel<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRaySmem) !=
            cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        allowed[dev] = 1;
    }
    const int width = (n + 31) / 32 * 32, sms = sm_count() > 0 ? sm_count() : 1;
    int views = (int)((long long)V * B / sms);  // about one CTA per SM ...
    if (views < 4) views = 4;
    if (views > 1024 / width) views = 1024 / width;  // ... of at most 1024 threads
    if (views > kRayViews) views = kRayViews;
    if (views < 1) views = 1;
    if (views > V) views = V;
    ray_smem_kernel<OP>
        <<<dim3((V + views - 1) / views, B), dim3(width, views), smem, st>>>(n, P, V, dx, mu, F, tab, out);
    return true;
}

void attenuation_table(const boac_geom* g, int B, const float* mu, float* tab, cudaStream_t st) {
    if (!ray_smem_launch<RayOp::kTable>(g->n, g->n_views, B, g->pixel_cm, mu, nullptr, nullptr, tab, st))
        attenuation_table_kernel<<<ray_global_grid(g, B), kRayGlobalThreads, 0, st>>>(g->n, g->n_views, g->pixel_cm, mu,
                                                                                      tab);
}
void project_rays(const boac_geom* g, int B, const float* mu, const float* F, float* q, cudaStream_t st) {
    if (!ray_smem_launch<RayOp::kProject>(g->n, g->n_views, B, g->pixel_cm, mu, F, nullptr, q, st))
        project_otf_kernel<<<ray_global_grid(g, B), kRayGlobalThreads, 0, st>>>(g->n, g->n_views, g->pixel_cm, mu, F,
                                                                                q);
}
void project_table_rays(const boac_geom* g, int B, float dx, const float* tab, const float* F, float* q,
                        cudaStream_t st) {
    if (!ray_smem_launch<RayOp::kProjectTable>(g->n, g->n_views, B, dx, nullptr, F, tab, q, st))
        project_table_kernel<<<ray_global_grid(g, B), kRayGlobalThreads, 0, st>>>(g->n, g->n_views, dx, tab, F, q);
}

// q = A F with a precomputed attenuation table
__global__ void project_table_kernel(int n, int V, float dx, const float* __restrict__ tab,
                                     const float* __restrict__ F, float* __restrict__ q) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x, v = blockIdx.y, cand = blockIdx.z;
    const size_t nn = (size_t)n * n;
    const float* t = tab + ((size_t)cand * V + v) * nn;
    const float* f_img = F + cand * nn;
    float cs, sn;
    cta_view_cos_sin(v, V, &cs, &sn);
    if (b >= n) return;
    const float c = 0.5f * (float)(n - 1);
    float acc = 0.0f;
    walk_ray(
        n,
        [&](int k) { return make_float2(__ldg(t + (size_t)k * n + b), ray_sample(f_img, n, k, b, cs, sn, c)); },
        [&](int, float2 s) { acc = fmaf(s.x, s.y, acc); });
    q[((size_t)cand * V + v) * n + b] = dx * acc;
}

// out[cand] (+)= scale * sum_v B_v^T (tab_v * y_v) (y == nullptr: y = 1), as
// a per-pixel gather: with tab = attenuation and scale = dx this is A^T y.
// The weights of a pixel's window are the geometry's, so a thread works them
// out once for C candidates; kViewLanes lanes of a warp take a pixel's views
// in turn, and every one of them adds up all views' sums in view order (one
// thread per pixel left the GPU waiting where the images are few and small: 4
// candidates of 100 x 100 and 75 views took 196 us, with 16 lanes and C = 2 62;
// with 8 lanes 67, C = 4 80).
template <int C, int kViewLanes>
__global__ void __launch_bounds__(kPixThreads)
    backproject_gather_kernel(int n, int V, int B, float scale, const float* __restrict__ tab,
                              const float* __restrict__ y, float* __restrict__ out, int accumulate) {
    extern __shared__ float csn[];  // [V][2]
    for (int v = threadIdx.x; v < V; v += blockDim.x) view_cos_sin(v, V, &csn[2 * v], &csn[2 * v + 1]);
    __syncthreads();
    constexpr int kPix = 32 / kViewLanes;  // pixels of a warp, side by side
    const int lane = threadIdx.x & 31, px = lane % kPix, vl = lane / kPix;
    const int cand0 = blockIdx.y * C;
    const int pix = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) / 32) * kPix + px;
    const bool mine = pix < n * n;  // (every lane stays for the shuffles)
    const int i = mine ? pix / n : 0, j = mine ? pix % n : 0;
    const size_t nn = (size_t)n * n;
    const float c = 0.5f * (float)(n - 1);
    const float jc = (float)j - c, ic = (float)i - c;
    float acc[C];
#pragma unroll
    for (int q = 0; q < C; ++q) acc[q] = 0.0f;
    for (int v0 = 0; v0 < V; v0 += kViewLanes) {
        const int v = v0 + vl;
        float vacc[C];
#pragma unroll
        for (int q = 0; q < C; ++q) vacc[q] = 0.0f;
        if (mine && v < V) {
            const float cs = csn[2 * v], sn = csn[2 * v + 1];
            // continuous (k', b') of the pixel centre on this view's sample grid
            const float bp = c + jc * cs + ic * sn;
            const float kp = c - jc * sn + ic * cs;
            int kmin = (int)floorf(kp - 1.4143f) + 1, kmax = (int)floorf(kp + 1.4143f);
            int bmin = (int)floorf(bp - 1.4143f) + 1, bmax = (int)floorf(bp + 1.4143f);
            kmin = max(kmin, 0);
            bmin = max(bmin, 0);
            kmax = min(kmax, n - 1);
            bmax = min(bmax, n - 1);
#pragma unroll
            for (int db = 0; db < 3; ++db) {  // the window is at most 3 x 3
                const int b = bmin + db;
                if (b > bmax) break;
                float bacc[C];
#pragma unroll
                for (int q = 0; q < C; ++q) bacc[q] = 0.0f;
                // the weights of the three samples, their loads in flight
                // together, then the sums
                float wt[3], t[3][C];
#pragma unroll
                for (int dk = 0; dk < 3; ++dk) {
                    const int k = kmin + dk;
                    wt[dk] = 0.0f;
                    if (k <= kmax) {
                        float u, w;
                        sample_uw(k, b, cs, sn, c, &u, &w);
                        wt[dk] = pixel_weight(u, w, i, j, n);
                    }
                }
                const float* tp = tab + ((size_t)cand0 * V + v) * nn + (size_t)kmin * n + b;
#pragma unroll
                for (int dk = 0; dk < 3; ++dk)
#pragma unroll
                    for (int q = 0; q < C; ++q)
                        t[dk][q] = wt[dk] != 0.0f && (C == 1 || cand0 + q < B) ? __ldg(tp + (size_t)q * V * nn + dk * n) : 0.0f;
#pragma unroll
                for (int dk = 0; dk < 3; ++dk)
                    if (wt[dk] != 0.0f)
#pragma unroll
                        for (int q = 0; q < C; ++q) bacc[q] = fmaf(wt[dk], t[dk][q], bacc[q]);
#pragma unroll
                for (int q = 0; q < C; ++q)
                    if (C == 1 || cand0 + q < B)
                        vacc[q] = fmaf(bacc[q], y ? __ldg(y + ((size_t)(cand0 + q) * V + v) * n + b) : 1.0f, vacc[q]);
            }
        }
        // the views of this turn, in order
#pragma unroll
        for (int l = 0; l < kViewLanes; ++l)
            if (v0 + l < V)
#pragma unroll
                for (int q = 0; q < C; ++q) acc[q] += __shfl_sync(0xffffffffu, vacc[q], l * kPix + px);
    }
    if (!mine || vl != 0) return;
#pragma unroll
    for (int q = 0; q < C; ++q)
        if (C == 1 || cand0 + q < B) {
            float* o = out + (size_t)(cand0 + q) * nn + pix;
            *o = accumulate ? *o + scale * acc[q] : scale * acc[q];
        }
}

template <int C, int LANES>
static void gather_launch(int n, int V, int B, float scale, const float* tab, const float* y, float* out, int accumulate,
                          cudaStream_t st) {
    const size_t warps = ((size_t)n * n * LANES + 31) / 32;
    const unsigned blocks = (unsigned)((warps * 32 + kPixThreads - 1) / kPixThreads);
    backproject_gather_kernel<C, LANES><<<dim3(blocks, (B + C - 1) / C), kPixThreads, sizeof(float) * 2 * V, st>>>(
        n, V, B, scale, tab, y, out, accumulate);
}

void backproject_gather(int n, int V, int B, float scale, const float* tab, const float* y, float* out,
                        int accumulate, cudaStream_t st) {
    // Two candidates share a thread's weights, and a pixel's views go to as few
    // lanes as leave the SMs enough threads: more lanes idle where the views do
    // not fill their last turn, and each adds up all views' sums.  That is about
    // 1600 threads each, or 3400 from 32 views on, where the turns are full, with
    // 16 lanes only for what 8 leave below 1600.  (Whole back-projections, us with
    // 1 / 2 / 4 / 8 / 16 lanes: 64 images of 200 x 200 and 9 views 390 / 445 / 540 /
    // 729 / 978, 64 of 100 x 100 and 120 views 1229 / 1149 / 1138 / 1185 / 1394; 8 of
    // 200 x 200 and 240 1527 / 1306 / 1211 / 1217 / 1338, 8 of 100 x 100 and 75 218 /
    // 155 / 151 / 140 / 144; 4 of 100 x 100 and 75 209 / 131 / 101 / 103 / 100.)
    const long long items = (long long)n * n * ((B + 1) / 2), sms = sm_count() > 0 ? sm_count() : 1;
    int lanes = 1;
    while (lanes < 8 && items * lanes < (V < 32 ? 1600 : 3400) * sms) lanes *= 2;
    if (lanes == 8 && items * 8 < 1600 * sms) lanes = 16;
#define X(L)                                                                                                   \
    if (lanes == L) {                                                                                          \
        (B == 1 ? gather_launch<1, L> : gather_launch<2, L>)(n, V, B, scale, tab, y, out, accumulate, st); \
        return;                                                                                                \
    }
    X(1) X(2) X(4) X(8) X(16)
#undef X
}

__global__ void ratio_kernel(int count, const float* __restrict__ S, const float* __restrict__ q,
                             float* __restrict__ r) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const float qi = q[i];
        r[i] = qi > 0.0f ? __ldg(S + i) / qi : 0.0f;
    }
}

__global__ void update_kernel(int count, float* __restrict__ F, const float* __restrict__ bp,
                              const float* __restrict__ sens) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        const float s = sens[i];
        F[i] = s > 0.0f ? F[i] * bp[i] / s : 0.0f;
    }
}

__device__ __forceinline__ double loglik_term_plain(double s, double q, bool include_lgamma) {
    double term;
    if (s > 0.0) term = q > 0.0 ? s * log(q) - q : -INFINITY;
    else term = -q;
    if (include_lgamma) term -= lgamma(s + 1.0);
    return term;
}

// L[cand] = sum_i S_i ln q_i - q_i [- lgamma(S_i + 1)] in float64.  Fixed
// per-thread strides and a fixed reduction tree: deterministic.  With lgS
// (candidates sharing one sinogram) the ln S! term is its precomputed sum,
// subtracted once, instead of a term per bin.
__global__ void loglik_kernel(int nbin, const float* __restrict__ q, const float* __restrict__ S,
                              long long s_stride, int include_lgamma, double* __restrict__ L,
                              const double* __restrict__ lgS, int* status) {
    __shared__ double part[32];
    const int cand = blockIdx.x;
    const float* qc = q + (size_t)cand * nbin;
    const float* Sc = S + (size_t)cand * s_stride;
    double acc = 0.0;
    for (int i = threadIdx.x; i < nbin; i += blockDim.x) {
        acc += loglik_term_plain((double)__ldg(Sc + i), (double)__ldg(qc + i), include_lgamma && !lgS);
    }
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
        L[cand] = include_lgamma && lgS ? t - *lgS : t;
        if (status && t == -INFINITY) atomicCAS(status, BOAC_OK, BOAC_ENONFINITE);
    }
}

// loglik_kernel's sums by a cluster of CTAs per candidate: the terms (a float64
// logarithm each, at two float64 operations per SM and cycle) are spread over
// the cluster's SMs, rank r's share [r chunk, (r + 1) chunk) in its shared
// memory; then rank 0 adds them in loglik_kernel's order.  8 candidates of
// 96 x 96 and 90 views: 107 -> 19 us.
__global__ void __launch_bounds__(256) loglik_cluster_kernel(int nbin, int chunk, const float* __restrict__ q,
                                                            const float* __restrict__ S, long long s_stride,
                                                            int include_lgamma, double* __restrict__ L,
                                                            const double* __restrict__ lgS, int* status) {
    extern __shared__ __align__(16) double terms[];  // [chunk], then [32] (no static array: see loglik_launch)
    double* part = terms + chunk;
    cg::cluster_group cl = cg::this_cluster();
    const int ranks = (int)cl.num_blocks(), rank = (int)cl.block_rank(), cand = blockIdx.x / ranks;
    const float* qc = q + (size_t)cand * nbin;
    const float* Sc = S + (size_t)cand * s_stride;
    for (int t = threadIdx.x; t < chunk; t += blockDim.x) {
        const int i = rank * chunk + t;
        if (i < nbin) terms[t] = loglik_term_plain((double)__ldg(Sc + i), (double)__ldg(qc + i), include_lgamma && !lgS);
    }
    cl.sync();
    if (rank == 0) {
        double acc = 0.0;
#pragma unroll 8
        for (int i = threadIdx.x; i < nbin; i += 256) acc += cl.map_shared_rank(terms, i / chunk)[i % chunk];
        for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
            L[cand] = include_lgamma && lgS ? t - *lgS : t;
            if (status && t == -INFINITY) atomicCAS(status, BOAC_OK, BOAC_ENONFINITE);
        }
    }
    cl.sync();  // rank 0 has read every rank's terms
}

int loglik_launch(int nbin, int B, const float* q, const float* S, long long s_stride, int include_lgamma, double* L,
                  const double* lgS, int* status, cudaStream_t st) {
    // Eight CTAs per candidate where their terms and partial sums fit 48 KB
    // each, all the shared memory (static arrays included) that a launch gets
    // without an attribute, and the batch leaves SMs idle (one CTA per
    // candidate reaches every SM at 152).
    constexpr int kRanks = 8;
    const int chunk = (nbin + kRanks - 1) / kRanks;
    const size_t smem = sizeof(double) * ((size_t)chunk + 32);
    if (B > 64 || smem > 48 * 1024) {
        loglik_kernel<<<B, 256, 0, st>>>(nbin, q, S, s_stride, include_lgamma, L, lgS, status);
        return launch_status();
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kRanks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(B * kRanks), 1, 1);
    cfg.blockDim = dim3(256, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, loglik_cluster_kernel, nbin, chunk, q, S, s_stride, include_lgamma, L, lgS, status) !=
        cudaSuccess)
        return launch_status();
    return launch_status();
}

// sum_i lgamma(S_i + 1) over one sinogram (the ln S! term of Eq. 5, equal
// for every candidate that shares the sinogram), float64: block b adds bins
// b * blockDim + t, b * blockDim + t + G blockDim, ... into part[b] with a
// fixed reduction tree; one thread then adds part[0..G) in order.
__global__ void lgamma_partial_kernel(int nbin, const float* __restrict__ S, double* __restrict__ part) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nbin; i += gridDim.x * blockDim.x)
        acc += lgamma((double)__ldg(S + i) + 1.0);
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
        part[blockIdx.x] = t;
    }
}

__global__ void lgamma_final_kernel(int nparts, const double* __restrict__ part, double* __restrict__ out) {
    double t = 0.0;
    for (int i = 0; i < nparts; ++i) t += part[i];
    *out = t;
}

const double* lgamma_sum(int nbin, const float* S, double* scratch, cudaStream_t st) {
    int parts = (nbin + 255) / 256;
    if (parts > kLgammaScratchDoubles - 1) parts = kLgammaScratchDoubles - 1;
    if (parts < 1) parts = 1;
    lgamma_partial_kernel<<<parts, 256, 0, st>>>(nbin, S, scratch + 1);
    lgamma_final_kernel<<<1, 1, 0, st>>>(parts, scratch + 1, scratch);
    return scratch;
}

dim3 ray_grid(const boac_geom* g, int B) {
    return dim3((g->n + kRayThreads - 1) / kRayThreads, g->n_views, B);
}

int grid_1d(long long count, int threads) {
    long long b = (count + threads - 1) / threads;
    long long cap = 16LL * (sm_count() > 0 ? sm_count() : 1);
    return (int)(b < cap ? b : cap);
}

}  // namespace boac

using namespace boac;

extern "C" int boac_project(const boac_geom* g, const float* mu, const float* F, int B, float* q,
                            void* stream) {
    BOAC_RANGE("boac_project");
    if (!geom_ok(g) || !mu || !F || !q || B < 1 || B > 65535) return BOAC_EINVAL;
    if (ops_on_grids(g)) return project_on_grids(g, mu, F, B, q, as_stream(stream));
    project_rays(g, B, mu, F, q, as_stream(stream));
    return launch_status();
}

extern "C" int boac_backproject(const boac_geom* g, const float* mu, const float* y, int B,
                                float* out, void* ws, size_t ws_bytes, void* stream) {
    BOAC_RANGE("boac_backproject");
    if (!geom_ok(g) || !mu || !out || B < 1 || B > 65535) return BOAC_EINVAL;
    const size_t nn = (size_t)g->n * g->n;
    const size_t per = backproject_candidate_bytes(g);  // one candidate's table + partials
    if (!ws || ws_bytes < per + 2 * 256) return BOAC_EWORKSPACE;
    const size_t fit = (ws_bytes - 2 * 256) / per;
    const int chunk = (int)(fit < (size_t)B ? fit : (size_t)B);
    cudaStream_t st = as_stream(stream);
    char* base = static_cast<char*>(ws);
    float* tab = reinterpret_cast<float*>(base);
    float* partial = reinterpret_cast<float*>(
        base + align256(sizeof(float) * (size_t)chunk * g->n_views * nn));
    for (int c0 = 0; c0 < B; c0 += chunk) {
        const int cb = (B - c0) < chunk ? (B - c0) : chunk;
        if (ops_on_grids(g)) {  // no table
            const int s = backproject_on_grids(g, mu + c0 * nn, y ? y + (size_t)c0 * g->n_views * g->n_bins : nullptr, cb,
                                               out + c0 * nn, partial, st);
            if (s != BOAC_OK) return s;
            continue;
        }
        attenuation_table(g, cb, mu + c0 * nn, tab, st);
        int s = launch_status();
        if (s != BOAC_OK) return s;
        s = backproject_table(g, cb, tab, y ? y + (size_t)c0 * g->n_views * g->n_bins : nullptr,
                              g->pixel_cm, out + c0 * nn, 0, partial, st);
        if (s != BOAC_OK) return s;
    }
    return BOAC_OK;
}

extern "C" int boac_loglik(const boac_geom* g, const float* q, const float* S, long long s_stride,
                           int B, int include_lgamma, double* L, void* stream) {
    BOAC_RANGE("boac_loglik");
    if (!geom_ok(g) || !q || !S || !L || B < 1 || s_stride < 0) return BOAC_EINVAL;
    return loglik_launch(g->n_views * g->n_bins, B, q, S, s_stride, include_lgamma, L, nullptr, nullptr,
                         as_stream(stream));
}

extern "C" int boac_score(const boac_geom* g, const float* mu, const float* S, long long s_stride,
                          const float* F, int B, int include_lgamma, double* L, void* ws,
                          size_t ws_bytes, void* stream) {
    BOAC_RANGE("boac_score");
    if (!geom_ok(g) || !mu || !S || !F || !L || B < 1 || B > 65535 || s_stride < 0)
        return BOAC_EINVAL;
    const size_t vb = (size_t)g->n_views * g->n_bins;
    if (!ws || ws_bytes < sizeof(float) * vb * B) return BOAC_EWORKSPACE;
    float* q = static_cast<float*>(ws);
    int s = boac_project(g, mu, F, B, q, stream);
    if (s != BOAC_OK) return s;
    return boac_loglik(g, q, S, s_stride, B, include_lgamma, L, stream);
}

extern "C" int boac_mlem_plain(const boac_geom* g, const float* mu, const float* S,
                               long long s_stride, float* F, int K, int B, double* L,
                               int include_lgamma, void* ws, size_t ws_bytes, void* stream) {
    BOAC_RANGE("boac_mlem_plain");
    if (!geom_ok(g) || !mu || !S || !F || B < 1 || K < 0 || s_stride < 0) return BOAC_EINVAL;
    if (!ws || ws_bytes < plain_candidate_bytes(g)) return BOAC_EWORKSPACE;
    const size_t nn = (size_t)g->n * g->n, vb = (size_t)g->n_views * g->n_bins;
    char* base = static_cast<char*>(ws);
    float* tab = reinterpret_cast<float*>(base);
    base += align256(sizeof(float) * vb * g->n);
    float* sens = reinterpret_cast<float*>(base);
    base += align256(sizeof(float) * nn);
    float* bp = reinterpret_cast<float*>(base);
    base += align256(sizeof(float) * nn);
    float* q = reinterpret_cast<float*>(base);
    base += align256(sizeof(float) * vb);
    float* r = reinterpret_cast<float*>(base);
    base += align256(sizeof(float) * vb);
    float* partial = reinterpret_cast<float*>(base);
    cudaStream_t st = as_stream(stream);
    const float dx = g->pixel_cm;
    for (int cand = 0; cand < B; ++cand) {
        const float* m_c = mu + cand * nn;
        const float* S_c = S + (size_t)cand * s_stride;
        float* F_c = F + cand * nn;
        attenuation_table(g, 1, m_c, tab, st);
        int s = backproject_table(g, 1, tab, nullptr, dx, sens, 0, partial, st);
        if (s != BOAC_OK) return s;
        for (int it = 0; it < K; ++it) {
            s = project_table(g, 1, tab, F_c, dx, q, st);
            if (s != BOAC_OK) return s;
            ratio_kernel<<<grid_1d((long long)vb, 256), 256, 0, st>>>((int)vb, S_c, q, r);
            s = backproject_table(g, 1, tab, r, dx, bp, 0, partial, st);
            if (s != BOAC_OK) return s;
            update_kernel<<<grid_1d((long long)nn, 256), 256, 0, st>>>((int)nn, F_c, bp, sens);
        }
        if (L) {
            s = project_table(g, 1, tab, F_c, dx, q, st);
            if (s != BOAC_OK) return s;
            s = loglik_launch((int)vb, 1, q, S_c, 0, include_lgamma, L + cand, nullptr, nullptr, st);
            if (s != BOAC_OK) return s;
        }
        s = launch_status();
        if (s != BOAC_OK) return s;
    }
    return BOAC_OK;
}

#ifdef BOAC_CHECKED
namespace boac {
BOAC_FAULT_READER(bounds_faults_plain)
}  // namespace boac
#endif
