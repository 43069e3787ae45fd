// boac_ops.cu -- the bare operators q = A^mu F and z = (A^mu)^T y (Eq. 1-2 and
// the adjoint) for 64 x 64, 96 x 96 and 128 x 128 images with an even view
// count, on the fused kernels' sample grids: four views (two, where the view
// count is not a multiple of 4) share one bilinear sampling of the images in
// shared memory, and the attenuation of their samples stays on chip.  One CTA
// takes a run of one candidate's grids.  The per-ray projector walks mu and F
// once per view through L1 with 128 dependent steps, and the table-based
// back-projector writes and reads every attenuation factor (8 MB per candidate
// at 128 x 128 and 120 views); other sizes still use them (boac_plain.cu).
// Measured, 64 candidates at 128 x 128 and 120 views: projection 126 us
// (880), back-projection 165 us (780).
#include <cuda_runtime.h>
#include <math.h>

#include "boac_device.cuh"
#include "boac_fused.h"
#include "boac_internal.h"
#include "boac_ops.h"
#include "boac_plain_kernels.cuh"
#include "boac_sched.cuh"

namespace boac {

namespace {

template <int N>
struct OpShape {
    static constexpr int NT = 8 * N, P = N + 1, WP = N + 4;
    static constexpr int IMG = ((N + 1) * (N + 2) + 1 + kScatterPad + 3) & ~3;
    static constexpr int NSEG = 8, SEG = N / 8;  // a ray's segments, one per thread
    static constexpr size_t SMEM = sizeof(float) * (2 * (size_t)IMG + (size_t)N * WP + 4 * NSEG * N + 4 * N);
};

// The views of grid gi, and the bin of grid coordinate j in the vi-th of them.
template <bool QUAD>
__device__ __forceinline__ int grid_view(int gi, int vi, int V) {
    return gi + (vi == 0 ? 0 : vi == 1 ? V / 2 : vi == 2 ? V / 4 : 3 * V / 4);
}
template <int N>
__device__ __forceinline__ int grid_bin(int vi, int j) { return (vi & 1) ? N - 1 - j : j; }

// Sums of the segments before and after this thread's (part[seg][lb]).
template <int N, int NSEG>
__device__ __forceinline__ void segment_sums(const float* part, int lb, int seg, float* before, float* after) {
    float b = 0.0f, a = 0.0f;
#pragma unroll
    for (int s = 0; s < NSEG; ++s) {
        const float v = part[s * N + lb];
        if (s < seg) b += v;
        if (s > seg) a += v;
    }
    *before = b;
    *after = a;
}

// 2^x.  TINY: results below 2^-126 kept (ex2 flushes them to 0: up to 27 % of a
// pixel behind 60 cm at 8 / cm).  Only the CTAs whose mu can lead there do (see
// load_scaled); on all, the operators on 64 images take 128 + 171 us instead of
// 126 + 165.
template <bool TINY>
__device__ __forceinline__ float factor(float x) {
    if constexpr (!TINY) return ex2(x);
    float y;
    asm("ex2.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// A thread's run of SEG samples m of a ray, scaled for base 2 (load_scaled):
// the factors towards the ray's end (e[2 s]: the half-cell sum of the samples
// behind it) and towards its start (e[2 s + 1]).
template <bool TINY, int SEG>
__device__ __forceinline__ void run_factors(const float (&m)[SEG], float before, float after, float (&e)[2 * SEG]) {
#pragma unroll
    for (int s = 0; s < SEG; ++s) {
        e[2 * s + 1] = factor<TINY>(fmaf(0.5f, m[s], before));
        before += m[s];
    }
#pragma unroll
    for (int s = SEG - 1; s >= 0; --s) {
        e[2 * s] = factor<TINY>(fmaf(0.5f, m[s], after));
        after += m[s];
    }
}

template <int N, int NT, int P>
__device__ __forceinline__ void load_image(float* img, const float* __restrict__ src) {
#pragma unroll 4
    for (int i = threadIdx.x; i < N * N; i += NT) img[(i / N + 1) * P + (i % N) + 1] = __ldg(src + i);
}

// mu times -dx log2(e), the product rounded once (the factor in two floats), so
// that the sums along a ray are exponents of 2.  A rounded factor applied to
// the rounded sum instead put both errors, which grow with the exponent, on
// every attenuation factor: back-projections at 128 x 128, 120 views and 2 / cm
// were 9.5e-7 off (root mean square of the pixels' relative errors against 64
// bits), now 9.0e-7; with expf of the sum 9.0e-7 and 160 + 196 us instead of
// 126 + 165 for the operators on 64 images.  (The factor comes from the host:
// its float64 product by each of 1024 threads takes 1 us.)
//
// Returns whether a factor below 2^-126 is possible: an exponent is at most the
// sum of a ray's samples, N times the largest |mu| (to rounding, 125 for 126).
// Called by all threads; ends with a barrier.
template <int N, int NT, int P>
__device__ __forceinline__ bool load_scaled(float* img, const float* __restrict__ src, float2 scale) {
    bool dense = false;
#pragma unroll 4
    for (int i = threadIdx.x; i < N * N; i += NT) {
        const float v = __ldg(src + i);
        const float x = fabsf(v) < INFINITY ? fmaf(v, scale.x, v * scale.y) : v * scale.x;  // (inf - inf is not inf)
        img[(i / N + 1) * P + (i % N) + 1] = x;
        dense |= !(fabsf(x) < 125.0f / N);  // (or not a number)
    }
    return __syncthreads_or(dense);
}

// q of one candidate's grids [g0, g1), their directions in csn, its images in
// shared memory.
template <int N, bool QUAD, bool TINY>
__device__ __forceinline__ void project_grids(int V, float dx, int g0, int g1, const float* csn, float* smem,
                                              float* __restrict__ q) {
    using O = OpShape<N>;
    constexpr int NT = O::NT, P = O::P, WP = O::WP, IMG = O::IMG, NSEG = O::NSEG, SEG = O::SEG;
    const float* img0 = smem;        // F
    const float* img1 = img0 + IMG;  // mu, scaled
    float* W = smem + 2 * IMG;       // [N][WP] samples of mu, then of F
    float* red = W + N * WP;         // [4][NSEG][N]
    const int tid = threadIdx.x, lb = tid % N, seg = tid / N, k0 = seg * SEG;
    const float c = 0.5f * (float)(N - 1);
    for (int gi = g0; gi < g1; ++gi) {
        const float cs = csn[2 * (gi - g0)], sn = csn[2 * (gi - g0) + 1];
        float f[SEG], e[2 * SEG];
        {
            float m[SEG], sum = 0.0f;
            ColumnWalk walk(k0, lb, cs, sn, c);
#pragma unroll
            for (int s = 0; s < SEG; ++s) {
                const Cell<N, P> x(walk.next());
                m[s] = f[s] = 0.0f;
                if (x.in && index_ok(x.cell, (long long)P * (N + 1))) {
                    m[s] = bilerp_cell<P>(img1 + x.cell, x.frac);
                    f[s] = bilerp_cell<P>(img0 + x.cell, x.frac);
                }
                if (QUAD) W[(k0 + s) * WP + lb] = m[s];
                sum += m[s];
            }
            red[seg * N + lb] = sum;
            __syncthreads();
            float before, after;
            segment_sums<N, NSEG>(red, lb, seg, &before, &after);
            run_factors<TINY, SEG>(m, before, after, e);
        }
        float a1 = 0.0f, a2 = 0.0f;
#pragma unroll
        for (int s = 0; s < SEG; ++s) {
            a1 = fmaf(e[2 * s], f[s], a1);
            a2 = fmaf(e[2 * s + 1], f[s], a2);
        }
        float a3 = 0.0f, a4 = 0.0f;
        if (QUAD) {
            // rows: phi + pi/2 has its detector towards b = 0, phi + 3pi/2
            // towards the row's end
            float m[SEG], sum = 0.0f;
#pragma unroll
            for (int s = 0; s < SEG; s += 4) {
                const float4 m4 = *reinterpret_cast<const float4*>(W + lb * WP + k0 + s);
                m[s] = m4.x, m[s + 1] = m4.y, m[s + 2] = m4.z, m[s + 3] = m4.w;
                sum += m4.x + m4.y + (m4.z + m4.w);
            }
            red[(NSEG + seg) * N + lb] = sum;
            __syncthreads();
            float before, after;
            segment_sums<N, NSEG>(red + NSEG * N, lb, seg, &before, &after);
            run_factors<TINY, SEG>(m, before, after, e);
#pragma unroll
            for (int s = 0; s < SEG; ++s) W[(k0 + s) * WP + lb] = f[s];
            __syncthreads();
#pragma unroll
            for (int s = 0; s < SEG; s += 4) {
                const float4 f4 = *reinterpret_cast<const float4*>(W + lb * WP + k0 + s);
                const float ff[4] = {f4.x, f4.y, f4.z, f4.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    a3 = fmaf(e[2 * (s + j) + 1], ff[j], a3);
                    a4 = fmaf(e[2 * (s + j)], ff[j], a4);
                }
            }
        } else {
            __syncthreads();  // the segment sums read
        }
        red[seg * N + lb] = a1;
        red[(NSEG + seg) * N + lb] = a2;
        if (QUAD) {
            red[(2 * NSEG + seg) * N + lb] = a3;
            red[(3 * NSEG + seg) * N + lb] = a4;
        }
        __syncthreads();
        for (int t = tid; t < (QUAD ? 4 : 2) * N; t += NT) {
            const int vi = t / N, j = t % N;
            float sum = 0.0f;
#pragma unroll
            for (int s = 0; s < NSEG; ++s) sum += red[(vi * NSEG + s) * N + j];
            q[(size_t)grid_view<QUAD>(gi, vi, V) * N + grid_bin<N>(vi, j)] = dx * sum;
        }
        __syncthreads();
    }
}

// q of grids [blockIdx.x share) of candidate blockIdx.y.  Bounded by the two
// gathers of every sample (shared memory) and the barriers between the column
// and row passes, as the fused MLEM kernel's forward half.
template <int N, bool QUAD>
__global__ void __launch_bounds__(8 * N, 1)
    project_grids_kernel(int V, float dx, float2 scale, const float* __restrict__ mu, const float* __restrict__ F,
                         float* __restrict__ q) {
    using O = OpShape<N>;
    constexpr int NT = O::NT, P = O::P, IMG = O::IMG;
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, cand = blockIdx.y, ngrid = QUAD ? V / 4 : V / 2;
    const int g0 = (int)((long long)blockIdx.x * ngrid / gridDim.x);
    const int g1 = (int)((long long)(blockIdx.x + 1) * ngrid / gridDim.x);
    __shared__ float csn[kMaxViews];  // the share's grids (at most half the views)
    for (int gi = g0 + tid; gi < g1; gi += NT) view_cos_sin(gi, V, &csn[2 * (gi - g0)], &csn[2 * (gi - g0) + 1]);
    for (int i = tid; i < 2 * IMG; i += NT) smem[i] = 0.0f;
    __syncthreads();
    load_image<N, NT, P>(smem, F + (size_t)cand * N * N);
    const bool dense = load_scaled<N, NT, P>(smem + IMG, mu + (size_t)cand * N * N, scale);
    float* qc = q + (size_t)cand * V * N;
    if (dense) project_grids<N, QUAD, true>(V, dx, g0, g1, csn, smem, qc);
    else project_grids<N, QUAD, false>(V, dx, g0, g1, csn, smem, qc);
}

// z of one candidate's grids [g0, g1) into the accumulator img1.
template <int N, bool QUAD, bool SCHED, bool TINY>
__device__ __forceinline__ void backproject_grids(int V, float dx, int g0, int g1, const float* csn, float* smem,
                                                  const float* __restrict__ y,
                                                  const unsigned short* __restrict__ sched) {
    using O = OpShape<N>;
    constexpr int NT = O::NT, P = O::P, WP = O::WP, IMG = O::IMG, NSEG = O::NSEG, SEG = O::SEG;
    const float* img0 = smem;       // mu, scaled
    float* img1 = smem + IMG;       // accumulator
    float* W = img1 + IMG;          // [N][WP] samples of mu, then weights
    float* red = W + N * WP;        // [2][NSEG][N]
    float* yy = red + 4 * NSEG * N;  // [4][N] dx y by grid coordinate
    const int tid = threadIdx.x, lb = tid % N, seg = tid / N, k0 = seg * SEG;
    const float c = 0.5f * (float)(N - 1);
    for (int gi = g0; gi < g1; ++gi) {
        const float cs = csn[2 * (gi - g0)], sn = csn[2 * (gi - g0) + 1];
        for (int t = tid; t < (QUAD ? 4 : 2) * N; t += NT) {
            const int vi = t / N, j = t % N;
            yy[t] = dx * (y ? __ldg(y + (size_t)grid_view<QUAD>(gi, vi, V) * N + grid_bin<N>(vi, j)) : 1.0f);
        }
        float e[2 * SEG], gc[SEG];
        {
            float m[SEG], sum = 0.0f;
            ColumnWalk walk(k0, lb, cs, sn, c);
#pragma unroll
            for (int s = 0; s < SEG; ++s) {
                m[s] = bilerp_pos<N, P>(img0, walk.next());
                if (QUAD) W[(k0 + s) * WP + lb] = m[s];
                sum += m[s];
            }
            red[seg * N + lb] = sum;
            __syncthreads();
            float before, after;
            segment_sums<N, NSEG>(red, lb, seg, &before, &after);
            run_factors<TINY, SEG>(m, before, after, e);
        }
        {
            const float y1 = yy[lb], y2 = yy[N + lb];
#pragma unroll
            for (int s = 0; s < SEG; ++s) gc[s] = fmaf(e[2 * s], y1, e[2 * s + 1] * y2);
        }
        if (QUAD) {
            float m[SEG], sum = 0.0f;
#pragma unroll
            for (int s = 0; s < SEG; s += 4) {
                const float4 m4 = *reinterpret_cast<const float4*>(W + lb * WP + k0 + s);
                m[s] = m4.x, m[s + 1] = m4.y, m[s + 2] = m4.z, m[s + 3] = m4.w;
                sum += m4.x + m4.y + (m4.z + m4.w);
            }
            red[(NSEG + seg) * N + lb] = sum;
            __syncthreads();
            float before, after;
            segment_sums<N, NSEG>(red + NSEG * N, lb, seg, &before, &after);
            run_factors<TINY, SEG>(m, before, after, e);
        }
#pragma unroll
        for (int s = 0; s < SEG; ++s) W[(k0 + s) * WP + lb] = gc[s];
        const unsigned short* gs = SCHED ? sched + (size_t)gi * 9 * SchedShape<N>::CLS_ENTRIES : nullptr;
        SchedSlots<N, NT> sched0;
        if constexpr (SCHED) sched0.load(gs);
        __syncthreads();
        if (QUAD) {
            const float y3 = yy[2 * N + lb], y4 = yy[3 * N + lb];
#pragma unroll
            for (int s = 0; s < SEG; s += 4) {
                float4* w4 = reinterpret_cast<float4*>(W + lb * WP + k0 + s);
                float4 v = *w4;
                v.x += fmaf(e[2 * s + 1], y3, e[2 * s] * y4);
                v.y += fmaf(e[2 * s + 3], y3, e[2 * s + 2] * y4);
                v.z += fmaf(e[2 * s + 5], y3, e[2 * s + 4] * y4);
                v.w += fmaf(e[2 * s + 7], y3, e[2 * s + 6] * y4);
                *w4 = v;
            }
            __syncthreads();
        }
        if constexpr (SCHED) scatter_scheduled<N, NT, P, WP>(W, img1, cs, sn, c, gs, sched0);
        else scatter_classes<N, NT, P, WP>(W, img1, cs, sn, c);
    }
}

// z of grids [blockIdx.x share) of candidate blockIdx.y into its partial
// image.  SCHED: the scatter runs in the order of a kept schedule; elsewhere
// in lattice order, with the same sums (one image at 128 x 128 and 120 views: a
// schedule of the call's own takes about 190 us to build, all else 33 us;
// 8 images with 230 views in lattice order, both operators: 297 us, with the
// per-ray and per-grid table kernels 630).
template <int N, bool QUAD, bool SCHED>
__global__ void __launch_bounds__(8 * N, 1)
    backproject_grids_kernel(int V, float dx, float2 scale, const float* __restrict__ mu, const float* __restrict__ y,
                             const unsigned short* __restrict__ sched, float* __restrict__ partial) {
    using O = OpShape<N>;
    constexpr int NT = O::NT, P = O::P, IMG = O::IMG;
    extern __shared__ __align__(16) float smem[];
    const int tid = threadIdx.x, cand = blockIdx.y, ngrid = QUAD ? V / 4 : V / 2;
    const int g0 = (int)((long long)blockIdx.x * ngrid / gridDim.x);
    const int g1 = (int)((long long)(blockIdx.x + 1) * ngrid / gridDim.x);
    __shared__ float csn[kMaxViews];  // the share's grids (at most half the views)
    for (int gi = g0 + tid; gi < g1; gi += NT) view_cos_sin(gi, V, &csn[2 * (gi - g0)], &csn[2 * (gi - g0) + 1]);
    for (int i = tid; i < 2 * IMG; i += NT) smem[i] = 0.0f;
    __syncthreads();
    const bool dense = load_scaled<N, NT, P>(smem, mu + (size_t)cand * N * N, scale);
    const float* yc = y ? y + (size_t)cand * V * N : nullptr;
    if (dense) backproject_grids<N, QUAD, SCHED, true>(V, dx, g0, g1, csn, smem, yc, sched);
    else backproject_grids<N, QUAD, SCHED, false>(V, dx, g0, g1, csn, smem, yc, sched);
    float* out = partial + ((size_t)cand * gridDim.x + blockIdx.x) * N * N;
    for (int i = tid; i < N * N; i += NT) out[i] = smem[IMG + (i / N + 1) * P + (i % N) + 1];
}

// -dx log2(e) in two floats (load_scaled).
float2 exponent_scale(float dx) {
    const double s = -1.44269504088896340736 * (double)dx;
    return make_float2((float)s, (float)(s - (double)(float)s));
}

// CTAs per candidate for B candidates of ngrid grids: the least rounds over
// the SMs (one CTA each) times the grids of a CTA, a CTA's image loads and
// start counted as one grid.
int grid_shares(int B, int ngrid) {
    const int sms = sm_count() > 0 ? sm_count() : 1;
    int best = 1;
    long long best_t = -1;
    for (int s = 1; s <= ngrid; ++s) {
        const long long t = (((long long)B * s + sms - 1) / sms) * ((ngrid + s - 1) / s + 1);
        if (best_t < 0 || t < best_t) {
            best = s;
            best_t = t;
        }
    }
    return best;
}

template <class Kernel>
int allow_smem(Kernel k, size_t bytes, bool* done) {
    constexpr int kDev = 64;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDev) return launch_status();
    if (!done[dev]) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess)
            return launch_status();
        done[dev] = true;
    }
    return BOAC_OK;
}

template <int N, bool QUAD>
int project_t(int V, float dx, const float* mu, const float* F, int B, float* q, cudaStream_t st) {
    static bool done[64];
    const int s = allow_smem(project_grids_kernel<N, QUAD>, OpShape<N>::SMEM, done);
    if (s != BOAC_OK) return s;
    project_grids_kernel<N, QUAD>
        <<<dim3(grid_shares(B, QUAD ? V / 4 : V / 2), B), 8 * N, OpShape<N>::SMEM, st>>>(V, dx, exponent_scale(dx), mu,
                                                                                         F, q);
    return launch_status();
}

template <int N, bool QUAD>
int backproject_t(int V, float dx, const float* mu, const float* y, int B, float* out, float* partial,
                  cudaStream_t st) {
    static bool done[2][64];
    int s = BOAC_OK;
    const int ngrid = QUAD ? V / 4 : V / 2, shares = grid_shares(B, ngrid);
    const unsigned short* sched = sched_prepare(N, V, ngrid, OpShape<N>::WP, nullptr, st, &s);
    if (s != BOAC_OK) return s;
    auto kernel = sched ? backproject_grids_kernel<N, QUAD, true> : backproject_grids_kernel<N, QUAD, false>;
    s = allow_smem(kernel, OpShape<N>::SMEM, done[sched != nullptr]);
    if (s != BOAC_OK) return s;
    kernel<<<dim3(shares, B), 8 * N, OpShape<N>::SMEM, st>>>(V, dx, exponent_scale(dx), mu, y, sched, partial);
    return sum_partial_images(B, shares, N * N, partial, out, st);
}

}  // namespace

bool ops_on_grids(const boac_geom* g) {
    return (g->n == 64 || g->n == 96 || g->n == 128) && g->n_views % 2 == 0;
}

#define BOAC_OPS(CALL)                                   \
    switch (g->n) {                                      \
        case 64: return quad ? CALL(64, true) : CALL(64, false);    \
        case 96: return quad ? CALL(96, true) : CALL(96, false);    \
        case 128: return quad ? CALL(128, true) : CALL(128, false); \
        default: return BOAC_EUNSUPPORTED;               \
    }

int project_on_grids(const boac_geom* g, const float* mu, const float* F, int B, float* q, cudaStream_t st) {
    const bool quad = g->n_views % 4 == 0;
#define CALL(NV, QUAD) project_t<NV, QUAD>(g->n_views, g->pixel_cm, mu, F, B, q, st)
    BOAC_OPS(CALL)
#undef CALL
}

int backproject_on_grids(const boac_geom* g, const float* mu, const float* y, int B, float* out, float* partial,
                         cudaStream_t st) {
    const bool quad = g->n_views % 4 == 0;
#define CALL(NV, QUAD) backproject_t<NV, QUAD>(g->n_views, g->pixel_cm, mu, y, B, out, partial, st)
    BOAC_OPS(CALL)
#undef CALL
}
#undef BOAC_OPS

#ifdef BOAC_CHECKED
BOAC_FAULT_READER(bounds_faults_ops)
#endif

}  // namespace boac
