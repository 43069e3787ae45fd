// boac_fused_kernel.cuh -- the fused MLEM kernel (see boac_fused.cu) and the
// record of a launch shape, for the translation units that instantiate it:
// boac_fused.cu (one CTA per candidate) and boac_split.cu (a cluster of CTAs
// per candidate).
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <math.h>

#include "boac_device.cuh"
#include "boac_fused.h"
#include "boac_internal.h"
#include "boac_plain_kernels.cuh"
#include "boac_sched.cuh"
#include "boac_tmem.cuh"

namespace cg = cooperative_groups;

namespace boac {

// Shared-memory and work layout of one CTA (image side N, NT threads).
template <int N, int NT>
struct FusedShape {
    // Padded image: pixel (i, j), i, j in [-1, n], at (i+1) P + (j+1) with
    // P = n + 1, so the right padding column of row i and the left padding
    // column of row i+1 are the same zero cell; P = 1 (mod 32) for n a
    // multiple of 32 spreads rotated rows of samples over the banks.
    static constexpr int P = N + 1;
    static constexpr int IMG = (N + 1) * (N + 2) + 1;
    static constexpr int IMGA = (IMG + kScatterPad + 3) & ~3;  // an image's floats, rounded to 16 bytes
    static constexpr int NN = N * N;
    // Sample-buffer pitch: rows start 16 bytes apart in whole groups, and a
    // quarter-warp's 16-byte row accesses (threads on consecutive rows) fall
    // on 8 different 16-byte bank groups since (N + 4) / 4 is odd.
    static constexpr int WP = N + 4;
    static constexpr int NSEG = NT / N;      // segments per column / row
    static constexpr int SEG = N / NSEG;     // samples per segment
    static_assert(NT % N == 0 && N % NSEG == 0, "segmentation");
};

// Views that share one sample grid: 4 (phi + j pi/2, needs V % 4 == 0) or 2
// (phi, phi + pi).  Attenuation exponents stored per grid, already scaled by
// -dx log2(e) so that a = exp2(y):
//   Xc[k][b] = view phi        (detector at k -> +inf, suffix along k)
//   Uc[b]    = whole-column sum: the view phi + pi exponent is Uc - Xc
//   XrT[b][k] = view phi + pi/2 (detector at b -> -inf, prefix along b),
//               stored transposed for row-parallel access
// (the planes in the interleaved order of tab_ix below)
//   Ur[k]    = whole-row sum: the view phi + 3pi/2 exponent is Ur - XrT
// because for one ray the half-cell sums towards both ends add up to the
// ray's total: a_phi * a_{phi+pi} = exp(-dx sum_k mu_k).
__host__ __device__ constexpr size_t fused_group_floats(int n, bool quad) {
    return quad ? 2 * (size_t)n * n + 2 * (size_t)n : (size_t)n * n + (size_t)n;
}
__host__ __device__ constexpr size_t fused_tab_floats(int n, int V) {
    // V/4 groups of 4 views or V/2 groups of 2: the same total
    return (size_t)(V / 2) * ((size_t)n * n + (size_t)n);
}
// The attenuation exponents one CTA keeps: all grids (G = 1), or in cluster
// mode the grids of one of G ranks, at most ceil(grids / G).
__host__ __device__ constexpr size_t fused_tab_floats(int n, int V, bool quad, int G) {
    return G <= 1 ? fused_tab_floats(n, V)
                  : (size_t)(((quad ? V / 4 : V / 2) + G - 1) / G) * fused_group_floats(n, quad);
}

// Whether the images of an n x n candidate live in global memory.
__host__ __device__ constexpr bool fused_global_images(int n) { return n > 128; }

template <int N, int NT>
__host__ __device__ constexpr size_t fused_image_floats() {
    using L = FusedShape<N, NT>;
    return 2 * (size_t)L::IMGA + (size_t)N * L::WP;
}

// A 96 x 96 CTA takes all of its SM's tensor memory (288 of the 512 columns
// used, and allocations are powers of two) but only half of its shared memory.
// It asks for enough of the latter that no 64 x 64 CTA of another launch (56
// KB, 128 columns) fits beside it, where one of the two would wait for the
// other's tensor memory until that kernel ends.
constexpr size_t kSoleSmem = 176 * 1024;

template <int N, int NT>
__host__ __device__ constexpr size_t fused_smem_bytes(int V) {
    using L = FusedShape<N, NT>;
    const size_t need = sizeof(float) * ((fused_global_images(N) ? 0 : fused_image_floats<N, NT>()) +
                                         4 * L::NSEG * N + 10 * N + 2 * ((V + 1) / 2) * 2) +
                        sizeof(double) * 33;
    return N == 96 && need < kSoleSmem ? kSoleSmem : need;
}

// CTAs per SM the register allocation is sized for: as many as shared memory
// allows (three 64x64 CTAs, one of the larger sizes), but no fewer than 64
// registers per thread.
template <int N, int NT>
constexpr int fused_min_blocks() {
    return (N <= 64 ? 3 : 1) < 1024 / NT ? (N <= 64 ? 3 : 1) : (1024 / NT > 0 ? 1024 / NT : 1);
}

// Tensor memory of a CTA (see the kernel): floats per thread, and the columns
// they take; 0 where they are more than an SM has and nothing is kept there.
template <int N, int NT, bool QUAD>
constexpr int fused_stash() {
    return (QUAD ? 4 : 2) * FusedShape<N, NT>::SEG;
}
template <int N, int NT, bool QUAD>
constexpr int fused_tmem_columns() {
    constexpr int c = tmem_columns(NT / 32, fused_stash<N, NT, QUAD>());
    return c <= kTmemColumns ? c : 0;
}

// A thread's exponents of one grid, from the workspace planes into tensor
// memory: chunk i is four samples of its column run, or (i >= SEG / 4) of its
// row run.  A run's exponents lie in the upper half of the columns that its
// factors will fill: the forward pass reads chunk c (columns SEG + 4 c ..)
// before it writes that chunk's factors (8 c ..), and those never reach a
// later chunk's exponents.  As the class scatter's side work the next grid's
// chunks are loaded one class and stored the next, so their L2 latency, which
// the forward passes waited for, passes during the scatter.  32 candidates x
// 20 iterations, 128 x 128, 120 views: 2.13 -> 2.05 ms; 256 x 50: 28.6 -> 28.2.
template <int N, int SEG, bool QUAD>
struct ExponentFetch {
    static constexpr int kRun = SEG / 4, kChunks = (QUAD ? 2 : 1) * kRun;
    static constexpr int kPerClass = (kChunks + 7) / 8;
    const float* planes;  // this thread's first sample of its column run
    unsigned stash;
    float4 v[kPerClass];
    __device__ __forceinline__ ExponentFetch(const float* Xc, int k0, int lb, unsigned stash_)
        : planes(Xc + tab_ix(N, k0, lb)), stash(stash_) {}
    __device__ __forceinline__ static constexpr int column(int i) {
        return i < kRun ? SEG + 4 * i : 2 * SEG + SEG + 4 * (i - kRun);
    }
    __device__ __forceinline__ float4 load(int i) const {
        return *reinterpret_cast<const float4*>(planes + 4 * N * i + (i < kRun ? 0 : N * N - 4 * N * kRun));
    }
    __device__ __forceinline__ void begin(int cls) {
#pragma unroll
        for (int j = 0; j < kPerClass; ++j) {
            const int i = cls * kPerClass + j, before = i - kPerClass;
            if (before >= 0 && before < kChunks) tmem_st4(stash + column(before), v[j]);
            if (i < kChunks) v[j] = load(i);
        }
    }
    // the whole grid at once
    __device__ __forceinline__ void all() {
#pragma unroll 4
        for (int i = 0; i < kChunks; ++i) tmem_st4(stash + column(i), load(i));
    }
};

// The scatter schedule of grid gi (images up to 128 x 128 only).
template <int N>
__device__ __forceinline__ const unsigned short* grid_sched(const FusedArgs& a, int gi) {
    return a.sched + (size_t)gi * 9 * SchedShape<(N <= 128 ? N : 128)>::CLS_ENTRIES;
}

// G = 1: one CTA per candidate at a time (the batch's iterations split over
// the CTAs).  G > 1 (cluster mode, for batches too small to fill the GPU one
// CTA per candidate): a thread-block cluster of G CTAs per candidate, CTA
// rank r working on the sample grids [r V' / G, (r + 1) V' / G) (V' grids)
// with its own copy of F and its own accumulator; after every iteration's
// grids the G accumulators are summed through distributed shared memory,
// each rank updating its share of the image rows and writing them into
// every rank's F.
template <int N, int NT, bool QUAD, int G = 1>
__global__ void __launch_bounds__(NT, (G > 1 ? 1 : fused_min_blocks<N, NT>())) mlem_fused_kernel(FusedArgs a) {
    using Lay = FusedShape<N, NT>;
    constexpr int P = Lay::P, IMG = Lay::IMG, IMGA = Lay::IMGA, NN = Lay::NN, WP = Lay::WP;
    constexpr int NSEG = Lay::NSEG, SEG = Lay::SEG;
    constexpr float kLog2e = 1.44269504088896340736f;

    class_begin(a);
    extern __shared__ __align__(16) float smem[];
    float* const img_base = fused_global_images(N)
                                ? a.img + (size_t)blockIdx.x * fused_image_floats<N, NT>()
                                : smem;
    float* img0 = img_base;             // F (mu during set-up), padded
    float* img1 = img0 + IMGA;          // back-projection accumulator, padded
    float* W = img1 + IMGA;             // [N][WP] grid samples / weights
    float* redc = fused_global_images(N) ? smem : W + N * WP;  // [2][NSEG][N] column partial sums
    float* redr = redc + 2 * NSEG * N;  // [2][NSEG][N] row partial sums
    float* rr = redr + 2 * NSEG * N;    // [4][N] ratios r = S / q per view
    float* Sg = rr + 4 * N;             // [4][N] the grid's sinogram rows (cp.async)
    float* Us = Sg + 4 * N;             // [2][N] the grid's whole-ray exponents Uc, Ur (cp.async)
    float* csn = Us + 2 * N;            // [V][2]
    double* dred = reinterpret_cast<double*>(csn + 2 * ((a.V + 1) / 2) * 2);

    const int tid = threadIdx.x;
    const int V = a.V;
    const int ngrid = QUAD ? V / 4 : V / 2;
    const float c = 0.5f * (float)(N - 1);
    const float dx = a.dx;
    const float ndl = -dx * kLog2e;
    // column mapping: thread owns column `lb`, samples k in [k0, k0 + SEG);
    // row mapping: thread owns row `lb`, samples b in [k0, k0 + SEG)
    const int lb = tid % N, seg = tid / N;
    const int k0 = seg * SEG;
    const size_t gstride = fused_group_floats(N, QUAD);
    // scatter in schedule order: images up to 128 x 128
    constexpr int SN = N <= 128 ? N : 128;
    constexpr bool use_sched = N <= 128;

    for (int v = tid; v < V; v += NT) view_cos_sin(v, V, &csn[2 * v], &csn[2 * v + 1]);

    // Attenuation factors of the grid in flight, in tensor memory: two per
    // sample of the thread's column run, two more per sample of its row run
    // (64 floats per thread, all 256 KB, at 128 x 128).  The weight passes
    // were a second read of the exponents through L2 (131 KB per grid, a
    // fifth of the kernel's L2 traffic) and a second set of exponentials.
    // 256 candidates x 50 iterations, 128 x 128, 120 views: 33.5 -> 31.5 ms.
    // 256 x 256 images (four times the samples per thread) do not fit and
    // read the exponents twice.  CTAs that share an SM (64 x 64 only, at most
    // three by shared memory) take 128 columns each.
    constexpr int kStash = fused_stash<N, NT, QUAD>(), kTmemCols = fused_tmem_columns<N, NT, QUAD>();
    constexpr bool kStashed = kTmemCols > 0;
    __shared__ unsigned tmem_addr;
    unsigned stash = 0;
    if constexpr (kStashed) {
        if (tid < 32) tmem_alloc<kTmemCols>(&tmem_addr);
        __syncthreads();
        stash = tmem_mine(tmem_addr, tid, kStash);
    }
    // The two factors of each of four samples, from their exponents.
    auto factors4 = [](const float (&y)[4], float total, float (&e)[8]) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            e[2 * j] = ex2(y[j]);
            e[2 * j + 1] = ex2(total - y[j]);
        }
    };
    auto plane4 = [](const float* p, float (&y)[4]) {
        const float4 y4 = *reinterpret_cast<const float4*>(p);
        y[0] = y4.x, y[1] = y4.y, y[2] = y4.z, y[3] = y4.w;
    };

    float* tab = a.tab + (size_t)blockIdx.x * fused_tab_floats(N, V, QUAD, G);
    float* sens = a.sens + (size_t)blockIdx.x * NN;
    // this CTA's sample grids [g0, g1) and (cluster mode) update rows [R0, R1)
    int rank = 0, g0 = 0, g1 = ngrid, R0 = 0, R1 = N;
    if constexpr (G > 1) {
        rank = (int)cg::this_cluster().block_rank();
        g0 = rank * ngrid / G;
        g1 = (rank + 1) * ngrid / G;
        R0 = rank * N / G;
        R1 = (rank + 1) * N / G;
    }

    __shared__ int wait_ok;
    __shared__ long long t_begin;  // the clock at the candidate's start
    const long long units = a.job_start ? a.job_start[a.B] : (long long)a.B * (a.K > 0 ? a.K : 1);
    const long long m0 = (long long)blockIdx.x * a.cap;
    const long long m1 = m0 + a.cap < units ? m0 + a.cap : units;
    // candidate whose units contain x
    auto job_of = [&](long long x) -> int {
        if (!a.job_start) return (int)(x / (a.K > 0 ? a.K : 1));
        int lo = 0, hi = a.B - 1;  // largest j with job_start[j] <= x
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (a.job_start[mid] <= x) lo = mid;
            else hi = mid - 1;
        }
        return lo;
    };
    const int j_first = m0 < m1 ? job_of(m0) : 0;
    const int j_last = m0 < m1 ? job_of(m1 - 1) : -1;

    // cluster mode: cluster h takes candidates h, h + H, h + 2 H, ... whole
    const int n_holders = G > 1 ? (int)(gridDim.x / G) : 1;
    const int holder = G > 1 ? (int)(blockIdx.x / G) : 0;
    // (one loop form for both modes: a counter besides cand costs the one-CTA
    // kernel a register spill)
    for (int cand = (G == 1 ? j_last : holder); G == 1 ? cand >= j_first : cand < a.B;
         cand += (G == 1 ? -1 : n_holders)) {
        const RaggedDesc* d = a.desc ? a.desc + cand : nullptr;
        const float* __restrict__ S = a.S + (d ? d->S_off : (long long)cand * a.s_stride);
        const float* __restrict__ mu = a.mu + (d ? d->mu_off : (long long)cand * NN);
        float* Fc = a.F + (d ? d->F_off : (long long)cand * NN);
        const int Kc = d ? d->K : a.K;
        const int lidx = d ? d->out : cand;
        // this CTA's part of the candidate: iterations [it0, it1)
        const long long js = a.job_start ? a.job_start[cand] : (long long)cand * (a.K > 0 ? a.K : 1);
        const long long jl = Kc > 0 ? Kc : 1;
        const long long u0 = G > 1 ? 0 : (m0 - js > 0 ? m0 - js : 0);
        const long long u1 = G > 1 ? jl : (m1 - js < jl ? m1 - js : jl);
        const bool first = (u0 == 0), last = (u1 == jl);
        const int it0 = (int)(u0 < Kc ? u0 : Kc), it1 = (int)(u1 < Kc ? u1 : Kc);

        // ---- set-up: mu -> img0 (zero ring), img1 = 0
        if (tid == 0) t_begin = clock64();
        for (int i = tid; i < IMG; i += NT) {
            img0[i] = 0.0f;
            img1[i] = 0.0f;
        }
        __syncthreads();
        for (int i = tid; i < NN; i += NT) img0[(i / N + 1) * P + (i % N) + 1] = __ldg(mu + i);
        __syncthreads();

        // ---- system matrix (attenuation exponents) + sensitivity A^T 1
        // (loops unrolled by 8, as in the iterations below: +0.8 % measured)
        for (int gi = g0; gi < g1; ++gi) {
            const float cs = csn[2 * gi], sn = csn[2 * gi + 1];
            SchedSlots<SN, NT> sched0;  // this grid's scatter slots of class 0
            if (use_sched) sched0.load(grid_sched<N>(a, gi));
            float* Xc = tab + (gi - g0) * gstride;
            float* XrT = Xc + NN;
            float* Uc = QUAD ? Xc + 2 * NN : Xc + NN;
            float* Ur = Uc + N;
            float ps = 0.0f;
            ColumnWalk walk(k0, lb, cs, sn, c);
#pragma unroll 8
            for (int s = 0; s < SEG; ++s) {
                const float m = bilerp_pos<N, P>(img0, walk.next());
                W[(k0 + s) * WP + lb] = m;
                ps += m;
            }
            redc[seg * N + lb] = ps;
            __syncthreads();
            {   // columns: suffix sums towards k = N-1
                float after = 0.0f, total = 0.0f;
#pragma unroll
                for (int s2 = 0; s2 < NSEG; ++s2) {
                    const float v = redc[s2 * N + lb];
                    total += v;
                    if (s2 > seg) after += v;
                }
                float suf = after;
#pragma unroll 8
                for (int s = SEG - 1; s >= 0; --s) {
                    const int k = k0 + s;
                    const float m = W[k * WP + lb];
                    Xc[tab_ix(N, k, lb)] = ndl * (0.5f * m + suf);
                    suf += m;
                }
                if (seg == 0) Uc[lb] = ndl * total;
            }
            if (QUAD) {  // rows: prefix sums from b = 0
                float pr = 0.0f;
#pragma unroll 2
                for (int s4 = 0; s4 < SEG; s4 += 4) {
                    const float4 m4 = *reinterpret_cast<const float4*>(W + lb * WP + k0 + s4);
                    pr += m4.x;
                    pr += m4.y;
                    pr += m4.z;
                    pr += m4.w;
                }
                redr[seg * N + lb] = pr;
                __syncthreads();
                float before = 0.0f, total = 0.0f;
#pragma unroll
                for (int s2 = 0; s2 < NSEG; ++s2) {
                    const float v = redr[s2 * N + lb];
                    total += v;
                    if (s2 < seg) before += v;
                }
                float pre = before;
#pragma unroll 2
                for (int s4 = 0; s4 < SEG; s4 += 4) {
                    const float4 m4 = *reinterpret_cast<const float4*>(W + lb * WP + k0 + s4);
                    const float mm[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        XrT[tab_ix(N, k0 + s4 + j, lb)] = ndl * (0.5f * mm[j] + pre);
                        pre += mm[j];
                    }
                }
                if (seg == 0) Ur[lb] = ndl * total;
            }
            __syncthreads();
            {   // G = dx (sum of the grid's views' attenuation factors)
                const float uc = Uc[lb];
#pragma unroll 8
                for (int s = 0; s < SEG; ++s) {
                    const int k = k0 + s;
                    const float y = Xc[tab_ix(N, k, lb)];
                    W[k * WP + lb] = dx * (ex2(y) + ex2(uc - y));
                }
            }
            if (QUAD) {
                __syncthreads();
                const float ur = Ur[lb];
#pragma unroll 2
                for (int s4 = 0; s4 < SEG; s4 += 4) {
                    float4* w4 = reinterpret_cast<float4*>(W + lb * WP + k0 + s4);
                    const float4 y4 = *reinterpret_cast<const float4*>(XrT + tab_ix(N, k0 + s4, lb));
                    float4 v = *w4;
                    v.x += dx * (ex2(y4.x) + ex2(ur - y4.x));
                    v.y += dx * (ex2(y4.y) + ex2(ur - y4.y));
                    v.z += dx * (ex2(y4.z) + ex2(ur - y4.z));
                    v.w += dx * (ex2(y4.w) + ex2(ur - y4.w));
                    *w4 = v;
                }
            }
            __syncthreads();
            if constexpr (use_sched) scatter_scheduled<SN, NT, P, WP>(W, img1, cs, sn, c, grid_sched<N>(a, gi), sched0);
            else scatter_classes<N, NT, P, WP>(W, img1, cs, sn, c);
        }
        if (tid == 0) {  // second part of a cut candidate: wait for the first
            int ok = 1;
            if (!first) {
                const long long t0 = clock64(), limit = wait_limit(a, u0, t0 - t_begin);
                for (;;) {
                    int f;
                    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(f) : "l"(a.ready + cand) : "memory");
                    if (f) break;
                    if (clock64() - t0 > limit) {
                        ok = 0;
                        atomicExch(a.status, BOAC_ETIMEOUT);
                        break;
                    }
                    __nanosleep(256);
                }
            }
            wait_ok = ok;
        }
        __syncthreads();
        if (!wait_ok) {  // give up on this part: no F written, score NaN
            if (tid == 0 && last && a.L) a.L[lidx] = __longlong_as_double(0x7ff8000000000000LL);
            __syncthreads();
            continue;
        }
        if constexpr (G > 1) {
            // the sensitivity of this rank's rows: the ranks' partial images
            // summed in rank order
            cg::cluster_group cl = cg::this_cluster();
            cl.sync();
            for (int i = tid; i < (R1 - R0) * N; i += NT) {
                const int pi = (R0 + i / N + 1) * P + (i % N) + 1;
                sens[i] = rank_sum<G>(img1, pi);
            }
            cl.sync();
            for (int i = tid; i < NN; i += NT) img0[(i / N + 1) * P + (i % N) + 1] = Fc[i];
        } else {
            for (int i = tid; i < NN; i += NT) {
                const int pi = (i / N + 1) * P + (i % N) + 1;
                sens[i] = img1[pi];
                img0[pi] = first ? Fc[i] : __ldcg(Fc + i);  // L2: written by another SM
            }
        }
        __syncthreads();
        for (int i = tid; i < IMG; i += NT) img1[i] = 0.0f;
        __syncthreads();

        // What grid gi needs besides its schedule, ahead of its passes: its
        // sinogram rows and whole-ray exponents copied to shared memory...
        auto stage = [&](int gi) {
            for (int t = tid; t < (QUAD ? 4 * N : 2 * N); t += NT) {
                const int vi = t / N;  // views gi, gi + V/2 (columns), gi + V/4, gi + 3V/4 (rows)
                const int v = gi + (vi == 0 ? 0 : vi == 1 ? V / 2 : vi == 2 ? V / 4 : 3 * V / 4);
                copy_async4(Sg + t, S + (size_t)v * N + (t % N));
            }
            const float* U = tab + (gi - g0) * gstride + (QUAD ? 2 * NN : NN);
            for (int t = tid; t < (QUAD ? 2 * N : N); t += NT) copy_async4(Us + t, U + t);
            copy_async_commit();
        };
        // ...and its exponents in tensor memory (or, where they do not fit,
        // read by the passes)
        using Fetch = ExponentFetch<N, SEG, QUAD>;
        auto fetch = [&](int gi) { return Fetch(tab + (gi - g0) * gstride, k0, lb, stash); };
        auto prepare_now = [&](int gi) {
            stage(gi);
            if constexpr (kStashed) {
                fetch(gi).all();
                tmem_wait_st();
            }
            copy_async_wait_all();
            __syncthreads();
        };

        // ---- MLEM iterations, then one more forward pass for the score
        double lacc = 0.0;
        prepare_now(g0);
        for (int it = it0; it <= it1; ++it) {
            const bool scoring = (it == Kc);
            if (it == it1 && !(last && a.L)) break;
            for (int gi = g0; gi < g1; ++gi) {
                const float cs = csn[2 * gi], sn = csn[2 * gi + 1];
                const float* Xc = tab + (gi - g0) * gstride;
                const float* XrT = Xc + NN;
                const int gn = gi + 1 < g1 ? gi + 1 : g0;
                {   // the next grid's exponent planes are read from DRAM
                    // once per iteration: start that read now (one 128-byte
                    // line per thread, 2 n^2 floats per grid)
                    const float* nxt = tab + (gn - g0) * gstride;
                    constexpr int kLines = (int)((2 * (size_t)NN * sizeof(float) + 127) / 128);
                    for (int l = tid; l < (QUAD ? kLines : kLines / 2); l += NT) prefetch_l2(nxt + 32 * l);
                }
                // forward, column views: sample F on the grid.  (Unrolled by
                // 8 samples; the whole run at once takes 31.7 instead of 28.2
                // ms, the row pass is best unrolled by 16.)
                {
                    const float uc = Us[lb];
                    float acc1 = 0.0f, acc2 = 0.0f;
                    ColumnWalk walk(k0, lb, cs, sn, c);
#pragma unroll 2
                    for (int s4 = 0; s4 < SEG; s4 += 4) {
                        float y[4], e[8];
                        if constexpr (kStashed) {
                            tmem_ld4(stash + SEG + s4, y);
                            tmem_wait_ld(y);
                        } else {
                            plane4(Xc + tab_ix(N, k0 + s4, lb), y);
                        }
                        factors4(y, uc, e);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int k = k0 + s4 + j;
                            const float f = bilerp_pos<N, P>(img0, walk.next());
                            if (QUAD) W[k * WP + lb] = f;
                            acc1 = fmaf(e[2 * j], f, acc1);
                            acc2 = fmaf(e[2 * j + 1], f, acc2);
                        }
                        if constexpr (kStashed) tmem_st8(stash + 2 * s4, e);
                    }
                    redc[seg * N + lb] = acc1;
                    redc[(NSEG + seg) * N + lb] = acc2;
                }
                if (QUAD) {  // forward, row views: the samples back from W
                    __syncthreads();
                    const float ur = Us[N + lb];
                    float acc3 = 0.0f, acc4 = 0.0f;
#pragma unroll 4
                    for (int s4 = 0; s4 < SEG; s4 += 4) {
                        float y[4], e[8];
                        if constexpr (kStashed) tmem_ld4(stash + 3 * SEG + s4, y);
                        else plane4(XrT + tab_ix(N, k0 + s4, lb), y);
                        const float4 f4 = *reinterpret_cast<const float4*>(W + lb * WP + k0 + s4);
                        const float ff[4] = {f4.x, f4.y, f4.z, f4.w};
                        if constexpr (kStashed) tmem_wait_ld(y);
                        factors4(y, ur, e);
#pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            acc3 = fmaf(e[2 * j], ff[j], acc3);
                            acc4 = fmaf(e[2 * j + 1], ff[j], acc4);
                        }
                        if constexpr (kStashed) tmem_st8(stash + 2 * (SEG + s4), e);
                    }
                    redr[seg * N + lb] = acc3;
                    redr[(NSEG + seg) * N + lb] = acc4;
                }
                if constexpr (kStashed) tmem_wait_st();
                __syncthreads();
                // q, then r = S / q (or the Eq. 5 terms when scoring)
                for (int t = tid; t < (QUAD ? 4 * N : 2 * N); t += NT) {  // one ray per thread
                    const int j = t % N, vi = t / N;
                    const float* rp = (vi >= 2 ? redr : redc) + ((vi & 1) ? NSEG * N : 0);
                    float q = 0.0f;
#pragma unroll
                    for (int s2 = 0; s2 < NSEG; ++s2) q += rp[s2 * N + j];
                    q *= dx;
                    const float Sv = Sg[vi * N + ((vi & 1) ? N - 1 - j : j)];
                    if (scoring) lacc += loglik_term(Sv, q, a.include_lgamma && !a.lgS);
                    else rr[vi * N + j] = q > 0.0f ? Sv / q : 0.0f;
                }
                __syncthreads();
                if (scoring) {
                    prepare_now(gn);
                    continue;
                }
                stage(gn);
                SchedSlots<SN, NT> sched0;  // in flight during the weight passes
                if (use_sched) sched0.load(grid_sched<N>(a, gi));
                // back-projection weights of the grid's views, from the stashed
                // factors
                {
                    const float r1 = dx * rr[lb], r2 = dx * rr[N + lb];
                    [[maybe_unused]] const float uc = kStashed ? 0.0f : Xc[(QUAD ? 2 * NN : NN) + lb];
#pragma unroll 2
                    for (int s4 = 0; s4 < SEG; s4 += 4) {
                        float e[8];
                        if constexpr (kStashed) {
                            tmem_ld8(stash + 2 * s4, e);
                            tmem_wait_ld(e);
                        } else {
                            float y[4];
                            plane4(Xc + tab_ix(N, k0 + s4, lb), y);
                            factors4(y, uc, e);
                        }
#pragma unroll
                        for (int j = 0; j < 4; ++j) W[(k0 + s4 + j) * WP + lb] = fmaf(e[2 * j], r1, e[2 * j + 1] * r2);
                    }
                }
                if (QUAD) {
                    __syncthreads();
                    const float r3 = dx * rr[2 * N + lb], r4 = dx * rr[3 * N + lb];
                    [[maybe_unused]] const float ur = kStashed ? 0.0f : Xc[2 * NN + N + lb];
#pragma unroll 2
                    for (int s4 = 0; s4 < SEG; s4 += 4) {
                        float e[8];
                        float4* w4 = reinterpret_cast<float4*>(W + lb * WP + k0 + s4);
                        float4 v = *w4;
                        if constexpr (kStashed) {
                            tmem_ld8(stash + 2 * (SEG + s4), e);
                            tmem_wait_ld(e);
                        } else {
                            float y[4];
                            plane4(XrT + tab_ix(N, k0 + s4, lb), y);
                            factors4(y, ur, e);
                        }
                        v.x += fmaf(e[0], r3, e[1] * r4);
                        v.y += fmaf(e[2], r3, e[3] * r4);
                        v.z += fmaf(e[4], r3, e[5] * r4);
                        v.w += fmaf(e[6], r3, e[7] * r4);
                        *w4 = v;
                    }
                }
                copy_async_wait_all();
                __syncthreads();
                if constexpr (use_sched)
                    scatter_scheduled<SN, NT, P, WP, false>(W, img1, cs, sn, c, grid_sched<N>(a, gi), sched0, fetch(gn));
                else
                    scatter_classes<N, NT, P, WP>(W, img1, cs, sn, c);
                if constexpr (kStashed) tmem_wait_st();
            }
            if (scoring) break;
            if constexpr (G > 1) {
                // this rank's rows: back-projection summed over the ranks in
                // rank order, multiplicative update, written into every
                // rank's F; then the accumulator is cleared
                cg::cluster_group cl = cg::this_cluster();
                cl.sync();
                for (int i = tid; i < (R1 - R0) * N; i += NT) {
                    const int pi = (R0 + i / N + 1) * P + (i % N) + 1;
                    const float sv = sens[i];
                    const float bp = rank_sum<G>(img1, pi);
                    rank_put<G>(img0, pi, sv > 0.0f ? img0[pi] * bp / sv : 0.0f);
                }
                cl.sync();
                for (int i = tid; i < IMG; i += NT) img1[i] = 0.0f;
                __syncthreads();
            } else {
                // multiplicative update; clears the accumulator for the next pass
                for (int i = tid; i < IMG; i += NT) {
                    const int row = i / P, col = i % P;
                    if (row >= 1 && row <= N && col >= 1 && col <= N) {
                        const float sv = sens[(row - 1) * N + (col - 1)];
                        img0[i] = sv > 0.0f ? img0[i] * img1[i] / sv : 0.0f;
                    }
                    img1[i] = 0.0f;
                }
                __syncthreads();
            }
        }

        // ---- Eq. 5: deterministic block reduction of the float64 terms
        if (last && a.L) {
            for (int off = 16; off > 0; off >>= 1) lacc += __shfl_down_sync(0xffffffffu, lacc, off);
            if ((tid & 31) == 0) dred[tid >> 5] = lacc;
            __syncthreads();
            if (tid == 0) {
                double t = 0.0;
                for (int wi = 0; wi < NT / 32; ++wi) t += dred[wi];
                if constexpr (G > 1) {
                    dred[32] = t;  // this rank's terms
                } else {
                    a.L[lidx] = a.include_lgamma && a.lgS ? t - *a.lgS : t;
                    if (t == -INFINITY) atomicCAS(a.status, BOAC_OK, BOAC_ENONFINITE);
                }
            }
            if constexpr (G > 1) {  // the ranks' terms added in rank order
                cg::cluster_group cl = cg::this_cluster();
                cl.sync();
                if (rank == 0 && tid == 0) {
                    double t = 0.0;
                    for (int r = 0; r < G; ++r) t += cl.map_shared_rank(dred, r)[32];
                    a.L[lidx] = a.include_lgamma && a.lgS ? t - *a.lgS : t;
                    if (t == -INFINITY) atomicCAS(a.status, BOAC_OK, BOAC_ENONFINITE);
                }
            }
        }

        // ---- F out (F^K, or the state handed to the candidate's second part;
        // cluster mode: each rank its rows)
        for (int i = R0 * N + tid; i < R1 * N; i += NT) Fc[i] = img0[(i / N + 1) * P + (i % N) + 1];
        if constexpr (G > 1) cg::this_cluster().sync();  // no rank still reads another's memory
        __syncthreads();
        if (!last && tid == 0 && cand != a.withhold) {
            __threadfence();
            asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(a.ready + cand), "r"(1) : "memory");
        }
    }
    if constexpr (kStashed) {
        __syncthreads();
        if (tid < 32) tmem_free<kTmemCols>(tmem_addr);
    }
    class_end(a);
}

// ---------------------------------------------------------------- host side
struct FusedVariant {
    int n, nt;
    bool quad;
    int nb;  // CTAs per candidate in the band kernel's cluster (1 otherwise)
    size_t (*smem)(int V);
    const void* func;
    // what the geometry needs before the kernel: the scatter schedule (its
    // place left in a->sched) or the ray-run records
    int (*prepare)(FusedArgs* a, cudaStream_t st);
    // `holders`: CTAs (nb == 1, g == 1) or clusters that share the work
    int (*launch)(const FusedArgs& a, int holders, cudaStream_t st);
    int g;   // CTAs per candidate in the fused kernel's cluster mode (1 otherwise)
    int (*max_clusters)();  // cluster mode: clusters resident at once
    size_t image_floats;    // one-CTA kernel: F, accumulator and sample buffer of a CTA
    int tmem_cols;          // columns of tensor memory of a CTA (0: none)
};

template <int N, int NT, bool QUAD>
static int fused_prepare_t(FusedArgs* a, cudaStream_t st) {
    int s = BOAC_OK;
    if constexpr (N <= 128)
        a->sched = sched_prepare(N, a->V, QUAD ? a->V / 4 : a->V / 2, FusedShape<N, NT>::WP,
                                 const_cast<unsigned short*>(a->sched), st, &s);
    return s;
}

template <int N, int NT>
static size_t smem_of(int V) { return fused_smem_bytes<N, NT>(V); }

// The cluster-mode variants of an image side, kSplitConfigs of them (nullptr:
// none).
constexpr int kSplitConfigs = 8;
const FusedVariant* split_variants(int n);

}  // namespace boac
