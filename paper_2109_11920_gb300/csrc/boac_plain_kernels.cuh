// boac_plain_kernels.cuh -- the unfused kernels of boac_plain.cu, declared
// for reuse by the gradient path (boac_grad.cu).  All are batched over
// candidates (grid z or y) and documented at their definitions.
#pragma once

#include <cuda_runtime.h>

#include "boac_internal.h"

namespace boac {

constexpr int kRayThreads = 128;   // ray kernels: one thread per (candidate, view, bin)
constexpr int kPixThreads = 256;   // pixel kernels: one thread per (candidate, pixel)

__global__ void attenuation_table_kernel(int n, int V, float dx, const float* __restrict__ mu,
                                         float* __restrict__ tab);
__global__ void project_otf_kernel(int n, int V, float dx, const float* __restrict__ mu,
                                   const float* __restrict__ F, float* __restrict__ q);
__global__ void project_table_kernel(int n, int V, float dx, const float* __restrict__ tab,
                                     const float* __restrict__ F, float* __restrict__ q);
// The same with their images in shared memory where those fit (same bits).
void attenuation_table(const boac_geom* g, int B, const float* mu, float* tab, cudaStream_t st);
void project_rays(const boac_geom* g, int B, const float* mu, const float* F, float* q, cudaStream_t st);
void project_table_rays(const boac_geom* g, int B, float dx, const float* tab, const float* F, float* q,
                        cudaStream_t st);
// out[cand] (+)= scale sum_v B_v^T (tab_v y_v), per-pixel gather (boac_plain.cu).
void backproject_gather(int n, int V, int B, float scale, const float* tab, const float* y, float* out,
                        int accumulate, cudaStream_t st);
__global__ void ratio_kernel(int count, const float* __restrict__ S, const float* __restrict__ q,
                             float* __restrict__ r);
__global__ void update_kernel(int count, float* __restrict__ F, const float* __restrict__ bp,
                              const float* __restrict__ sens);
// status (nullable): set to BOAC_ENONFINITE (unless already non-zero) when
// a candidate's score is -inf (q = 0 on a bin with S > 0).
__global__ void loglik_kernel(int nbin, const float* __restrict__ q, const float* __restrict__ S,
                              long long s_stride, int include_lgamma, double* __restrict__ L,
                              const double* __restrict__ lgS, int* status = nullptr);
// Launch it for B candidates, on clusters where that is faster (same bits).
// (The launchers below read, and so clear, the CUDA error: the status they
// return is the only report of a refused launch.)
[[nodiscard]] int loglik_launch(int nbin, int B, const float* q, const float* S, long long s_stride, int include_lgamma,
                                double* L, const double* lgS, int* status, cudaStream_t st);
// sum_i lgamma(S_i + 1) of one sinogram S[nbin] into scratch[0]
// (scratch: kLgammaScratchDoubles doubles, 8-byte aligned); returns scratch.
constexpr int kLgammaScratchDoubles = 31;
const double* lgamma_sum(int nbin, const float* S, double* scratch, cudaStream_t st);
// r = S / q over B candidates (0 where q <= 0), S rows s_stride apart (boac_grad.cu).
__global__ void ratio_batched_kernel(int B, int nbin, const float* __restrict__ S, long long s_stride,
                                     const float* __restrict__ q, float* __restrict__ r);

dim3 ray_grid(const boac_geom* g, int B);
int grid_1d(long long count, int threads);

// out[cand] (+)= scale * sum_v B_v^T (tab_v * y_v) for B candidates from an
// attenuation table [B][V][n][n] (boac_bpgroup.cu): grouped shared-memory
// scatter with per-grid partial images in `partial` (bp_partial_floats(g, B)
// floats), or the per-pixel gather where the geometry has no grouped kernel
// (then `partial` may be null).
size_t bp_partial_floats(const boac_geom* g, int B);
// q[cand][v][bin] = dx * sum_k tab_v[k][bin] F(sample (k, bin) of view v) for
// B candidates (boac_bpgroup.cu): one CTA per candidate and sample grid with
// F in shared memory, or one thread per ray where no grouped kernel exists.
[[nodiscard]] int project_table(const boac_geom* g, int B, const float* tab, const float* F, float dx, float* q,
                                cudaStream_t st);
// One whole MLEM iteration F <- F A^T(S / A F) / sens from the table, for
// geometries with grouped kernels (mlem_grouped): two launches, `partial` as
// above, sched from mlem_group_sched (nullptr where none is kept).
bool mlem_grouped(const boac_geom* g);
const unsigned short* mlem_group_sched(const boac_geom* g, cudaStream_t st, int* status);
[[nodiscard]] int mlem_group_iteration(const boac_geom* g, int B, float dx, const float* tab, const float* S,
                                       long long s_stride, float* F, const float* sens, const unsigned short* sched,
                                       float* partial, cudaStream_t st);
[[nodiscard]] int backproject_table(const boac_geom* g, int B, const float* tab, const float* y, float scale, float* out,
                                    int accumulate, float* partial, cudaStream_t st);

}  // namespace boac
