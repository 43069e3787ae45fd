// boac_ops.h -- the bare operators on shared sample grids (boac_ops.cu).
#pragma once

#include <cuda_runtime.h>

#include "../../include/boac.h"

namespace boac {

// Whether the geometry has these kernels (64 / 96 / 128 images, even views).
bool ops_on_grids(const boac_geom* g);
int project_on_grids(const boac_geom* g, const float* mu, const float* F, int B, float* q, cudaStream_t st);
// partial: bp_partial_floats(g, B) floats.
int backproject_on_grids(const boac_geom* g, const float* mu, const float* y, int B, float* out, float* partial,
                         cudaStream_t st);
// out[cand] = sum over shares of partial[cand][share], in order (boac_bpgroup.cu).
int sum_partial_images(int B, int shares, int nn, const float* partial, float* out, cudaStream_t st);

}  // namespace boac
