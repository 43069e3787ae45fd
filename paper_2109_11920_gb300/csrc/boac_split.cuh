// boac_split.cuh -- launches of the fused MLEM kernel's cluster mode, for the
// translation units that instantiate it.
#pragma once

#include "boac_fused_kernel.cuh"

namespace boac {

// Cluster-mode launches: dynamic shared memory and (16 CTAs) the
// non-portable cluster size allowed once per device, then the kernel on
// `clusters` clusters of G CTAs.
template <int N, int NT, int G>
static int split_attrs() {
    constexpr int kDev = 64;
    static bool done[kDev];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDev) return launch_status();
    if (!done[dev]) {
        if (cudaFuncSetAttribute(mlem_fused_kernel<N, NT, true, G>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)fused_smem_bytes<N, NT>(kMaxViews)) != cudaSuccess)
            return launch_status();
        if (G > 8 && cudaFuncSetAttribute(mlem_fused_kernel<N, NT, true, G>,
                                          cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return launch_status();
        done[dev] = true;
    }
    return BOAC_OK;
}

template <int N, int NT, int G>
static cudaLaunchConfig_t split_config(int clusters, int V, cudaStream_t st, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = G;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(clusters * G), 1, 1);
    cfg.blockDim = dim3(NT, 1, 1);
    cfg.dynamicSmemBytes = fused_smem_bytes<N, NT>(V);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

template <int N, int NT, int G>
static int split_max_clusters_t() {
    constexpr int kDev = 64;
    static int cached[kDev];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDev) {
        cudaGetLastError();
        return 0;
    }
    if (cached[dev]) return cached[dev];
    if (split_attrs<N, NT, G>() != BOAC_OK) {
        cudaGetLastError();
        return 0;
    }
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = split_config<N, NT, G>(64, kMaxViews, nullptr, attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, mlem_fused_kernel<N, NT, true, G>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    cached[dev] = n;
    return n;
}

template <int N, int NT, int G>
static int split_launch_t(const FusedArgs& a, int clusters, cudaStream_t st) {
    int s = split_attrs<N, NT, G>();
    if (s != BOAC_OK) return s;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = split_config<N, NT, G>(clusters, a.V, st, attr);
    overlap_attribute(&attr[1], a);
    cfg.numAttrs = 2;
    if (cudaLaunchKernelEx(&cfg, mlem_fused_kernel<N, NT, true, G>, a) != cudaSuccess) return launch_status();
    return launch_status();
}

template <int N, int G>
static FusedVariant make_split_variant() {
    return FusedVariant{N, 8 * N, true, 1, smem_of<N, 8 * N>, (const void*)mlem_fused_kernel<N, 8 * N, true, G>,
                        fused_prepare_t<N, 8 * N, true>, split_launch_t<N, 8 * N, G>, G, split_max_clusters_t<N, 8 * N, G>,
                        fused_image_floats<N, 8 * N>(), fused_tmem_columns<N, 8 * N, true>()};
}

// The cluster sizes of split_variants (configuration ids 9 ..).
#define BOAC_SPLIT(NV)                                                                        \
    make_split_variant<NV, 2>(), make_split_variant<NV, 3>(), make_split_variant<NV, 4>(),  \
        make_split_variant<NV, 6>(), make_split_variant<NV, 8>(), make_split_variant<NV, 9>(), \
        make_split_variant<NV, 12>(), make_split_variant<NV, 16>()

}  // namespace boac
