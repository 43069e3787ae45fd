// boac_split.cu -- the fused MLEM kernel's cluster mode (boac_fused.cu: G > 1,
// a thread-block cluster of G CTAs per candidate, each on its share of the
// sample grids), instantiated here and handed to boac_fused.cu as a table.
#include <cuda_runtime.h>

#include "boac_split.cuh"

namespace boac {

const FusedVariant* split_variants(int n) {
    static const FusedVariant t64[kSplitConfigs] = {BOAC_SPLIT(64)};
    static const FusedVariant t96[kSplitConfigs] = {BOAC_SPLIT(96)};
    static const FusedVariant t128[kSplitConfigs] = {BOAC_SPLIT(128)};
    return n == 64 ? t64 : n == 96 ? t96 : n == 128 ? t128 : nullptr;
}

#ifdef BOAC_CHECKED
BOAC_FAULT_READER(bounds_faults_split)
#endif

}  // namespace boac
