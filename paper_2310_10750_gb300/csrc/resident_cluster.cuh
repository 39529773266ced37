// The resident solve of lattices one SM cannot hold, or whose disc rows reach too far for
// resident_strip.cuh: interface of resident_cluster.cu.
#pragma once

#include "step_kernels.cuh"

namespace mfmc {

// n = 128 (one CTA a sample) with R = 5, 6 or 8, n = 256 (a cluster of four) with R = 4, 6 or 8.
constexpr bool resident_cluster_shape(int n, int R) {
    return (n == 128 && (R == 5 || R == 6 || R == 8)) || (n == 256 && (R == 4 || R == 6 || R == 8));
}
mfmc_status launch_resident_cluster(int R, const ResidentArgs &a, cudaStream_t st);

}  // namespace mfmc
