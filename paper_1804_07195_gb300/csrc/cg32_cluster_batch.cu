// The batched instances of the FP32 CG on thread block clusters (cg32_cluster.cuh).
#include "cg32_cluster.cuh"

namespace hmc {

const void* cluster_kernel_batch(const TilePlan& p) { return cluster_kernel_of<true>(p); }

}  // namespace hmc
