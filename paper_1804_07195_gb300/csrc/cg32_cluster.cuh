// The kernel of cg32_cluster.cu: its instances for single systems and for batches
// are two translation units.
#pragma once

#include "cg_tile.h"

namespace hmc {

// Bytes between the padded arrays: the small one leaves room for several
// blocks on an SM.
constexpr int kStrideSmall = 12 * 1024, kStrideLarge = 44 * 1024;

// BATCH: a list of systems, one cluster each, with wide scalars; otherwise `one`.
template <int CW, int S, int AS, bool BATCH>
__global__ void __launch_bounds__(tile_max_threads<float, CW, S>(), 1)
    k_cg32_cluster(const TileSys* __restrict__ list, const __grid_constant__ TileSys one, unsigned extra, long long limit) {
  extern __shared__ float4 s_tile[];
  __shared__ TileSys ts;
  static_assert(sizeof(TileSys) % 4 == 0, "copied by words");
  const unsigned* src = BATCH ? (const unsigned*)(list + blockIdx.x / cluster_size()) : (const unsigned*)&one;
  for (unsigned i = threadIdx.x; i < sizeof(TileSys) / 4; i += blockDim.x) ((unsigned*)&ts)[i] = src[i];
  __syncthreads();
  cg_tile_solve<float, CW, S, true, AS, false, BATCH>(ts, GridSync{nullptr, nullptr, nullptr, extra, limit},
                                                      (int)cluster_rank(), (char*)s_tile);
}

template <bool BATCH>
const void* cluster_kernel_of(const TilePlan& p) {
#define HMC_CASE(cw_, s_)                                                                       \
  if (p.cw == cw_ && p.S == s_)                                                                 \
    return p.stride == kStrideSmall ? (const void*)k_cg32_cluster<cw_, s_, kStrideSmall, BATCH> \
                                    : (const void*)k_cg32_cluster<cw_, s_, kStrideLarge, BATCH>;
  HMC_CASE(1, 1) HMC_CASE(1, 2) HMC_CASE(1, 4) HMC_CASE(1, 8) HMC_CASE(1, 8 + kXInMemory)
  HMC_CASE(2, 1) HMC_CASE(2, 2) HMC_CASE(2, 4) HMC_CASE(2, 4 + kXInMemory)
#undef HMC_CASE
  return nullptr;
}

const void* cluster_kernel_batch(const TilePlan& p);

}  // namespace hmc
