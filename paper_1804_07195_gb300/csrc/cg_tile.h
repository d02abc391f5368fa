// Host side of the resident-tile CG (cg_tile.cuh): plans and launches.
#pragma once

#include "cg_tile.cuh"
#include "ctx.h"

namespace hmc {

// Slices per column of the FP32 kernel instances (0 ends the list) and their
// largest blocks.
const int* tile_slices32(int cw);
int max_threads32(int cw, int S);

// Lets kernel k use all the shared memory a block may have (the same value for
// every caller, so that plans of different lattices do not undo each other's).
inline bool tile_allow_smem(const hmc_ctx* c, const void* k) {
  int optin = 0;
  cudaFuncAttributes a;
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device) == cudaSuccess &&
      cudaFuncGetAttributes(&a, k) == cudaSuccess &&
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)a.sharedSizeBytes) == cudaSuccess)
    return true;
  cudaGetLastError();
  return false;
}

TileSys make_tile_sys(const Geo& g, const TilePlan& p, const void* ph, void* x, void* r, void* U, CGScal* sc);

}  // namespace hmc
