// Host side of the resident-tile CG (cg_tile.cuh): plans and launches.
#pragma once

#include "cg_tile.cuh"
#include "ctx.h"

#include <vector>

namespace hmc {

// Tiles for one cooperative launch over all SMs: every tile resident, within the
// shared memory a block may use; false when there are none. real: bytes of a
// real number; slices: the kernel instances (0 ends the list) with their largest
// blocks.
bool tile_plan_grid(const hmc_ctx* c, const Geo& g, int cw, int real, const int* slices, int (*max_threads)(int, int),
                    TilePlan* out);
hmc_status tile_grid_launch(hmc_ctx* c, int id, const void* kfn, const TilePlan& p, const TileSys& system);

// The FP32 kernel instances (0 ends the list) and their largest blocks.
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

TileSys make_tile_sys(const Geo& g, const TilePlan& p, const void* ph, void* x, void* r, void* U, CGScal* sc,
                      void* gtab = nullptr);

// One launch of a batch: systems whose plans share a kernel instance and a
// cluster size (2^log2 blocks). plan: the instance, with the block and the
// shared memory of the launch; stream: the context's side stream it runs on.
struct ClusterGroup {
  int log2 = 0, stream = 0;
  TilePlan plan;
  std::vector<int> sys;        // indices into the batch, longest first
  std::vector<TilePlan> plans;  // theirs
};
// Groups for a batch of systems on the lattices geos; iters: expected
// iterations, up to a common factor. false: a lattice does not fit a cluster.
bool cg32_cluster_batch(hmc_ctx* c, const std::vector<Geo>& geos, const std::vector<double>& iters,
                        std::vector<ClusterGroup>* groups);
// Solve them all: list holds the systems in the order of the groups; ordered
// on c->stream.
hmc_status cg32_cluster_batch_launch(hmc_ctx* c, const std::vector<ClusterGroup>& groups, const TileSys* list);

}  // namespace hmc
