// Resident-tile CG over all SMs in FP64, one cooperative launch per solve
// (cg_tile.cuh): the plain FP64 CG of Section 3 on lattices whose tiles fit the
// chip (up to about 500,000 sites).
#include "cg_tile.h"
#include "launch.cuh"

namespace hmc {

template <int S>
__global__ void __launch_bounds__(tile_max_threads<double, 1, S>(), 1) k_cg64_resident(TileSys ts, GridSync gs) {
  extern __shared__ float4 s_tile[];
  cg_tile_solve<double, 1, S, false, kTileStride>(ts, gs, blockIdx.x, (char*)s_tile);
}

static const int kSlices64[] = {1, 2, 4 + kXInMemory, 0};
static int max_threads64(int, int S) {
  switch (S) {
    case 1: return tile_max_threads<double, 1, 1>();
    case 2: return tile_max_threads<double, 1, 2>();
    case 4 + kXInMemory: return tile_max_threads<double, 1, 4 + kXInMemory>();
  }
  return 0;
}
static const void* kernel64(int S) {
  switch (S) {
    case 1: return (const void*)k_cg64_resident<1>;
    case 2: return (const void*)k_cg64_resident<2>;
    case 4 + kXInMemory: return (const void*)k_cg64_resident<4 + kXInMemory>;
  }
  return nullptr;
}

bool cg64_resident_ok(hmc_ctx* c, const Geo& g) {
  TilePlan& p = c->tile_plan64;
  if (p.cw == 0 && !tile_plan_grid(c, g, 1, sizeof(double), kSlices64, max_threads64, &p)) p.cw = -1;
  return p.cw > 0;
}

hmc_status cg64_resident_launch(hmc_ctx* c, const Geo& g, double2* x, double2* r, double2* u, CGScal* sc) {
  if (!cg64_resident_ok(c, g)) return fail(c, HMC_ERR_INVALID, "resident CG tiles do not fit on chip");
  const TilePlan& p = c->tile_plan64;
  const TileSys ts = make_tile_sys(g, p, phase_of<double>(c).E, x, r, u, sc);
  return tile_grid_launch(c, K_CG_RES64, kernel64(p.S), p, ts);
}

}  // namespace hmc
