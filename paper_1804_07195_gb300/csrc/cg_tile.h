// Host side of the resident-tile CG (cg_tile.cuh): plans and launches.
#pragma once

#include "cg_tile.cuh"
#include "ctx.h"

namespace hmc {

// Tiles for one cooperative launch: every tile resident, within the shared
// memory a block may use. Among the plans that fit, the one with the fewest
// cells per tile, then the fewest padding rows and slices per cell.
template <typename R>
bool tile_plan_grid(const hmc_ctx* c, const Geo& g, int cw, TilePlan* out);
// Tiles for one cluster of cs blocks (cs = 1, 2, 4, 8 or 16).
template <typename R>
bool tile_plan_cluster(const hmc_ctx* c, const Geo& g, int cw, int cs, TilePlan* out);

TileSys make_tile_sys(const Geo& g, const TilePlan& p, const void* ph, void* x, void* r, void* U, CGScal* sc);

}  // namespace hmc
