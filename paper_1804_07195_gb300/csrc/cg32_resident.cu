// Resident-tile CG over all SMs, one cooperative launch per solve (cg_tile.cuh):
// plans, kernel instances and launches, FP32 (the inner solver of Section 3 and
// Algorithm A.1).
#include <algorithm>
#include <cstdint>

#include "cg_tile.h"
#include "launch.cuh"

namespace hmc {

// One cell per column, and two (n even: 16-byte complex64 pairs).
template <int S>
__global__ void __launch_bounds__(tile_max_threads<float, 1, S>(), 1) k_cg32_resident(TileSys ts, GridSync gs) {
  extern __shared__ float4 s_tile[];
  cg_tile_solve<float, 1, S, false, kTileStride>(ts, gs, blockIdx.x, (char*)s_tile);
}
template <int S>
__global__ void __launch_bounds__(tile_max_threads<float, 2, S>(), 1) k_cg32_resident2(TileSys ts, GridSync gs) {
  extern __shared__ float4 s_tile[];
  cg_tile_solve<float, 2, S, false, kTileStride>(ts, gs, blockIdx.x, (char*)s_tile);
}

// Lattices whose tiles leave no room for the padding's table: arrays up to the whole
// of shared memory, the table in global memory, where a thread's own entries cost it a
// trip to L2 twice an iteration. (us per iteration, in brackets the best of the designs
// that run it from L2: 106x106x64 13.3, 108x108x64 16.4 (19.6), 110x110x64 16.7 (20.1),
// 99x99x64 16.7 (17.5), 105x105x64 16.9 (19.1). Pairs in columns of eight slices are the
// slowest: 352 threads; single cells in 672 threads take 16.8 at 108x108x64.)
constexpr int kStrideAll = 57856;
template <int CW, int S>
__global__ void __launch_bounds__(tile_max_threads<float, CW, S>(), 1) k_cg32_resident_large(TileSys ts, GridSync gs) {
  extern __shared__ float4 s_tile[];
  cg_tile_solve<float, CW, S, false, kStrideAll, true>(ts, gs, blockIdx.x, (char*)s_tile);
}

const int* tile_slices32(int cw) {
  static const int one[] = {1, 2, 4, 4 + kXInMemory, 8, 8 + kXInMemory, 0}, two[] = {1, 2, 2 + kXInMemory, 4, 4 + kXInMemory, 0};
  return cw == 2 ? two : one;
}

int max_threads32(int cw, int S) {
  if (cw == 1) switch (S) {
      case 1: return tile_max_threads<float, 1, 1>();
      case 2: return tile_max_threads<float, 1, 2>();
      case 4: return tile_max_threads<float, 1, 4>();
      case 4 + kXInMemory: return tile_max_threads<float, 1, 4 + kXInMemory>();
      case 8: return tile_max_threads<float, 1, 8>();
      case 8 + kXInMemory: return tile_max_threads<float, 1, 8 + kXInMemory>();
    }
  switch (S) {
    case 1: return tile_max_threads<float, 2, 1>();
    case 2: return tile_max_threads<float, 2, 2>();
    case 2 + kXInMemory: return tile_max_threads<float, 2, 2 + kXInMemory>();
    case 4: return tile_max_threads<float, 2, 4>();
    case 4 + kXInMemory: return tile_max_threads<float, 2, 4 + kXInMemory>();
  }
  return 0;
}

static size_t smem_cap(const hmc_ctx* c, size_t statics) {
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
  return optin > (int)statics ? (size_t)optin - statics : 0;
}

bool tile_plan_grid(const hmc_ctx* c, const Geo& g, int cw, int real, const int* slices, int (*max_threads)(int, int),
                    TilePlan* out) {
  if (g.n % cw) return false;
  const size_t cap = smem_cap(c, real == 8 ? 7168 : 2048);  // static arrays and the driver's 1 KB
  constexpr size_t AS = kTileStride;
  const int nq = g.n / cw;
  bool found = false;
  double best = 0.0;
  for (const int* S = slices; *S; ++S)
    for (int nseg = 1, fits = 1; fits && (nseg - 1) * tile_slices(*S) < g.nt; ++nseg)
      for (int J = 1; J <= g.m; ++J) {
        TilePlan p;
        p.cw = cw;
        p.S = *S;
        p.nseg = nseg;
        p.J = J;
        p.T = nseg * tile_slices(*S);
        p.tiles_j = (g.m + J - 1) / J;
        p.tiles_t = (g.nt + p.T - 1) / p.T;
        const size_t one = (size_t)(p.T + 1) * (J + 1) * g.n * 2 * real;
        const long long th = ((long long)nq * J * nseg + 31) / 32 * 32;
        const size_t table = (size_t)2 * (p.T + J) * nq * sizeof(uint2);
        if (one > AS || 3 * AS + one + table > cap || th > max_threads(cw, *S)) {
          fits = J > 1;  // larger J, and for J = 1 larger nseg, only grow them
          break;
        }
        if ((long long)p.tiles_j * p.tiles_t > std::min(c->nsm, kTileMaxGroup)) continue;
        p.threads = (int)th;
        p.tab = (int)(3 * AS + one);
        p.smem = p.tab + table;
        // the work of the largest tile: its cells, the padding it exchanges (about
        // a third of a cell's work each), a little for every slice of a column
        // (fewer, longer columns overlap less)
        const int Tmax = std::min(p.T, g.nt);
        const double cost = (double)J * Tmax * nq + 0.7 * (J + Tmax) * nq + 8.0 * tile_slices(*S);
        if (!found || cost < best) {
          found = true;
          best = cost;
          *out = p;
        }
      }
  return found;
}

TileSys make_tile_sys(const Geo& g, const TilePlan& p, const void* ph, void* x, void* r, void* U, CGScal* sc, void* gtab) {
  TileSys ts;
  ts.g = g;
  ts.J = p.J;
  ts.T = p.T;
  ts.tiles_j = p.tiles_j;
  ts.tiles_t = p.tiles_t;
  ts.nseg = p.nseg;
  ts.tab = p.tab;
  ts.rp = p.rp;
  ts.fq = make_fastdiv((uint32_t)(g.n / p.cw));
  ts.ph = ph;
  ts.x = x;
  ts.r = r;
  ts.U = U;
  ts.gtab = (uint2*)gtab;
  ts.sc = sc;
  return ts;
}

static const void* grid_kernel32(int cw, int S) {
  if (cw == 1) switch (S) {
      case 1: return (const void*)k_cg32_resident<1>;
      case 2: return (const void*)k_cg32_resident<2>;
      case 4: return (const void*)k_cg32_resident<4>;
      case 4 + kXInMemory: return (const void*)k_cg32_resident<4 + kXInMemory>;
      case 8: return (const void*)k_cg32_resident<8>;
      case 8 + kXInMemory: return (const void*)k_cg32_resident<8 + kXInMemory>;
    }
  switch (S) {
    case 1: return (const void*)k_cg32_resident2<1>;
    case 2: return (const void*)k_cg32_resident2<2>;
    case 2 + kXInMemory: return (const void*)k_cg32_resident2<2 + kXInMemory>;
    case 4: return (const void*)k_cg32_resident2<4>;
    case 4 + kXInMemory: return (const void*)k_cg32_resident2<4 + kXInMemory>;
  }
  return nullptr;
}

// The partials, the arrival word and the error mark of the exchanges, kept
// with the context. A launch leaves the word with all low bits zero, so it is
// cleared only when new and after a solve whose wait gave up.
static hmc_status grid_sync(hmc_ctx* c, int blocks, GridSync* gs) {
  const size_t bytes = sizeof(double) * 2 * kTileMaxGroup + 256;
  if (!c->tile_sync) {
    HMC_CUDA(c, cudaMalloc(&c->tile_sync, bytes));
    c->tile_sync_stale = true;
  }
  if (c->tile_sync_stale) HMC_CUDA(c, cudaMemsetAsync(c->tile_sync, 0, bytes, c->stream));
  c->tile_sync_stale = false;
  gs->part = (double*)c->tile_sync;
  gs->word = (unsigned*)(gs->part + 2 * kTileMaxGroup);
  gs->err = (int*)(gs->word + 32);
  gs->need = (unsigned)blocks + (unsigned)c->bar_extra;
  gs->limit = c->bar_limit > 0 ? c->bar_limit : 2000000000LL;
  return HMC_OK;
}

hmc_status tile_grid_launch(hmc_ctx* c, int id, const void* kfn, const TilePlan& p, const TileSys& system) {
  if (!tile_allow_smem(c, kfn)) return fail(c, HMC_ERR_CUDA, "resident CG shared memory");
  const int blocks = p.tiles_j * p.tiles_t;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kfn, p.threads, p.smem) != cudaSuccess ||
      (long long)occ * c->nsm < blocks) {
    cudaGetLastError();
    return fail(c, HMC_ERR_INVALID, "resident CG tiles cannot all be resident");
  }
  TileSys ts = system;
  GridSync gs;
  HMC_TRY(grid_sync(c, blocks, &gs));
  void* args[] = {&ts, &gs};
  cudaError_t le = cudaSuccess;
  HMC_TRY(launch_b(c, id, 0.0, [&] {
    le = cudaLaunchCooperativeKernel(kfn, dim3(blocks), dim3(p.threads), args, p.smem, c->stream);
  }));
  return le == cudaSuccess ? HMC_OK : cuda_fail(c, le, "resident CG launch");
}

// The context's plan for its lattice with cw cells per column, searched once.
static const TilePlan* plan32(hmc_ctx* c, const Geo& g, int cw) {
  TilePlan& p = c->tile_plan32[cw - 1];
  if (p.cw == 0 && !tile_plan_grid(c, g, cw, sizeof(float), tile_slices32(cw), max_threads32, &p)) p.cw = -1;
  return p.cw > 0 ? &p : nullptr;
}

// The same for lattices that plan32 finds no tiles for. T need not be a multiple
// of the slices a column has. table: bytes of global memory at hand for the table.
static const int* slices_large(int cw) {
  static const int one[] = {8 + kXInMemory, 0}, two[] = {4 + kXInMemory, 8 + kXInMemory, 0};
  return cw == 2 ? two : one;
}
static int max_threads_large(int cw, int S) {
  if (cw == 1) return tile_max_threads<float, 1, 8 + kXInMemory>();
  return S == 4 + kXInMemory ? tile_max_threads<float, 2, 4 + kXInMemory>() : tile_max_threads<float, 2, 8 + kXInMemory>();
}
static const void* kernel_large(int cw, int S) {
  if (cw == 1) return (const void*)k_cg32_resident_large<1, 8 + kXInMemory>;
  return S == 4 + kXInMemory ? (const void*)k_cg32_resident_large<2, 4 + kXInMemory>
                             : (const void*)k_cg32_resident_large<2, 8 + kXInMemory>;
}
static bool plan_large(const hmc_ctx* c, const Geo& g, int cw, TilePlan* out) {
  if (g.n % cw) return false;
  const size_t cap = smem_cap(c, 1024), table = sizeof(float2) * (size_t)g.N;
  const int nq = g.n / cw;
  bool found = false;
  double best = 0.0;
  for (const int* S = slices_large(cw); *S; ++S)
    for (int T = 1; T <= g.nt && (size_t)(T + 1) * 2 * g.n * sizeof(float2) <= (size_t)kStrideAll; ++T)
      for (int J = 1; J <= g.m; ++J) {
        TilePlan p;
        p.cw = cw;
        p.S = *S;
        p.J = J;
        p.T = T;
        p.nseg = (T + tile_slices(*S) - 1) / tile_slices(*S);
        p.tiles_j = (g.m + J - 1) / J;
        p.tiles_t = (g.nt + T - 1) / T;
        p.stride = kStrideAll;
        const size_t one = (size_t)(T + 1) * (J + 1) * g.n * sizeof(float2);
        const long long th = ((long long)nq * J * p.nseg + 31) / 32 * 32;
        p.smem = 3 * (size_t)kStrideAll + one;
        if (one > (size_t)kStrideAll || p.smem > cap || th > max_threads_large(cw, *S)) break;
        const long long tiles = (long long)p.tiles_j * p.tiles_t;
        if (tiles > std::min(c->nsm, kTileMaxGroup) || tiles * 2 * (T + J) * nq * sizeof(uint2) > table) continue;
        p.threads = (int)th;
        const double cost = (double)J * T * nq + 0.7 * (J + T) * nq + 8.0 * tile_slices(*S);
        if (!found || cost < best) {
          found = true;
          best = cost;
          *out = p;
        }
      }
  return found;
}
static const TilePlan* plan32_large(hmc_ctx* c, const Geo& g, int cw) {
  TilePlan& p = c->tile_plan32_large[cw - 1];
  if (p.cw == 0 && !plan_large(c, g, cw, &p)) p.cw = -1;
  return p.cw > 0 ? &p : nullptr;
}

// two cells per column where n is even and every vector is 16-byte aligned
static const TilePlan* pick32(hmc_ctx* c, const Geo& g, bool aligned) {
  const TilePlan* p = aligned ? plan32(c, g, 2) : nullptr;
  if (!p) p = plan32(c, g, 1);
  if (!p && aligned) p = plan32_large(c, g, 2);
  return p ? p : plan32_large(c, g, 1);
}

bool cg32_resident_ok(hmc_ctx* c, const Geo& g) { return pick32(c, g, true) != nullptr; }

bool cg32_prefer_cluster(hmc_ctx* c, const Geo& g) {
  if (!cg32_cluster_ok(c, g)) return false;
  const TilePlan* p = pick32(c, g, true);
  if (!p) return true;
  // us per iteration over all SMs: two exchanges through L2, phase latency, work
  // (measured: 5.6 at 36x36x64, 7.95 at 72x72x64; 5.6 to 6.8 below 100,000 sites);
  // cluster_us has the cluster's. The line between them runs near 70,000 sites
  // (measured: 24x24x48 4.2 us on a cluster, 5.9 over all SMs; 25x25x48 7.2, 5.7;
  // 36x36x32 5.6, 5.6; 30x30x64 6.7, 5.6)
  const double cols = (double)p->J * std::min(p->T, g.nt) * (g.n / p->cw) * (p->cw == 2 ? 1.0 : 0.75);
  return c->cluster_us < 5.2 + 2.6e-3 * cols;
}

hmc_status cg32_resident_launch(hmc_ctx* c, const Geo& g, float2* x, float2* r, float2* u, float2* spare, CGScal* sc) {
  auto al16 = [](const void* v) { return ((uintptr_t)v & 15u) == 0; };
  const TilePlan* pp = pick32(c, g, al16(x) && al16(r) && al16(u));
  if (!pp) return fail(c, HMC_ERR_INVALID, "resident CG tiles do not fit on chip");
  const TilePlan& p = *pp;
  const void* kfn = p.stride == kStrideAll ? kernel_large(p.cw, p.S) : grid_kernel32(p.cw, p.S);
  const TileSys ts = make_tile_sys(g, p, phase_of<float>(c).phi, x, r, u, sc, spare);
  HMC_TRY(tile_grid_launch(c, K_CG_RES32, kfn, p, ts));
  c->shape[K_CG_RES32].tiled = p.cw == 2 ? 4 : 0;  // reported as the design
  c->shape[K_CG_RES32].waves = p.tiles_j * p.tiles_t;
  return HMC_OK;
}

}  // namespace hmc
