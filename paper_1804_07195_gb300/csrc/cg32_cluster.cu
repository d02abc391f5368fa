// Resident-tile FP32 CG on thread block clusters (cg_tile.cuh): one cluster
// solves one system, so a launch can hold any number of independent systems
// and none waits for another. Plans, kernel instances and launches.
//
// An exchange inside a cluster is a round of stores into the other blocks'
// shared memory and one cluster barrier: 0.65 us over 4 blocks, 0.75 over 8,
// 1.0 over 16 (128 threads a block), against 2.0 us between blocks that meet in
// L2; but the work is spread over 16 SMs at most.
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "cg_tile.h"
#include "launch.cuh"

namespace hmc {

// Bytes between the padded arrays: the small one leaves room for several
// blocks on an SM.
constexpr int kStrideSmall = 12 * 1024, kStrideLarge = 44 * 1024;

template <int CW, int S, int AS>
__global__ void __launch_bounds__(tile_max_threads<float, CW, S>(), 1)
    k_cg32_cluster(const TileSys* __restrict__ list, const __grid_constant__ TileSys one) {
  extern __shared__ float4 s_tile[];
  __shared__ TileSys ts;
  static_assert(sizeof(TileSys) % 4 == 0, "copied by words");
  const unsigned* src = list ? (const unsigned*)(list + blockIdx.x / cluster_size()) : (const unsigned*)&one;
  for (unsigned i = threadIdx.x; i < sizeof(TileSys) / 4; i += blockDim.x) ((unsigned*)&ts)[i] = src[i];
  __syncthreads();
  cg_tile_solve<float, CW, S, true, AS>(ts, GridSync{}, (int)cluster_rank(), (char*)s_tile);
}

static const void* cluster_kernel32(const TilePlan& p) {
#define HMC_CASE(cw_, s_)                                                          \
  if (p.cw == cw_ && p.S == s_)                                                    \
    return p.stride == kStrideSmall ? (const void*)k_cg32_cluster<cw_, s_, kStrideSmall> \
                                    : (const void*)k_cg32_cluster<cw_, s_, kStrideLarge>;
  HMC_CASE(1, 1) HMC_CASE(1, 2) HMC_CASE(1, 4) HMC_CASE(1, 8)
  HMC_CASE(2, 1) HMC_CASE(2, 2) HMC_CASE(2, 4)
#undef HMC_CASE
  return nullptr;
}

// us per iteration of a system on a cluster of cs blocks, from the size of its
// largest tile (pairs of cells; one cell per column counts 0.75): fixed phase
// latency, two exchanges, work. Fitted to measured iterations (6x6x16 2.7,
// 12x12x32 2.9, 18x18x48 3.9, 24x24x48 4.5 us); it only ranks the choices.
static double cluster_us(const TilePlan& p, const Geo& g, int cs) {
  const double exch = cs == 1 ? 0.35 : cs == 2 ? 0.6 : cs == 4 ? 0.7 : cs == 8 ? 0.85 : 1.15;
  const double cols = (double)p.J * std::min(p.T, g.nt) * (g.n / p.cw) * (p.cw == 2 ? 1.0 : 0.75);
  return 0.8 + 2.0 * exch + 1.9e-3 * cols;
}

// Tiles of one system for a cluster of cs blocks (cs a power of two): the split
// into rows and slices with the smallest largest tile, then the least padding.
static bool plan_cluster(const hmc_ctx* c, const Geo& g, int cs, TilePlan* out) {
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device);
  // static arrays (partials, the system) and the driver's 1 KB
  const long long cap = (long long)optin - (2 * kTileMaxCluster * kTileMaxWarps * (long long)sizeof(float2) + 2048);
  const int cw = g.n % 2 == 0 ? 2 : 1, nq = g.n / cw;
  const size_t VB = sizeof(float2) * cw;
  bool found = false;
  double best = 0.0;
  for (int tj = 1; tj <= cs; tj *= 2) {
    const int J = (g.m + tj - 1) / tj, T0 = (g.nt + cs / tj - 1) / (cs / tj);
    for (const int* S = tile_slices32(cw); *S; ++S) {
      TilePlan p;
      p.cw = cw;
      p.S = *S;
      p.J = J;
      p.nseg = (T0 + *S - 1) / *S;
      p.T = p.nseg * *S;
      const long long th = ((long long)nq * J * p.nseg + 31) / 32 * 32;
      if (th > max_threads32(cw, *S)) continue;
      const long long one = (long long)(p.T + 1) * (J + 1) * nq * (long long)VB;
      const long long cols = 2LL * (p.T + J) * nq;
      if (one > kStrideLarge) continue;
      p.stride = one <= kStrideSmall ? kStrideSmall : kStrideLarge;
      const long long tab = 3LL * p.stride + one, rp = (tab + cols * (long long)sizeof(uint2) + 15) / 16 * 16;
      const long long smem = rp + cols * (long long)VB;
      if (smem > cap) continue;
      p.tiles_j = (g.m + J - 1) / J;
      p.tiles_t = (g.nt + p.T - 1) / p.T;
      if (p.tiles_j * p.tiles_t > cs) continue;
      p.threads = (int)th;
      p.tab = (int)tab;
      p.rp = (int)rp;
      p.smem = (size_t)smem;
      const double cost = (double)J * p.T + 0.7 * (J + p.T);
      if (!found || cost < best) {
        found = true;
        best = cost;
        *out = p;
      }
      break;  // more slices per column would only leave fewer threads
    }
  }
  return found;
}

static void cluster_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, const TilePlan& p, int cs, int nsys,
                           cudaStream_t s) {
  *cfg = {};
  cfg->gridDim = dim3((unsigned)(cs * nsys));
  cfg->blockDim = dim3((unsigned)p.threads);
  cfg->dynamicSmemBytes = p.smem;
  cfg->stream = s;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = (unsigned)cs;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 1;
}

// Whether this GPU can run a cluster of the plan.
static bool cluster_runs(const hmc_ctx* c, const TilePlan& p, int cs) {
  const void* k = cluster_kernel32(p);
  if (!k) return false;
  if (!tile_allow_smem(c, k) ||
      (cs > 8 && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  cluster_config(&cfg, &attr, p, cs, 1, nullptr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return n > 0;
}

// The plans of one lattice by log2 of the cluster size (cw == 0: none).
struct ClusterPlans {
  TilePlan p[5];
  double us[5];
};
static ClusterPlans cluster_plans(const hmc_ctx* c, const Geo& g) {
  ClusterPlans cp;
  for (int k = 0; k < 5; ++k) {
    if (!plan_cluster(c, g, 1 << k, &cp.p[k]) || !cluster_runs(c, cp.p[k], 1 << k)) cp.p[k].cw = 0;
    cp.us[k] = cp.p[k].cw ? cluster_us(cp.p[k], g, 1 << k) : 0.0;
  }
  return cp;
}

bool cg32_cluster_ok(hmc_ctx* c, const Geo& g) {
  if (c->cluster_log2 == -2) {
    const ClusterPlans cp = cluster_plans(c, g);
    c->cluster_log2 = -1;
    for (int k = 0; k < 5; ++k)
      if (cp.p[k].cw && (c->cluster_log2 < 0 || cp.us[k] < cp.us[c->cluster_log2])) c->cluster_log2 = k;
    if (c->cluster_log2 >= 0) {
      c->cluster_plan = cp.p[c->cluster_log2];
      c->cluster_us = cp.us[c->cluster_log2];
    }
  }
  return c->cluster_log2 >= 0;
}

hmc_status cg32_cluster_launch(hmc_ctx* c, const Geo& g, float2* x, float2* r, CGScal* sc) {
  if (!cg32_cluster_ok(c, g)) return fail(c, HMC_ERR_INVALID, "resident CG tiles do not fit a cluster");
  const TilePlan& p = c->cluster_plan;
  const TileSys one = make_tile_sys(g, p, phase_of<float>(c).phi, x, r, nullptr, sc);
  const TileSys* list = nullptr;
  void* args[] = {(void*)&list, (void*)&one};
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  cluster_config(&cfg, &attr, p, 1 << c->cluster_log2, 1, c->stream);
  cudaError_t le = cudaSuccess;
  HMC_TRY(launch_b(c, K_CG_RES32, 0.0, [&] { le = cudaLaunchKernelExC(&cfg, cluster_kernel32(p), args); }));
  if (le != cudaSuccess) return cuda_fail(c, le, "resident CG cluster launch");
  c->shape[K_CG_RES32].tiled = p.cw == 2 ? 4 : 0;  // reported as the design
  return HMC_OK;
}

}  // namespace hmc
