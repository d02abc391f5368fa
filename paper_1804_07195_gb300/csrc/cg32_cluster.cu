// Resident-tile FP32 CG on thread block clusters (cg_tile.cuh): one cluster
// solves one system, so a launch can hold any number of independent systems
// and none waits for another. Plans and launches.
//
// An exchange inside a cluster is a round of stores into the other blocks'
// shared memory, each reporting its bytes to a barrier word there, and the wait
// for one's own: two of them and the phases between take 2.2 us on 2 to 16 blocks
// of the smallest tiles (5x5x16), where two exchanges through L2 alone take 3.8; but
// the work is spread over 16 SMs at most.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <functional>
#include <queue>
#include <utility>

#include "cg32_cluster.cuh"
#include "launch.cuh"

namespace hmc {

static const void* cluster_kernel(const TilePlan& p, bool batch) { return batch ? cluster_kernel_batch(p) : cluster_kernel_of<false>(p); }

// us per iteration of a system on a cluster of 2^k blocks: the cells of its largest
// tile, and the partials every warp sends to and takes from every block, twice. It
// only ranks the choices. Fitted to 151 measured plans (4x43x20 to 36x36x48, odd and
// even n; rms error 8 %; the cluster it ranks first is 0.2 % slower than the fastest on
// average, 3.6 % at most), for instance on 1, 2, 4, 8, 16 blocks (a dash: does not fit):
//   6x6x16 2.61, 2.36, 2.29, 2.33, 2.42   12x12x32 9.29, 4.47, 3.40, 2.74, 2.59
//   13x13x32 -, 5.62, 4.04, 3.50, 2.85    18x18x48 -, -, 6.26, 4.11, 3.49
//   24x24x48 -, -, -, 6.06, 4.23          25x25x48 -, -, -, 12.7, 7.24
//   36x36x48 -, -, -, -, 6.46 (over all SMs 5.60)
static double cluster_us(const TilePlan& p, const Geo& g, int k) {
  const double cols = (double)p.J * std::min(p.T, g.nt) * (g.n / p.cw);
  const double slope = (p.cw == 1 ? 1.35e-3 : 1.95e-3) + (p.S >= kXInMemory ? 1.25e-3 : 0.0);
  return 1.95 + 0.07 * k + 0.0034 * (p.threads / 32) * (1 << k) + slope * cols;
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
    for (const int* inst = tile_slices32(cw); *inst; ++inst) {
      // x out of registers: only the longest columns, it streams through L2 here
      if (*inst > kXInMemory && *inst != (cw == 1 ? 8 : 4) + kXInMemory) continue;
      const int S = tile_slices(*inst);
      TilePlan p;
      p.cw = cw;
      p.S = *inst;
      p.J = J;
      p.nseg = (T0 + S - 1) / S;
      p.T = p.nseg * S;
      const long long th = ((long long)nq * J * p.nseg + 31) / 32 * 32;
      if (th > max_threads32(cw, *inst)) continue;
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

// The waits of an exchange: by the wait test for sums that nobody sends, and the
// cycles after which a block gives up. Not below 50 us: a block that has given up
// leaves once all have, and by then every store on its way to it must have landed.
static void cluster_waits(const hmc_ctx* c, unsigned* extra, long long* limit) {
  *extra = (unsigned)c->bar_extra;
  *limit = c->bar_limit > 0 ? std::max(c->bar_limit, 100000LL) : 2000000000LL;
}

// How many clusters of the plan this GPU can run at a time with an SM to each block.
// (Blocks of small tiles can share one, but then take longer: counted that way, 100
// systems of 4x4 to 8x8 cells take 3.8 ms instead of 3.35.)
static int cluster_count(const hmc_ctx* c, const TilePlan& p, int cs, bool batch) {
  const void* k = cluster_kernel(p, batch);
  if (!k) return 0;
  if (!tile_allow_smem(c, k) ||
      (cs > 8 && cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  TilePlan alone = p;
  alone.smem = std::max(p.smem, (size_t)120 * 1024);  // more than half of an SM's
  cluster_config(&cfg, &attr, alone, cs, 1, nullptr);
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

static ClusterPlans cluster_plans(const hmc_ctx* c, const Geo& g, bool batch) {
  ClusterPlans cp;
  for (int k = 0; k < 5; ++k) {
    cp.count[k] = plan_cluster(c, g, 1 << k, &cp.p[k]) ? cluster_count(c, cp.p[k], 1 << k, batch) : 0;
    if (cp.count[k] < 1) cp.p[k].cw = 0;
    cp.us[k] = cp.p[k].cw ? cluster_us(cp.p[k], g, k) : 0.0;
  }
  return cp;
}

bool cg32_cluster_ok(hmc_ctx* c, const Geo& g) {
  if (c->cluster_log2 == -2) {
    const ClusterPlans cp = cluster_plans(c, g, false);
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
  unsigned extra = 0;
  long long limit = 0;
  cluster_waits(c, &extra, &limit);
  void* args[] = {(void*)&list, (void*)&one, &extra, &limit};
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  cluster_config(&cfg, &attr, p, 1 << c->cluster_log2, 1, c->stream);
  cudaError_t le = cudaSuccess;
  HMC_TRY(launch_b(c, K_CG_RES32, 0.0, [&] { le = cudaLaunchKernelExC(&cfg, cluster_kernel(p, false), args); }));
  if (le != cudaSuccess) return cuda_fail(c, le, "resident CG cluster launch");
  c->shape[K_CG_RES32].tiled = p.cw == 2 ? 4 : 0;  // reported as the design
  c->shape[K_CG_RES32].waves = -(1 << c->cluster_log2);
  return HMC_OK;
}

// ---------------------------------------------------------------------------
// Batches: every system on a cluster of its own. Before, all systems of a batch
// went through an iteration together, two launches (or grid barriers) each, until
// the last had converged; 48 systems of 16 lattices took 22.8 ms, now 10.5, and
// a trajectory of 8 chains 345 ms, now 123.

bool cg32_cluster_batch(hmc_ctx* c, const std::vector<Geo>& geos, const std::vector<double>& iters,
                        std::vector<ClusterGroup>* groups) {
  const int ns = (int)geos.size();
  if (c->batch_plans.size() > 512) c->batch_plans.clear();
  std::vector<const ClusterPlans*> cp(ns);
  std::vector<int> pick(ns);
  for (int i = 0; i < ns; ++i) {
    const std::array<int, 3> key{geos[i].n, geos[i].m, geos[i].nt};
    auto it = c->batch_plans.find(key);
    if (it == c->batch_plans.end()) it = c->batch_plans.emplace(key, cluster_plans(c, geos[i], true)).first;
    cp[i] = &it->second;
  }
  // For a time T every system takes the smallest cluster (the least SM time)
  // that is expected to finish within T, or its fastest; the batch's end is that
  // of running them longest first on the SMs that are free. Of up to 32 values
  // of T, spread over the systems' possible times, the best end wins.
  std::vector<double> cand;
  auto time_at = [&](int i, int k) { return iters[i] * cp[i]->us[k]; };
  for (int i = 0; i < ns; ++i) {
    int any = 0;
    for (int k = 0; k < 5; ++k)
      if (cp[i]->p[k].cw > 0) {
        cand.push_back(time_at(i, k));
        any = 1;
      }
    if (!any) return false;
  }
  std::sort(cand.begin(), cand.end());
  std::vector<int> trial(ns), order(ns);
  std::vector<double> ends, times;
  std::vector<std::vector<int>> trials;
  const int ncand = (int)cand.size(), tries = std::min(ncand, 32);
  for (int v = 0; v < tries; ++v) {
    const double T = cand[tries == ncand ? v : (size_t)v * (ncand - 1) / (tries - 1)];
    for (int i = 0; i < ns; ++i) {
      int k = -1;
      for (int l = 0; l < 5; ++l)
        if (cp[i]->p[l].cw > 0 && (k < 0 || time_at(i, k) > T) && (k < 0 || time_at(i, l) < time_at(i, k))) k = l;
      trial[i] = k;
      order[i] = i;
    }
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return time_at(a, trial[a]) > time_at(b, trial[b]); });
    std::priority_queue<std::pair<double, double>, std::vector<std::pair<double, double>>, std::greater<>> running;
    double free = c->nsm, now = 0.0, end = 0.0;
    for (int i : order) {
      // SMs a cluster takes of this GPU: clusters must lie in one of its groups of SMs
      // and leave some unused (152, 76, 36, 15 and 7 of 1 to 16 blocks at a time on 152
      // SMs)
      const double need = (double)c->nsm / cp[i]->count[trial[i]];
      while (free < need && !running.empty()) {
        now = running.top().first;
        free += running.top().second;
        running.pop();
      }
      const double done = now + time_at(i, trial[i]);
      running.push({done, need});
      free -= need;
      end = std::max(end, done);
    }
    ends.push_back(end);
    times.push_back(T);
    trials.push_back(trial);
  }
  // Of values that end together the largest T (the least SM time), but the systems'
  // iterations differ from what is expected: below 0.65 of the end, where there is
  // one. (ms for 48 systems of 5x5x16 to 19x19x32, 24 of 12x12 to 24x24, 12 of 6x6 to
  // 24x24, with the largest T, the smallest, and this one: 5.0, 4.3, 4.3; 6.1, 6.3, 6.5;
  // 8.05, 9.1, 8.05; eight chains 115, 104, 109.)
  const double best = *std::min_element(ends.begin(), ends.end());
  int take = -1;
  for (int v = 0; v < tries; ++v)
    if (ends[v] <= 1.01 * best && (take < 0 || times[v] <= 0.65 * best)) take = v;
  pick = trials[take];
  auto time_of = [&](int i) { return time_at(i, pick[i]); };
  // one launch per instance and cluster size, with the largest block and shared
  // memory of its systems; the systems that run longest first
  for (int i = 0; i < ns; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return time_of(a) > time_of(b); });
  groups->clear();
  double load[hmc_ctx::kSideStreams] = {};
  for (int i : order) {
    const TilePlan& p = cp[i]->p[pick[i]];
    ClusterGroup* g = nullptr;
    for (ClusterGroup& h : *groups)
      if (h.log2 == pick[i] && h.plan.cw == p.cw && h.plan.S == p.S && h.plan.stride == p.stride) g = &h;
    if (!g) {
      groups->push_back(ClusterGroup{});
      g = &groups->back();
      g->log2 = pick[i];
      g->plan = p;
      // the launches of one stream run one after another: the one that has the
      // least to do so far
      int s = 0;
      for (int k = 1; k < hmc_ctx::kSideStreams; ++k)
        if (load[k] < load[s]) s = k;
      g->stream = s;
      load[s] += time_of(i);
    }
    g->plan.smem = std::max(g->plan.smem, p.smem);
    g->plan.threads = std::max(g->plan.threads, p.threads);
    g->sys.push_back(i);
    g->plans.push_back(p);
  }
  for (const ClusterGroup& g : *groups)
    if (cluster_count(c, g.plan, 1 << g.log2, true) < 1) return false;
  return true;
}

hmc_status cg32_cluster_batch_launch(hmc_ctx* c, const std::vector<ClusterGroup>& groups, const TileSys* list) {
  // all that can fail for want of memory before the first launch
  if (!c->side_start) HMC_CUDA(c, cudaEventCreateWithFlags(&c->side_start, cudaEventDisableTiming));
  for (const ClusterGroup& g : groups) {
    const int i = g.stream;
    if (!c->side[i]) HMC_CUDA(c, cudaStreamCreateWithFlags(&c->side[i], cudaStreamNonBlocking));
    if (!c->side_done[i]) HMC_CUDA(c, cudaEventCreateWithFlags(&c->side_done[i], cudaEventDisableTiming));
  }
  bool on[hmc_ctx::kSideStreams] = {};
  HMC_CUDA(c, cudaEventRecord(c->side_start, c->stream));
  unsigned extra = 0;
  long long limit = 0;
  cluster_waits(c, &extra, &limit);
  int first = 0;
  hmc_status st = HMC_OK;
  for (size_t k = 0; k < groups.size() && st == HMC_OK; ++k) {
    const ClusterGroup& g = groups[k];
    const int i = g.stream;
    if (!on[i]) {
      const cudaError_t e = cudaStreamWaitEvent(c->side[i], c->side_start, 0);
      if (e != cudaSuccess) {
        st = cuda_fail(c, e, "batched CG side stream");
        break;
      }
    }
    on[i] = true;
    const TileSys* mine = list + first;
    const TileSys one{};
    void* args[] = {(void*)&mine, (void*)&one, &extra, &limit};
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr;
    cluster_config(&cfg, &attr, g.plan, 1 << g.log2, (int)g.sys.size(), c->side[i]);
    const cudaError_t e = cudaLaunchKernelExC(&cfg, cluster_kernel(g.plan, true), args);
    if (e != cudaSuccess) st = cuda_fail(c, e, "batched CG cluster launch");
    c->prof.launches[K_BATCH_CG32]++;
    first += (int)g.sys.size();
  }
  // also after a failure: nothing outlives the call, whose buffers go back to the pool
  for (int i = 0; i < hmc_ctx::kSideStreams; ++i) {
    if (!on[i]) continue;
    cudaError_t e = cudaEventRecord(c->side_done[i], c->side[i]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(c->stream, c->side_done[i], 0);
    if (e != cudaSuccess) {
      cudaStreamSynchronize(c->side[i]);
      if (st == HMC_OK) st = cuda_fail(c, e, "batched CG side stream");
    }
  }
  return st;
}

}  // namespace hmc
