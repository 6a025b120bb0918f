// cluster.cu -- plan and dispatch of the register-resident recursion (cluster.cuh).
#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.h"

namespace cbdg {

// one translation unit per kernel: tiles of 4 x by sites that cover the lattice
// as `rag` says (4 x 10 has no kernel of its own for the exact case)
#define CBDG_CLUSTER(by, rag)                                                                          \
  cudaError_t launch_cluster_##by##_##rag(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s); \
  int cluster_slots_##by##_##rag(const ClusterPlan &p);
#define CBDG_CLUSTERS(X) \
  X(4, 0) X(4, 1) X(4, 2) X(6, 0) X(6, 1) X(6, 2) X(8, 0) X(8, 1) X(8, 2) X(10, 1) X(10, 2)
CBDG_CLUSTERS(CBDG_CLUSTER)
#undef CBDG_CLUSTER

namespace {

int slots_of(const ClusterPlan &p) {
#define CBDG_SLOTS(b, r) \
  if (p.by == b && p.rag == r) return cluster_slots_##b##_##r(p);
  CBDG_CLUSTERS(CBDG_SLOTS)
#undef CBDG_SLOTS
  return 0;
}

}  // namespace

// Tile height, CTAs per cluster and tile rows per CTA for ncols start vectors:
// the candidate with the least rounds x cycles of a step.  A round is as many
// columns as run at once -- asked of the device, whose clusters stay within
// groups of SMs, for the candidates that look best: a cluster of 3 that should
// have fitted 101 times took twice the time of one of 2.  A step costs an SM 28
// to 31 cycles (40 with tiles of 10, whose registers leave no room to reorder) for
// each tile row of each of its warps, rounded up to its four schedulers, 500 for the latency of its barriers, edge
// loads and sums, and 250 for every doubling of the cluster (all columns of 64 x 64, M = 512:
// 4.37, 4.83 and 5.43 ms with tiles of 8 rows in clusters of 1, 2 and 4).  (The cycles were fitted
// with plain sums; the compensated ones add up to a tenth to every candidate and leave the order.)
// High tiles exchange fewer edges per site and win where they fill the SM (4.37
// against 4.65 ms with 4 rows there; 128 x 128, M = 512: 76.1 against 82.5 ms), tiles of 6
// and 10 hold more sites per SM (96 x 96: 21.1 ms with 6 in one CTA against 31.9
// and 33.1 with 4 and 8; 500 x 320 fits on chip only with 10), low ones leave more
// warps to a lattice that leaves SMs idle (33 x 21, two iterations: 0.82 against 0.93 ms).
bool plan_cluster(int Lx, int Ly, int px, int py, int ncols, ClusterPlan *p) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  struct Candidate {
    ClusterPlan plan;
    int warps, per_sm;
    bool asked;
    double cost;
  };
  const auto price = [&](Candidate &c, long long slots) {
    const int nw = c.plan.threads / 32, by = c.plan.by;
    const long long ctas = static_cast<long long>(ncols) * c.plan.cluster;
    const long long rounds = (ncols + slots - 1) / slots;
    const int busy = static_cast<int>(std::min<long long>(c.per_sm, (ctas + sms - 1) / sms));  // CTAs on an SM
    const double row_cycles = by == 4 ? 31.0 : by == 6 ? 29.3 : by == 8 ? 28.4 : 40.0;
    const double ragged = c.plan.rag == 2 ? 1.4 : 1.0;  // selects, waits without work in between
    c.cost = static_cast<double>(rounds) * (500.0 + 250.0 * std::log2(static_cast<double>(c.plan.cluster)) +
                                            ragged * row_cycles * ((busy * nw + 3) / 4 * 4) * by);
  };
  const int TX = (Lx + 3) / 4;
  std::vector<Candidate> list;
  for (int by : {4, 6, 8, 10}) {
    const int TY = (Ly + by - 1) / by;
    const int warps = by == 4 ? 16 : by == 6 ? 12 : 8;                    // an SM's registers hold
    const int quads = by == 4 ? 21 : by == 6 ? 27 : by == 8 ? 25 : 39;    // a thread's record (Record<BY>)
    const int per_ghost = by < 8 ? 2 : 3;
    const int rag = (Lx % 4 && px) || (Ly % by && py) ? 2 : Lx % 4 || Ly % by || by == 10 ? 1 : 0;
    for (int cluster = 1; cluster <= kMaxCluster && cluster <= TY; ++cluster) {
      const int rows = (TY + cluster - 1) / cluster, nw = (TX * rows + 31) / 32;
      if ((TY + rows - 1) / rows != cluster || nw > warps) continue;
      const int ghosts = cluster > 1 ? (TX + per_ghost - 1) / per_ghost : 0;
      const size_t smem = static_cast<size_t>(nw * 32 + ghosts + 1) * quads * 16 +
                          static_cast<size_t>(cluster) * 3 * kClusterBatch * 8 + 2 * kClusterBatch * 3 * nw * 8;
      if (smem > kClusterSmem) continue;
      Candidate c{ClusterPlan{by, cluster, rows, nw * 32, rag, smem}, nw,
                  std::min(warps / nw, static_cast<int>(kClusterSmem / (smem + 1024))), false, 0.0};
      price(c, std::max(1, sms * c.per_sm / cluster));
      list.push_back(c);
    }
  }
  while (!list.empty()) {
    auto best = std::min_element(list.begin(), list.end(), [](const Candidate &x, const Candidate &y) { return x.cost < y.cost; });
    if (best->asked) {
      *p = best->plan;
      return true;
    }
    const int slots = slots_of(best->plan);
    if (slots < 1) {
      list.erase(best);
      continue;
    }
    best->asked = true;
    price(*best, slots);
  }
  return false;
}

cudaError_t launch_cluster(ClusterArgs a, const ClusterPlan &p, cudaStream_t s) {
  if (a.ncols <= 0) return cudaSuccess;
  a.cluster = p.cluster;
  a.rows = p.rows;
#define CBDG_LAUNCH(b, r) \
  if (p.by == b && p.rag == r) return launch_cluster_##b##_##r(a, p, s);
  CBDG_CLUSTERS(CBDG_LAUNCH)
#undef CBDG_LAUNCH
  return cudaErrorInvalidValue;
}

}  // namespace cbdg
