// cluster.cu -- plan and dispatch of the register-resident recursion (cluster.cuh).
#include <algorithm>
#include <cmath>

#include "internal.h"

namespace cbdg {

#define CBDG_CLUSTER(by)                                                                        \
  cudaError_t launch_cluster_##by##_0(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s); \
  cudaError_t launch_cluster_##by##_1(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s); \
  cudaError_t launch_cluster_##by##_2(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s);
CBDG_CLUSTER(4)
CBDG_CLUSTER(6)
CBDG_CLUSTER(8)
#undef CBDG_CLUSTER

// Tile height, CTAs per cluster and tile rows per CTA for ncols start vectors:
// the candidate with the least rounds x cycles of a step, where a round is as
// many columns as run at once and a step costs an SM 28 to 31 cycles for each
// tile row of each of its warps (arithmetic; the warps rounded up to its four
// schedulers), 500 for the latency of its barriers, edge loads and sums, and 250
// for every doubling of the cluster
// (64 x 64, M = 512, all columns: 4.21, 4.65 and 5.27 ms with tiles of 8 rows in
// clusters of 1, 2 and 4).  High tiles exchange fewer edges per site and win
// where they fill the SM (4.21 against 4.32 ms with 4 rows there; 128 x 128:
// 73.7 against 78.6 ms), tiles of 6 hold more sites per SM (96 x 96: 19.9 ms in
// one CTA against 27.4 and 31.1), low ones leave more warps to a lattice that
// leaves SMs idle (33 x 21: 0.53 against 0.61 ms).
bool plan_cluster(int Lx, int Ly, int ncols, ClusterPlan *p) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int TX = (Lx + 3) / 4;
  double best = 0.0;
  for (int by : {4, 6, 8}) {
    const int TY = (Ly + by - 1) / by;
    const int warps = by == 4 ? 16 : by == 6 ? 12 : 8;   // an SM's registers hold
    const int quads = by == 4 ? 21 : by == 6 ? 27 : 25;  // a thread's record (Record<BY>)
    const double row_cycles = by == 4 ? 31.0 : by == 6 ? 29.3 : 28.4;
    for (int cluster = 1; cluster <= kMaxCluster && cluster <= TY; ++cluster) {
      const int rows = (TY + cluster - 1) / cluster, nw = (TX * rows + 31) / 32;
      if ((TY + rows - 1) / rows != cluster || nw > warps) continue;
      const size_t smem = static_cast<size_t>(nw * 32 + (cluster > 1 ? TX : 0) + 1) * quads * 16 +
                          static_cast<size_t>(cluster) * 3 * kClusterBatch * 8 + 2 * kClusterBatch * 3 * nw * 4;
      if (smem > kClusterSmem) continue;
      const int per_sm = std::min(warps / nw, static_cast<int>(kClusterSmem / (smem + 1024)));
      const long long slots = std::max(1, sms * per_sm / cluster), ctas = static_cast<long long>(ncols) * cluster;
      const long long rounds = (ncols + slots - 1) / slots;
      const int busy = static_cast<int>(std::min<long long>(per_sm, (ctas + sms - 1) / sms));  // CTAs on an SM
      const double step = 500.0 + 250.0 * std::log2(static_cast<double>(cluster)) + row_cycles * ((busy * nw + 3) / 4 * 4) * by;
      const double cost = static_cast<double>(rounds) * step;
      if (best == 0.0 || cost < best) {
        best = cost;
        *p = ClusterPlan{by, cluster, rows, nw * 32, smem};
      }
    }
  }
  return best > 0.0;
}

cudaError_t launch_cluster(ClusterArgs a, const ClusterPlan &p, cudaStream_t s) {
  if (a.ncols <= 0) return cudaSuccess;
  a.cluster = p.cluster;
  a.rows = p.rows;
  const int rag = (a.Lx % 4 && a.px) || (a.Ly % p.by && a.py) ? 2 : a.Lx % 4 || a.Ly % p.by ? 1 : 0;
  switch (p.by * 4 + rag) {
    case 16: return launch_cluster_4_0(a, p, s);
    case 17: return launch_cluster_4_1(a, p, s);
    case 18: return launch_cluster_4_2(a, p, s);
    case 24: return launch_cluster_6_0(a, p, s);
    case 25: return launch_cluster_6_1(a, p, s);
    case 26: return launch_cluster_6_2(a, p, s);
    case 32: return launch_cluster_8_0(a, p, s);
    case 33: return launch_cluster_8_1(a, p, s);
    case 34: return launch_cluster_8_2(a, p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace cbdg
