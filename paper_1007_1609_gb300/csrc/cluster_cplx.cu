// cluster_cplx.cu -- plan and dispatch of the register-resident recursion of
// general lattices (cluster_cplx.cuh).
#include <algorithm>
#include <cmath>
#include <tuple>

#include "internal.h"
#include "slot_table.h"

namespace cbdg {

#define CBDG_CPLX(nnn, bond)                                                                                     \
  int cplx_slots_##nnn##_##bond(const ClusterPlan &p);                                                           \
  cudaError_t cplx_launch_##nnn##_##bond(const CplxClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s);
CBDG_CPLX(0, 0)
CBDG_CPLX(0, 1)
CBDG_CPLX(1, 0)
CBDG_CPLX(1, 1)
#undef CBDG_CPLX

namespace {

constexpr int kRecord = 33, kCols = 2, kMaxThreads = 384;  // as in cluster_cplx.cuh

// p.rag: nnn + 2 bond + 4 for periodic sides that the tiles do not divide
int slots_of(const ClusterPlan &p) {
  static SlotTable<std::tuple<int, int, int, int, size_t>> known;
  int dev = 0;
  cudaGetDevice(&dev);
  return known.get(std::make_tuple(dev, p.rag, p.cluster, p.threads, p.smem), [&] {
    const int kind = p.rag & 3;
    return kind == 0   ? cplx_slots_0_0(p)
           : kind == 1 ? cplx_slots_1_0(p)
           : kind == 2 ? cplx_slots_0_1(p)
                       : cplx_slots_1_1(p);
  });
}

}  // namespace

// Cycles of a step of all columns, by clusters: a round takes 900 for the chain through shared
// memory, 250 for each doubling of the cluster (its barrier) and the shared-memory wavefronts of
// the warps on an SM, 1500 every pass of the threads over the targets after the first; fitted to 32 .. 800 columns of 16 x 16 .. 140 x 120 sites, within 15 %.
// Falls short (false) where the streamed kernels are expected to be faster.
bool plan_cluster_cplx(int Lx, int Ly, int px, int py, int nnn, int bond, int ncols, int n_t, ClusterPlan *p, int *clusters) {
  if (ncols < 1) return false;
  const int rag = (px && Lx % 4) || (py && Ly % 2) ? 4 : 0;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int TX = (Lx + 3) / 4, TY = (Ly + 1) / 2, pairs = (ncols + kCols - 1) / kCols;
  const double wide = nnn ? (bond ? 355.0 : 285.0) : (bond ? 255.0 : 215.0);
  double best = 0.0;
  for (int cluster = 1; cluster <= kMaxCluster && cluster <= TY; ++cluster) {
    const int rows = (TY + cluster - 1) / cluster, threads = (TX * rows + 31) / 32 * 32 * kCols;
    if ((TY + rows - 1) / rows != cluster || threads > kMaxThreads) continue;
    ClusterPlan q{2, cluster, rows, threads, nnn + 2 * bond + rag,
                  static_cast<size_t>(TX * rows + (cluster > 1 ? TX : 0) + 1) * 2 * kRecord * 16};
    if (q.smem > kCplxClusterSmem) continue;
    const int slots = slots_of(q);
    if (slots < 1) continue;
    const int nw = threads / 32;
    const int per_sm = std::max(1, std::min(12 / nw, static_cast<int>(kClusterSmem / (q.smem + 4096))));
    const long long rounds = (pairs + slots - 1) / slots, ctas = static_cast<long long>(pairs) * cluster;
    const int busy = static_cast<int>(std::min<long long>(per_sm, (ctas + sms - 1) / sms));
    const double warp_cycles = (threads > 256 ? wide : 0.78 * wide) * (rag ? 1.1 : 1.0);  // (the two kernels of cluster_cplx.cuh)
    const double cost = static_cast<double>(rounds) *
                        (900.0 + 250.0 * std::log2(static_cast<double>(cluster)) + warp_cycles * busy * nw +
                         1500.0 * ((kCols * n_t + threads - 1) / threads - 1));
    if (best == 0.0 || cost < best) {
      best = cost;
      *p = q;
      *clusters = std::min(slots, pairs);
    }
  }
  // The streamed kernels take 21,000 cycles a step (launches, latency) and 0.0165 a site and
  // vector.  Streamed -> on chip, ms, eight hoppings and bond pairing, M = 400: 40 x 36,
  // 400 columns: 6.0 -> 2.3; 64 x 64: 9.3 -> 5.5; 96 x 96: 18.3 -> 9.8; 1000 columns:
  // 41.8 -> 28.3; 120 x 120: 57.2 -> 48.5; 100 x 98: 45.0 -> 42.2.  Clusters of 13 to 16 CTAs
  // fit the chip only seven times (112 of the 152 SMs): 128 x 128, 512 columns: 31.5 -> 30.8, and
  // more of them stay streamed.
  // Many targets: 64 x 64, 16 columns, M = 200: 256 targets 2.58 -> 0.66, 1024: 2.58 -> 1.52, 4096 would
  // take 17.8 (streamed 3.0); 128 x 128, 64 columns: 256: 3.66 -> 2.93, 512: 4.52 (streamed 3.80).
  // Ragged periodic sides: 33 x 33, 512 columns: 6.0 -> 1.6; 75 x 90, 1000: 35.2 -> 19.0; 98 x 98: 41.4 ->
  // 36.7; 121 x 119 would take 1.08 of the streamed time, so they are given a margin.
  return best > 0.0 && best * (rag ? 1.15 : 1.0) < 21000.0 + 0.0165 * Lx * Ly * ncols;
}

cudaError_t launch_cluster_cplx(CplxClusterArgs a, int bond, const ClusterPlan &p, int clusters, cudaStream_t s) {
  a.cluster = p.cluster;
  a.rows = p.rows;
  if (bond) return p.rag & 1 ? cplx_launch_1_1(a, p, clusters, s) : cplx_launch_0_1(a, p, clusters, s);
  return p.rag & 1 ? cplx_launch_1_0(a, p, clusters, s) : cplx_launch_0_0(a, p, clusters, s);
}

}  // namespace cbdg
