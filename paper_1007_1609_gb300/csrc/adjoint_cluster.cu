// adjoint_cluster.cu -- plan, dispatch and final sums of the register-resident
// adjoint (adjoint_cluster.cuh).
#include <algorithm>
#include <cmath>
#include <tuple>

#include "internal.h"
#include "slot_table.h"

namespace cbdg {

int adjoint_slots_0(const ClusterPlan &p);
int adjoint_slots_1(const ClusterPlan &p);
cudaError_t adjoint_launch_0(const AdjointClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s);
cudaError_t adjoint_launch_1(const AdjointClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s);

namespace {

constexpr int kQuads = 41, kGhosts = 2;  // as in adjoint_cluster.cuh
constexpr int kMaxM = 4096;                             // the column's source table is in shared memory

int slots_of(const ClusterPlan &p) {
  static SlotTable<std::tuple<int, int, int, int, size_t>> known;
  int dev = 0;
  cudaGetDevice(&dev);
  return known.get(std::make_tuple(dev, p.rag, p.cluster, p.threads, p.smem),
                   [&] { return p.rag ? adjoint_slots_1(p) : adjoint_slots_0(p); });
}

// Sums over the clusters (heads and tails in FP64); one thread per site.
__global__ void adjoint_cluster_final_kernel(int Lx, int Ly, int px, int py, int cluster, int rows, int threads,
                                             int clusters, const float2 *acc, const double *scal, double *g_eps,
                                             double *g_hop, double *g_delta) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Lx * Ly) return;
  const double a = scal[kScalA];
  const int TX = (Lx + 3) / 4;
  auto sum = [&](int kind, int x, int y) {
    const int ty = y / 4, rank = ty / rows, t = (ty - rank * rows) * TX + x / 4;
    const int k = kind * 16 + (y % 4) * 4 + x % 4;
    double s = 0.0;
    for (int c = 0; c < clusters; ++c) {
      const float2 v = acc[(static_cast<size_t>(c * cluster + rank) * 64 + k) * threads + t];
      s += static_cast<double>(v.x) + static_cast<double>(v.y);
    }
    return s / a;
  };
  const int x = i % Lx, y = i / Lx;
  if (g_eps) g_eps[i] = sum(0, x, y);
  if (g_delta) g_delta[i] = sum(1, x, y);
  if (g_hop) {
    const int xl = x > 0 ? x - 1 : px ? Lx - 1 : -1, yl = y > 0 ? y - 1 : py ? Ly - 1 : -1;
    g_hop[static_cast<size_t>(i) * 4 + 0] = x + 1 < Lx || px ? sum(2, x, y) : 0.0;
    g_hop[static_cast<size_t>(i) * 4 + 1] = xl >= 0 ? sum(2, xl, y) : 0.0;
    g_hop[static_cast<size_t>(i) * 4 + 2] = y + 1 < Ly || py ? sum(3, x, y) : 0.0;
    g_hop[static_cast<size_t>(i) * 4 + 3] = yl >= 0 ? sum(3, x, yl) : 0.0;
  }
}

}  // namespace

// The least rounds x cycles of a step among the clusters the device holds, as
// plan_cluster (a step back takes an SM about four times a step of the moments).
bool plan_adjoint_cluster(int Lx, int Ly, int px, int py, int ncols, int M, ClusterPlan *p, int *clusters,
                          size_t *ck_bytes, size_t *acc_bytes) {
  if ((px && Lx % 4) || (py && Ly % 4) || M > kMaxM || ncols < 1) return false;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int TX = (Lx + 3) / 4, TY = (Ly + 3) / 4;
  double best = 0.0;
  for (int cluster = 1; cluster <= kMaxCluster && cluster <= TY; ++cluster) {
    const int rows = (TY + cluster - 1) / cluster, nw = (TX * rows + 31) / 32;
    if ((TY + rows - 1) / rows != cluster || nw > 8) continue;
    const int ghosts = cluster > 1 ? (TX + kGhosts - 1) / kGhosts : 0;
    ClusterPlan q{4, cluster, rows, nw * 32, Lx % 4 || Ly % 4 ? 1 : 0,
                  static_cast<size_t>(nw * 32 + ghosts + 1) * kQuads * 16 + static_cast<size_t>(M) * 8};
    if (q.smem > kClusterSmem) continue;
    const int slots = slots_of(q);
    if (slots < 1) continue;
    const int per_sm = std::min(8 / nw, static_cast<int>(kClusterSmem / (q.smem + 1024)));
    const long long rounds = (ncols + slots - 1) / slots, ctas = static_cast<long long>(ncols) * cluster;
    const int busy = static_cast<int>(std::min<long long>(std::max(1, per_sm), (ctas + sms - 1) / sms));
    const double cost = static_cast<double>(rounds) *
                        (900.0 + 250.0 * std::log2(static_cast<double>(cluster)) + 250.0 * ((busy * nw + 3) / 4 * 4));
    if (best == 0.0 || cost < best) {
      best = cost;
      *p = q;
      *clusters = std::min(slots, ncols);
    }
  }
  if (best == 0.0) return false;
  const size_t lanes = static_cast<size_t>(p->cluster) * p->threads;
  *ck_bytes = lanes * (M - 1) * 8 * sizeof(float4);
  *acc_bytes = lanes * 64 * sizeof(float2);
  return true;
}

cudaError_t launch_adjoint_cluster(AdjointClusterArgs a, const ClusterPlan &p, int clusters, cudaStream_t s) {
  a.cluster = p.cluster;
  a.rows = p.rows;
  return p.rag ? adjoint_launch_1(a, p, clusters, s) : adjoint_launch_0(a, p, clusters, s);
}

cudaError_t launch_adjoint_cluster_final(const AdjointClusterArgs &a, const ClusterPlan &p, int clusters, double *g_eps,
                                         double *g_hop, double *g_delta, cudaStream_t s) {
  adjoint_cluster_final_kernel<<<(a.Lx * a.Ly + 127) / 128, 128, 0, s>>>(
      a.Lx, a.Ly, a.px, a.py, p.cluster, p.rows, p.threads, clusters, a.acc, a.scal, g_eps, g_hop, g_delta);
  return cudaGetLastError();
}

}  // namespace cbdg
