// The register-resident recursion (cluster.cuh): tiles 4 x 6, sticking out over open edges.
#include "cluster.cuh"

namespace cbdg {

cudaError_t launch_cluster_6_1(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s) {
  return launch_one<6, 1>(a, p, s);
}

int cluster_slots_6_1(const ClusterPlan &p) { return slots_one<6, 1>(p); }

}  // namespace cbdg
