// The register-resident recursion (cluster.cuh): tiles 4 x 10, sticking out over a periodic edge.
#include "cluster.cuh"

namespace cbdg {

cudaError_t launch_cluster_10_2(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s) {
  return launch_one<10, 2>(a, p, s);
}

int cluster_slots_10_2(const ClusterPlan &p) { return slots_one<10, 2>(p); }

}  // namespace cbdg
