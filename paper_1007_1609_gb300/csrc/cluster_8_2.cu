// The register-resident recursion (cluster.cuh): tiles 4 x 8, sticking out over a periodic edge.
#include "cluster.cuh"

namespace cbdg {

cudaError_t launch_cluster_8_2(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s) {
  return launch_one<8, 2>(a, p, s);
}

int cluster_slots_8_2(const ClusterPlan &p) { return slots_one<8, 2>(p); }

}  // namespace cbdg
