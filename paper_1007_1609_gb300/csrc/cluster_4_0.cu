// The register-resident recursion (cluster.cuh): tiles 4 x 4, covering the lattice exactly.
#include "cluster.cuh"

namespace cbdg {

cudaError_t launch_cluster_4_0(const ClusterArgs &a, const ClusterPlan &p, cudaStream_t s) {
  return launch_one<4, 0>(a, p, s);
}

int cluster_slots_4_0(const ClusterPlan &p) { return slots_one<4, 0>(p); }

}  // namespace cbdg
