// The register-resident adjoint (adjoint_cluster.cuh), tiles sticking out over open edges.
#include "adjoint_cluster.cuh"

namespace cbdg {

int adjoint_slots_1(const ClusterPlan &p) { return adjoint_slots_one<1>(p); }
cudaError_t adjoint_launch_1(const AdjointClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s) {
  return adjoint_launch_one<1>(a, p, clusters, s);
}

}  // namespace cbdg
