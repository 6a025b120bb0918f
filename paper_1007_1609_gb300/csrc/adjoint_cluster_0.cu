// The register-resident adjoint (adjoint_cluster.cuh), tiles covering the lattice exactly.
#include "adjoint_cluster.cuh"

namespace cbdg {

int adjoint_slots_0(const ClusterPlan &p) { return adjoint_slots_one<0>(p); }
cudaError_t adjoint_launch_0(const AdjointClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s) {
  return adjoint_launch_one<0>(a, p, clusters, s);
}

}  // namespace cbdg
