// The register-resident recursion of general lattices (cluster_cplx.cuh): next-nearest neighbours, bond pairing.
#include "cluster_cplx.cuh"

namespace cbdg {

int cplx_slots_1_1(const ClusterPlan &p) { return cplx_slots_one<true, true>(p); }
cudaError_t cplx_launch_1_1(const CplxClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s) {
  return cplx_launch_one<true, true>(a, p, clusters, s);
}

}  // namespace cbdg
