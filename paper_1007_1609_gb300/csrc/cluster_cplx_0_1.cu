// The register-resident recursion of general lattices (cluster_cplx.cuh): nearest neighbours, bond pairing.
#include "cluster_cplx.cuh"

namespace cbdg {

int cplx_slots_0_1(const ClusterPlan &p) { return cplx_slots_one<false, true>(p); }
cudaError_t cplx_launch_0_1(const CplxClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s) {
  return cplx_launch_one<false, true>(a, p, clusters, s);
}

}  // namespace cbdg
