// The register-resident recursion of general lattices (cluster_cplx.cuh): next-nearest neighbours, on-site pairing.
#include "cluster_cplx.cuh"

namespace cbdg {

int cplx_slots_1_0(const ClusterPlan &p) { return cplx_slots_one<true, false>(p); }
cudaError_t cplx_launch_1_0(const CplxClusterArgs &a, const ClusterPlan &p, int clusters, cudaStream_t s) {
  return cplx_launch_one<true, false>(a, p, clusters, s);
}

}  // namespace cbdg
