// Instantiations of the p-phase kernel for the cluster-per-problem launch of
// batched node solves with the backtracking step rule (a translation unit of
// their own: compiled in parallel with the grid instantiations).
#include "launch.cuh"

namespace relax {

const void* pphase_cluster_kernel(int ept) {
  return ept == PEPT ? reinterpret_cast<const void*>(&pphase_kernel<double, PEPT, true, true>)
                     : reinterpret_cast<const void*>(&pphase_kernel<double, PEPT_CLUSTER, true, true>);
}

}  // namespace relax
