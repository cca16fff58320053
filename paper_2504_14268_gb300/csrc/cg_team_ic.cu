// The team solver's instantiation with the IC(0) preconditioner (a translation unit of its own,
// compiled in parallel).
#include "team.cuh"

namespace mpcg {

cudaError_t team_setup_ic(size_t smem_max) {
  const cudaError_t e =
      cudaFuncSetAttribute(cg_team<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(cg_team<true, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

cudaError_t launch_cg_team_ic(const Launch& L, int cluster, int grid, size_t smem, cudaStream_t s) {
  return team_launch_cluster(cg_team<true, true>, L, cluster, grid, smem, s);
}

}  // namespace mpcg
