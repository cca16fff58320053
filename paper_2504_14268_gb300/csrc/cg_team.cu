// Launch of the team solver (team.cuh).
#include "team.cuh"


namespace mpcg {

namespace {
constexpr size_t kTeamSmemMax = 227 * 1024;
}

size_t team_max_heap() { return kTeamSmemMax - kTeamFixed; }

// Sets the kernels' limits; *max_cluster receives the largest cluster that fits the device,
// resident[i] how many clusters of 2^i CTAs run at a time.
cudaError_t team_setup(int* max_cluster, int resident[5]) {
  cudaError_t e = cudaFuncSetAttribute(cg_team<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTeamSmemMax);
  if (e == cudaSuccess) e = team_setup_grid(kTeamSmemMax);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(cg_team<true, false>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) e = team_setup_ic(kTeamSmemMax);
  if (e != cudaSuccess) return e;
  *max_cluster = 0;
  for (int i = 0, c = 1; c <= kTeamMaxCluster; ++i, c *= 2) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(kTT);
    cfg.dynamicSmemBytes = kTeamSmemMax;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    resident[i] = 0;
    if (cudaOccupancyMaxActiveClusters(&n, cg_team<true, false>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    resident[i] = n;
    if (n > 0) *max_cluster = c;
  }
  return cudaSuccess;
}

cudaError_t launch_cg_team(const Launch& L, int cluster, int grid, cudaStream_t s) {
  if (cluster == 0) return launch_cg_team_grid(L, grid, s);
  const size_t smem = kTeamFixed + (size_t)L.team_heap;
  if (L.ic) return launch_cg_team_ic(L, cluster, grid, smem, s);
  return team_launch_cluster(cg_team<true, false>, L, cluster, grid, smem, s);
}

}  // namespace mpcg
