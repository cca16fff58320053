// The team solver's whole-grid form: one system, one CTA per SM (a translation unit of its own,
// compiled in parallel).
#include "team.cuh"

namespace mpcg {

cudaError_t team_setup_grid(size_t smem_max) {
  return cudaFuncSetAttribute(cg_team<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_max);
}

cudaError_t launch_cg_team_grid(const Launch& L, int grid, cudaStream_t s) {
  void* args[] = {(void*)&L};
  return cudaLaunchCooperativeKernel((const void*)cg_team<false, false>, dim3(grid), dim3(kTT), args,
                                     kTeamFixed + (size_t)L.team_heap, s);
}

}  // namespace mpcg
