// Launcher of the rollout kernel k_forward_blk for every other robot.
#include "dp_blk_fwd.cuh"
#include "dp_kernels.h"

cudaError_t forward_groups_blk_dyn(const DevTopo& T4, int* n) {
  const size_t smem = (size_t)T4.sm_total * 128;
  cudaError_t e = cudaFuncSetAttribute(k_forward_blk<true, BlkDyn>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k_forward_blk<true, BlkDyn>, 32 * T4.blk_nw, smem);
}
cudaError_t launch_forward_blk_dyn(const DevTopo& T, const DevPtrs& D, const float* x0, int t0, int nsteps, int rollout,
                                   int record, cudaStream_t s) {
  return record ? launch_forward_blk_t<true, BlkDyn>(T, D, x0, t0, nsteps, rollout, s)
                : launch_forward_blk_t<false, BlkDyn>(T, D, x0, t0, nsteps, rollout, s);
}
