// Launcher of the rollout kernel k_forward_blk for the uneven batch's arms.
#include "dp_blk_fwd.cuh"
#include "dp_kernels.h"

cudaError_t launch_forward_blk_arm(const DevTopo& T, const DevPtrs& D, const float* x0, int t0, int nsteps, int rollout,
                                   int record, cudaStream_t s) {
  return record ? launch_forward_blk_t<true, BlkArm>(T, D, x0, t0, nsteps, rollout, s)
                : launch_forward_blk_t<false, BlkArm>(T, D, x0, t0, nsteps, rollout, s);
}
