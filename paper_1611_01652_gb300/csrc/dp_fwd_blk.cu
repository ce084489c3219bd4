// Launcher of the rollout kernel k_forward_blk for the quadruped's worlds, and the choice
// between the kernels.
#include "dp_blk_fwd.cuh"
#include "dp_kernels.h"

cudaError_t launch_forward_blk_quad(const DevTopo& T, const DevPtrs& D, const float* x0, int t0, int nsteps, int rollout,
                                   int record, cudaStream_t s) {
  return record ? launch_forward_blk_t<true, BlkQuad>(T, D, x0, t0, nsteps, rollout, s)
                : launch_forward_blk_t<false, BlkQuad>(T, D, x0, t0, nsteps, rollout, s);
}
cudaError_t launch_forward_blk(const DevTopo& T, const DevPtrs& D, const float* x0, int t0, int nsteps, int rollout,
                               int record, cudaStream_t s) {
  // compiled topologies carry their own controller width (or the fp32-arithmetic path, which every
  // kernel has); the rest dispatch on the width at run time
  if (T.topo_id == 0) return launch_forward_blk_dyn(T, D, x0, t0, nsteps, rollout, record, s);
  if (T.mlp_tc && T.widths[1] == BlkArm::CTRL_H) return launch_forward_blk_arm(T, D, x0, t0, nsteps, rollout, record, s);
  return launch_forward_blk_quad(T, D, x0, t0, nsteps, rollout, record, s);
}
