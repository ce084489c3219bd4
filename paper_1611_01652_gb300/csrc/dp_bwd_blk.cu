// Launchers of the reverse kernels on blocks for the quadruped's worlds, and the choice
// between the kernels.
#include "dp_blk_bwd.cuh"
#include "dp_kernels.h"

cudaError_t launch_backward_blk_quad(const DevTopo& T, const DevTopo& Ts, const DevPtrs& D, cudaStream_t s) {
  return launch_backward_blk_t<BlkQuad>(T, Ts, D, s);
}
cudaError_t launch_backward_blk(const DevTopo& T, const DevTopo& Ts, const DevPtrs& D, cudaStream_t s) {
  if (T.topo_id == 0) return launch_backward_blk_dyn(T, Ts, D, s);
  if (T.mlp_tc && T.widths[1] == BlkArm::CTRL_H) return launch_backward_blk_arm(T, Ts, D, s);
  return launch_backward_blk_quad(T, Ts, D, s);
}
// (the wide controller's launches run no network: one kernel for every compiled topology)
cudaError_t launch_backward_ext_blk(const DevTopo& T, const DevPtrs& D, int t, cudaStream_t s) {
  if (T.topo_id == 0) return launch_backward_ext_blk_dyn(T, D, t, s);
  return launch_backward_ext_blk_t<BlkQuad>(T, D, t, s);
}
