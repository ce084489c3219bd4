// Launchers of the reverse kernels on blocks for every other robot.
#include "dp_blk_bwd.cuh"
#include "dp_kernels.h"

cudaError_t launch_backward_blk_dyn(const DevTopo& T, const DevTopo& Ts, const DevPtrs& D, cudaStream_t s) {
  return launch_backward_blk_t<BlkDyn>(T, Ts, D, s);
}
cudaError_t launch_backward_ext_blk_dyn(const DevTopo& T, const DevPtrs& D, int t, cudaStream_t s) {
  return launch_backward_ext_blk_t<BlkDyn>(T, D, t, s);
}
