// Launchers of the reverse kernels on blocks for the uneven batch's arms.
#include "dp_blk_bwd.cuh"
#include "dp_kernels.h"

cudaError_t launch_backward_blk_arm(const DevTopo& T, const DevTopo& Ts, const DevPtrs& D, cudaStream_t s) {
  return launch_backward_blk_t<BlkArm>(T, Ts, D, s);
}
