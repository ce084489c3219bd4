// Launchers of the one-warp reverse-mode kernel k_backward, and the choice between it and the
// kernels on blocks (dp_bwd_blk.cu).
#include "dp_steps.cuh"
#include "dp_kernels.h"

template <class Q>
static cudaError_t launch_backward_q(const DevTopo& T, const DevPtrs& D, cudaStream_t s) {
  size_t smem = SM_BYTES(T);
  cudaError_t e = cudaFuncSetAttribute(k_backward<Q>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_backward<Q><<<T.Bp / 32, 32, smem, s>>>(T, D);
  return cudaGetLastError();
}
cudaError_t launch_backward(const DevTopo& T, const DevTopo& Ts, const DevPtrs& D, cudaStream_t s) {
  if (T.blk_bwd) return launch_backward_blk(T, Ts, D, s);
  if (T.topo_id == QuadrupedTopo::id) return launch_backward_q<QuadrupedTopo>(T, D, s);
  return launch_backward_q<DynTopo>(T, D, s);
}
