// sweep_packed.cu -- the FP64 batch kernels that gather the integrals from
// the packed array (the compound index of Algorithm hash) instead of the
// context's four-index layout: used by the no-allocation entry point, whose
// only copy of the integrals is the caller's packed one.
#include "sweep_impl.cuh"

namespace qp {

cudaError_t launch_batch_packed(int nint, const SweepParams& p, int grid, size_t smem, cudaStream_t st) {
  return batch_launch<double, false, false, false>(nint, p, grid, smem, st);
}

int batch_blocks_per_sm_packed(int nint, size_t smem) {
  return nint == 1 ? blocks_per_sm<batch_kernel<1, double, false, false, false>>(kThreads, smem)
                   : blocks_per_sm<batch_kernel<2, double, false, false, false>>(kThreads, smem);
}

}  // namespace qp
