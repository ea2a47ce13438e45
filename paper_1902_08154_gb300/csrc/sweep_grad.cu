// sweep_grad.cu -- the batch kernel in gradient mode (FP64): it rebuilds the
// accumulators A(R) of each batch exactly as the sweep does, then scatters the
// derivative of E_PT2 with respect to h and the packed integrals (recomputing
// the matrix elements; nothing is stored from the forward sweep).
#include "sweep_impl.cuh"

namespace qp {

cudaError_t launch_batch_grad(int nint, const SweepParams& p, int grid, size_t smem, cudaStream_t st) {
  return batch_launch<double, true>(nint, p, grid, smem, st);
}

}  // namespace qp
