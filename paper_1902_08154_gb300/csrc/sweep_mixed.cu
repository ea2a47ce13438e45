// sweep_mixed.cu -- the mixed-precision batch kernels (FP32 integral gathers and
// products; exact accumulation, denominators and reductions as in the FP64
// sweep); see sweep_impl.cuh.
#include "sweep_impl.cuh"

namespace qp {

cudaError_t launch_batch_mixed(int nint, const SweepParams& p, int grid, size_t smem, cudaStream_t st) {
  return batch_launch<float>(nint, p, grid, smem, st);
}

cudaError_t launch_wave_multi_mixed(int nint, const MultiWaveInline& m, int total_slots, int grid, size_t smem,
                                    cudaStream_t st) {
  return multi_wave_launch<float>(nint, m, total_slots, grid, smem, st);
}

cudaError_t launch_compact_multi_mixed(int nint, const SweepParams* ps, int n, int grid, cudaStream_t st) {
  return multi_compact_launch<float>(nint, ps, n, grid, st);
}

int batch_multi_blocks_per_sm_mixed(int nint, size_t smem) { return multi_blocks_per_sm<float>(nint, smem); }

int batch_blocks_per_sm_mixed(int nint, size_t smem) {
  return nint == 1 ? blocks_per_sm<batch_kernel<1, float>>(kThreads, smem) : blocks_per_sm<batch_kernel<2, float>>(kThreads, smem);
}

}  // namespace qp
