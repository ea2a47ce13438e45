// sweep.cu -- the FP64 sweep kernels (prep, batch) and their launch helpers;
// the kernels themselves are in sweep_impl.cuh, the mixed-precision batch
// kernels in sweep_mixed.cu.
#include "sweep_impl.cuh"

namespace qp {

// a + b and its rounding error.
__device__ __forceinline__ void two_sum(double& s, double& c, double v) {
  const double u = s + v;
  c += fabs(s) >= fabs(v) ? (s - u) + v : (v - u) + s;
  s = u;
}

// Per generator of the wave and per state: eps_I and sum A^2/D^2 from the
// items' slots, added with Neumaier's compensation, so that they are the same
// bits on every run and every grid size: lane l adds the items l, l + 32, ...
// in order, and the lanes' sums are added by a fixed tree.  (One thread per
// generator was a chain of 8 dependent FP64 additions per item: 25 us for 50
// generators, 104 us for 1,201 of 153 items; this takes 4 and 8 us.)
__device__ __forceinline__ void reduce_items(const SweepParams& p, const int t) {
  const int lane = threadIdx.x & 31, nst = p.nst > 1 ? p.nst : 1;
  if (t >= p.wave_slots * nst) return;
  const int slot = t / nst, st = t - slot * nst;
  const int g = p.meta[slot].g;
  const double* its = p.it_sum + (size_t)slot * p.nper * p.it_stride + 2 * st;
  double se = 0.0, ce = 0.0, ss = 0.0, cs = 0.0;
  for (int j = lane; j < p.nper; j += 32) {
    two_sum(se, ce, its[(size_t)j * p.it_stride]);
    two_sum(ss, cs, its[(size_t)j * p.it_stride + 1]);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const double ve = __shfl_xor_sync(0xffffffffu, se, o), vs = __shfl_xor_sync(0xffffffffu, ss, o);
    ce += __shfl_xor_sync(0xffffffffu, ce, o);
    cs += __shfl_xor_sync(0xffffffffu, cs, o);
    two_sum(se, ce, ve);
    two_sum(ss, cs, vs);
  }
  if (g < 0 || lane) return;
  p.eps[(size_t)st * p.ndet + g] = se + ce;
  p.s2[(size_t)st * p.ndet + g] = ss + cs;
}

constexpr int kReduceThreads = 128;  // four generators per block

__global__ void reduce_items_kernel(const __grid_constant__ SweepParams p) {
  reduce_items(p, (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5));
}

// Instance blockIdx.y of a multi-instance wave.
__global__ void reduce_items_multi_kernel(const SweepParams* __restrict__ ps) {
  reduce_items(ps[blockIdx.y], (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5));
}

cudaError_t launch_reduce_items(const SweepParams& p, cudaStream_t st) {
  const int n = p.wave_slots * (p.nst > 1 ? p.nst : 1), per = kReduceThreads / 32;
  if (n > 0) reduce_items_kernel<<<(n + per - 1) / per, kReduceThreads, 0, st>>>(p);
  return cudaGetLastError();
}

// max_slots: the most slots any of the n instances has in this wave (one
// state each).
cudaError_t launch_reduce_items_multi(const SweepParams* ps, int n, int max_slots, cudaStream_t st) {
  const int per = kReduceThreads / 32;
  if (n > 0 && max_slots > 0)
    reduce_items_multi_kernel<<<dim3((max_slots + per - 1) / per, n), kReduceThreads, 0, st>>>(ps);
  return cudaGetLastError();
}

cudaError_t launch_wave_multi_mixed(int nint, const MultiWaveInline& m, int total_slots, int grid, size_t smem,
                                    cudaStream_t st);
cudaError_t launch_compact_multi_mixed(int nint, const SweepParams* ps, int n, int grid, cudaStream_t st);
int batch_multi_blocks_per_sm_mixed(int nint, size_t smem);

// The prep and batch launches of one wave of several instances: the prep
// kernel reads the pieces' parameters from the device table m.ps, the batch
// kernel from its own parameters mi.
cudaError_t launch_wave_multi(int nint, int mixed, const MultiWave& m, const MultiWaveInline& mi, int total_slots,
                              int grid, size_t smem, cudaStream_t st) {
  if (total_slots <= 0) return cudaSuccess;
  size_t ps = 0;
  for (int i = 0; i < mi.n; i++) {
    const size_t b = 4 * (size_t)mi.ps[i].mask_w + 8 * (size_t)mi.ps[i].orb_w;
    ps = b > ps ? b : ps;
  }
  const cudaError_t e = nint == 1 ? launch_smem<prep_multi_kernel<1>>(m, total_slots, ps, st)
                                  : launch_smem<prep_multi_kernel<2>>(m, total_slots, ps, st);
  if (e != cudaSuccess) return e;
  if (mixed) return launch_wave_multi_mixed(nint, mi, total_slots, grid, smem, st);
  return multi_wave_launch<double>(nint, mi, total_slots, grid, smem, st);
}

cudaError_t launch_compact_multi(int nint, int mixed, const SweepParams* ps, int n, int grid, cudaStream_t st) {
  if (mixed) return launch_compact_multi_mixed(nint, ps, n, grid, st);
  return multi_compact_launch<double>(nint, ps, n, grid, st);
}

int batch_multi_blocks_per_sm(int nint, int mixed, size_t smem) {
  if (mixed) return batch_multi_blocks_per_sm_mixed(nint, smem);
  return multi_blocks_per_sm<double>(nint, smem);
}

template __global__ void prep_kernel<1>(const __grid_constant__ SweepParams);
template __global__ void prep_kernel<2>(const __grid_constant__ SweepParams);
template __global__ void grad_gen_kernel<1>(const __grid_constant__ SweepParams);
template __global__ void grad_gen_kernel<2>(const __grid_constant__ SweepParams);

cudaError_t launch_batch_grad(int nint, const SweepParams& p, int grid, size_t smem, cudaStream_t st);

cudaError_t launch_grad_gen(int nint, const SweepParams& p, int ngen, cudaStream_t st) {
  if (nint == 1) grad_gen_kernel<1><<<ngen, kThreads, 0, st>>>(p);
  else grad_gen_kernel<2><<<ngen, kThreads, 0, st>>>(p);
  return cudaGetLastError();
}

cudaError_t launch_batch_mixed(int nint, const SweepParams& p, int grid, size_t smem, cudaStream_t st);
int batch_blocks_per_sm_mixed(int nint, size_t smem);

// Dynamic shared memory of the prep kernel: a slot's ban masks.
static size_t prep_smem(const SweepParams& p) { return 4 * (size_t)p.mask_w + 8 * (size_t)p.orb_w; }

cudaError_t launch_prep(int nint, const SweepParams& p, int slots, cudaStream_t st) {
  const size_t smem = prep_smem(p);
  return nint == 1 ? launch_smem<prep_kernel<1>>(p, slots, smem, st) : launch_smem<prep_kernel<2>>(p, slots, smem, st);
}

cudaError_t launch_batch(int nint, const SweepParams& p, int grid, size_t smem, cudaStream_t st) {
  if (p.mixed) return launch_batch_mixed(nint, p, grid, smem, st);
  return batch_launch<double>(nint, p, grid, smem, st);
}

int batch_blocks_per_sm(int nint, int mixed, size_t smem) {
  if (mixed) return batch_blocks_per_sm_mixed(nint, smem);
  return nint == 1 ? blocks_per_sm<batch_kernel<1, double>>(kThreads, smem) : blocks_per_sm<batch_kernel<2, double>>(kThreads, smem);
}

int sweep_threads() { return kThreads; }

}  // namespace qp
