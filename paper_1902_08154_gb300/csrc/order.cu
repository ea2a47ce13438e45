// order.cu -- the generator order and the order of the selected determinants
// by counting: every element's rank is the number of elements before it.
// n^2 comparisons in one launch beat the radix sorts of 64-bit keys (8 passes
// each, two for the generators, one per key word and |e| for the selection)
// up to some 10^4 elements: 50 determinants and 100 candidates take 5 + 4 us
// instead of five single-tile sorts of 14.5 us and their 7 helper kernels.
#include <cuda_runtime.h>

#include "common.cuh"

namespace qp {

// A call that sweeps one generator, counting against sorting: 4,096
// determinants 183 against 340 us, 10^4 386 against 439 (count_rank_kernel 168
// of it), 12,288 443 against 458, 16,384 606 against 485; two words per spin
// 12,288 531 against 549, 16,384 677 against 559.
constexpr int64_t kCountRankMax = 12288;
// A sweep of 60 determinants, 40 orbitals: 1,000 candidates 486 against 598 us,
// 4,000 601 against 949, 8,000 803 against 1,080 (two words 1,024 against
// 1,510).  Counting was still ahead with 20,000 (1,747 against 1,830), where
// its n^2 is near the sorts' cost; the line keeps a margin.
constexpr int kCountSelectMax = 8192;

int64_t count_rank_max() { return kCountRankMax; }
int count_select_max() { return kCountSelectMax; }

namespace {

constexpr int kT = 256;  // a block ranks 32 elements, a warp comparing them with every eighth tile row

// Occupations and coefficients checked (flags as validate_kernel sets them),
// duplicates found by comparison, and the generator order: decreasing c^2
// (increasing ~bits(c*c)), ties by index.
template <int NINT>
__global__ void __launch_bounds__(kT) count_rank_kernel(int n, int norb, int na, int nb, const uint64_t* __restrict__ dets,
                                                        const double* __restrict__ coefs, int32_t* order, int32_t* rank_of,
                                                        int* err, unsigned long long* cmax, unsigned long long* min_den) {
  constexpr int NW = 2 * NINT;
  __shared__ uint64_t tw[NW][kT];
  __shared__ unsigned long long tk[kT];
  __shared__ int cnt[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, i = blockIdx.x * 32 + lane;
  if (blockIdx.x == 0 && tid == 0) *min_den = 0x7FF0000000000000ull;
  if (tid < 32) cnt[tid] = 0;
  uint64_t w[NW];
  double c = 0.0;
#pragma unroll
  for (int k = 0; k < NW; k++) w[k] = i < n ? dets[(size_t)i * NW + k] : 0ull;
  if (i < n) c = coefs[i];
  const unsigned long long key = ~(unsigned long long)__double_as_longlong(c * c);
  if (warp == 0) {
    int bad = 0;
    unsigned long long m = 0;
    if (i < n) {
#pragma unroll
      for (int s = 0; s < 2; s++) {
        int e = 0;
#pragma unroll
        for (int k = 0; k < NINT; k++) {
          const uint64_t x = w[s * NINT + k];
          const int lim = norb - 64 * k;  // orbitals of this word
          e += __popcll(x);
          if (lim < 64 && (x & (lim <= 0 ? ~0ull : ~((1ull << lim) - 1)))) bad |= 1;
        }
        if (e != (s == 0 ? na : nb)) bad |= 1;
      }
      if (!isfinite(c)) bad |= 4;
      else m = (unsigned long long)__double_as_longlong(fabs(c));
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const unsigned long long v = __shfl_xor_sync(0xffffffffu, m, o);
      m = v > m ? v : m;
    }
    if (lane == 0) atomicMax(cmax, m);
    if (bad) atomicOr(err, bad);
  }
  int before = 0;
  bool dup = false;
  for (int t0 = 0; t0 < n; t0 += kT) {
    __syncthreads();
    const int j = t0 + tid;
    if (j < n) {
#pragma unroll
      for (int k = 0; k < NW; k++) tw[k][tid] = dets[(size_t)j * NW + k];
      const double cj = coefs[j];
      tk[tid] = ~(unsigned long long)__double_as_longlong(cj * cj);
    }
    __syncthreads();
    const int e = min(32 * warp + 32, n - t0);
#pragma unroll 4
    for (int r = 32 * warp; r < e; r++) {
      const unsigned long long kj = tk[r];
      before += kj < key || (kj == key && t0 + r < i);
      bool same = t0 + r != i;
#pragma unroll
      for (int k = 0; k < NW; k++) same = same && tw[k][r] == w[k];
      dup |= same;
    }
  }
  atomicAdd(&cnt[lane], before);
  __syncthreads();
  if (i < n && dup) atomicOr(err, 2);
  if (warp == 0 && i < n) {
    rank_of[i] = cnt[lane];
    order[cnt[lane]] = i;
  }
}

// The best min(n, k) of n = *ncand distinct candidates, best first: |e|
// decreasing, then the key words increasing.  More candidates than this
// kernel is for: left to the sorts.
template <int NINT>
__global__ void __launch_bounds__(kT) count_select_kernel(const int* __restrict__ ncand, long long k,
                                                          const double* __restrict__ ce, const double* __restrict__ ca,
                                                          const uint64_t* __restrict__ ck, uint64_t* sel, double* se,
                                                          double* sn) {
  constexpr int NW = 2 * NINT;
  const int n = *ncand;
  if (n > kCountSelectMax || (int)blockIdx.x * 32 >= n) return;
  __shared__ unsigned long long te[kT];
  __shared__ int cnt[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, i = blockIdx.x * 32 + lane;
  if (tid < 32) cnt[tid] = 0;
  const unsigned long long e0 = i < n ? (unsigned long long)__double_as_longlong(fabs(ce[i])) : 0ull;
  int before = 0;
  for (int t0 = 0; t0 < n; t0 += kT) {
    __syncthreads();
    if (t0 + tid < n) te[tid] = (unsigned long long)__double_as_longlong(fabs(ce[t0 + tid]));
    __syncthreads();
    const int e = min(32 * warp + 32, n - t0);
#pragma unroll 4
    for (int r = 32 * warp; r < e; r++) {
      bool b = te[r] > e0;
      if (te[r] == e0 && i < n && t0 + r != i) {  // a tie in |e|: the keys decide
        const uint64_t *x = ck + (size_t)(t0 + r) * NW, *y = ck + (size_t)i * NW;
        int w = 0;
        while (w < NW - 1 && x[w] == y[w]) w++;
        b = x[w] < y[w];
      }
      before += b;
    }
  }
  atomicAdd(&cnt[lane], before);
  __syncthreads();
  const int r = cnt[lane];
  if (warp == 0 && i < n && r < k) {
    if (sel)
#pragma unroll
      for (int w = 0; w < NW; w++) sel[(size_t)r * NW + w] = ck[(size_t)i * NW + w];
    if (se) se[r] = ce[i];
    if (sn) sn[r] = ca[i];
  }
}

}  // namespace

cudaError_t launch_count_rank(int nint, int64_t n, int norb, int na, int nb, const uint64_t* dets, const double* coefs,
                              int32_t* order, int32_t* rank_of, int* err, unsigned long long* cmax,
                              unsigned long long* min_den, cudaStream_t st) {
  const unsigned grid = (unsigned)((n + 31) / 32);
  if (nint == 1)
    count_rank_kernel<1><<<grid, kT, 0, st>>>((int)n, norb, na, nb, dets, coefs, order, rank_of, err, cmax, min_den);
  else
    count_rank_kernel<2><<<grid, kT, 0, st>>>((int)n, norb, na, nb, dets, coefs, order, rank_of, err, cmax, min_den);
  return cudaGetLastError();
}

cudaError_t launch_count_select(int nint, size_t maxn, const int* ncand, int64_t k, const double* ce, const double* ca,
                                const uint64_t* ck, uint64_t* sel, double* se, double* sn, cudaStream_t st) {
  const size_t n = maxn < (size_t)kCountSelectMax ? maxn : (size_t)kCountSelectMax;
  const unsigned grid = (unsigned)((n + 31) / 32);
  if (grid == 0) return cudaSuccess;
  if (nint == 1) count_select_kernel<1><<<grid, kT, 0, st>>>(ncand, k, ce, ca, ck, sel, se, sn);
  else count_select_kernel<2><<<grid, kT, 0, st>>>(ncand, k, ce, ca, ck, sel, se, sn);
  return cudaGetLastError();
}

}  // namespace qp
