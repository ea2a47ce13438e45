// davidson.cu -- the Hamiltonian over Psi0 and its lowest eigenpair on sm_103a
// (Quantum Package 2.0, arXiv:1902.08154, Sec. "Davidson diagonalization":
// the variational step of CIPSI, E0 and c_I as the lowest eigenpair of H in
// the internal space).
//
//   * H is built once per call as a CSR matrix of the pairs (I, J) at
//     excitation degree 1 or 2 (Slater-Condon rules, Eqs. Hij), plus its
//     diagonal.  Pairs are found through the spin-up and spin-down strings
//     of the determinants (the paper's DISCIUS-like search, see below) into
//     a bit map per row, read off with ascending columns, or, as a
//     cross-check, by a tiled all-pairs test (each CTA keeps a tile of rows in
//     shared memory and streams every determinant once) whose pairs are then
//     sorted by column within each row; the products below add in a fixed order.
//   * sigma = H u by a warp per row, a block for the longest rows.
//   * Davidson's method (E. R. Davidson, J. Comput. Phys. 17, 87 (1975)) with
//     the diagonal preconditioner t = r / (theta - H_II): basis vectors,
//     their products with H and every dot product stay on the device; only
//     the small subspace matrix goes to the host, where its lowest
//     eigenpair is found through a tridiagonal matrix (Golub & Van Loan,
//     Secs. 8.3 and 8.4).
#include <cuda_runtime.h>

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>
#include <cub/device/device_segmented_radix_sort.cuh>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "../../include/qp_pt2.h"
#include "common.cuh"
#include "lowest_eigenpair.h"

namespace qp {
namespace {

constexpr int kRows = 64;  // rows of H per CTA in the pair search
constexpr int kMaxBasis = 32;

#define DV_TRY(expr)                                                \
  do {                                                              \
    cudaError_t e_ = (expr);                                        \
    if (e_ != cudaSuccess) return report(QP_ECUDA, cudaGetErrorString(e_)); \
  } while (0)

// Up to two set bits of m (spin-orbital codes base + bit), in ascending order.
template <int NINT>
__device__ __forceinline__ void take_bits(const uint64_t* m, int base, int* out, int* n) {
#pragma unroll
  for (int w = 0; w < NINT; w++) {
    uint64_t b = m[w];
    while (b && *n < 2) {
      out[(*n)++] = base + 64 * w + __ffsll((long long)b) - 1;
      b &= b - 1;
    }
  }
}

// <I|H|J> for two determinants at excitation degree 1 or 2: holes are the
// spin orbitals of I missing from J, particles those of J missing from I.
template <int NINT>
__device__ double hij_pair(const uint64_t* I, const uint64_t* J, int norb, const double* h, const double* eri) {
  int ho[2], pa[2], nh = 0, np = 0;
  for (int s = 0; s < 2; s++) {
    uint64_t x[NINT], y[NINT];
#pragma unroll
    for (int w = 0; w < NINT; w++) {
      x[w] = I[s * NINT + w] & ~J[s * NINT + w];
      y[w] = J[s * NINT + w] & ~I[s * NINT + w];
    }
    take_bits<NINT>(x, s * norb, ho, &nh);
    take_bits<NINT>(y, s * norb, pa, &np);
  }
  if (nh == 1) {  // single a -> b: h_ab + sum_{q in I} [(ab|qq) - delta (aq|qb)]
    const int s = ho[0] >= norb, a = ho[0] - s * norb, b = pa[0] - s * norb;
    double v = h[a * norb + b];
    for (int t = 0; t < 2; t++) {
#pragma unroll
      for (int w = 0; w < NINT; w++) {
        uint64_t bits = I[t * NINT + w];
        while (bits) {
          const int q = 64 * w + __ffsll((long long)bits) - 1;
          bits &= bits - 1;
          v += eri[eri_index(a, b, q, q)];
          if (t == s) v -= eri[eri_index(a, q, q, b)];
        }
      }
    }
    const int par = count_between<NINT>(I + s * NINT, a < b ? a : b, a < b ? b : a) & 1;
    return par ? -v : v;
  }
  // double: holes h1 < h2 and particles p1 < p2 (codes), paired 1-1 and 2-2
  const int s1 = ho[0] >= norb, s2 = ho[1] >= norb;
  const int h1 = ho[0] - s1 * norb, h2 = ho[1] - s2 * norb;
  const int p1 = pa[0] - s1 * norb, p2 = pa[1] - s2 * norb;
  uint64_t w1[NINT];
#pragma unroll
  for (int w = 0; w < NINT; w++) w1[w] = I[s1 * NINT + w];
  int par = count_between<NINT>(w1, h1 < p1 ? h1 : p1, h1 < p1 ? p1 : h1);
#pragma unroll
  for (int w = 0; w < NINT; w++) {  // apply h1 -> p1, then count h2 -> p2 on the result
    if (w == (h1 >> 6)) w1[w] &= ~(1ull << (h1 & 63));
    if (w == (p1 >> 6)) w1[w] |= 1ull << (p1 & 63);
  }
  par += (s1 == s2) ? count_between<NINT>(w1, h2 < p2 ? h2 : p2, h2 < p2 ? p2 : h2)
                    : count_between<NINT>(I + s2 * NINT, h2 < p2 ? h2 : p2, h2 < p2 ? p2 : h2);
  double v = eri[eri_index(h1, p1, h2, p2)];
  if (s1 == s2) v -= eri[eri_index(h1, p2, h2, p1)];
  return (par & 1) ? -v : v;
}

// H_II = sum_i h_ii + sum_{i<j} [(ii|jj) - delta_spin (ij|ji)] over I's spin orbitals.
template <int NINT>
__global__ void diag_kernel(int64_t n, const uint64_t* dets, int norb, const double* h, const double* Jm,
                            const double* Km, double* diag) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t* d = dets + i * 2 * NINT;
  int occ[kMaxElec], ne = 0;
  for (int s = 0; s < 2; s++)
    for (int w = 0; w < NINT; w++) {
      uint64_t b = d[s * NINT + w];
      while (b && ne < kMaxElec) {
        occ[ne++] = s * norb + 64 * w + __ffsll((long long)b) - 1;
        b &= b - 1;
      }
    }
  double e = 0.0;
  for (int a = 0; a < ne; a++) {
    const int sa = occ[a] >= norb, pa = occ[a] - sa * norb;
    e += h[pa * norb + pa];
    for (int b = 0; b < a; b++) {
      const int sb = occ[b] >= norb, pb = occ[b] - sb * norb;
      e += Jm[pa * norb + pb];
      if (sa == sb) e -= Km[pa * norb + pb];
    }
  }
  diag[i] = e;
}

// Pair search over a tile of kRows rows: COUNT pass writes row counts,
// otherwise (col, <I|H|J>) pairs go to each row's next free slots.
template <int NINT, bool COUNT>
__global__ void pairs_kernel(int64_t n, const uint64_t* dets, int norb, const double* h, const double* eri,
                             int64_t* rowcnt, const int64_t* rowptr, int* cursor, int* cols, double* vals, int* err) {
  constexpr int NW = 2 * NINT;
  __shared__ uint64_t rows[kRows][NW];
  __shared__ int cnt[kRows];
  const int64_t r0 = (int64_t)blockIdx.x * kRows;
  const int nr = (int)((n - r0) < kRows ? (n - r0) : kRows);
  for (int t = threadIdx.x; t < nr * NW; t += blockDim.x) rows[t / NW][t % NW] = dets[(r0 + t / NW) * NW + t % NW];
  if (threadIdx.x < kRows) cnt[threadIdx.x] = 0;
  __syncthreads();
  for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
    uint64_t J[NW];
#pragma unroll
    for (int w = 0; w < NW; w++) J[w] = dets[j * NW + w];
    for (int r = 0; r < nr; r++) {
      int x = 0;
#pragma unroll
      for (int w = 0; w < NW; w++) x += __popcll(rows[r][w] ^ J[w]);
      if (x > 4) continue;
      if (x == 0) {
        if (r0 + r != j) atomicOr(err, 1);  // a repeated determinant
        continue;
      }
      if (COUNT) {
        atomicAdd(&cnt[r], 1);
      } else {
        const int64_t pos = rowptr[r0 + r] + atomicAdd(&cursor[r0 + r], 1);
        cols[pos] = (int)j;
        vals[pos] = hij_pair<NINT>(rows[r], J, norb, h, eri);
      }
    }
  }
  if (COUNT) {
    __syncthreads();
    if (threadIdx.x < nr) rowcnt[r0 + threadIdx.x] = cnt[threadIdx.x];
  }
}

// ---------------------------------------------------------------------------
// Connected pairs through the alpha and beta strings (Appendix "Davidson
// diagonalization": Psi0 = sum C_IJ |I_up J_dn>, same-spin excitations found
// along a row or a column of C, opposite-spin doubles by a spin-up single
// excitation followed by a spin-down one).  The determinants are grouped by
// their spin-up string and by their spin-down string; for row I:
//   (a) J with the spin-down string of I: spin-up excitation of degree 1 or 2;
//   (b) J with the spin-up string of I: spin-down excitation of degree 1 or 2;
//   (c) J whose spin-up string is a single excitation of I's (the string
//       neighbour lists) and whose spin-down string is a single excitation of
//       I's: the opposite-spin doubles.
// Every connected pair is met exactly once, and the work per row is the
// length of its lists instead of N_det.
// ---------------------------------------------------------------------------
struct SpinStrings {
  int nu = 0;             // distinct strings
  int* sid = nullptr;     // [n] string index of each determinant
  int* ptr = nullptr;     // [nu + 1] offsets into grp
  int* grp = nullptr;     // [n] determinants ordered by string
  uint64_t* ukey = nullptr;  // [nu][nint] the distinct strings
  int* nb_ptr = nullptr;  // [nu + 1] single-excitation neighbours (spin-up strings only)
  int* nb = nullptr;
};

__global__ void str_key_kernel(int64_t n, int nw, int off, const uint64_t* dets, const int* perm,
                               unsigned long long* key, int* val) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int j = perm ? perm[i] : (int)i;
  key[i] = dets[(size_t)j * nw + off];
  val[i] = j;
}

template <int NINT>
__global__ void str_flag_kernel(int64_t n, int spin, const uint64_t* dets, const int* grp, int* flag) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int f = (i == 0);
  if (i > 0) {
    const uint64_t* a = dets + (size_t)grp[i] * 2 * NINT + spin * NINT;
    const uint64_t* b = dets + (size_t)grp[i - 1] * 2 * NINT + spin * NINT;
#pragma unroll
    for (int w = 0; w < NINT; w++) f |= (a[w] != b[w]);
  }
  flag[i] = f;
}

template <int NINT>
__global__ void str_index_kernel(int64_t n, int spin, const uint64_t* dets, const int* grp, const int* flag,
                                 const int* incl, int* sid, int* ptr, uint64_t* ukey) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int id = incl[i] - 1;
  sid[grp[i]] = id;
  if (flag[i]) {
    ptr[id] = (int)i;
#pragma unroll
    for (int w = 0; w < NINT; w++) ukey[(size_t)id * NINT + w] = dets[(size_t)grp[i] * 2 * NINT + spin * NINT + w];
  }
}

// Single-excitation neighbours among the distinct strings (count, then fill),
// a warp per string (a thread per string took 190 us for 3,000 of them).
template <int NINT, bool COUNT>
__global__ void str_nb_kernel(int nu, const uint64_t* ukey, int* cnt, const int* nb_ptr, int* nb) {
  const int u = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (u >= nu) return;
  uint64_t a[NINT];
#pragma unroll
  for (int w = 0; w < NINT; w++) a[w] = ukey[(size_t)u * NINT + w];
  int c = COUNT ? 0 : nb_ptr[u];
  for (int v0 = 0; v0 < nu; v0 += 32) {
    const int v = v0 + lane;
    int d = 0;
    if (v < nu)
#pragma unroll
      for (int w = 0; w < NINT; w++) d += __popcll(a[w] ^ ukey[(size_t)v * NINT + w]);
    const unsigned hit = __ballot_sync(0xffffffffu, d == 2);
    if (!COUNT && d == 2) nb[c + __popc(hit & ((1u << lane) - 1u))] = v;
    c += __popc(hit);
  }
  if (COUNT && lane == 0) cnt[u] = c;
}

template <int NINT>
__device__ __forceinline__ int spin_degree(const uint64_t* I, const uint64_t* J, int spin) {
  int d = 0;
#pragma unroll
  for (int w = 0; w < NINT; w++) d += __popcll(I[spin * NINT + w] ^ J[spin * NINT + w]);
  return d >> 1;
}

// One block per row I.  COUNT: the number of connected J; otherwise they are
// marked in a bit map of the determinants (shared memory; `win` of them at a
// time) and the columns read off it in ascending order, so that nothing is
// sorted.  A row with so few that the map's words would cost more than
// comparing them with each other is ranked by counting instead (10^6
// determinants without connections to speak of: 138 ms with the map for every
// row and in both passes, 22.9 for a warp per row and the sort, 12.7 so).
// Spin-up neighbour strings with few determinants take a thread
// each, the others a warp.  (A warp per row that evaluated each element as it
// found it and drew its slot from a global counter, and a segmented sort of
// the pairs, took 2.9 ms for 10^4 determinants, 6.2e6 elements; the two passes
// of this kernel and the values take 0.58.)
constexpr int kMapThreads = 256;
constexpr int kMapQueue = 512;
constexpr int kFew = 512;  // columns ranked by counting at most
constexpr int64_t kMapMax = 1 << 20;  // determinants per window: 128 KB of map

template <int NINT, bool COUNT>
__global__ void __launch_bounds__(kMapThreads) str_pairs_kernel(
    int64_t n, int win, const uint64_t* __restrict__ dets, const int* __restrict__ aid, const int* __restrict__ aptr,
    const int* __restrict__ agrp, const int* __restrict__ anb_ptr, const int* __restrict__ anb,
    const int* __restrict__ bid, const int* __restrict__ bptr, const int* __restrict__ bgrp, int64_t* rowcnt,
    const int64_t* rowptr, int* cols, int* err) {
  constexpr int NW = 2 * NINT;
  extern __shared__ uint32_t map[];
  __shared__ int queue[kMapQueue], nq, wsum[kMapThreads / 32], hit[COUNT ? 1 : kFew], nhit;
  const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint64_t I[NW];
#pragma unroll
  for (int w = 0; w < NW; w++) I[w] = dets[(size_t)row * NW + w];
  const int a = aid[row], b = bid[row];
  const int64_t q0 = COUNT ? 0 : rowptr[row], len = COUNT ? 0 : rowptr[row + 1] - q0;
  if (!COUNT && len == 0) return;
  // comparisons against three passes over the map's words
  const bool few = !COUNT && len <= kFew && len * ((len + kMapThreads - 1) / kMapThreads * kMapThreads) <= 3 * (n / 32);
  int found = 0;  // COUNT: by this thread
  int64_t done = 0;
  for (int64_t lo = 0; lo < n; lo += COUNT || few ? n : win) {
    const int nbits = (int)(n - lo < win ? n - lo : win), nwords = COUNT || few ? 0 : (nbits + 31) / 32;
    for (int w = tid; w < nwords; w += kMapThreads) map[w] = 0u;
    if (tid == 0) nq = nhit = 0;
    __syncthreads();
    auto mark = [&](int j) {
      if (COUNT) {
        found++;
        return;
      }
      if (few) {
        const int at = atomicAdd(&nhit, 1);
        if (at < kFew) hit[COUNT ? 0 : at] = j;
        return;
      }
      const int64_t at = j - lo;
      if (at >= 0 && at < nbits) atomicOr(&map[at >> 5], 1u << (at & 31));
    };
    for (int k = bptr[b] + tid; k < bptr[b + 1]; k += kMapThreads) {  // (a) the same spin-down string
      const int j = bgrp[k];
      if (j == row) continue;
      const int d = spin_degree<NINT>(I, dets + (size_t)j * NW, 0);
      if (d == 0) atomicOr(err, 1);  // a repeated determinant
      else if (d <= 2) mark(j);
    }
    for (int k = aptr[a] + tid; k < aptr[a + 1]; k += kMapThreads) {  // (b) the same spin-up string
      const int j = agrp[k];
      if (j == row) continue;
      const int d = spin_degree<NINT>(I, dets + (size_t)j * NW, 1);
      if (d >= 1 && d <= 2) mark(j);
    }
    auto pair = [&](int k) {
      const int j = agrp[k];
      if (spin_degree<NINT>(I, dets + (size_t)j * NW, 1) == 1) mark(j);
    };
    for (int q = anb_ptr[a] + tid; q < anb_ptr[a + 1]; q += kMapThreads) {  // (c) spin-up single, then spin-down single
      const int a2 = anb[q], k0 = aptr[a2], k1 = aptr[a2 + 1];
      if (k1 - k0 > 8) {
        const int at = atomicAdd(&nq, 1);
        if (at < kMapQueue) {
          queue[at] = a2;
          continue;
        }
      }
      for (int k = k0; k < k1; k++) pair(k);
    }
    __syncthreads();
    const int nbig = nq < kMapQueue ? nq : kMapQueue;
    for (int q = warp; q < nbig; q += kMapThreads / 32)
      for (int k = aptr[queue[q]] + lane, e = aptr[queue[q] + 1]; k < e; k += 32) pair(k);
    __syncthreads();
    if (few) {
      for (int i = tid; i < (int)len; i += kMapThreads) {
        const int j = hit[COUNT ? 0 : i];
        int before = 0;
#pragma unroll 4
        for (int k = 0; k < (int)len; k++) before += hit[COUNT ? 0 : k] < j;
        cols[q0 + before] = j;
      }
      return;
    }
    if (COUNT) break;
    // a contiguous run of words per thread, of odd length: 32 banks
    const int per = ((nwords + kMapThreads - 1) / kMapThreads) | 1, w0 = min(tid * per, nwords), w1 = min(w0 + per, nwords);
    int c = 0;
    for (int w = w0; w < w1; w++) c += __popc(map[w]);
    int at = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += v;
    }
    if (lane == 31) wsum[warp] = at;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int w = 0; w < kMapThreads / 32; w++) {
      before += w < warp ? wsum[w] : 0;
      all += wsum[w];
    }
    int* out = cols + q0 + done + before + at - c;
    for (int w = w0; w < w1; w++)
      for (uint32_t m = map[w]; m; m &= m - 1) *out++ = (int)(lo + 32 * w + __ffs((int)m) - 1);
    done += all;
    __syncthreads();
  }
  if (COUNT) {
    found = __reduce_add_sync(0xffffffffu, found);
    if (lane == 0) wsum[warp] = found;
    __syncthreads();
    if (tid == 0) {
      int64_t all = 0;
      for (int w = 0; w < kMapThreads / 32; w++) all += wsum[w];
      rowcnt[row] = all;
    }
  }
}

// The elements of the columns found: a block per row, a thread per element;
// single excitations, whose sums run over the occupied orbitals, are listed
// and taken together, so that a warp of doubles does not wait for one of them
// (533 -> 200 us for 6.2e6 elements).
constexpr int kValThreads = 128, kSingles = 1024;
template <int NINT>
__global__ void __launch_bounds__(kValThreads) str_vals_kernel(const uint64_t* __restrict__ dets, int norb,
                                                               const double* __restrict__ h,
                                                               const double* __restrict__ eri,
                                                               const int64_t* __restrict__ rowptr,
                                                               const int* __restrict__ cols, double* __restrict__ vals) {
  constexpr int NW = 2 * NINT;
  __shared__ int single[kSingles], ns;
  const int64_t row = blockIdx.x, q0 = rowptr[row];
  const int len = (int)(rowptr[row + 1] - q0);
  uint64_t I[NW];
#pragma unroll
  for (int w = 0; w < NW; w++) I[w] = dets[(size_t)row * NW + w];
  if (threadIdx.x == 0) ns = 0;
  __syncthreads();
  auto element = [&](int k) {
    uint64_t J[NW];
    const uint64_t* p = dets + (size_t)cols[q0 + k] * NW;
#pragma unroll
    for (int w = 0; w < NW; w++) J[w] = p[w];
    vals[q0 + k] = hij_pair<NINT>(I, J, norb, h, eri);
  };
  for (int k = threadIdx.x; k < len; k += kValThreads) {
    const uint64_t* p = dets + (size_t)cols[q0 + k] * NW;
    int x = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) x += __popcll(I[w] ^ p[w]);
    if (x == 2) {
      const int at = atomicAdd(&ns, 1);
      if (at < kSingles) {
        single[at] = k;
        continue;
      }
    }
    element(k);
  }
  __syncthreads();
  for (int q = threadIdx.x, e = ns < kSingles ? ns : kSingles; q < e; q += kValThreads) element(single[q]);
}

// Y[k] = H X[k] for nvec vectors of length n: a warp per row, and the whole
// block for those of its rows that are longer than kLongRow (the row of the
// reference holds fifteen times the average; a block's rows lie apart, as the
// long ones are often neighbours).  A product costs a warp 19 cycles of the
// SM's FP64 unit, and so does each step of a sum over lanes: for the 6.2e6
// elements of 10^4 rows 12.8 us and 4, and their 75 MB take 11 us from HBM.
// 33 us; a warp per row throughout took 130 (85 of it the longest row alone),
// four warps per row 35, long rows from 1,536 on 34, and one block per SM with
// x in shared memory 34: neither the sums nor the gathers are the bound, but
// the chain of loads in each row.
constexpr int kLongRow = 4096, kSpmvLoads = 8, kSpmvThreads = 256, kSpmvRows = kSpmvThreads / 32;
__device__ __forceinline__ double row_part(int len, int first, int step, const int* __restrict__ c,
                                           const double* __restrict__ v, const double* x) {
  double a = 0.0, b = 0.0;
  for (int q = first; q < len; q += kSpmvLoads * step) {
    int cc[kSpmvLoads];
    double vv[kSpmvLoads];
#pragma unroll
    for (int u = 0; u < kSpmvLoads; u++) {
      const bool ok = q + u * step < len;
      cc[u] = ok ? c[q + u * step] : -1;
      vv[u] = ok ? v[q + u * step] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < kSpmvLoads; u += 2) {
      if (cc[u] >= 0) a = fma(vv[u], x[cc[u]], a);
      if (cc[u + 1] >= 0) b = fma(vv[u + 1], x[cc[u + 1]], b);
    }
  }
  a += b;
#pragma unroll
  for (int o = 16; o; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}

__global__ void __launch_bounds__(kSpmvThreads) spmv_kernel(int64_t n, int nvec, const int64_t* __restrict__ rowptr,
                                                            const int* __restrict__ cols,
                                                            const double* __restrict__ vals,
                                                            const double* __restrict__ diag,
                                                            const double* __restrict__ X, double* __restrict__ Y) {
  __shared__ double part[kSpmvRows];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t own = blockIdx.x + (int64_t)warp * gridDim.x;
  const int64_t row = own < n ? own : n - 1, q0 = rowptr[row];
  const int len = own < n ? (int)(rowptr[row + 1] - q0) : -1;  // -1: no row
  const int any = __syncthreads_or(len > kLongRow);
  for (int k = 0; k < nvec; k++) {
    const double* x = X + (size_t)k * n;
    double* y = Y + (size_t)k * n;
    if (len >= 0 && len <= kLongRow) {
      const double s = row_part(len, lane, 32, cols + q0, vals + q0, x);
      if (lane == 0) y[row] = fma(diag[row], x[row], s);
    }
    if (!any) continue;
    for (int64_t r = blockIdx.x; r < n; r += gridDim.x) {
      const int64_t p0 = rowptr[r], p1 = rowptr[r + 1];
      if (p1 - p0 <= kLongRow) continue;
      const double s = row_part((int)(p1 - p0), threadIdx.x, kSpmvThreads, cols + p0, vals + p0, x);
      if (lane == 0) part[warp] = s;
      __syncthreads();
      if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kSpmvRows; w++) t += part[w];
        y[r] = fma(diag[r], x[r], t);
      }
      __syncthreads();
    }
  }
}

// out[kDotParts k + p] = part p of V[k] . y for k < m, and of z . z at k = m
// where z is given.  A block per part: one SM's FP64 unit alone takes 3 us for
// a product over 10^4 elements.
constexpr int kDotThreads = 256, kDotParts = 8;
__global__ void __launch_bounds__(kDotThreads) dots_kernel(int64_t n, int m, const double* __restrict__ V,
                                                           const double* __restrict__ y, const double* __restrict__ z,
                                                           double* out) {
  const int k = blockIdx.x / kDotParts, p = blockIdx.x % kDotParts;
  const double* a = k < m ? V + (size_t)k * n : z;
  const double* b = k < m ? y : z;
  const int64_t lo = n * p / kDotParts, hi = n * (p + 1) / kDotParts;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  int64_t i = lo + threadIdx.x;
  for (; i + 3 * kDotThreads < hi; i += 4 * kDotThreads)
#pragma unroll
    for (int u = 0; u < 4; u++) acc[u] = fma(a[i + u * kDotThreads], b[i + u * kDotThreads], acc[u]);
#pragma unroll
  for (int u = 0; u < 3; u++)
    if (i + u * kDotThreads < hi) acc[u] = fma(a[i + u * kDotThreads], b[i + u * kDotThreads], acc[u]);
  double s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
  __shared__ double part[kDotThreads / 32];
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    s = 0.0;
    for (int w = 0; w < kDotThreads / 32; w++) s += part[w];
    out[blockIdx.x] = s;
  }
}
// A product from its parts, the same sum on the host and on the device.
__host__ __device__ inline double dot_sum(const double* p) {
  double s = 0.0;
  for (int i = 0; i < kDotParts; i++) s += p[i];
  return s;
}

// The lowest Ritz vector's coefficients, passed by value.
struct Ritz {
  double s[kMaxBasis], theta;
};

// x = sum_k s_k V_k, w = sum_k s_k W_k, r = w - theta x, t = r / (theta - H_II)
// with |theta - H_II| kept above 1e-6.  restart: x and w become the first
// basis vector and its product.
__global__ void __launch_bounds__(128) ritz_kernel(int64_t n, int m, int restart, const __grid_constant__ Ritz z, double* V,
                                                   double* W, const double* __restrict__ diag, double* x, double* w,
                                                   double* r, double* t) {
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (i >= n) return;
  double xi = 0.0, wi = 0.0;
#pragma unroll 4
  for (int k = 0; k < m; k++) {
    xi += z.s[k] * V[(size_t)k * n + i];
    wi += z.s[k] * W[(size_t)k * n + i];
  }
  const double ri = wi - z.theta * xi;
  double den = z.theta - diag[i];
  if (fabs(den) < 1e-6) den = den < 0 ? -1e-6 : 1e-6;
  x[i] = xi;
  w[i] = wi;
  r[i] = ri;
  t[i] = ri / den;
  if (restart) {
    V[i] = xi;
    W[i] = wi;
  }
}

// t - sum_k d_k V_k; norm: divided by its norm, whose square is t.t - sum d_k^2
// (d_k the second pass's products, at the rounding level of t), into out.
// d: parts of the products, t.t last.
__global__ void __launch_bounds__(128) orth_kernel(int64_t n, int m, int norm, const double* __restrict__ V,
                                                   const double* __restrict__ d, const double* t, double* out) {
  __shared__ double c[kMaxBasis + 1], rn;
  const int64_t i = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (threadIdx.x < 32) {
    const int k = threadIdx.x;
    double v = k < m ? dot_sum(d + k * kDotParts) : 0.0;
    c[k] = v;
    if (norm) {
      v *= v;
#pragma unroll
      for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (k == 0) {
        const double nn = dot_sum(d + m * kDotParts) - v;
        rn = nn > 1e-28 ? sqrt(nn) : 0.0;
      }
    }
  }
  __syncthreads();
  if (i >= n) return;
  double acc = 0.0;
#pragma unroll 4
  for (int k = 0; k < m; k++) acc += c[k] * V[(size_t)k * n + i];
  acc = t[i] - acc;
  if (norm) acc = rn > 0.0 ? acc / rn : 0.0;
  out[i] = acc;
}

// Device buffers of one call: cut from the context's workspace as far as it
// goes (one call at a time holds it), the rest allocated and freed on scope
// exit.  A call that needed more than the workspace, and not more than
// kKeepBytes in all, leaves one of the size it needed.
constexpr size_t kKeepBytes = (size_t)256 << 20;
struct DevMem {
  const CtxView& c;
  bool held;
  void* ws = nullptr;
  size_t ws_bytes = 0, off = 0, need = 0;
  std::vector<void*> ptrs;
  explicit DevMem(const CtxView& v) : c(v), held(ctx_ws_take(v.ctx, &ws, &ws_bytes)) {}
  DevMem(const DevMem&) = delete;
  ~DevMem() {
    cudaStreamSynchronize(c.st);  // nothing of this call may still run
    for (void* p : ptrs) cudaFree(p);
    if (held) ctx_ws_give(c.ctx, need <= kKeepBytes ? need : 0);
  }
  template <typename T>
  T* alloc(size_t count) {
    const size_t bytes = (sizeof(T) * (count ? count : 1) + 255) & ~(size_t)255;
    need += bytes;
    if (off + bytes <= ws_bytes) {
      T* p = reinterpret_cast<T*>(static_cast<unsigned char*>(ws) + off);
      off += bytes;
      return p;
    }
    void* p = nullptr;
    if (cudaMalloc(&p, bytes) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    ptrs.push_back(p);
    return static_cast<T*>(p);
  }
};

struct HMat {
  int64_t n = 0, nnz = 0;
  int64_t* rowptr = nullptr;
  int* cols = nullptr;
  double *vals = nullptr, *diag = nullptr;
};

// The determinants grouped by their string of one spin (radix sort of the
// string words, least significant word first), the distinct strings, and
// for the spin-up strings their single-excitation neighbours.
int build_strings(const CtxView& c, int64_t n, const uint64_t* d_dets, int spin, bool neighbours, DevMem& mem,
                  SpinStrings* S) {
  cudaStream_t st = c.st;
  const int nint = c.nint, nw = 2 * nint;
  const unsigned nb = (unsigned)((n + 255) / 256);
  unsigned long long* key = mem.alloc<unsigned long long>(n);
  unsigned long long* key2 = mem.alloc<unsigned long long>(n);
  int* val = mem.alloc<int>(n);
  int* perm = mem.alloc<int>(n);
  int* flag = mem.alloc<int>(n);
  int* incl = mem.alloc<int>(n);
  S->sid = mem.alloc<int>(n);
  S->grp = perm;
  if (!key || !key2 || !val || !perm || !flag || !incl || !S->sid)
    return report(QP_ENOMEM, "device allocation for the spin strings failed");
  size_t tmp = 0, tmp2 = 0;
  cub::DeviceRadixSort::SortPairs(nullptr, tmp, key, key2, val, perm, (int)n, 0, 64, st);
  cub::DeviceScan::InclusiveSum(nullptr, tmp2, flag, incl, (int)n, st);
  void* d_tmp = mem.alloc<unsigned char>(tmp > tmp2 ? tmp : tmp2);
  if (!d_tmp) return report(QP_ENOMEM, "device allocation for the spin strings failed");
  for (int w = nint - 1; w >= 0; w--) {  // least significant word first; the sorts are stable
    str_key_kernel<<<nb, 256, 0, st>>>(n, nw, spin * nint + w, d_dets, w == nint - 1 ? nullptr : perm, key, val);
    DV_TRY(cub::DeviceRadixSort::SortPairs(d_tmp, tmp, key, key2, val, perm, (int)n, 0, 64, st));
  }
  if (nint == 1) str_flag_kernel<1><<<nb, 256, 0, st>>>(n, spin, d_dets, perm, flag);
  else str_flag_kernel<2><<<nb, 256, 0, st>>>(n, spin, d_dets, perm, flag);
  DV_TRY(cub::DeviceScan::InclusiveSum(d_tmp, tmp2, flag, incl, (int)n, st));
  int nu = 0;
  DV_TRY(cudaMemcpyAsync(&nu, incl + (n - 1), sizeof(int), cudaMemcpyDeviceToHost, st));
  DV_TRY(cudaStreamSynchronize(st));
  S->nu = nu;
  S->ptr = mem.alloc<int>((size_t)nu + 1);
  S->ukey = mem.alloc<uint64_t>((size_t)nu * nint);
  if (!S->ptr || !S->ukey) return report(QP_ENOMEM, "device allocation for the spin strings failed");
  if (nint == 1) str_index_kernel<1><<<nb, 256, 0, st>>>(n, spin, d_dets, perm, flag, incl, S->sid, S->ptr, S->ukey);
  else str_index_kernel<2><<<nb, 256, 0, st>>>(n, spin, d_dets, perm, flag, incl, S->sid, S->ptr, S->ukey);
  const int nn = (int)n;
  DV_TRY(cudaMemcpyAsync(S->ptr + nu, &nn, sizeof(int), cudaMemcpyHostToDevice, st));
  if (!neighbours) return QP_OK;
  int* cnt = mem.alloc<int>((size_t)nu + 1);
  S->nb_ptr = mem.alloc<int>((size_t)nu + 1);
  if (!cnt || !S->nb_ptr) return report(QP_ENOMEM, "device allocation for the spin strings failed");
  DV_TRY(cudaMemsetAsync(cnt, 0, sizeof(int) * ((size_t)nu + 1), st));
  const unsigned nbu = (unsigned)(((int64_t)nu * 32 + 127) / 128);
  if (nint == 1) str_nb_kernel<1, true><<<nbu, 128, 0, st>>>(nu, S->ukey, cnt, nullptr, nullptr);
  else str_nb_kernel<2, true><<<nbu, 128, 0, st>>>(nu, S->ukey, cnt, nullptr, nullptr);
  size_t tmp3 = 0;
  cub::DeviceScan::ExclusiveSum(nullptr, tmp3, cnt, S->nb_ptr, nu + 1, st);
  void* d_tmp3 = mem.alloc<unsigned char>(tmp3);
  if (!d_tmp3) return report(QP_ENOMEM, "device allocation for the spin strings failed");
  DV_TRY(cub::DeviceScan::ExclusiveSum(d_tmp3, tmp3, cnt, S->nb_ptr, nu + 1, st));
  int tot = 0;
  DV_TRY(cudaMemcpyAsync(&tot, S->nb_ptr + nu, sizeof(int), cudaMemcpyDeviceToHost, st));
  DV_TRY(cudaStreamSynchronize(st));
  S->nb = mem.alloc<int>((size_t)tot);
  if (!S->nb) return report(QP_ENOMEM, "device allocation for the spin strings failed");
  if (nint == 1) str_nb_kernel<1, false><<<nbu, 128, 0, st>>>(nu, S->ukey, nullptr, S->nb_ptr, S->nb);
  else str_nb_kernel<2, false><<<nbu, 128, 0, st>>>(nu, S->ukey, nullptr, S->nb_ptr, S->nb);
  DV_TRY(cudaGetLastError());
  return QP_OK;
}

// search: 0, the spin strings; 1, the tiled test of every pair, O(N_det^2),
// kept as a cross-check.
int build_h(const CtxView& c, int64_t n, const uint64_t* d_dets, DevMem& mem, HMat* H, int search = 0) {
  cudaStream_t st = c.st;
  H->n = n;
  int64_t* cnt = mem.alloc<int64_t>(n + 1);
  int* err = mem.alloc<int>(1);
  H->rowptr = mem.alloc<int64_t>(n + 1);
  H->diag = mem.alloc<double>(n);
  size_t tmp = 0;
  cub::DeviceScan::ExclusiveSum(nullptr, tmp, cnt, H->rowptr, (int)(n + 1), st);
  void* d_tmp = mem.alloc<unsigned char>(tmp);
  if (!cnt || !err || !H->rowptr || !H->diag || !d_tmp)
    return report(QP_ENOMEM, "device allocation for the Hamiltonian failed");
  DV_TRY(cudaMemsetAsync(err, 0, sizeof(int), st));
  DV_TRY(cudaMemsetAsync(cnt, 0, sizeof(int64_t) * (n + 1), st));
  const unsigned tiles = (unsigned)((n + kRows - 1) / kRows), nb = (unsigned)((n + 255) / 256);
  const int win = (int)(n < kMapMax ? n : kMapMax);  // determinants per bit map
  const size_t smem = 4 * (size_t)((win + 31) / 32);
  SpinStrings SA, SB;
  int rc;
  if (search == 0) {
    if ((rc = build_strings(c, n, d_dets, 0, true, mem, &SA)) || (rc = build_strings(c, n, d_dets, 1, false, mem, &SB)))
      return rc;
  }
  int* cursor = nullptr;
  if (search == 1) {
    cursor = mem.alloc<int>(n);
    if (!cursor) return report(QP_ENOMEM, "device allocation for the Hamiltonian failed");
    DV_TRY(cudaMemsetAsync(cursor, 0, sizeof(int) * n, st));
  }
  // one pass of the pair search: row counts, or the columns (and, all pairs,
  // the elements in any order)
  auto strings = [&](auto nint, auto count, int* cols) -> cudaError_t {
    constexpr bool kCount = decltype(count)::value;
    constexpr auto* k = str_pairs_kernel<decltype(nint)::value, kCount>;
    const cudaError_t e = allow_smem<k>();
    if (e != cudaSuccess) return e;
    k<<<(unsigned)n, kMapThreads, kCount ? 0 : smem, st>>>(n, win, d_dets, SA.sid, SA.ptr, SA.grp, SA.nb_ptr, SA.nb, SB.sid,
                                              SB.ptr, SB.grp, cnt, H->rowptr, cols, err);
    return cudaGetLastError();
  };
  auto pairs = [&](auto nint, auto count, int* cols, double* vals) -> cudaError_t {
    pairs_kernel<decltype(nint)::value, decltype(count)::value><<<tiles, 256, 0, st>>>(
        n, d_dets, c.norb, c.h, c.eri, cnt, H->rowptr, cursor, cols, vals, err);
    return cudaGetLastError();
  };
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  if (c.nint == 1) diag_kernel<1><<<nb, 256, 0, st>>>(n, d_dets, c.norb, c.h, c.Jm, c.Km, H->diag);
  else diag_kernel<2><<<nb, 256, 0, st>>>(n, d_dets, c.norb, c.h, c.Jm, c.Km, H->diag);
  if (search == 0)
    DV_TRY(c.nint == 1 ? strings(I1{}, std::true_type{}, nullptr) : strings(I2{}, std::true_type{}, nullptr));
  else
    DV_TRY(c.nint == 1 ? pairs(I1{}, std::true_type{}, nullptr, nullptr) : pairs(I2{}, std::true_type{}, nullptr, nullptr));
  DV_TRY(cub::DeviceScan::ExclusiveSum(d_tmp, tmp, cnt, H->rowptr, (int)(n + 1), st));
  int herr = 0;
  DV_TRY(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
  DV_TRY(cudaMemcpyAsync(&H->nnz, H->rowptr + n, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  DV_TRY(cudaStreamSynchronize(st));
  if (herr) return report(QP_EDUP, "duplicate determinant in Psi0");
  if (H->nnz >= (1ll << 31)) return report(QP_ENOTSUP, "Hamiltonian above 2^31 entries");
  H->cols = mem.alloc<int>(H->nnz);
  H->vals = mem.alloc<double>(H->nnz);
  if (!H->cols || !H->vals) return report(QP_ENOMEM, "device allocation for the Hamiltonian failed");
  if (H->nnz == 0) return QP_OK;
  if (search == 0) {
    DV_TRY(c.nint == 1 ? strings(I1{}, std::false_type{}, H->cols) : strings(I2{}, std::false_type{}, H->cols));
    if (c.nint == 1) str_vals_kernel<1><<<(unsigned)n, 128, 0, st>>>(d_dets, c.norb, c.h, c.eri, H->rowptr, H->cols, H->vals);
    else str_vals_kernel<2><<<(unsigned)n, 128, 0, st>>>(d_dets, c.norb, c.h, c.eri, H->rowptr, H->cols, H->vals);
    DV_TRY(cudaGetLastError());
    return QP_OK;
  }
  int* cols2 = mem.alloc<int>(H->nnz);
  double* vals2 = mem.alloc<double>(H->nnz);
  if (!cols2 || !vals2) return report(QP_ENOMEM, "device allocation for the Hamiltonian failed");
  DV_TRY(c.nint == 1 ? pairs(I1{}, std::false_type{}, cols2, vals2) : pairs(I2{}, std::false_type{}, cols2, vals2));
  // columns ascending within each row: a fixed order of the sums
  size_t tmp2 = 0;
  cub::DeviceSegmentedRadixSort::SortPairs(nullptr, tmp2, cols2, H->cols, vals2, H->vals, (int)H->nnz, (int)n,
                                           H->rowptr, H->rowptr + 1, 0, 32, st);
  void* d_tmp2 = mem.alloc<unsigned char>(tmp2);
  if (!d_tmp2) return report(QP_ENOMEM, "device allocation for the Hamiltonian failed");
  DV_TRY(cub::DeviceSegmentedRadixSort::SortPairs(d_tmp2, tmp2, cols2, H->cols, vals2, H->vals, (int)H->nnz, (int)n,
                                                  H->rowptr, H->rowptr + 1, 0, 32, st));
  return QP_OK;
}

int spmv(const CtxView& c, const HMat& H, int nvec, const double* X, double* Y) {
  spmv_kernel<<<(unsigned)((H.n + kSpmvRows - 1) / kSpmvRows), kSpmvThreads, 0, c.st>>>(H.n, nvec, H.rowptr, H.cols,
                                                                                        H.vals, H.diag, X, Y);
  DV_TRY(cudaGetLastError());
  return QP_OK;
}

int check_inputs(const CtxView& c, int64_t n, const uint64_t* dets) {
  if (n < 1) return report(QP_EINVAL, "ndet must be positive");
  if (n >= (1ll << 31)) return report(QP_EINVAL, "ndet must be below 2^31");
  if (!dets) return report(QP_EINVAL, "dets is NULL");
  (void)c;
  return QP_OK;
}

// Copies a caller array to the device unless it is there already.
template <typename T>
int to_device(const T* src, size_t count, cudaStream_t st, DevMem& mem, const T** out) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, src) == cudaSuccess &&
      (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged)) {
    *out = src;
    return QP_OK;
  }
  cudaGetLastError();
  T* d = mem.alloc<T>(count);
  if (!d) return report(QP_ENOMEM, "device allocation failed");
  DV_TRY(cudaMemcpyAsync(d, src, sizeof(T) * count, cudaMemcpyHostToDevice, st));
  *out = d;
  return QP_OK;
}

// Occupation counts and bits beyond norb.
__global__ void check_dets_kernel(int64_t n, int nint, int norb, int na, int nb, const uint64_t* dets, int* bad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int f = 0;
  for (int s = 0; s < 2; s++) {
    int cnt = 0;
    for (int w = 0; w < nint; w++) {
      const uint64_t b = dets[(size_t)i * 2 * nint + s * nint + w];
      const int lim = norb - 64 * w;  // orbitals held by this word
      const uint64_t valid = lim >= 64 ? ~0ull : (lim <= 0 ? 0ull : (1ull << lim) - 1);
      if (b & ~valid) f |= 1;
      cnt += __popcll(b);
    }
    if (cnt != (s ? nb : na)) f |= 2;
  }
  if (f) atomicOr(bad, f);
}

int validate(const CtxView& c, int64_t n, const uint64_t* d_dets, DevMem& mem) {
  int* bad = mem.alloc<int>(1);
  if (!bad) return report(QP_ENOMEM, "device allocation failed");
  DV_TRY(cudaMemsetAsync(bad, 0, sizeof(int), c.st));
  check_dets_kernel<<<(unsigned)((n + 255) / 256), 256, 0, c.st>>>(n, c.nint, c.norb, c.nalpha, c.nbeta, d_dets, bad);
  DV_TRY(cudaGetLastError());
  int f = 0;
  DV_TRY(cudaMemcpyAsync(&f, bad, sizeof(int), cudaMemcpyDeviceToHost, c.st));
  DV_TRY(cudaStreamSynchronize(c.st));
  if (f & 1) return report(QP_EINVAL, "a bit beyond norb is set");
  if (f & 2) return report(QP_EINVAL, "a determinant has the wrong occupation");
  return QP_OK;
}

}  // namespace
}  // namespace qp

using namespace qp;

extern "C" int qp_pt2_sigma(qp_pt2_ctx* ctx, int64_t ndet, const uint64_t* dets, int nvec, const double* U,
                            double* S) {
  CtxView c;
  int rc = ctx_view(ctx, &c);
  if (rc) return rc;
  if ((rc = check_inputs(c, ndet, dets))) return rc;
  if (nvec < 1 || !U || !S) return report(QP_EINVAL, "nvec must be positive and U, S non-NULL");
  DevMem mem(c);
  const uint64_t* d_dets;
  const double* d_u;
  if ((rc = to_device(dets, (size_t)ndet * 2 * c.nint, c.st, mem, &d_dets))) return rc;
  if ((rc = validate(c, ndet, d_dets, mem))) return rc;
  if ((rc = to_device(U, (size_t)ndet * nvec, c.st, mem, &d_u))) return rc;
  HMat H;
  if ((rc = build_h(c, ndet, d_dets, mem, &H))) return rc;
  double* d_s = mem.alloc<double>((size_t)ndet * nvec);
  if (!d_s) return report(QP_ENOMEM, "device allocation failed");
  if ((rc = spmv(c, H, nvec, d_u, d_s))) return rc;
  DV_TRY(cudaMemcpyAsync(S, d_s, sizeof(double) * ndet * nvec, cudaMemcpyDefault, c.st));
  DV_TRY(cudaStreamSynchronize(c.st));
  return QP_OK;
}

extern "C" int qp_pt2_hamiltonian(qp_pt2_ctx* ctx, int64_t ndet, const uint64_t* dets, int search, int64_t* nnz,
                                  int64_t* rowptr, int32_t* cols, double* vals, double* diag, double* build_ms) {
  CtxView c;
  int rc = ctx_view(ctx, &c);
  if (rc) return rc;
  if ((rc = check_inputs(c, ndet, dets))) return rc;
  if (!nnz) return report(QP_EINVAL, "nnz is NULL");
  if (search != 0 && search != 1) return report(QP_EINVAL, "search must be 0 (spin strings) or 1 (all pairs)");
  DevMem mem(c);
  const uint64_t* d_dets;
  if ((rc = to_device(dets, (size_t)ndet * 2 * c.nint, c.st, mem, &d_dets))) return rc;
  if ((rc = validate(c, ndet, d_dets, mem))) return rc;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  cudaEventRecord(e0, c.st);
  HMat H;
  rc = build_h(c, ndet, d_dets, mem, &H, search);
  cudaEventRecord(e1, c.st);
  cudaEventSynchronize(e1);
  float ms = 0.f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  *nnz = H.nnz;
  if (build_ms) *build_ms = ms;
  if (rowptr) DV_TRY(cudaMemcpyAsync(rowptr, H.rowptr, sizeof(int64_t) * (ndet + 1), cudaMemcpyDefault, c.st));
  if (cols && H.nnz) DV_TRY(cudaMemcpyAsync(cols, H.cols, sizeof(int) * H.nnz, cudaMemcpyDefault, c.st));
  if (vals && H.nnz) DV_TRY(cudaMemcpyAsync(vals, H.vals, sizeof(double) * H.nnz, cudaMemcpyDefault, c.st));
  if (diag) DV_TRY(cudaMemcpyAsync(diag, H.diag, sizeof(double) * ndet, cudaMemcpyDefault, c.st));
  DV_TRY(cudaStreamSynchronize(c.st));
  return QP_OK;
}

extern "C" int qp_pt2_davidson(qp_pt2_ctx* ctx, int64_t ndet, const uint64_t* dets, const double* guess,
                               double tol, int max_iter, double* coefs, double* e0, qp_pt2_davidson_info* info) {
  CtxView c;
  int rc = ctx_view(ctx, &c);
  if (rc) return rc;
  if ((rc = check_inputs(c, ndet, dets))) return rc;
  if (!coefs || !e0) return report(QP_EINVAL, "coefs or e0 is NULL");
  if (!(tol > 0.0) || max_iter < 1) return report(QP_EINVAL, "tol must be positive and max_iter at least 1");
  cudaStream_t st = c.st;
  const int64_t n = ndet;
  const unsigned nb = (unsigned)((n + 127) / 128);
  DevMem mem(c);
  const uint64_t* d_dets;
  if ((rc = to_device(dets, (size_t)n * 2 * c.nint, st, mem, &d_dets))) return rc;
  if ((rc = validate(c, n, d_dets, mem))) return rc;
  struct Events {  // destroyed on every return
    cudaEvent_t e[3] = {nullptr, nullptr, nullptr};
    Events() {
      for (auto& x : e) cudaEventCreate(&x);
    }
    ~Events() {
      for (auto& x : e)
        if (x) cudaEventDestroy(x);
    }
  } evs;
  cudaEvent_t ev0 = evs.e[0], ev1 = evs.e[1], ev2 = evs.e[2];
  cudaEventRecord(ev0, st);
  HMat H;
  if ((rc = build_h(c, n, d_dets, mem, &H))) return rc;
  cudaEventRecord(ev1, st);
  const int mmax = (int)(n < kMaxBasis ? n : kMaxBasis);
  double* V = mem.alloc<double>((size_t)mmax * n);
  double* W = mem.alloc<double>((size_t)mmax * n);
  double* x = mem.alloc<double>(n);
  double* w = mem.alloc<double>(n);
  double* r = mem.alloc<double>(n);
  double* t = mem.alloc<double>(n);
  // products of the two orthogonalisation passes (with r.r and t.t) and of the
  // new column of the subspace matrix
  constexpr int kProducts = (kMaxBasis + 1) * kDotParts;
  double* d_small = mem.alloc<double>(3 * kProducts);
  if (!V || !W || !x || !w || !r || !t || !d_small) return report(QP_ENOMEM, "device allocation for Davidson failed");
  // first basis vector: the guess, or the determinant of lowest H_II
  std::vector<double> hv((size_t)n);
  if (guess) {
    DV_TRY(cudaMemcpyAsync(hv.data(), guess, sizeof(double) * n, cudaMemcpyDefault, st));
    DV_TRY(cudaStreamSynchronize(st));
  } else {
    DV_TRY(cudaMemcpyAsync(hv.data(), H.diag, sizeof(double) * n, cudaMemcpyDeviceToHost, st));
    DV_TRY(cudaStreamSynchronize(st));
    int64_t best = 0;
    for (int64_t i = 1; i < n; i++)
      if (hv[i] < hv[best]) best = i;
    std::fill(hv.begin(), hv.end(), 0.0);
    hv[best] = 1.0;
  }
  double nrm = 0.0;
  for (double v : hv) nrm += v * v;
  if (!(nrm > 0.0) || !std::isfinite(nrm)) return report(QP_EINVAL, "the guess vector is zero or not finite");
  for (double& v : hv) v /= std::sqrt(nrm);
  DV_TRY(cudaMemcpyAsync(V, hv.data(), sizeof(double) * n, cudaMemcpyHostToDevice, st));
  auto dot = [&](const double* a, const double* b, double* out_host) -> int {
    double parts[kDotParts];
    dots_kernel<<<kDotParts, kDotThreads, 0, st>>>(n, 1, a, b, nullptr, d_small);
    DV_TRY(cudaMemcpyAsync(parts, d_small, sizeof(parts), cudaMemcpyDeviceToHost, st));
    DV_TRY(cudaStreamSynchronize(st));
    *out_host = dot_sum(parts);
    return QP_OK;
  };
  double *d1 = d_small, *d2 = d1 + kProducts, *d3 = d2 + kProducts;
  if ((rc = spmv(c, H, 1, V, W))) return rc;
  std::vector<double> G((size_t)kMaxBasis * kMaxBasis, 0.0), a;
  double hs[3 * kProducts];
  const double *h1 = hs, *h2 = h1 + kProducts, *h3 = h2 + kProducts;
  if ((rc = dot(V, W, G.data()))) return rc;
  int m = 1, it = 0;
  double theta = G[0], rnorm = INFINITY;
  bool converged = false;
  // One iteration: the lowest Ritz pair of the subspace matrix on the host,
  // then seven launches without a wait between them (the Ritz vector, its
  // residual and correction; two orthogonalisation passes; the product with
  // H; the subspace matrix's new column), and one read-back.  The residual is
  // known with it: the extension of the last iteration is not used.
  for (;;) {
    a.resize((size_t)m * m);
    for (int i = 0; i < m; i++)
      for (int j = 0; j < m; j++) a[(size_t)i * m + j] = 0.5 * (G[(size_t)i * kMaxBasis + j] + G[(size_t)j * kMaxBasis + i]);
    Ritz z{};
    z.theta = theta = lowest_eigenpair(m, a, z.s);
    const int restart = m == mmax ? 1 : 0, mb = restart ? 1 : m;  // full: restart from the Ritz vector
    ritz_kernel<<<nb, 128, 0, st>>>(n, m, restart, z, V, W, H.diag, x, w, r, t);
    dots_kernel<<<(mb + 1) * kDotParts, kDotThreads, 0, st>>>(n, mb, V, t, r, d1);
    orth_kernel<<<nb, 128, 0, st>>>(n, mb, 0, V, d1, t, t);
    dots_kernel<<<(mb + 1) * kDotParts, kDotThreads, 0, st>>>(n, mb, V, t, t, d2);
    // (a basis that is restarted at its full length leaves room for one more)
    double *vn = V + (size_t)mb * n, *wn = W + (size_t)mb * n;
    const bool room = mb < mmax;
    if (room) {
      orth_kernel<<<nb, 128, 0, st>>>(n, mb, 1, V, d2, t, vn);
      if ((rc = spmv(c, H, 1, vn, wn))) return rc;
      dots_kernel<<<(mb + 1) * kDotParts, kDotThreads, 0, st>>>(n, mb + 1, V, wn, nullptr, d3);
    }
    DV_TRY(cudaGetLastError());
    DV_TRY(cudaMemcpyAsync(hs, d_small, sizeof(hs), cudaMemcpyDeviceToHost, st));
    DV_TRY(cudaStreamSynchronize(st));
    rnorm = std::sqrt(dot_sum(h1 + mb * kDotParts));
    if (rnorm <= tol) {
      converged = true;
      break;
    }
    if (++it > max_iter) break;
    if (restart) {
      G[0] = theta;
      m = 1;
    }
    double tt = dot_sum(h2 + m * kDotParts);
    for (int i = 0; i < m; i++) {
      const double d = dot_sum(h2 + i * kDotParts);
      tt -= d * d;
    }
    if (!room || !(tt > 1e-28)) break;  // no new direction
    for (int i = 0; i <= m; i++) {
      const double g = dot_sum(h3 + i * kDotParts);
      G[(size_t)i * kMaxBasis + m] = g;
      G[(size_t)m * kMaxBasis + i] = g;
    }
    m++;
  }
  // output: x normalised, with coefs[0] >= 0
  DV_TRY(cudaMemcpyAsync(hv.data(), x, sizeof(double) * n, cudaMemcpyDeviceToHost, st));
  cudaEventRecord(ev2, st);
  DV_TRY(cudaStreamSynchronize(st));
  double xx = 0.0;
  for (double v : hv) xx += v * v;
  const double sc = (hv[0] < 0 ? -1.0 : 1.0) / std::sqrt(xx);
  for (double& v : hv) v *= sc;
  // E0 as the Rayleigh quotient of the returned vector
  DV_TRY(cudaMemcpyAsync(x, hv.data(), sizeof(double) * n, cudaMemcpyHostToDevice, st));
  if ((rc = spmv(c, H, 1, x, w))) return rc;
  double xhx;
  if ((rc = dot(x, w, &xhx))) return rc;
  DV_TRY(cudaMemcpyAsync(coefs, x, sizeof(double) * n, cudaMemcpyDefault, st));
  DV_TRY(cudaStreamSynchronize(st));
  *e0 = xhx;
  if (info) {
    float a = 0.f, b = 0.f;
    cudaEventElapsedTime(&a, ev0, ev1);
    cudaEventElapsedTime(&b, ev1, ev2);
    info->iterations = it;
    info->residual = rnorm;
    info->nnz = H.nnz;
    info->converged = converged ? 1 : 0;
    info->build_ms = a;
    info->solve_ms = b;
  }
  return converged ? QP_OK : report(QP_ENOTCONV, "Davidson did not reach the residual tolerance");
}
