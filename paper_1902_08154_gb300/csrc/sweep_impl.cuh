// sweep_impl.cuh -- sm_103a kernels of the deterministic EN-PT2 + selection sweep
// (Quantum Package 2.0, arXiv:1902.08154, Appendix "CIPSI selection and PT2
// energy").
//
// Generators are taken in rank order (decreasing c_I^2) in waves of slots.
// Per wave two kernels run:
//
//  prep_kernel (one CTA per generator I of the wave)
//    - the Fock diagonal of I, so that <alpha|H|alpha> costs a few flops per
//      alpha (Appendix: "pre-compute the diagonal of the Fock matrix");
//    - the coarse filter: every internal J within excitation degree 4 of I,
//      stored as a record (its words, c_J, the holes of I missing from J as a
//      mask over I's occupied list, the particles of J outside I, and whether
//      J ranks before I);
//    - the fine filter, done once per generator: a batch is a hole set H of I
//      (|H| = 1 or 2) holding the alpha = I - H + R for the particle sets R
//      outside I with the spins of H.  With K = I - H, t = |K - J| and
//      X = J - K, deg(J, alpha) = t + |H| - |R n X|, so J reaches batch H only
//      if t <= 2.  With Q the holes of J (d = |Q|), t = d - |Q n H|: J with
//      d <= 2 reaches every batch, d = 3 the batches meeting Q, d = 4 the
//      batches inside Q.  The bans of J ranked before I with d <= 3 go into
//      bit masks (one for every batch, one per hole); the other J that reach
//      a cell these leave go to one shared list (d <= 2), to a list per hole
//      (d <= 3) and to a bucket per pair of holes (d >= 2).
//
//  batch_kernel (persistent CTAs, one (generator, batch) item at a time, in
//  the order of the prep kernel's list: large waves by kind, see by_kind)
//    bans:   the masks, then the bucket's J ranked before I; a later J equal
//            to some alpha bans it;
//    loop 2: J ranked at or after I add c_J <J|H|alpha> into the shared-memory
//            accumulator A(R) of the cells they reach that are not banned.
//            A row of cells is a warp's, a lane per cell; J reaching a few
//            cells are a thread's; J reaching every cell go through pair
//            tables in the cells pass;
//    cells:  every cell left is a perturber of I: e = A^2/(E0 - H_aa) with
//            H_aa from per-batch row and column sums in fixed point (FP64 where
//            its unit is too coarse), added to eps_I and offered to the CTA's
//            selection buffer.
// Matrix elements follow the Slater-Condon rules (Eqs. Hij) with phases from
// a masked popcount of J's spin string.
//
// Numerator precision: the batch kernel is a template on NT, the type of the
// integrals it gathers and of the products c_J <J|H|alpha>.  NT = double is
// the plain FP64 sweep; NT = float gathers FP32 integrals and forms FP32
// products, while each product is still added into the exact accumulator
// A(R), and the denominators, e_alpha and every reduction are those of the
// FP64 sweep.
// sweep.cu instantiates the FP64 kernels, sweep_mixed.cu the mixed ones.
#pragma once
#include <cfloat>
#include <cstdio>
#include <type_traits>

#include "common.cuh"

namespace qp {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kChunk = 512;  // bucket entries classified per round
constexpr int kGroup = 6;     // J reaching every cell, handled together
constexpr unsigned kFull = 0xffffffffu;
// Bit of a bucket entry's particle word that flags a J ranked before I (see
// part_code below).
constexpr uint64_t kBeforeBit = 1ull << 15;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ unsigned long long warp_sum_u(unsigned long long v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ unsigned long long warp_xor_u(unsigned long long v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v ^= __shfl_xor_sync(kFull, v, o);
  return v;
}
__device__ __forceinline__ unsigned long long warp_min_u(unsigned long long v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    unsigned long long w = __shfl_xor_sync(kFull, v, o);
    v = w < v ? w : v;
  }
  return v;
}

// Block-wide exclusive scan of a 0/1 flag; returns this thread's position and
// the block total.  wsum: kWarps ints of shared memory.
__device__ __forceinline__ int block_scan_flag(bool f, int* wsum, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned b = __ballot_sync(kFull, f);
  int before = __popc(b & ((1u << lane) - 1));
  if (lane == 0) wsum[warp] = __popc(b);
  __syncthreads();
  int off = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < kWarps; w++) {
    int c = wsum[w];
    off += (w < warp) ? c : 0;
    tot += c;
  }
  __syncthreads();
  *total = tot;
  return off + before;
}

// Integrals in the numerator precision.
// E4: the four-index layout of the context (eri4_index); else the packed
// array (the no-allocation entry point, which has only the caller's copy).
template <typename NT, bool E4>
__device__ __forceinline__ const NT* numer_eri(const SweepParams& p) {
  if constexpr (sizeof(NT) == 8) return reinterpret_cast<const NT*>(E4 ? p.eri4 : p.eri);
  else return reinterpret_cast<const NT*>(E4 ? p.eri4_32 : p.eri32);
}

// Position of (pq|rs) in the gather layout.
template <bool E4>
__device__ __forceinline__ int gidx(int p, int q, int r, int s, int norb) {
  if constexpr (E4) return eri4_index(p, q, r, s, norb);
  else return eri_index(p, q, r, s);
}
template <typename NT>
__device__ __forceinline__ const NT* numer_h(const SweepParams& p);
template <>
__device__ __forceinline__ const double* numer_h<double>(const SweepParams& p) { return p.h; }
template <>
__device__ __forceinline__ const float* numer_h<float>(const SweepParams& p) { return p.h32; }

// ---------------------------------------------------------------------------
// Denominators D = E0 - H_aa as 64-bit integers in units of 2^-S, and A/D by
// integer arithmetic.  An FP64 warp instruction takes 19 cycles of an SM here
// (a 64-bit integer add 1, a high 64-bit product 5.5), so the two FP64
// additions of D and the five operations of its reciprocal were most of the
// cells pass.  S is the same for a whole sweep:
// |D| <= |E0| + n_el max|h| + n_el (n_el - 1) max|(pq|rs)| < 2^(63 - S), and
// sums of table entries on the way may wrap.
// That bound is over all orbitals, whichever a perturber has: one large entry
// of h or of the integrals (a level-shifted orbital, a tight virtual one) makes
// the unit coarse for every D, while FP64 sums lose digits only where they
// contain it.  So a generator has this form only where the unit is at most
// 2^-55 of the sums that make up its H_II (or of E0 where that is larger),
// whose rounding each of its FP64 denominators carries; otherwise its energies
// and denominators stay in FP64 (den_form) and its items go to the FP64 form
// of the batch kernel.  2^62 units against those sums: 2^2.4 to 2^4.7 on the
// workloads of 14 to 64 orbitals and 3 to 26 electrons, up to 2^7.2 with 64
// electrons; with one h_pp of 10^4 2^12, where D is up to 18 times further off
// than in FP64, with one of 10^6 2^19 and 8,000 times.
// Two states at once, 2,000 determinants, 64 orbitals: 43 to 33.8 ms (two
// quotients per cell); one state, 10^4 determinants 113.3 to 111.8 ms; 10^3
// determinants, 128 orbitals 87.1 to 84.1 ms.  The FP64 form of the present
// kernels (all generators of 10^4 determinants, 64 orbitals, one h_pp of 10^6):
// 95.0 ms against 73.4, two states 44.1 against 23.6.
// ---------------------------------------------------------------------------
constexpr int kDenFp64 = 1 << 20;  // in the place of S: energies as the bits of FP64 numbers
__device__ __forceinline__ int den_scale(const SweepParams& p) {
  const double hmx = __longlong_as_double((long long)p.hmax_bits[0]);
  const double emx = __longlong_as_double((long long)p.hmax_bits[1]);
  double e0 = fabs(p.e0);
  for (int s = 0; s < p.nst; s++) e0 = fmax(e0, fabs(p.st_e0[s]));
  const double n = (double)(p.nel + 2), bound = e0 + n * hmx + n * (n - 1.0) * emx;
  if (!(bound < 1e300)) return kDenFp64;  // or not finite
  const int e = (int)((((unsigned long long)__double_as_longlong(bound)) >> 52) & 0x7FF) - 1023;
  return 62 - e < 900 ? 62 - e : 900;
}
// 2^e, e within the normal exponents.
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }
// x in units of 2^-S.
__device__ __forceinline__ long long den_fix(double x, int S) {
  return S == kDenFp64 ? 0ll : __double2ll_rn(x * pow2(S));
}
__device__ __forceinline__ double den_double(unsigned long long um, int S) { return (double)um * pow2(-S); }
// The form of a generator's denominators: S, or kDenFp64 where that unit is
// too coarse.  sum: of |h_ii| and |F(i)| over its orbitals, twice what H_II's
// partial sums reach.
__device__ __forceinline__ int den_form(const SweepParams& p, int S, double sum) {
  if (S == kDenFp64) return S;
  double e0 = fabs(p.nst > 0 ? p.st_e0[0] : p.e0);
  for (int s = 1; s < p.nst; s++) e0 = fmin(e0, fabs(p.st_e0[s]));
  return pow2(62 - S) <= kDenRange * fmax(e0, 0.5 * sum) ? S : kDenFp64;
}

// a / (d 2^-S) for a quotient outside the normal range, a zero denominator
// or operands that are not finite.
static __device__ __noinline__ double div_slow(double a, long long d, int S) { return a / ((double)d * pow2(-S)); }

// a / (d 2^-S): the reciprocal of the normalised 64-bit magnitude m of d from
// the FP32 approximation of its top 24 bits (relative error e below 2^-21) by
// two Newton steps in integers (e^2 and the 32 bits of m left out of the
// first step, then 2^-60), the product with a's mantissa, one rounding to
// FP64 (half away from zero).
// *bad: the result is not this one but div_rest's (one test for all of them).
// SMALL: denominators below 2^32 units are done here too; without it they go
// to div_rest, where they are exact in FP64, and the leading zeros of one word
// are counted (two states 26.6 -> 25.4 ms with SMALL, one state, 10^4
// determinants 78.8 -> 78.5 ms without).
template <bool SMALL>
__device__ __forceinline__ double div_core(double a, long long d, int S, bool* bad) {
  const unsigned long long ab = (unsigned long long)__double_as_longlong(a);
  const int ea = (int)((ab >> 52) & 0x7FF);
  unsigned long long m = d < 0 ? 0ull - (unsigned long long)d : (unsigned long long)d;
  const bool small = SMALL ? m == 0ull : (m >> 32) == 0ull;
  const int n = SMALL ? __clzll((long long)m) : __clz((int)(m >> 32));
  m <<= n & 63;
  const unsigned int mh = (unsigned int)(m >> 32);
  float rf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(__uint2float_rn(mh)));
  const unsigned int r0 = __float2uint_rz(rf * 9.223372036854775808e18f);  // 2^63 / mh, at most 2^32 - 1
  const long long e1 = (long long)(0x8000000000000000ull - (unsigned long long)mh * r0);
  unsigned long long r = ((unsigned long long)r0 << 32) + (unsigned long long)(((long long)(int)(e1 >> 20) * (long long)r0) >> 11);
  const long long e2 = (long long)(0x7FFFFFFFFFFFFFFFull - __umul64hi(m, r));
  r += (unsigned long long)(((long long)(r >> 34) * e2) >> 29);  // 2^127 / m
  unsigned long long q = __umul64hi(((ab & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 11, r);
  const int up = (int)(q >> 63);
  q <<= 1 - up;
  const int ex = ea + S + n - 64 + up;
  *bad = small || (unsigned)(ex - 1) > 2044u || (unsigned)(ea - 1) > 2045u;
  const unsigned long long v = ((unsigned long long)(unsigned int)(ex - 1) << 52) + (q >> 11) + ((q >> 10) & 1ull);
  return __longlong_as_double((long long)(v | ((ab ^ (unsigned long long)d) & 0x8000000000000000ull)));
}
__device__ __forceinline__ double div_rest(double a, long long d, int S) {
  if (((__double_as_longlong(a) >> 52) & 0x7FF) == 0 && d != 0) return 0.0;
  return div_slow(a, d, S);
}
template <bool SMALL>
__device__ __forceinline__ double div_fix(double a, long long d, int S) {
  bool bad;
  const double q = div_core<SMALL>(a, d, S, &bad);
  return bad ? div_rest(a, d, S) : q;
}

// Nanoseconds of the device's global timer.
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Bit pattern of |x|.  The mask is applied in inline PTX: written in C++ the
// compiler recognises it as fabs and issues it on the FP64 pipe.
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  unsigned long long b;
  asm("and.b64 %0, %1, 0x7FFFFFFFFFFFFFFF;" : "=l"(b) : "l"((unsigned long long)__double_as_longlong(x)));
  return b;
}

// v with its sign flipped when neg: a bit operation, no floating-point pipe.
__device__ __forceinline__ double flip_sign(double v, bool neg) {
  return __longlong_as_double(__double_as_longlong(v) ^ ((long long)neg << 63));
}
__device__ __forceinline__ float flip_sign(float v, bool neg) {
  return __int_as_float(__float_as_int(v) ^ ((int)neg << 31));
}

// ---------------------------------------------------------------------------
// Exact accumulation of the numerator A_alpha = sum_J c_J <J|H|alpha> in the
// one-state sweep.  Each product (FP64, or FP32 in the mixed form) is
// converted, with one rounding at 2^-F, to a 96-bit two's-complement integer
// in units of 2^-F and added with integer arithmetic, so that A_alpha does
// not depend on the order of the additions: the J of a batch reach a cell
// from different warps, and integer sums give the same bits on every run
// and every grid.  F is the same for a whole sweep: with
// B = max_I |c_I| * N_det * Hmax, where Hmax bounds every |<J|H|alpha>|
// (max |h| + 2 (n_el + 1) max |(pq|rs)|), |A_alpha| <= B < 2^(94 - F), so no
// sum leaves the 95-bit range and every product lies below 2^94 * 2^-F.  The
// sum is rounded once to FP64 in the cells pass; it keeps everything above
// 2^-F (about 1e-21 on the workloads here), more than an FP64 sum of the
// same products keeps.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int fix_scale(const SweepParams& p) {
  const double cmax = __longlong_as_double((long long)*p.cmax_bits);
  const double hmx = __longlong_as_double((long long)p.hmax_bits[0]);
  const double emx = __longlong_as_double((long long)p.hmax_bits[1]);
  const double hmax = hmx + 2.0 * (double)(p.nel + 1) * emx;
  const double bound = cmax * (double)p.ndet * hmax;
  if (!(bound > 0.0)) return 100;
  // floor(log2(bound)) from the exponent field; 2^(e+1) > bound
  const int e = (int)((((unsigned long long)__double_as_longlong(bound)) >> 52) & 0x7FF) - 1023;
  int F = 93 - e;
  if (F > 126) F = 126;
  if (F < 0) {  // coefficients times integrals beyond 2^93: not representable
    atomicOr(p.err, 64);
    F = 0;
  }
  return F;
}

// m * 2^sh as a 96-bit integer (lo, hi), negated when neg; m < 2^53 and
// m * 2^sh < 2^94, so sh < 64; for sh < 0 the bits below 2^0 are rounded (half
// up).
__device__ __forceinline__ void fix_of_mant(unsigned long long m, int sh, bool neg, unsigned long long& lo,
                                            int& hi) {
  unsigned long long l;
  unsigned int h = 0u;
  if (sh <= 0) {
    const int r = -sh < 63 ? -sh : 63;
    l = (m + ((1ull << r) >> 1)) >> r;
  } else {
    l = m << sh;
    h = (unsigned int)((m >> 1) >> (63 - sh));
  }
  const unsigned int s = neg ? ~0u : 0u;
  l = (l ^ (((unsigned long long)s << 32) | s)) + (neg ? 1ull : 0ull);
  h = (h ^ s) + (neg && l == 0ull ? 1u : 0u);
  lo = l;
  hi = (int)h;
}

__device__ __forceinline__ void fix_of(double x, int F, unsigned long long& lo, int& hi) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF);
  // zero, or below 2^-1022: nothing at 2^-F (F <= 126)
  fix_of_mant(e == 0 ? 0ull : (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull, e - 1075 + F, (b >> 63) != 0ull, lo,
              hi);
}

__device__ __forceinline__ void fix_of(float x, int F, unsigned long long& lo, int& hi) {
  const unsigned int b = (unsigned int)__float_as_int(x);
  const int e = (int)((b >> 23) & 0xFF);
  fix_of_mant(e == 0 ? 0ull : (unsigned long long)((b & 0x7FFFFFu) | 0x800000u) << 29, e - 179 + F, (b >> 31) != 0u, lo,
              hi);
}

__device__ __forceinline__ void fix_add(unsigned long long& lo, int& hi, unsigned long long l2, int h2) {
  lo += l2;
  hi += h2 + (lo < l2 ? 1 : 0);
}

// Adds (l, h) into the shared-memory accumulator of a cell, kept as three
// 32-bit words in arrays of their own (a 64-bit shared-memory add is a
// compare-and-swap loop: 116 cycles against 44 for a 32-bit one): each carry
// out of a word is added to the next, so the total is exact whatever the
// order of the atomics.
__device__ __forceinline__ void fix_atomic_add(uint32_t* A0, uint32_t* A1, uint32_t* A2, int cc, unsigned long long l,
                                               int h) {
  const uint32_t l0 = (uint32_t)l, l1 = (uint32_t)(l >> 32);
  const uint32_t o0 = atomicAdd(&A0[cc], l0);
  const uint32_t c0 = o0 + l0 < o0 ? 1u : 0u, t1 = l1 + c0;
  const uint32_t o1 = atomicAdd(&A1[cc], t1);
  const uint32_t dh = (uint32_t)h + (t1 < c0 ? 1u : 0u) + (o1 + t1 < o1 ? 1u : 0u);
  if (dh) atomicAdd(&A2[cc], dh);
}

// (lo, hi) * 2^-F rounded to FP64 (nearest, ties away from zero): the top
// 53 bits of the magnitude, with integer operations only.  The magnitude's
// leading word is moved to the front, the words shifted left by its leading
// zeros; the rounding bit's carry goes on into the exponent (64 orbitals, 10^4
// determinants 79.5 -> 78.8 ms).
__device__ __forceinline__ double fix_to_double(unsigned long long lo, int hi, int F) {
  const unsigned int sg = (unsigned int)(hi >> 31);
  const unsigned long long s2 = ((unsigned long long)sg << 32) | sg;
  const unsigned long long l = (lo ^ s2) - s2;  // + 1 when negative
  unsigned int w2 = ((unsigned int)hi ^ sg) + (sg & (l == 0ull ? 1u : 0u));
  unsigned int w1 = (unsigned int)(l >> 32), w0 = (unsigned int)l;
  int n = 1023 + 95 - F;  // biased exponent of the leading bit
  if (w2 == 0u) {
    w2 = w1;
    w1 = w0;
    w0 = 0u;
    n -= 32;
    if (w2 == 0u) {
      w2 = w1;
      w1 = 0u;
      n -= 32;
      if (w2 == 0u) return 0.0;
    }
  }
  const int z = __clz((int)w2);
  const unsigned int h = __funnelshift_l(w1, w2, z), m = __funnelshift_l(w0, w1, z);
  const unsigned long long top = ((unsigned long long)h << 32) | m;
  const unsigned long long v = ((unsigned long long)(unsigned int)(n - z - 1) << 52) + (top >> 11) + ((m >> 10) & 1u);
  return __longlong_as_double((long long)(v | ((unsigned long long)(sg & 0x80000000u) << 32)));
}

__device__ __forceinline__ int pair_batch(int nel, int i, int j) {  // i < j
  return nel + j * (j - 1) / 2 + i;
}

// A bucket entry's particle word: four 16-bit fields, each the spin-orbital
// code s*norb + q (< 256) of a particle of J outside I, or kNoPart.  Bit 15
// (the top bit of the first field, which always holds a particle when it is
// set) flags a J ranked before I, so that one 16-byte load of the entry
// (hole mask, particle word) is all the classification reads.
constexpr int kNoPart = 0x7FFF;
__device__ __forceinline__ int part_code(uint64_t part, int i) { return (int)((part >> (16 * i)) & 0x7FFF); }

// Keep bits of a record's particle word (the free top bits of its fields,
// set and used by the prep kernel only): d <= 2: list J in the shared bucket;
// d = 3: list J with its i-th hole.
constexpr uint64_t kKeep0 = 1ull << 31, kKeep1 = 1ull << 47, kKeep2 = 1ull << 63;

// Buckets of a record of degree 3 at most with hole mask hm and particle word
// pt (see prep_slot); dead: bits of the batches banned as a whole, whose
// buckets nothing reads.
template <typename Fn>
__device__ __forceinline__ void for_buckets(uint64_t hm, uint64_t pt, int nel, int nbat, const uint32_t* dead,
                                            Fn&& fn) {
  const int d = __popcll(hm);
  const bool before = pt & kBeforeBit;
  int Q[3], n = 0;
  uint64_t m = hm;
  while (m && n < 3) {
    Q[n++] = __ffsll((long long)m) - 1;
    m &= m - 1;
  }
  if (before && d <= 2) return;  // in the masks as a whole
  if (d == 0 || (d <= 2 && (pt & kKeep0))) fn(nbat);
  if (!before) {
#pragma unroll
    for (int i = 0; i < 3; i++)
      if (i < d && (d < 3 || (pt & (kKeep0 << (16 * i))))) fn(Q[i]);
  }
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int j = i + 1; j < 3; j++) {
      if (j >= d) continue;
      const int b = pair_batch(nel, Q[i], Q[j]);
      if (!((dead[b >> 5] >> (b & 31)) & 1u)) fn(b);
    }
}

// Buckets of a record of degree 4: the six pairs of its holes.
template <typename Fn>
__device__ __forceinline__ void for_pairs4(uint64_t hm, int nel, const uint32_t* dead, Fn&& fn) {
  int Q[4];
#pragma unroll
  for (int i = 0; i < 4; i++) {
    Q[i] = __ffsll((long long)hm) - 1;
    hm &= hm - 1;
  }
#pragma unroll
  for (int j = 1; j < 4; j++) {
    const int row = nel + Q[j] * (Q[j] - 1) / 2;
#pragma unroll
    for (int i = 0; i < j; i++) {
      const int b = row + Q[i];
      if (!((dead[b >> 5] >> (b & 31)) & 1u)) fn(b);
    }
  }
}

struct Batch {
  int h;            // number of holes (1, 2)
  int kind;         // 0 single, 1 same-spin double, 2 opposite-spin double
  int ia, ib;       // occupied indices of the holes in I
  int ca, cb;       // their spin-orbital codes
  int sa, sb;       // their spins
  int qa, qb;       // their orbitals
  uint64_t hm;      // hole mask over I's occupied list
  int ncell;
  int clo, nct;     // this work item's cells: [clo, clo + nct) (a tile of the batch)
};


// Work items of a large wave are taken by kind, same-spin and one-hole ones
// first, so that the code of one kind at a time is in the instruction caches
// (10^4 determinants, 64 orbitals 78.5 -> 73.9 ms with a cells pass per kind,
// 79.0 without the order; opposite-spin first 74.4).  By kind against as they
// come: 67,200 items 2.88 against 3.05 ms, 84,000 items of 400 generators of a
// space of 10^4 12.2 against 12.9, 184,000 4.90 against 5.27.  Below the line
// it depends on the items: 50,400 2.23 against 2.35 ms (64 orbitals) and 22,950
// 0.83 against 0.87, but 25,200 items of 120 heavy generators 9.1 against 8.1
// and 9,900 425 against 415 us; so the line lies above all sizes at which the
// order was seen to lose.  The last wave of a large sweep may fall below it.
// (Not where the back of the list is the FP64 form's, den64.)
constexpr long long kItemsByKind = 65536;
__device__ __forceinline__ bool by_kind(const SweepParams& p) {
  return !p.den64 && (long long)p.wave_slots * p.nper >= kItemsByKind;
}

// Batch and tile of work item j of a generator: j < nbat is batch j (the first
// row tile of a split batch), j >= nbat row tile 1 + (j - nbat) / (n_alpha
// n_beta) of opposite-spin batch (j - nbat) % (n_alpha n_beta).
__device__ __forceinline__ int item_batch(const SweepParams& p, int j, int* tile) {
  *tile = 0;
  if (j < p.nbat) return j;
  const int na = p.nalpha, nab = p.nalpha * p.nbeta, k = (j - p.nbat) % nab;
  *tile = 1 + (j - p.nbat) / nab;
  const int ia = k % na, ib = na + k / na;
  return p.nel + ib * (ib - 1) / 2 + ia;
}

// The holes, kind and cells of batch b, tile `tile` (the orbitals of the
// holes are filled in from the generator's occupied list).  The occupied list
// is ordered spin-up first, so the indices give the spins.
__device__ __forceinline__ void batch_geometry(const SweepParams& p, int b, int tile, Batch& B) {
  const int nv0 = p.norb - p.nalpha, nv1 = p.norb - p.nbeta;
  if (b < p.nel) {
    B.h = 1;
    B.ia = b;
    B.ib = -1;
    B.sa = b >= p.nalpha;
    B.sb = -1;
    B.kind = 0;
    B.hm = 1ull << b;
    B.ncell = B.sa ? nv1 : nv0;
  } else {
    const int t = b - p.nel;
    int y = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)t)) * 0.5f);
    while (y * (y - 1) / 2 > t) y--;
    while ((y + 1) * y / 2 <= t) y++;
    B.h = 2;
    B.ib = y;
    B.ia = t - y * (y - 1) / 2;
    B.sa = B.ia >= p.nalpha;
    B.sb = B.ib >= p.nalpha;
    B.kind = B.sa == B.sb ? 1 : 2;
    B.hm = (1ull << B.ia) | (1ull << B.ib);
    const int nv = B.sa ? nv1 : nv0;
    B.ncell = B.kind == 1 ? nv * (nv - 1) / 2 : nv0 * nv1;
  }
  B.clo = 0;
  B.nct = B.ncell;
  if (p.ntile > 1 && B.kind == 2) {  // rows [tile h, min((tile + 1) h, nv0))
    const int h = (nv0 + p.ntile - 1) / p.ntile;
    const int r0 = tile * h, r1 = min(r0 + h, nv0);
    B.clo = r0 * nv1;
    B.nct = (r1 - r0) * nv1;
  }
}

// ---------------------------------------------------------------------------
// prep kernel: one CTA per generator slot of the wave
// ---------------------------------------------------------------------------
template <int NINT>
__device__ __forceinline__ void prep_slot(const SweepParams& p, const int slot) {
  constexpr int NW = 2 * NINT;
  __shared__ int s_cnt[kMaxBatch + 2];
  __shared__ uint32_t s_dead[(kMaxBatch + 31) / 32];
  __shared__ uint64_t sI[NW];
  __shared__ int s_occ[kMaxElec];
  __shared__ unsigned char s_vidx[2][kMaxOrb];
  __shared__ double s_F[2 * kMaxOrb];
  __shared__ int s_nrec[2];    // records of degree 3 at most, of degree 4
  __shared__ int s_form;       // den_form of I, and H_II (with den64)
  __shared__ double s_hii;
  __shared__ int s_below[NW];  // I's electrons in the words before
  extern __shared__ __align__(16) unsigned char dyn[];
  uint32_t* sm = reinterpret_cast<uint32_t*>(dyn);               // cell masks (MaskDims)
  uint64_t* so = reinterpret_cast<uint64_t*>(sm + p.mask_w);     // orbital masks (orb_mask_words)
  const int tid = threadIdx.x;
  const int norb = p.norb, nel = p.nel, nbat = p.nbat;
  GenMeta* M = p.meta + slot;
  // the slot's per-item sums start from zero (an item that adds nothing
  // does not write its sums)
  for (int j = tid; j < p.nper * p.it_stride; j += kThreads) p.it_sum[(size_t)slot * p.nper * p.it_stride + j] = 0.0;
  const long long t = (long long)p.wave_start + slot;
  const long long gg = p.gen_list ? (long long)p.gen_list[t] : p.shard_index + t * (long long)p.shard_count;
  // determinants of unequal electron counts (a batch's graph runs on after
  // the check has flagged them): no work, as the particle lists below are
  // taken to be as long as the hole lists
  if (gg >= p.ndet || (*p.err & kErrOcc)) {
    if (tid == 0) {
      M->g = -1;
      M->nrec = 0;
    }
    return;
  }
  const int g = (int)gg, gi = p.order[g];
  if (tid < NW) sI[tid] = p.dets[(size_t)gi * NW + tid];
  __syncthreads();
  if (tid == 0) {
    int n = 0;
    for (int s = 0; s < 2; s++)
      for (int q = 0; q < norb; q++)
        if ((sI[s * NINT + (q >> 6)] >> (q & 63)) & 1ull) s_occ[n++] = s * norb + q;
    M->g = g;
    M->cI = p.coefs[gi];
    for (int w = 0, below = 0; w < 4; w++) {
      M->I[w] = w < NW ? sI[w] : 0ull;
      if (w >= NW) continue;
      s_below[w] = below;
      below += __popcll(sI[w]);
    }
    s_nrec[0] = s_nrec[1] = 0;
  }
  __syncthreads();
  if (tid < nel) M->occ[tid] = s_occ[tid];
  const int S = den_scale(p);
  if (slot == 0)  // the denominators' tables, once per wave
    for (int x = tid; x < norb * norb; x += kThreads) {
      const long long j = den_fix(p.Jm[x], S);
      p.Ji[x] = j;
      p.Wi[x] = j - den_fix(p.Km[x], S);
    }
  // Fock diagonal F_s(q) = h_qq + sum_{j in I} [(qq|jj) - delta_s (qj|jq)]
  for (int x = tid; x < 2 * norb; x += kThreads) {
    const int s = x / norb, q = x - s * norb;
    double f = p.h[q * norb + q];
    for (int i = 0; i < nel; i++) {
      const int c = s_occ[i], sj = c >= norb, j = c - sj * norb;
      f += p.Jm[q * norb + j];
      if (sj == s) f -= p.Km[q * norb + j];
    }
    M->F[s][q] = den_fix(f, S);
    s_F[x] = f;
  }
  __syncthreads();
  if (tid == 0) {  // H_II = 1/2 sum_i (h_ii + F(i))
    double e = 0.0;
    for (int i = 0; i < nel; i++) {
      const int c = s_occ[i], s = c >= norb, q = c - s * norb;
      e += p.h[q * norb + q] + s_F[c];
    }
    M->hii = den_fix(0.5 * e, S);
    if (p.den64) s_hii = 0.5 * e;
  } else if (p.den64 && tid >> 5 == 1) {
    double sum = 0.0;
    for (int i = tid & 31; i < nel; i += 32) {
      const int c = s_occ[i], q = c >= norb ? c - norb : c;
      sum += fabs(p.h[q * norb + q]) + fabs(s_F[c]);
    }
    sum = warp_sum(sum);
    if (tid == 32) s_form = den_form(p, S, sum);
  }

  // ---- coarse filter: J within degree 4 of I (I itself included): those of
  // degree 4, most of a large space, from the back of the slot's arrays, the
  // others from the front, so that the passes below do not run the branches
  // of one kind with a few lanes of it in every warp (10^4 determinants, 64
  // orbitals: prep 7.5 -> 5.9 ms, the sweep 81.1 -> 79.5 ms) ----
  const size_t rb = (size_t)slot * (size_t)p.ndet;
  uint64_t* rw = p.r_words + rb * NW;
  double* rc = p.r_coef + rb;
  uint64_t* rh = p.r_hmask + rb;
  uint64_t* rp = p.r_part + rb;
  uint64_t Iw[NW];
#pragma unroll
  for (int w = 0; w < NW; w++) Iw[w] = sI[w];
  const int lane = tid & 31;
  for (long long base = tid - lane; base < p.ndet; base += kThreads) {
    const long long j = base + lane;
    int d = 9;  // degree
    uint64_t Jw[NW];
    if (j < p.ndet) {
      int x = 0;
#pragma unroll
      for (int w = 0; w < NW; w++) {
        Jw[w] = p.dets[(size_t)j * NW + w];
        x += __popcll(Jw[w] ^ Iw[w]);
      }
      d = x >> 1;
    }
    const unsigned b3 = __ballot_sync(kFull, d <= 3), b4 = __ballot_sync(kFull, d == 4);
    if (!(b3 | b4)) continue;
    int at = 0;
    if (lane < 2) at = atomicAdd(&s_nrec[lane], __popc(lane ? b4 : b3));
    const int at3 = __shfl_sync(kFull, at, 0), at4 = __shfl_sync(kFull, at, 1);
    if (d <= 4) {
      const unsigned before = (1u << lane) - 1u;
      const size_t r = d == 4 ? (size_t)p.ndet - 1 - (size_t)(at4 + __popc(b4 & before)) : (size_t)(at3 + __popc(b3 & before));
      uint64_t hmask = 0, part = 0x7FFF7FFF7FFF7FFFull;  // four unused fields (kNoPart)
      uint64_t miss[NW], extra[NW];
#pragma unroll
      for (int w = 0; w < NW; w++) {
        miss[w] = Iw[w] & ~Jw[w];
        extra[w] = Jw[w] & ~Iw[w];
      }
#pragma unroll
      for (int k = 0; k < 4; k++) {  // the k-th hole and particle, spin up first
        if (k >= d) break;
        uint64_t m = miss[NW - 1], iw = Iw[NW - 1], e = extra[NW - 1];
        int hb = s_below[NW - 1], eb = norb + 64 * (NINT - 1);
#pragma unroll
        for (int w = NW - 2; w >= 0; w--) {
          if (miss[w]) {
            m = miss[w];
            iw = Iw[w];
            hb = s_below[w];
          }
          if (extra[w]) {
            e = extra[w];
            eb = (w / NINT) * norb + 64 * (w % NINT);
          }
        }
        const uint64_t low = m & (0ull - m), elow = e & (0ull - e);
        hmask |= 1ull << (hb + __popcll(iw & (low - 1)));
        part ^= (uint64_t)(kNoPart ^ (eb + __popcll(elow - 1))) << (16 * k);
        bool mdone = false, edone = false;
#pragma unroll
        for (int w = 0; w < NW; w++) {  // clear the bits taken, in the first words that have any
          if (!mdone && miss[w]) {
            miss[w] &= miss[w] - 1;
            mdone = true;
          }
          if (!edone && extra[w]) {
            extra[w] &= extra[w] - 1;
            edone = true;
          }
        }
      }
#pragma unroll
      for (int w = 0; w < NW; w++) rw[r * NW + w] = Jw[w];
      rc[r] = p.coefs[j];
      for (int st = 1; st < p.nst; st++) rc[st * p.rc_stride + r] = p.coefs[(size_t)st * p.ndet + j];
      rh[r] = hmask;
      rp[r] = part | (p.rank_of[j] < g ? kBeforeBit : 0ull);
    }
  }

  // ---- bans by J ranked before I, once per generator.  With Q the holes of
  // J, P its particles and H the holes of a batch, t = |Q - H|:
  //  - t = 0 (one hole: t <= 1) bans the batch (dead);
  //  - t = 1 bans the rows of cells holding a particle of P, t = 2 the cells
  //    inside P.
  // d = |Q| = 2 has t = 2 for the batches that miss Q, t = 1 for those with
  // one of its holes (their rows include the cell P) and t = 0 for H = Q: so
  // the cell P is banned in every pair batch (base mask), the rows of P in
  // the batches holding a hole of Q (that hole's row mask).  d = 1 bans the
  // rows of its particle in every pair batch.  d = 3 bans the cells inside P
  // in the batches holding one of its holes (that hole's cell mask; with two
  // of them the rows are banned through the pair's bucket), and in the
  // one-hole batches of Q the cells of P.  Only d = 3 (rows) and d = 4 (cells)
  // are left to the pair buckets.  So a batch starts from base | hole | hole
  // masks, and J ranked after I whose cells those masks ban are not listed.
  // 10^4 determinants, 64 orbitals, 10+10 electrons: a batch reads 123 entries
  // instead of 1,190 and bans and classification fall from 23% to 12% of a
  // CTA's time; with the row pass below the sweep went from 134 to 113 ms. ----
  const MaskDims md = mask_dims(norb, p.nalpha, p.nbeta);
  const int mbase = md.ca + md.cb + md.cm, hmix = md.ca > md.cb ? md.ca : md.cb, nv1 = norb - p.nbeta;
  for (int x = tid; x < p.mask_w; x += kThreads) sm[x] = 0u;
  for (int x = tid; x < p.orb_w; x += kThreads) so[x] = 0ull;
  const int dw = (nbat + 31) / 32;
  for (int w = tid; w < dw; w += kThreads) s_dead[w] = 0u;
  for (int b = tid; b <= nbat + 1; b += kThreads) s_cnt[b] = 0;
  for (int x = tid; x < 2 * norb; x += kThreads) {
    const int s = x / norb, q = x - s * norb;
    int below = 0;
#pragma unroll
    for (int w = 0; w < NINT; w++) {
      const int lim = q - 64 * w;
      if (lim >= 64) below += __popcll(sI[s * NINT + w]);
      else if (lim > 0) below += __popcll(sI[s * NINT + w] & ((1ull << lim) - 1));
    }
    s_vidx[s][q] = (unsigned char)(q - below);
  }
  __syncthreads();
  const bool den64 = p.den64 && s_form == kDenFp64;
  if (den64) {
    for (int x = tid; x < 2 * norb; x += kThreads) M->F[x >= norb][x >= norb ? x - norb : x] = __double_as_longlong(s_F[x]);
    if (tid == 0) M->hii = __double_as_longlong(s_hii);
  }
  const int nlow = s_nrec[0], nfour = s_nrec[1];
  const size_t r4 = (size_t)p.ndet - nfour;  // first record of degree 4
  if (tid == 0) M->nrec = nlow + nfour;
  // cell of two particles: 0, 1 same spin, 2 opposite; its index in the batch
  auto pair_of = [&](int c0, int c1, int* idx) {
    const int s0 = c0 >= norb, s1 = c1 >= norb;
    const int x = s_vidx[s0][c0 - s0 * norb], y = s_vidx[s1][c1 - s1 * norb];
    if (s0 == s1) {
      const int lo = x < y ? x : y, hi = x < y ? y : x;
      *idx = hi * (hi - 1) / 2 + lo;
      return s0;
    }
    *idx = s0 ? y * nv1 + x : x * nv1 + y;
    return 2;
  };
  auto set_orb = [&](uint64_t* w, int c, int spins) {  // bit of code c in masks [spins][NINT]
    const int s = c >= norb, q = c - s * norb;
    atomicOr(reinterpret_cast<unsigned long long*>(w + (spins == 2 ? s * NINT : 0) + (q >> 6)), 1ull << (q & 63));
  };
  auto has_orb = [&](const uint64_t* w, int c, int spins) {
    const int s = c >= norb, q = c - s * norb;
    return (bool)((w[(spins == 2 ? s * NINT : 0) + (q >> 6)] >> (q & 63)) & 1ull);
  };
  auto kill = [&](int b) { atomicOr(&s_dead[b >> 5], 1u << (b & 31)); };
  uint64_t* brow = so;                // rows banned in every pair batch
  uint64_t* bone = so + 2 * NINT;     // cells banned in every one-hole batch
  auto hole_row = [&](int q) { return so + (4 + 3 * q) * NINT; };
  auto hole_one = [&](int q) { return so + (6 + 3 * q) * NINT; };
  auto hole_mask = [&](int q) { return sm + mbase + q * md.hs; };
  for (int r = tid; r < nlow; r += kThreads) {
    const uint64_t pt = rp[r], hm = rh[r];
    if (!(pt & kBeforeBit)) continue;
    const int d = __popcll(hm);
    const int c0 = part_code(pt, 0), c1 = part_code(pt, 1), c2 = part_code(pt, 2);
    if (d == 1) {
      const int q = __ffsll((long long)hm) - 1;
      for (int i = 0; i < nel; i++) kill(i);
      for (int o = 0; o < nel; o++)
        if (o != q) kill(pair_batch(nel, q < o ? q : o, q < o ? o : q));
      set_orb(brow, c0, 2);
    } else if (d == 2) {
      const int q1 = __ffsll((long long)hm) - 1, q2 = __ffsll((long long)(hm & (hm - 1))) - 1;
      kill(q1);
      kill(q2);
      kill(pair_batch(nel, q1, q2));
      int idx;
      const int kd = pair_of(c0, c1, &idx);
      atomicOr(&sm[(kd == 0 ? 0 : kd == 1 ? md.ca : md.ca + md.cb) + (idx >> 5)], 1u << (idx & 31));
      set_orb(bone, c0, 2);
      set_orb(bone, c1, 2);
      set_orb(hole_row(q1), c0, 2);
      set_orb(hole_row(q1), c1, 2);
      set_orb(hole_row(q2), c0, 2);
      set_orb(hole_row(q2), c1, 2);
    } else if (d == 3) {
      uint64_t m = hm;
      for (int i = 0; i < 3; i++) {
        const int q = __ffsll((long long)m) - 1, sq = s_occ[q] >= norb;
        m &= m - 1;
#pragma unroll
        for (int j = 0; j < 3; j++) {
          const int u = j == 2 ? c1 : c0, v = j == 0 ? c1 : c2, w = j == 0 ? c0 : j == 1 ? c1 : c2;
          int idx;
          const int kd = pair_of(u, v, &idx);
          if (kd == 2 || kd == sq) atomicOr(&hole_mask(q)[(kd == 2 ? hmix : 0) + (idx >> 5)], 1u << (idx & 31));
          if ((w >= norb) == sq) set_orb(hole_one(q), w, 1);
        }
      }
    }
  }
  __syncthreads();
  // the slot's work items, without those of batches banned as a whole; by
  // kind: the opposite-spin ones from the back of the list, taken after the
  // others (den64: those of FP64 generators from the back)
  const bool mixed = !by_kind(p);
  for (int j0 = 0; j0 < p.nper; j0 += kThreads) {
    const int j = j0 + tid;
    bool live = false, first = false;
    if (j < p.nper) {
      int tile;
      const int b = item_batch(p, j, &tile);
      Batch B;
      batch_geometry(p, b, tile, B);
      live = B.nct > 0 && !((s_dead[b >> 5] >> (b & 31)) & 1u);
      first = mixed ? !den64 : B.kind != 2;
    }
    const unsigned lf = __ballot_sync(kFull, live && first), ll = __ballot_sync(kFull, live && !first);
    int at = 0;
    if (lane < 2 && (lane ? ll : lf)) at = atomicAdd(p.live_cnt + lane, __popc(lane ? ll : lf));
    const int af = __shfl_sync(kFull, at, 0), al = __shfl_sync(kFull, at, 1);
    const unsigned before = (1u << lane) - 1u;
    if (live)
      p.live[first ? af + __popc(lf & before) : p.wave_slots * p.nper - 1 - (al + __popc(ll & before))] =
          (uint32_t)(slot * p.nper + j);
  }
  bool one_alive = false;
  for (int i = 0; i < nel; i++) one_alive |= !((s_dead[i >> 5] >> (i & 31)) & 1u);

  // ---- buckets: counting sort of the entries left into the shared list,
  // one list per hole and one bucket per pair of holes ----
  for (int r = tid; r < nlow; r += kThreads) {
    const uint64_t hm = rh[r];
    uint64_t pt = rp[r];
    const int d = __popcll(hm);
    if (!(pt & kBeforeBit) && d >= 1 && d <= 3) {
      uint64_t keep = 0;
      const int c0 = part_code(pt, 0), c1 = part_code(pt, 1), c2 = part_code(pt, 2);
      if (d == 1) {
        if (!has_orb(brow, c0, 2)) keep = kKeep0;
      } else if (d == 2) {
        int idx;
        const int kd = pair_of(c0, c1, &idx);
        const bool ban = ((sm[(kd == 0 ? 0 : kd == 1 ? md.ca : md.ca + md.cb) + (idx >> 5)] >> (idx & 31)) & 1u) ||
                         has_orb(brow, c0, 2) || has_orb(brow, c1, 2);
        if (!ban || (one_alive && !(has_orb(bone, c0, 2) && has_orb(bone, c1, 2)))) keep = kKeep0;
      } else {
        uint64_t m = hm;
        for (int i = 0; i < 3; i++) {
          const int q = __ffsll((long long)m) - 1, sq = s_occ[q] >= norb;
          m &= m - 1;
          bool live = false;
#pragma unroll
          for (int j = 0; j < 3; j++) {
            const int u = j == 2 ? c1 : c0, v = j == 0 ? c1 : c2, w = j == 0 ? c0 : j == 1 ? c1 : c2;
            int idx;
            const int kd = pair_of(u, v, &idx);
            if (kd == 2 || kd == sq) {
              const uint32_t bw = sm[(kd == 0 ? 0 : kd == 1 ? md.ca : md.ca + md.cb) + (idx >> 5)] |
                                  hole_mask(q)[(kd == 2 ? hmix : 0) + (idx >> 5)];
              live |= !((bw >> (idx & 31)) & 1u) && !has_orb(brow, u, 2) && !has_orb(brow, v, 2) &&
                      !has_orb(hole_row(q), u, 2) && !has_orb(hole_row(q), v, 2);
            }
            if (one_alive && (w >= norb) == sq) live |= !has_orb(bone, w, 2) && !has_orb(hole_one(q), w, 1);
          }
          if (live) keep |= kKeep0 << (16 * i);
        }
      }
      if (keep) {
        pt |= keep;
        rp[r] = pt;
      }
    }
    for_buckets(hm, pt, nel, nbat, s_dead, [&](int b) { atomicAdd(&s_cnt[b], 1); });
  }
  for (int r = tid; r < nfour; r += kThreads)
    for_pairs4(rh[r4 + r], nel, s_dead, [&](int b) { atomicAdd(&s_cnt[b], 1); });
  __syncthreads();
  if (tid < 32) {  // exclusive scan of the counts
    int run = 0;
    for (int b0 = 0; b0 <= nbat; b0 += 32) {
      const int b = b0 + tid;
      const int c = b <= nbat ? s_cnt[b] : 0;
      int inc = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFull, inc, o);
        if (tid >= o) inc += v;
      }
      if (b <= nbat) s_cnt[b] = run + inc - c;
      run += __shfl_sync(kFull, inc, 31);
    }
    if (tid == 0) {
      s_cnt[nbat + 1] = run;
      if (run > p.ent_cap) atomicOr(p.err, 8);
    }
  }
  __syncthreads();
  int* ofs = p.b_ofs + (size_t)slot * (nbat + 2);
  for (int b = tid; b <= nbat + 1; b += kThreads) ofs[b] = s_cnt[b];
  uint32_t* gm = p.b_mask + (size_t)slot * p.mask_w;
  for (int x = tid; x < p.mask_w; x += kThreads) gm[x] = sm[x];
  uint64_t* go = p.o_mask + (size_t)slot * p.orb_w;
  for (int x = tid; x < p.orb_w; x += kThreads) go[x] = so[x];
  __syncthreads();
  ulonglong2* e_hp = p.e_hp + (size_t)slot * (size_t)p.ent_cap;
  uint32_t* e_rec = p.e_rec + (size_t)slot * (size_t)p.ent_cap;
  const long long cap = p.ent_cap;
  auto put = [&](int b, uint64_t hm, uint64_t pe, uint32_t rec) {
    const int o = atomicAdd(&s_cnt[b], 1);
    if (o < cap) {
      e_hp[o] = make_ulonglong2(hm, pe);
      e_rec[o] = rec;
    }
  };
  for (int r = tid; r < nlow; r += kThreads) {
    const uint64_t hm = rh[r], pt = rp[r], pe = pt & ~(kKeep0 | kKeep1 | kKeep2);
    const uint32_t rec = (uint32_t)r | (pt & kBeforeBit ? 1u << 31 : 0u);
    for_buckets(hm, pt, nel, nbat, s_dead, [&](int b) { put(b, hm, pe, rec); });
  }
  for (int i = tid; i < nfour; i += kThreads) {
    const size_t r = r4 + i;
    const uint64_t hm = rh[r], pt = rp[r];
    const uint32_t rec = (uint32_t)r | (pt & kBeforeBit ? 1u << 31 : 0u);
    for_pairs4(hm, nel, s_dead, [&](int b) { put(b, hm, pt, rec); });
  }
}

// One CTA per generator slot of the wave.
template <int NINT>
__global__ void __launch_bounds__(kThreads) prep_kernel(const __grid_constant__ SweepParams p) {
  prep_slot<NINT>(p, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Several instances in one launch (a wave of each of their sweeps).  ps[i] is
// instance i's parameters for this wave; slot_ofs / item_ofs number the
// instances' generator slots / work items one instance after the other.
// ---------------------------------------------------------------------------
static_assert(sizeof(SweepParams) % 8 == 0, "parameters are copied by 8-byte words");

// Copy the parameters of instance i to shared memory (all threads).
__device__ __forceinline__ void load_params(SweepParams& dst, const SweepParams* ps, int i) {
  const unsigned long long* src = reinterpret_cast<const unsigned long long*>(ps + i);
  unsigned long long* d = reinterpret_cast<unsigned long long*>(&dst);
  for (int w = threadIdx.x; w < (int)(sizeof(SweepParams) / 8); w += blockDim.x) d[w] = src[w];
}

// The last instance whose first slot (item) is at or below x.
template <typename T>
__device__ __forceinline__ int instance_of(const T* ofs, int n, long long x) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((long long)ofs[mid] <= x) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// One CTA per generator slot of every instance of the wave.
template <int NINT>
__global__ void __launch_bounds__(kThreads) prep_multi_kernel(const __grid_constant__ MultiWave m) {
  __shared__ SweepParams Ps;
  __shared__ int s_inst;
  if (threadIdx.x == 0) s_inst = instance_of(m.slot_ofs, m.n, blockIdx.x);
  __syncthreads();
  const int i = s_inst;
  load_params(Ps, m.ps, i);
  __syncthreads();
  prep_slot<NINT>(Ps, (int)blockIdx.x - m.slot_ofs[i]);
}

// ---------------------------------------------------------------------------
// batch kernel
// ---------------------------------------------------------------------------
template <int NINT, typename NT>
struct BatchShared {
  int occ[kMaxElec];
  // virtual orbitals of I by index and their indices by orbital (255: occupied)
  unsigned char vir[2][kMaxOrb], vidx[2][kMaxOrb];
  int nv[2];  // the sweep's virtual orbitals per spin
  float inv_nv1;
  // per virtual orbital of the cells' row and column: d in fixed point
  // (den_scale), E0 - H_II + ... of the row (E0 - base - u0) and the sum u of
  // the column for H_aa; the orbital; idx: <I|H|I - H + R> by pair tables like
  // those of the J reaching every cell (its particles are the hole pair H)
  struct __align__(16) Side {
    long long d;
    int idx, orb;
  } row[kMaxOrb], col[kMaxOrb];
  uint64_t hk0[kMaxOrb];  // digest fold of the spin-up words of a row's determinants
  NT cI;
  uint64_t kbase[2 * NINT];  // I with the batch's holes removed
  // rows (and columns) of cells banned as a whole by J ranked before I, bits
  // by orbital
  uint64_t rowban[2 * NINT];
  // the item's records and bucket entries (kept here, not in registers, over
  // the phases that do not touch them): words, coefficients, hole masks and
  // particle words; entries; the lists' offsets and first positions
  const uint64_t *rw, *rhm, *rpt;
  const double* rc;
  const ulonglong2* ehp;
  const uint32_t* erec;
  int seg_o[4], seg_s[4];
  Batch bt;  // the item's batch, read again by each phase
  int item[2];        // this work item and the next (-1: none)
  int inext, iend, nlive, nfirst;  // positions left of the last draw; live items of the wave, those listed from the front
  // storage of one phase of a work item at a time: the J lists, the
  // selection histogram, the per-thread sums of the reduction
  union {
    struct {
      // records of the J reaching every cell; of the J reaching rows (from
      // the front) and a few cells (from the back)
      int L0[kChunk], L12[kChunk];
    } l;
    int hist[256];
    double red_t[2][kThreads];  // per-thread e and (A/D)^2 sums of the item
  } u;
  int n0, n1, n2;
  int cnext;  // next unit of the row pass to draw
  // a group of J reaching every cell, J = K + {x1, x2}: per particle orbital
  // of each slot the offset of its integrals, with the phase parity in bit 31
  // and, for the particles of J, bit 30 (row) or 29 (column), so that a cell's
  // offset, sign and flags are one sum
  NT gcj[kGroup];
  int gx1[kGroup], gx2[kGroup], gB[kGroup];
  int gRow[kGroup][kMaxOrb], gCol[kGroup][kMaxOrb];
  int wsum[kWarps];
  // selection
  int tkcnt;
  unsigned long long tau;
  uint64_t pw[1 + 2 * NINT];
  uint64_t thr[1 + 2 * NINT];
  int need, group, found_w, found_sh;
  // reductions: warps that finished the item, their counts
  int arrive;
  unsigned long long red_na[kWarps], red_con[kWarps];
  double sw2;
  // totals over the sweep: digest sum and xor, min |D| (of a thread each), |A| < 1e-14
  unsigned long long td0[kThreads], td1[kThreads], tmin[kThreads];
  unsigned int tiny;
  int nlist;  // cells left after the bans
};

template <int NINT, typename NT, int KD = -1>  // KD: the batch's kind where it is known
__device__ __forceinline__ void cell_orbitals(const Batch& B, const BatchShared<NINT, NT>& S, int c, int* r,
                                              int* s, int* x, int* y) {
  const int kind = KD >= 0 ? KD : B.kind;
  if (kind == 0) {
    *x = c;
    *y = -1;
    *r = S.vir[B.sa][c];
    *s = -1;
  } else if (kind == 2) {
    const int nv1 = S.nv[1];
    int xx = __float2int_rz((float)c * S.inv_nv1);  // c < 2^14: exact up to one step
    if (xx * nv1 > c) xx--;
    if ((xx + 1) * nv1 <= c) xx++;
    *x = xx;
    *y = c - xx * nv1;
    *r = S.vir[0][xx];
    *s = S.vir[1][*y];
  } else {
    // c < 2^13: the square root is exact up to one step
    int yy = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)c)) * 0.5f);
    if (yy * (yy - 1) / 2 > c) yy--;
    if ((yy + 1) * yy / 2 <= c) yy++;
    *x = c - yy * (yy - 1) / 2;
    *y = yy;
    *r = S.vir[B.sa][*x];
    *s = S.vir[B.sa][yy];
  }
}

// The FP64 form of the denominators (kDenFp64): the rows' and columns' terms,
// u = F - W(q, a) [- W(q, b)] of a column, (E0 - base) - u of a row, base = H_II -
// F(a) [- F(b) + W(a, b)]; all threads, with S.vir set.
template <int NINT, typename NT>
__device__ __forceinline__ void den64_sides(const SweepParams& p, BatchShared<NINT, NT>& S, const Batch& B,
                                            const GenMeta* M, double e0) {
  const int norb = p.norb;
  auto F = [&](int s, int q) { return __longlong_as_double(M->F[s][q]); };
  auto W = [&](int x, int sx, int y, int sy) {
    const double j = p.Jm[x * norb + y];
    return sx == sy ? j - p.Km[x * norb + y] : j;
  };
  double base = __longlong_as_double(M->hii) - F(B.sa, B.qa);
  if (B.h == 2) base = base - F(B.sb, B.qb) + W(B.qa, B.sa, B.qb, B.sb);
  for (int c = 0; c < B.h; c++) {
    const int s = c ? B.sb : B.sa;
    for (int v = threadIdx.x; v < S.nv[s]; v += kThreads) {
      const int q = S.vir[s][v];
      double u = F(s, q) - W(q, s, B.qa, B.sa);
      if (B.h == 2) u -= W(q, s, B.qb, B.sb);
      if (c) S.col[v].d = __double_as_longlong(u);
      else S.row[v].d = __double_as_longlong((e0 - base) - u);
    }
  }
}
// a / D, D = (row - column - pair) + de of a cell with the orbitals of r and c
// (kind 0: row + de); *D becomes the bits of |D|.
template <typename Side>
__device__ __forceinline__ double den64_quot(const SweepParams& p, double a, const Side& r, const Side& c, int kind,
                                             double de, long long* D) {
  double d = __longlong_as_double(r.d);
  if (kind > 0) {
    const int at = r.orb * p.norb + c.orb;
    d -= __longlong_as_double(c.d) + (kind == 1 ? p.Jm[at] - p.Km[at] : p.Jm[at]);
  }
  d += de;
  *D = __double_as_longlong(fabs(d));
  return a / d;
}

// Bans cell c (an index over the whole batch) when it lies in this item's tile.
__device__ __forceinline__ void ban_cell(uint32_t* ban, const Batch& B, int c) {
  const int cc = c - B.clo;
  if ((unsigned)cc < (unsigned)B.nct) atomicOr(&ban[cc >> 5], 1u << (cc & 31));
}

__device__ __forceinline__ int pair_cell(int x, int y) {  // x != y virtual indices
  int lo = x < y ? x : y, hi = x < y ? y : x;
  return hi * (hi - 1) / 2 + lo;
}

// Small sets are packed 8 bits per entry into a 32-bit register (orbitals
// < 128, spin-orbital codes < 256) with the count kept beside them: arrays
// indexed at run time would live in local memory.
__device__ __forceinline__ int pk(uint32_t v, int i) { return (int)((v >> (8 * i)) & 0xFFu); }

// Particles of J outside I, filtered to a spin, as orbitals (packed).
__device__ __forceinline__ uint32_t particles_of_spin(uint64_t part, int norb, int spin, int* n) {
  uint32_t out = 0;
  int k = 0;
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int c = part_code(part, i);
    if (c == kNoPart) continue;
    const int s = c >= norb;
    if (s == spin) {
      out |= (uint32_t)(c - s * norb) << (8 * k);
      k++;
    }
  }
  *n = k;
  return out;
}

// Cells inside the particles of J (t = 2): visited by one thread.
template <int NINT, typename NT, typename Fn>
__device__ __forceinline__ void for_subset_cells(const Batch& B, const BatchShared<NINT, NT>& S, int norb,
                                                 uint64_t part, Fn&& fn) {
  if (B.kind == 0) {
    int np;
    const uint32_t P = particles_of_spin(part, norb, B.sa, &np);
#pragma unroll 1
    for (int i = 0; i < np; i++) fn(S.vidx[B.sa][pk(P, i)]);
  } else if (B.kind == 1) {
    int np;
    const uint32_t P = particles_of_spin(part, norb, B.sa, &np);
#pragma unroll 1
    for (int i = 0; i < np; i++)
#pragma unroll 1
      for (int j = i + 1; j < np; j++) fn(pair_cell(S.vidx[B.sa][pk(P, i)], S.vidx[B.sa][pk(P, j)]));
  } else {
    int na, nb;
    const uint32_t Pa = particles_of_spin(part, norb, 0, &na);
    const uint32_t Pb = particles_of_spin(part, norb, 1, &nb);
#pragma unroll 1
    for (int i = 0; i < na; i++)
#pragma unroll 1
      for (int j = 0; j < nb; j++) fn(S.vidx[0][pk(Pa, i)] * S.nv[1] + S.vidx[1][pk(Pb, j)]);
  }
}

// True when the row (column) of cells holding orbital q of spin s is banned
// as a whole (two-hole batches).
template <int NINT, typename NT>
__device__ __forceinline__ bool row_banned(const BatchShared<NINT, NT>& S, int s, int q) {
  return (S.rowban[s * NINT + (q >> 6)] >> (q & 63)) & 1ull;
}

// True when some cell inside the particles of J lies in this item's tile and
// is not banned: a J with t = 2 that reaches no such cell adds nothing and is
// dropped at classification.  Rows banned as a whole are tested by their
// flags (their cells may not be in the ban bits yet).
template <int NINT, typename NT>
__device__ __forceinline__ bool subset_live(const Batch& B, const BatchShared<NINT, NT>& S, int norb,
                                            uint64_t part, const uint32_t* ban) {
  bool live = false;
  if (B.h == 2)
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int c = part_code(part, i), s = c >= norb;
      if (c != kNoPart && row_banned<NINT, NT>(S, s, c - s * norb)) part |= 0x7FFFull << (16 * i);
    }
  for_subset_cells<NINT, NT>(B, S, norb, part, [&](int c) {
    const int cc = c - B.clo;
    live |= (unsigned)cc < (unsigned)B.nct && !((ban[cc >> 5] >> (cc & 31)) & 1u);
  });
  return live;
}

// True when some row or column of cells that a J with t = 1 reaches (the
// rows of its particles) is not banned as a whole.  Rows flagged in loop 1
// hold no live cell, so a J whose rows are all flagged adds nothing: it is
// dropped at classification (the rows and columns of a J ranked after I are
// mostly those of earlier J with the same particles).
template <int NINT, typename NT>
__device__ __forceinline__ bool row_live(const Batch& B, const BatchShared<NINT, NT>& S, int norb, uint64_t part) {
  bool live = false;
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int c = part_code(part, i);
    if (c == kNoPart) continue;
    const int s = c >= norb, q = c - s * norb;
    if (B.kind == 2 || s == B.sa) live |= !row_banned<NINT, NT>(S, s, q);
  }
  return live;
}

// X = (particles of J) + (holes of H that J keeps); T = holes of J not in H.
// Both sets are spin-orbital codes, packed (see pk).
template <int NINT, typename NT>
__device__ __forceinline__ void excitation_sets(const Batch& B, const BatchShared<NINT, NT>& S, uint64_t part,
                                                uint64_t hm, uint32_t* X, int* nx, uint32_t* T, int* nt) {
  int a = 0, b = 0;
  uint32_t xs = 0, ts = 0;
#pragma unroll
  for (int i = 0; i < 4; i++) {
    const int c = part_code(part, i);
    if (c != kNoPart && a < 4) xs |= (uint32_t)c << (8 * a++);
  }
  if (!((hm >> B.ia) & 1ull) && a < 4) xs |= (uint32_t)B.ca << (8 * a++);
  if (B.h == 2 && !((hm >> B.ib) & 1ull) && a < 4) xs |= (uint32_t)B.cb << (8 * a++);
  uint64_t tm = hm & ~B.hm;
  while (tm && b < 2) {
    const int i = __ffsll((long long)tm) - 1;
    tm &= tm - 1;
    ts |= (uint32_t)S.occ[i] << (8 * b++);
  }
  *X = xs;
  *nx = a;
  *T = ts;
  *nt = b;
}

// <J|H|alpha> for the double substitution u0 u1 -> q0 q1 of J (spin-orbital
// codes, u0 < u1 occupied, q0 < q1 empty).
template <int NINT, typename NT, bool E4>
__device__ __forceinline__ NT double_element(const NT* eri, int norb, const uint64_t* Jw, int u0, int u1, int q0,
                                             int q1) {
  const int s1 = u0 >= norb, s2 = u1 >= norb;
  const int h1 = u0 - s1 * norb, p1 = q0 - s1 * norb;
  const int h2 = u1 - s2 * norb, p2 = q1 - s2 * norb;
  uint64_t w1[NINT], w2[NINT];
#pragma unroll
  for (int w = 0; w < NINT; w++) {
    w1[w] = s1 ? Jw[NINT + w] : Jw[w];
    w2[w] = s2 ? Jw[NINT + w] : Jw[w];
    if (s1 == s2) {  // the second substitution counts on the result of the first
      if ((h1 >> 6) == w) w2[w] &= ~(1ull << (h1 & 63));
      if ((p1 >> 6) == w) w2[w] |= 1ull << (p1 & 63);
    }
  }
  const int n = count_between<NINT>(w1, h1 < p1 ? h1 : p1, h1 < p1 ? p1 : h1) +
                count_between<NINT>(w2, h2 < p2 ? h2 : p2, h2 < p2 ? p2 : h2);
  NT v = eri[gidx<E4>(h1, p1, h2, p2, norb)];
  if (s1 == s2) v -= eri[gidx<E4>(h1, p2, h2, p1, norb)];
  return flip_sign(v, n & 1);
}

// Phases of the substitutions u -> z of a string w (NINT words, u occupied)
// for every empty z at once: bit z of M is the parity of the occupied
// orbitals strictly between u and z, flipped when c is odd.  With P(x) the
// parity of the occupied orbitals below x (a prefix XOR of the string, the
// idea of Algorithm PhasemaskOfDet), that parity is P(z) ^ P(u) ^ [z > u].
template <int NINT>
__device__ __forceinline__ void phase_mask(const uint64_t* w, int u, int c, uint64_t* M) {
  uint64_t carry = 0;
  int pu = c & 1;
#pragma unroll
  for (int i = 0; i < NINT; i++) {
    uint64_t t = w[i];
    t ^= t << 1;
    t ^= t << 2;
    t ^= t << 4;
    t ^= t << 8;
    t ^= t << 16;
    t ^= t << 32;
    t ^= carry;                          // parity of the orbitals up to x
    carry = 0ull - (t >> 63);
    const uint64_t e = t ^ w[i];         // below x
    const int lu = u - 64 * i;
    if (lu >= 0 && lu < 64) pu ^= (int)((e >> lu) & 1ull);
    M[i] = e ^ (lu < 0 ? ~0ull : (lu < 64 ? (~0ull << lu) << 1 : 0ull));
  }
  const uint64_t f = 0ull - (uint64_t)pu;
#pragma unroll
  for (int i = 0; i < NINT; i++) M[i] ^= f;
}

template <int NINT>
__device__ __forceinline__ bool mask_bit(const uint64_t* M, int z) {
  const uint64_t w = NINT == 1 ? M[0] : (z < 64 ? M[0] : M[NINT - 1]);
  return (w >> (z & 63)) & 1ull;
}

template <int NINT>
__device__ __forceinline__ void shfl_words(const uint64_t* in, int src, uint64_t* out) {
#pragma unroll
  for (int w = 0; w < NINT; w++) out[w] = __shfl_sync(kFull, in[w], src);
}

template <typename NT>
__device__ __forceinline__ NT warp_sum_nt(NT v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Gradient of one matrix element: adds w * d<J|H|alpha>/d(theta) into dh
// (symmetric halves) and the packed integrals, by the cases of the
// excitation degree.
template <int NINT>
__device__ __noinline__ void element_grad(double* g_dh, double* g_deri, int norb, const uint64_t* Jw, uint32_t X,
                                          int nx, uint32_t T, int nt, int r, int s, double w) {
  int ho[2], pa[2], nh = 0, npp = 0;
  bool r_in = false, s_in = false;
  for (int i = 0; i < nx; i++) {
    const int x = pk(X, i);
    r_in |= (x == r);
    s_in |= (x == s);
    if (x != r && x != s && nh < 2) ho[nh++] = x;
  }
  for (int i = 0; i < nt && npp < 2; i++) pa[npp++] = pk(T, i);
  if (!r_in && npp < 2) pa[npp++] = r;
  if (s >= 0 && !s_in && npp < 2) pa[npp++] = s;
  if (nh == 0 || nh != npp) return;
  if (nh == 1) {
    const int sp = ho[0] >= norb, a = ho[0] - sp * norb, b = pa[0] - sp * norb;
    const uint64_t* sw = Jw + sp * NINT;
    const int lo = a < b ? a : b, hi = a < b ? b : a;
    const double ws = (count_between<NINT>(sw, lo, hi) & 1) ? -w : w;
    atomicAdd(&g_dh[a * norb + b], 0.5 * ws);
    atomicAdd(&g_dh[b * norb + a], 0.5 * ws);
#pragma unroll
    for (int t = 0; t < 2; t++) {
#pragma unroll
      for (int wd = 0; wd < NINT; wd++) {
        uint64_t bits = Jw[t * NINT + wd];
        while (bits) {
          const int q = 64 * wd + __ffsll((long long)bits) - 1;
          bits &= bits - 1;
          atomicAdd(&g_deri[eri_index(a, b, q, q)], ws);
          if (t == sp) atomicAdd(&g_deri[eri_index(a, q, q, b)], -ws);
        }
      }
    }
    return;
  }
  if (ho[0] > ho[1]) { const int t = ho[0]; ho[0] = ho[1]; ho[1] = t; }
  if (pa[0] > pa[1]) { const int t = pa[0]; pa[0] = pa[1]; pa[1] = t; }
  const int s1 = ho[0] >= norb, s2 = ho[1] >= norb;
  const int h1 = ho[0] - s1 * norb, p1 = pa[0] - s1 * norb;
  const int h2 = ho[1] - s2 * norb, p2 = pa[1] - s2 * norb;
  uint64_t w1[NINT];
#pragma unroll
  for (int wd = 0; wd < NINT; wd++) w1[wd] = Jw[s1 * NINT + wd];
  const int n1 = count_between<NINT>(w1, h1 < p1 ? h1 : p1, h1 < p1 ? p1 : h1);
  w1[h1 >> 6] &= ~(1ull << (h1 & 63));
  w1[p1 >> 6] |= (1ull << (p1 & 63));
  const int n2 = (s2 == s1) ? count_between<NINT>(w1, h2 < p2 ? h2 : p2, h2 < p2 ? p2 : h2)
                            : count_between<NINT>(Jw + s2 * NINT, h2 < p2 ? h2 : p2, h2 < p2 ? p2 : h2);
  const double ws = ((n1 + n2) & 1) ? -w : w;
  atomicAdd(&g_deri[eri_index(h1, p1, h2, p2)], ws);
  if (s1 == s2) atomicAdd(&g_deri[eri_index(h1, p2, h2, p1)], -ws);
}

// w * dW(x, y)/d(theta), W(x, y) = (xx|yy) - delta_spin (xy|yx)
__device__ __forceinline__ void w_grad(const SweepParams& p, int x, int sx, int y, int sy, double w) {
  atomicAdd(&p.g_deri[eri_index(x, x, y, y)], w);
  if (sx == sy) atomicAdd(&p.g_deri[eri_index(x, y, y, x)], -w);
}

// ---------------------------------------------------------------------------
// Selection buffer compaction: keep the k best entries (|e| descending, key
// ascending) of the CTA's buffer.  MSD radix select over the composite
// (~bits(|e|), key words), 8-bit digits, then an ordered in-place compaction.
// ---------------------------------------------------------------------------
// Selection histogram bins: the binary exponent of |e| (2^-100 .. 2^27) and
// the top 3 mantissa bits, so that a bin's lower edge is a double whose bits
// are easy to form.  Values below 2^-100 fall in bin 0, whose edge is taken as
// 0; values of 2^28 and above fall in the last bin, whose edge is below them.
__device__ __forceinline__ int sel_bin(unsigned long long ebits) {
  const int ex = (int)(ebits >> 52) - 923;
  if (ex < 0) return 0;
  if (ex > 127) return kSelBins - 1;
  return ex * 8 + (int)((ebits >> 49) & 7ull);
}
__device__ __forceinline__ unsigned long long sel_bin_edge(int b) {
  return ((unsigned long long)(b / 8 + 923) << 52) | ((unsigned long long)(b % 8) << 49);
}

// A lower bound of the k-th largest |e| of the whole sweep: the lower edge of
// the highest bin at which at least k distinct perturbers (each counted once,
// when offered to a selection buffer) have |e| at or above the edge.
static __device__ unsigned long long hist_threshold(const unsigned int* hist, long long k) {
  const int lane = threadIdx.x & 31;
  constexpr int per = kSelBins / 32;
  // lane l owns bins [l*per, (l+1)*per); sums from the top
  unsigned long long mine = 0;
  for (int b = 0; b < per; b++) mine += hist[lane * per + b];
  unsigned long long suffix = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long v = __shfl_down_sync(0xffffffffu, suffix, o);
    if (lane + o < 32) suffix += v;
  }
  // suffix = counts in bins of lanes >= lane; the lane whose block holds the
  // k-th count from the top walks its bins
  const unsigned long long above_me = suffix - mine;
  unsigned long long res = 0;
  const bool holder = (above_me < (unsigned long long)k) && (suffix >= (unsigned long long)k);
  if (holder) {
    unsigned long long cum = above_me;
    for (int b = per - 1; b >= 0; b--) {
      cum += hist[lane * per + b];
      if (cum >= (unsigned long long)k) {
        const int bin = lane * per + b;
        res = bin > 0 ? sel_bin_edge(bin) : 0ull;
        break;
      }
    }
  }
  // broadcast from the holder lane (at most one)
  const unsigned m = __ballot_sync(0xffffffffu, holder);
  if (m == 0) return 0ull;
  return __shfl_sync(0xffffffffu, res, __ffs(m) - 1);
}

template <int NINT>
__device__ __forceinline__ uint64_t composite_word(const double* te, const uint64_t* tk, int i, int w) {
  if (w == 0) return ~((unsigned long long)__double_as_longlong(te[i]) & 0x7FFFFFFFFFFFFFFFull);
  return tk[(size_t)i * (2 * NINT) + (w - 1)];
}

template <int NINT>
__device__ bool prefix_match(const double* te, const uint64_t* tk, int i, const uint64_t* pw, int w,
                             int keep_sh) {
  for (int v = 0; v < w; v++)
    if (composite_word<NINT>(te, tk, i, v) != pw[v]) return false;
  if (keep_sh >= 64) return true;
  return (composite_word<NINT>(te, tk, i, w) >> keep_sh) == (pw[w] >> keep_sh);
}

template <int NINT, typename NT>
__device__ __noinline__ void compact_selection(const SweepParams& p, BatchShared<NINT, NT>& S, double* te,
                                               double* ta, uint64_t* tk) {
  constexpr int NW = 1 + 2 * NINT;
  const int tid = threadIdx.x;
  __syncthreads();
  const int n = S.tkcnt;
  const long long k = p.k;
  if (n <= k) return;
  if (tid == 0) {
    S.need = (int)k;
    for (int w = 0; w < NW; w++) S.pw[w] = 0;
    S.group = n;
    S.found_w = NW - 1;
    S.found_sh = 0;
  }
  __syncthreads();
  bool done = false;
  for (int w = 0; w < NW && !done; w++) {
    for (int sh = 56; sh >= 0; sh -= 8) {
      for (int b = tid; b < 256; b += kThreads) S.u.hist[b] = 0;
      __syncthreads();
      for (int i = tid; i < n; i += kThreads)
        if (prefix_match<NINT>(te, tk, i, S.pw, w, sh + 8))
          atomicAdd(&S.u.hist[(composite_word<NINT>(te, tk, i, w) >> sh) & 255], 1);
      __syncthreads();
      if (tid == 0) {
        int c = 0, d = 255;
        for (int b = 0; b < 256; b++) {
          if (c + S.u.hist[b] >= S.need) {
            d = b;
            break;
          }
          c += S.u.hist[b];
        }
        S.need -= c;
        S.group = S.u.hist[d];
        S.pw[w] |= (uint64_t)d << sh;
        S.found_w = w;
        S.found_sh = sh;
      }
      __syncthreads();
      if (S.group <= 1) {
        done = true;
        break;
      }
    }
  }
  if (S.group == 1) {
    for (int i = tid; i < n; i += kThreads)
      if (prefix_match<NINT>(te, tk, i, S.pw, S.found_w, S.found_sh))
        for (int w = 0; w < NW; w++) S.thr[w] = composite_word<NINT>(te, tk, i, w);
  } else if (tid == 0) {
    for (int w = 0; w < NW; w++) S.thr[w] = S.pw[w];
  }
  __syncthreads();
  int out = 0;
  for (int base = 0; base < n; base += kThreads) {
    const int i = base + tid;
    bool keep = false;
    double e = 0, a = 0;
    uint64_t key[2 * NINT];
    if (i < n) {
      int cmp = 0;
      for (int w = 0; w < NW && cmp == 0; w++) {
        const uint64_t x = composite_word<NINT>(te, tk, i, w);
        cmp = x < S.thr[w] ? -1 : (x > S.thr[w] ? 1 : 0);
      }
      keep = cmp <= 0;
      e = te[i];
      a = ta[i];
#pragma unroll
      for (int w = 0; w < 2 * NINT; w++) key[w] = tk[(size_t)i * (2 * NINT) + w];
    }
    int total;
    const int pos = block_scan_flag(keep, S.wsum, &total);
    if (keep) {
      const int o = out + pos;
      te[o] = e;
      ta[o] = a;
#pragma unroll
      for (int w = 0; w < 2 * NINT; w++) tk[(size_t)o * (2 * NINT) + w] = key[w];
    }
    out += total;
  }
  __syncthreads();
  if (tid < 32) {
    const unsigned long long th = hist_threshold(p.sel_hist, k);
    if (tid == 0) {
      S.tkcnt = out;
      unsigned long long t = ~S.thr[0];
      t = th > t ? th : t;
      if (t > S.tau) S.tau = t;
      atomicMax(p.tau_bits, t);
    }
  }
  __syncthreads();
}

// The CTA's dynamic shared memory for the sweep of p and the sweep's sizes,
// formed by the kernel once (once per instance in the multi-instance kernel)
// and kept across work items.  Multi-state form: one FP64 accumulator per
// state (stride mc), then the ban bits, the CTA group's coefficients per
// state, c_I per state and the weights w_s; one-state form: the exact 96-bit
// accumulators (their low, middle and high words), then the ban bits.
struct ItemEnv {
  double* A;
  uint32_t *A0, *A1, *A2;
  uint32_t* ban;
  unsigned short* lst;  // one-state form: the cells left
  double *ms_gc, *ms_cI, *ms_w;
  long long* ms_de;  // E0_s - E0_0, fixed point
  int mc, nst, norb, nel, nbat, nper;
  int dscale;    // den_scale
  long long e0;  // E0 (state 0's) in those units
};

template <bool MS>
__device__ __forceinline__ ItemEnv item_env(const SweepParams& p) {
  extern __shared__ __align__(16) unsigned char dyn[];
  ItemEnv E;
  E.mc = p.max_cells;
  E.A = reinterpret_cast<double*>(dyn);
  E.A0 = reinterpret_cast<uint32_t*>(dyn);
  E.A1 = E.A0 + E.mc;
  E.A2 = E.A1 + E.mc;
  E.ban = MS ? reinterpret_cast<uint32_t*>(E.A + p.nst * E.mc) : E.A2 + ((E.mc + 1) & ~1);
  E.lst = reinterpret_cast<unsigned short*>(E.ban + (E.mc + 31) / 32);
  E.ms_gc = reinterpret_cast<double*>(E.ban + (((E.mc + 31) / 32 + 1) & ~1));
  E.ms_cI = E.ms_gc + kGroup * kMaxStates;
  E.ms_w = E.ms_cI + kMaxStates;
  E.ms_de = reinterpret_cast<long long*>(E.ms_w + kMaxStates);
  E.nst = MS ? p.nst : 1;
  E.norb = p.norb;
  E.nel = p.nel;
  E.nbat = p.nbat;
  E.nper = p.nper;
  E.dscale = den_scale(p);
  E.e0 = den_fix(MS ? p.st_e0[0] : p.e0, E.dscale);
  return E;
}

// This CTA's candidate buffers of the selection.
__device__ __forceinline__ double* buf_e(const SweepParams& p) { return p.tk_e + (size_t)blockIdx.x * (size_t)p.cap; }
__device__ __forceinline__ double* buf_a(const SweepParams& p) { return p.tk_a + (size_t)blockIdx.x * (size_t)p.cap; }
template <int NINT>
__device__ __forceinline__ uint64_t* buf_key(const SweepParams& p) {
  return p.tk_key + (size_t)blockIdx.x * (size_t)p.cap * (2 * NINT);
}

// One work item of the sweep of p (a generator slot's hole-set batch, or a
// row tile of one): bans, the accumulation of A_alpha, the cells pass and the
// item's sums.  Used by the kernel of one sweep and by the kernel whose queue
// spans the waves of several instances.  FP: its generator's denominators are
// in FP64.
//
// What bounds an item is latency, not a pipe (issue slots half used, FP64
// 26%): 256 threads share about 2,000 cells, and every phase that few of them
// work in, every dependent global load and every barrier shows.  So the
// set-up reads the generator straight from global memory in two dependent
// steps, the first round of bucket entries is in registers before the bans
// are, tables of the J reaching every cell are units of the row pass, their
// terms are formed in the cells pass, and the item's sums are finished by the
// last warp to arrive while the others wait at the next item's first barrier:
// five barriers where there were fifteen.
template <int NINT, typename NT, bool GRAD, bool MS, bool E4, bool FP>
__device__ __forceinline__ void batch_item(const SweepParams& p, BatchShared<NINT, NT>& S, const long long item,
                                           const int F, const ItemEnv& E,
                                           const NT* eri_n, const NT* h_n) {
  constexpr int NW = 2 * NINT;
  double* A = E.A;  // multi-state form
  uint32_t *A0 = E.A0, *A1 = E.A1, *A2 = E.A2;
  uint32_t* ban = E.ban;
  double* ms_gc = E.ms_gc;
  double* ms_cI = E.ms_cI;
  double* ms_w = E.ms_w;
  long long* ms_de = E.ms_de;
  const int mc = E.mc, nst = E.nst;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int norb = E.norb, nel = E.nel, nbat = E.nbat;
  const int nper = E.nper;

  const int slot = (int)(item / nper), jitem = (int)(item - (long long)slot * nper);
  int tile;
  const int b = item_batch(p, jitem, &tile);
  Batch B;
  batch_geometry(p, b, tile, B);
  const GenMeta* M = p.meta + slot;

  // ---- set-up ----
  // bucket lists (prep_slot): this batch's bucket (a one-hole batch's is its
  // hole's list), for a two-hole batch the lists of its two holes (a record
  // holding both is in the batch's bucket), then the shared list (a record
  // with a hole of the batch is in that hole's list)
  const int* ofs = p.b_ofs + (size_t)slot * (nbat + 2);
  const size_t eb = (size_t)slot * (size_t)p.ent_cap;
  ulonglong2 en0 = make_ulonglong2(0ull, 0ull);  // this thread's entry of the first round
  uint32_t rec0 = 0;
  {
    const int ob = ofs[b], nb_ = ofs[b + 1] - ob, oa = ofs[nbat], na_ = ofs[nbat + 1] - oa;
    const int o1 = (B.h == 2) ? ofs[B.ia] : 0, n1_ = (B.h == 2) ? ofs[B.ia + 1] - o1 : 0;
    const int o2 = (B.h == 2) ? ofs[B.ib] : 0, n2_ = (B.h == 2) ? ofs[B.ib + 1] - o2 : 0;
    const int s1 = nb_, s2 = s1 + n1_, s3 = s2 + n2_, s4 = s3 + na_;
    if (tid < s4) {
      const int o = tid < s1 ? ob + tid : (tid < s2 ? o1 + tid - s1 : (tid < s3 ? o2 + tid - s2 : oa + tid - s3));
      en0 = p.e_hp[eb + o];
      rec0 = p.e_rec[eb + o];
    }
    if (tid == 0) {
      S.seg_o[0] = ob;
      S.seg_o[1] = o1 - s1;
      S.seg_o[2] = o2 - s2;
      S.seg_o[3] = oa - s3;
      S.seg_s[0] = s1;
      S.seg_s[1] = s2;
      S.seg_s[2] = s3;
      S.seg_s[3] = s4;
      const size_t rb = (size_t)slot * (size_t)p.ndet;
      S.rw = p.r_words + rb * NW;
      S.rc = p.r_coef + rb;
      S.rhm = p.r_hmask + rb;
      S.rpt = p.r_part + rb;
      S.ehp = p.e_hp + eb;
      S.erec = p.e_rec + eb;
    }
  }
  unsigned long long gtau = 0;
  if (p.k > 0 && tid == 0) gtau = *((volatile unsigned long long*)p.tau_bits);
  // position of the i-th entry of this batch in the slot's entry arrays
  auto entry = [&](int i) {
    return i + S.seg_o[i < S.seg_s[0] ? 0 : i < S.seg_s[1] ? 1 : i < S.seg_s[2] ? 2 : 3];
  };
  auto dup = [&](int i, uint64_t hm) {
    return i >= S.seg_s[0] && (i < S.seg_s[2] ? (hm & B.hm) == B.hm : (hm & B.hm) != 0ull);
  };
  B.ca = M->occ[B.ia];
  B.qa = B.ca - B.sa * norb;
  B.cb = B.h == 2 ? M->occ[B.ib] : -1;
  B.qb = B.h == 2 ? B.cb - B.sb * norb : -1;
  const int ibase = B.h == 2 ? (B.qa * norb + B.qb) * norb * norb : 0;
#pragma unroll 1
  for (int x = tid; x < 2 * norb; x += kThreads) {  // a thread per orbital and spin
    const int s = x >= norb, q = x - s * norb;
    uint64_t sw[NINT];
    int below = 0;  // occupied orbitals of spin s below q
#pragma unroll
    for (int w = 0; w < NINT; w++) {
      sw[w] = M->I[s * NINT + w];
      const int lim = q - 64 * w;
      if (lim >= 64) below += __popcll(sw[w]);
      else if (lim > 0) below += __popcll(sw[w] & ((1ull << lim) - 1));
    }
    if (mask_bit<NINT>(sw, q)) {
      S.vidx[s][q] = 255;
      continue;
    }
    const int v = q - below;
    S.vidx[s][q] = (unsigned char)v;
    S.vir[s][v] = (unsigned char)q;
    auto W = [&](int y, int sy) { return (s == sy ? p.Wi : p.Ji)[q * norb + y]; };
    const bool isrow = s == B.sa, iscol = B.h == 2 && s == B.sb;
    if (isrow || iscol) {
      long long u = M->F[s][q] - W(B.qa, B.sa);
      if (B.h == 2) u -= W(B.qb, B.sb);
      if (isrow) {  // E0 - base - u0, base = H_II - F(a) [- F(b) + W(a, b)]
        long long base = M->hii - M->F[B.sa][B.qa];
        if (B.h == 2) base += (B.kind == 1 ? p.Wi : p.Ji)[B.qa * norb + B.qb] - M->F[B.sb][B.qb];
        int idx = 0;  // pair tables of J = I: its particles x1, x2 are the holes a, b
        if (B.h == 2) {
          const int par = count_between<NINT>(sw, q < B.qa ? q : B.qa, q < B.qa ? B.qa : q) & 1;
          idx = (E4 ? ibase + q * norb : tri(B.qa, q)) | (par << 31);
        }
        S.row[v].d = (E.e0 - base) - u;
        S.row[v].idx = idx;
        S.row[v].orb = q;
        // spin-up words: of the row's cells (opposite-spin batch), or I's
        uint64_t hk = 0;
#pragma unroll
        for (int w = 0; w < NINT; w++) {
          uint64_t up = s == 0 ? sw[w] : M->I[w];
          if (s == 0 && (B.qa >> 6) == w) up &= ~(1ull << (B.qa & 63));
          if (s == 0 && (q >> 6) == w) up |= 1ull << (q & 63);
          hk = splitmix64(hk ^ up);
        }
        S.hk0[v] = hk;
      }
      if (iscol) {
        const int lo = q < B.qb ? q : B.qb, hi = q < B.qb ? B.qb : q;
        int par = count_between<NINT>(sw, lo, hi) & 1;
        if (B.kind == 1) par ^= (B.qa > lo && B.qa < hi) ? 1 : 0;
        S.col[v].d = u;
        S.col[v].idx = (E4 ? q : tri(B.qb, q)) | (par << 31);
        S.col[v].orb = q;
      }
    }
  }
  if (tid < nel) S.occ[tid] = M->occ[tid];
  if (lane == 0) S.red_con[warp] = 0ull;
  if (tid == 0) {
    S.bt = B;
    S.cI = (NT)M->cI;
    S.n0 = S.n1 = S.n2 = S.cnext = 0;
#pragma unroll
    for (int w = 0; w < NW; w++) S.kbase[w] = M->I[w];
    S.kbase[B.sa * NINT + (B.qa >> 6)] &= ~(1ull << (B.qa & 63));
    if (B.h == 2) S.kbase[B.sb * NINT + (B.qb >> 6)] &= ~(1ull << (B.qb & 63));
  }
  if constexpr (MS) {
    if (tid < nst) {
      ms_cI[tid] = p.coefs[(size_t)tid * p.ndet + p.order[M->g]];
      const double m = __longlong_as_double((long long)p.st_cmax[tid]);
      ms_w[tid] = 1.0 / (m * m);
      ms_de[tid] = den_fix(p.st_e0[tid], E.dscale) - E.e0;
    }
    for (int st = 0; st < nst; st++)
#pragma unroll 1
      for (int c = tid; c < B.nct; c += kThreads) A[st * mc + c] = 0.0;
  } else {
#pragma unroll 1
    for (int c = tid; c < B.nct; c += kThreads) A0[c] = A1[c] = A2[c] = 0u;
  }
  // bans by J ranked before I: the masks of the slot and the batch's holes
  const uint64_t* om = p.o_mask + (size_t)slot * p.orb_w;
  if (B.h == 2) {
    const MaskDims md = mask_dims(norb, p.nalpha, p.nbeta);
    const uint32_t* gm = p.b_mask + (size_t)slot * p.mask_w;
    const int mbase = md.ca + md.cb + md.cm, mix = md.ca > md.cb ? md.ca : md.cb;
    const uint32_t* m0 = gm + (B.kind == 2 ? md.ca + md.cb : B.sa ? md.ca : 0);
    const uint32_t* m1 = gm + mbase + B.ia * md.hs + (B.kind == 2 ? mix : 0);
    const uint32_t* m2 = gm + mbase + B.ib * md.hs + (B.kind == 2 ? mix : 0);
    const int nw32 = (B.ncell + 31) / 32;
    auto word = [&](int w) { return w < nw32 ? m0[w] | m1[w] | m2[w] : 0u; };
#pragma unroll 1
    for (int w = tid; w < (B.nct + 31) / 32; w += kThreads) {
      const int at = (B.clo >> 5) + w;
      ban[w] = __funnelshift_r(word(at), (B.clo & 31) ? word(at + 1) : 0u, B.clo & 31);
    }
    if (tid < NW) S.rowban[tid] = om[tid] | om[(4 + 3 * B.ia) * NINT + tid] | om[(4 + 3 * B.ib) * NINT + tid];
  }
  __syncthreads();
  if constexpr (FP) den64_sides<NINT, NT>(p, S, B, M, MS ? p.st_e0[0] : p.e0);
  if (B.h == 1) {
    const uint64_t *b1 = om + (2 + B.sa) * NINT, *h1 = om + (6 + 3 * B.ia) * NINT;
#pragma unroll 1
    for (int c0 = 0; c0 < B.nct; c0 += kThreads) {
      const int c = c0 + tid, r = c < B.nct ? S.vir[B.sa][c] : 0;
      const unsigned f = __ballot_sync(kFull, c < B.nct && (((b1[r >> 6] | h1[r >> 6]) >> (r & 63)) & 1ull));
      if (lane == 0 && c < B.nct) ban[c >> 5] = f;
    }
    __syncthreads();
  }
  if (p.tgt_on) {  // cells outside the target space contribute nothing: ban them
#pragma unroll 1
    for (int cc = tid; cc < B.nct; cc += kThreads) {
      int ro, so, x, y;
      cell_orbitals<NINT, NT>(B, S, B.clo + cc, &ro, &so, &x, &y);
      const int kwr = B.sa * NINT + (ro >> 6), kws = (B.h == 2) ? B.sb * NINT + (so >> 6) : -1;
      bool ok = true;
      int moved = 0;
#pragma unroll
      for (int w = 0; w < NW; w++) {
        const uint64_t k = S.kbase[w] | (w == kwr ? 1ull << (ro & 63) : 0ull) | (w == kws ? 1ull << (so & 63) : 0ull);
        ok &= (k & p.tgt_core[w]) == p.tgt_core[w];
        ok &= (k & p.tgt_del[w]) == 0ull;
        moved += __popcll(k ^ p.tgt_ref[w]);
      }
      if (p.tgt_max_exc >= 0) ok &= (moved >> 1) <= p.tgt_max_exc;
      if (!ok) atomicOr(&ban[cc >> 5], 1u << (cc & 31));
    }
  }
  // ---- loop 1: bans by the entries of the batch's own bucket.  J ranked
  // before I: rows (t = 1) and cells (t = 2); a later J equal to a cell's
  // alpha bans that cell ----
#pragma unroll 1
  for (int i = tid; i < S.seg_s[0]; i += kThreads) {
    const ulonglong2 en = i < kThreads ? en0 : S.ehp[S.seg_o[0] + i];
    const uint64_t hm = en.x, part = en.y;
    if ((part & kBeforeBit) && __popcll(hm) == 3) {
#pragma unroll
      for (int k = 0; k < 3; k++) {
        const int c = part_code(part, k), s = c >= norb, q = c - s * norb;
        if (B.kind == 2 || s == B.sa)
          atomicOr(reinterpret_cast<unsigned long long*>(&S.rowban[s * NINT + (q >> 6)]), 1ull << (q & 63));
      }
    } else if ((part & kBeforeBit) || hm == B.hm) {
      for_subset_cells<NINT, NT>(B, S, norb, part, [&](int c) { ban_cell(ban, B, c); });
    }
  }
  if (gtau > S.tau) S.tau = gtau;  // thread 0
  const int tkcnt = S.tkcnt;       // unchanged until the last pass over the cells
  __syncthreads();
  if (B.h == 2) {  // flagged rows and columns as cell bans: a row per thread, 32 cells at a time
    const int scol = B.kind == 2 ? 1 : B.sa, srow = B.kind == 2 ? 0 : B.sa, nvc = S.nv[scol];
    const int x0 = B.kind == 2 ? B.clo / nvc : 0, x1 = B.kind == 2 ? x0 + B.nct / nvc : nvc;
#pragma unroll 1
    for (int y = 0; y < nvc; y += 32) {
      const unsigned fw =
          __ballot_sync(kFull, y + lane < nvc && row_banned<NINT, NT>(S, scol, S.vir[scol][(y + lane) & (kMaxOrb - 1)]));
#pragma unroll 1
      for (int x = x0 + tid; x < x1; x += kThreads) {
        const int len = B.kind == 2 ? nvc : x;  // same spin: the cells (y, x), y < x
        if (y >= len) continue;
        uint32_t pat = row_banned<NINT, NT>(S, srow, S.vir[srow][x]) ? ~0u : fw;
        if (len - y < 32) pat &= (1u << (len - y)) - 1u;
        if (!pat) continue;
        const int pos = (B.kind == 2 ? (x - x0) * nvc : x * (x - 1) / 2) + y;
        atomicOr(&ban[pos >> 5], pat << (pos & 31));
        if ((pos & 31) && (pat >> (32 - (pos & 31)))) atomicOr(&ban[(pos >> 5) + 1], pat >> (32 - (pos & 31)));
      }
      __syncwarp();
    }
  }

  // Pair table of a J reaching every cell (a two-hole batch; a warp).
  // J = K + {x1, x2}, x1 < x2; for a cell R disjoint from {x1, x2} the element
  // is the double substitution x1 x2 -> R, whose integrals and phase split
  // into a row and a column part.  The cells holding a particle of J (bit 30)
  // are single substitutions and go with the rows.
  auto build_table = [&](int j, int r) {
    uint32_t xs, ts;
    int nxs, nts;
    excitation_sets<NINT, NT>(B, S, S.rpt[r], S.rhm[r], &xs, &nxs, &ts, &nts);
    const int a = pk(xs, 0), bb = pk(xs, 1);
    const int sr = B.sa, sc = B.kind == 2 ? 1 : B.sa;
    const int x1 = (a < bb ? a : bb) - sr * norb, x2 = (a < bb ? bb : a) - sc * norb;
    const int gB = (x1 * norb + x2) * norb * norb;
    if (lane == 0) {
      S.gcj[j] = (NT)S.rc[r];
      S.gx1[j] = x1;
      S.gx2[j] = x2;
      S.gB[j] = gB;
      if constexpr (MS)
        for (int st = 0; st < nst; st++) ms_gc[j * kMaxStates + st] = S.rc[st * p.rc_stride + r];
    }
    uint64_t w1[NINT], w2[NINT], M1[NINT], M2[NINT];
#pragma unroll
    for (int w = 0; w < NINT; w++) {
      w1[w] = S.rw[(size_t)r * NW + sr * NINT + w];
      w2[w] = S.rw[(size_t)r * NW + sc * NINT + w];
      if (B.kind == 1 && (x1 >> 6) == w) w2[w] &= ~(1ull << (x1 & 63));
    }
    phase_mask<NINT>(w1, x1, 0, M1);
    phase_mask<NINT>(w2, x2, 0, M2);
#pragma unroll 1
    for (int v = lane; v < S.nv[sr]; v += 32) {
      const int q = S.vir[sr][v];
      const int ex = q == x1 || (B.kind == 1 && q == x2) ? 1 << 30 : 0;
      S.gRow[j][v] = (E4 ? gB + q * norb : tri(x1, q)) | ex | ((int)mask_bit<NINT>(M1, q) << 31);
    }
#pragma unroll 1
    for (int v = lane; v < S.nv[sc]; v += 32) {
      const int q = S.vir[sc][v];
      const int ex = q == x2 || (B.kind == 1 && q == x1) ? 1 << 29 : 0;
      S.gCol[j][v] = (E4 ? q : tri(x2, q)) | ex | ((int)mask_bit<NINT>(M2, q) << 31);
    }
  };

  // the gradient's weight 2 A/D of a cell (in place of its accumulator)
  auto a2d = [&](int cc) {
    return __longlong_as_double((long long)(A0[cc] | ((unsigned long long)A1[cc] << 32)));
  };
  (void)a2d;

  // ---- loop 2: A(R) += c_J <J|H|I - H + R> over J ranked at or after I.
  // In the one-state form every term goes into the exact accumulator, so
  // the order in which J are listed and cells are reached does not matter ----
  unsigned int con = 0;  // of a round (at most 512 entries); summed per warp after each
  auto add_con = [&]() {
    const unsigned int wcon = __reduce_add_sync(kFull, con);
    if (lane == 0) S.red_con[warp] += wcon;
    con = 0;
  };
  // The J of a round but for the tables' terms, drawn by the warps as they free
  // up (G: the gradient's scatter of the same terms): the rows of J
  // reaching every cell (a two-hole batch: the cells touching their
  // particles; a one-hole batch: all cells), J reaching rows, and J reaching
  // a few cells (one lane each, 32 per draw).
  //
  // Along a row everything but the cell's orbital z is fixed: the element of
  // a double substitution is one or two integrals at base + z (consecutive
  // lanes on consecutive entries) with a sign from a phase mask of J's
  // string.  A warp draws up to eight row J and sets up their rows side by
  // side, a lane per (J, particle).  The few cells holding two particles of
  // such a J (one, in a one-hole batch) are single substitutions of J; their
  // sum over J's orbitals is spread over the lanes.  A row of a J reaching
  // every cell holds single substitutions only: a unit of work is 32 of its
  // cells, each lane summing over J's orbitals, four at a time in flight.
  // (Each cell through the general element routine, a warp per J, took 8,000
  // cycles of a warp per J: two masked popcounts per cell, and a lane's chain
  // of 30 dependent loads wherever a row met a single substitution.)
  auto row_pass = [&](auto gp) {
    constexpr bool G = decltype(gp)::value;
    const int n0 = S.n0, nrow = S.n1, n2 = S.n2;
    const int ntab = B.h == 2 ? (n0 < kGroup ? n0 : kGroup) : 0;
    const int nvm = S.nv[0] > S.nv[1] ? S.nv[0] : S.nv[1], nch = (nvm + 31) / 32;
    // units: pair tables, rows of the J reaching every cell (J, particle slot,
    // 32 cells), row J, the rest
    const int nall = ntab + n0 * B.h * nch;
    int per = (nrow + kWarps - 1) / kWarps;
    per = per > 8 ? 8 : per;
    const int ndraw = nall + (per ? (nrow + per - 1) / per : 0);
    // c_J v into cell cc
    auto add = [&](int cc, NT v, int rj, NT cjj) {
      if constexpr (MS) {
#pragma unroll
        for (int st = 0; st < kMaxStates; st++)
          if (st < nst) atomicAdd(&A[st * mc + cc], S.rc[st * p.rc_stride + rj] * (double)v);
      } else {
        unsigned long long l;
        int hh;
        fix_of(cjj * v, F, l, hh);
        fix_atomic_add(A0, A1, A2, cc, l, hh);
      }
      con++;
    };
    auto live = [&](int cc) { return (unsigned)cc < (unsigned)B.nct && !((ban[cc >> 5] >> (cc & 31)) & 1u); };
    for (;;) {
      int jd = 0;
      if (lane == 0) jd = atomicAdd(&S.cnext, 1);
      jd = __shfl_sync(kFull, jd, 0);
      if (jd < ntab) {
        build_table(jd, S.u.l.L0[jd]);
      } else if (jd < nall) {
        const int ju = jd - ntab, j = ju / (B.h * nch), rem = ju - j * (B.h * nch), ip = rem / nch, y = (rem - ip * nch) * 32 + lane;
        const int r = S.u.l.L0[j];
        const uint64_t hm = S.rhm[r], part = S.rpt[r];
        uint32_t X, T;
        int nx, nt;
        excitation_sets<NINT, NT>(B, S, part, hm, &X, &nx, &T, &nt);
        // row of particle ip; the hole u of the substitutions u -> z is the
        // other entry of X (one-hole batch: the only entry)
        const int code = B.h == 2 ? part_code(part, ip) : -1;
        if (code == kNoPart) continue;
        const int s = code >= norb, x = code >= 0 ? S.vidx[s][code - s * norb] : 0;
        if (B.kind == 1 && s != B.sa) continue;
        const int sz = B.kind == 2 ? 1 - s : B.sa;
        if (B.h == 2 && row_banned<NINT, NT>(S, s, code - s * norb)) continue;
        const int x0 = pk(X, 0), uz = (x0 == code ? pk(X, 1) : x0) - sz * norb;
        uint64_t wz[NINT], M[NINT];
#pragma unroll
        for (int w = 0; w < NINT; w++) wz[w] = S.rw[(size_t)r * NW + sz * NINT + w];
        phase_mask<NINT>(wz, uz, 0, M);
        if (y >= S.nv[sz]) continue;
        const int z = S.vir[sz][y];
        const int cc = (B.kind == 0 ? y : B.kind == 1 ? pair_cell(x, y) : (s ? y * S.nv[1] + x : x * S.nv[1] + y)) - B.clo;
        // z a particle of J: that cell is J itself (banned)
        if (mask_bit<NINT>(wz, z) || (B.kind == 1 && x == y) || !live(cc)) continue;
        if constexpr (G) {
          const double ws = flip_sign(S.rc[r] * a2d(cc), mask_bit<NINT>(M, z));
          atomicAdd(&p.g_dh[uz * norb + z], 0.5 * ws);
          atomicAdd(&p.g_dh[z * norb + uz], 0.5 * ws);
#pragma unroll 1
          for (int w = 0; w < NW; w++) {
            const bool sp = w / NINT == sz;
#pragma unroll 1
            for (uint64_t bits = S.rw[(size_t)r * NW + w]; bits; bits &= bits - 1) {
              const int o = 64 * (w % NINT) + __ffsll((long long)bits) - 1;
              atomicAdd(&p.g_deri[eri_index(o, o, uz, z)], ws);
              if (sp) atomicAdd(&p.g_deri[eri_index(uz, o, o, z)], -ws);
            }
          }
          continue;
        }
        NT v = h_n[uz * norb + z];
        // J's orbitals in ascending order (the FP32 form's sum depends on
        // it), four at a time so that their loads overlap
#pragma unroll 1
        for (int w = 0; w < NW; w++) {
          uint64_t bits = S.rw[(size_t)r * NW + w];
          const bool sp = w / NINT == sz;
#pragma unroll 1
          while (bits) {
            int o[4];
            NT a[4], b[4];
#pragma unroll
            for (int i = 0; i < 4; i++) {
              o[i] = bits ? 64 * (w % NINT) + __ffsll((long long)bits) - 1 : -1;
              bits &= bits - 1;
              if (o[i] < 0) continue;
              a[i] = eri_n[gidx<E4>(o[i], o[i], uz, z, norb)];
              if (sp) b[i] = eri_n[gidx<E4>(uz, o[i], o[i], z, norb)];
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
              if (o[i] < 0) continue;
              v += a[i];
              if (sp) v -= b[i];
            }
          }
        }
        add(cc, flip_sign(v, mask_bit<NINT>(M, z)), r, (NT)S.rc[r]);
      } else if (jd < ndraw) {
        const int jl = (jd - nall) * per + (lane >> 2), ip = lane & 3;
        const bool have = (lane >> 2) < per && jl < nrow;
        int r = 0;
        NT cj = NT(0);
        uint64_t part = 0x7FFF7FFF7FFF7FFFull, hm = 0;
        uint64_t M[NINT];         // phase of the row's substitution by z
        uint64_t EX[NINT];        // particles of J with the spin of z
        // orbitals: uz (hole paired with z) | uo (hole paired with q) << 8 |
        // q << 16 | same spin << 24
        uint32_t iw = 0;
        int geo = 0;              // virtual index of the row's particle, its spin << 8
        bool act = false;
        // the single substitution of the pair of particles ip: cell and
        // sign << 31, hole w | q << 8 | spin << 16
        bool sact = false;
        uint32_t scell = 0, sw = 0;
#pragma unroll
        for (int w = 0; w < NINT; w++) M[w] = EX[w] = 0;
        if (have) {
          r = S.u.l.L12[jl];
          part = S.rpt[r];
          hm = S.rhm[r];
          cj = (NT)S.rc[r];
          uint32_t X, T;
          int nx, nt;
          excitation_sets<NINT, NT>(B, S, part, hm, &X, &nx, &T, &nt);
          const int q = pk(T, 0), sq = q >= norb ? 1 : 0, qo = q - sq * norb;
          uint64_t Jw[NW];
#pragma unroll
          for (int w = 0; w < NW; w++) Jw[w] = S.rw[(size_t)r * NW + w];
          // the row's particle (a one-hole batch has one row per J and no
          // fixed particle)
          const int code = B.h == 2 ? part_code(part, ip) : (ip == 0 ? -1 : kNoPart);
          if (code != kNoPart) {
            const int s = code >= norb, x = code >= 0 ? S.vidx[s][code - s * norb] : 0;
            const int sz = B.kind == 2 ? 1 - s : B.sa;
            act = B.h == 1 || ((B.kind == 2 || s == B.sa) && !row_banned<NINT, NT>(S, s, code - s * norb));
            geo = x | (s << 8);
            int u0 = -1, u1 = -1;  // X without the row's particle
#pragma unroll
            for (int i = 0; i < 3; i++) {
              if (i >= nx) break;
              const int xc = pk(X, i);
              if (xc != code) {
                if (u0 < 0) u0 = xc;
                else u1 = xc;
              }
            }
            const bool same = (u0 >= norb) == (u1 >= norb);
            const bool second = same || (u1 >= norb) == (sz != 0);
            const int uz = second ? u1 : u0, uo = second ? u0 : u1;
            const int so = uo >= norb, zo = uz - sz * norb, oo = uo - so * norb;
            uint64_t wo[NINT], wz[NINT];
#pragma unroll
            for (int w = 0; w < NINT; w++) {
              wo[w] = so ? Jw[NINT + w] : Jw[w];
              wz[w] = sz ? Jw[NINT + w] : Jw[w];
              if (same) {
                if ((oo >> 6) == w) wz[w] &= ~(1ull << (oo & 63));
                if ((qo >> 6) == w) wz[w] |= 1ull << (qo & 63);
              }
            }
            const int c = count_between<NINT>(wo, oo < qo ? oo : qo, oo < qo ? qo : oo) & 1;
            phase_mask<NINT>(wz, zo, c, M);
            iw = (uint32_t)zo | ((uint32_t)oo << 8) | ((uint32_t)qo << 16) | ((uint32_t)same << 24);
#pragma unroll
            for (int i = 0; i < 4; i++) {
              const int pc = part_code(part, i);
              if (pc == kNoPart || (pc >= norb) != (sz != 0)) continue;
              const int po = pc - sz * norb;
#pragma unroll
              for (int w = 0; w < NINT; w++)
                if ((po >> 6) == w) EX[w] |= 1ull << (po & 63);
            }
          }
          if (ip < 3) {  // two-hole batch: pairs (0, 1), (0, 2), (1, 2) of J's particles; one-hole: its particles
            const int c0_ = part_code(part, B.h == 2 && ip == 2 ? 1 : (B.h == 2 ? 0 : ip));
            const int c1_ = B.h == 2 ? part_code(part, ip == 0 ? 1 : 2) : -1;
            if (c0_ != kNoPart && c1_ != kNoPart) {
              const int sx = c0_ >= norb, sy = c1_ >= norb;
              if (B.kind == 2 ? sx != sy : (sx == B.sa && (c1_ < 0 || sy == B.sa))) {
                const int vx = S.vidx[sx][c0_ - sx * norb], vy = c1_ < 0 ? 0 : S.vidx[sy][c1_ - sy * norb];
                const int cc = (B.kind == 0 ? vx : B.kind == 1 ? pair_cell(vx, vy) : (sx ? vy * S.nv[1] + vx : vx * S.nv[1] + vy)) - B.clo;
                if (live(cc)) {
                  int w = 0;  // X without the cell's particles: the hole, with q's spin
#pragma unroll
                  for (int i = 0; i < 3; i++) {
                    const int xc = pk(X, i);
                    if (i < nx && xc != c0_ && xc != c1_) w = xc;
                  }
                  const int wo = w - sq * norb;
                  uint64_t ws[NINT];
#pragma unroll
                  for (int i = 0; i < NINT; i++) ws[i] = sq ? Jw[NINT + i] : Jw[i];
                  const int neg = count_between<NINT>(ws, wo < qo ? wo : qo, wo < qo ? qo : wo) & 1;
                  sact = true;
                  scell = (uint32_t)cc | ((uint32_t)neg << 31);
                  sw = (uint32_t)wo | ((uint32_t)qo << 8) | ((uint32_t)sq << 16);
                }
              }
            }
          }
        }
#pragma unroll 1
        for (unsigned m = __ballot_sync(kFull, act); m; m &= m - 1) {
          const int src = __ffs((int)m) - 1;
          const uint32_t iwr = __shfl_sync(kFull, iw, src);
          const int gr = __shfl_sync(kFull, geo, src), rj = __shfl_sync(kFull, r, src);
          const NT cjr = __shfl_sync(kFull, cj, src);
          uint64_t Mr[NINT], Er[NINT];
          shfl_words<NINT>(M, src, Mr);
          shfl_words<NINT>(EX, src, Er);
          const int x = gr & 0xFF, s = gr >> 8, sz = B.kind == 2 ? 1 - s : B.sa;
          const int uz = iwr & 0xFF, uo = (iwr >> 8) & 0xFF, q = (iwr >> 16) & 0xFF;
          const bool same = (iwr >> 24) & 1u;
          const int nz = S.nv[sz], nv1 = S.nv[1];
          // the integrals at b1 + z and (same spin) b2 + z
          const NT* e1 = eri_n + ((uo * norb + uz) * norb + q) * norb;
          const NT* e2 = eri_n + ((uz * norb + uo) * norb + q) * norb;
          // cell of z's index y: cb + y cs, or (same spin) a pair
          const int cs = B.kind == 2 && s ? nv1 : 1;
          const int cb = (B.kind == 2 ? (s ? x : x * nv1) : 0) - B.clo, xx = x * (x - 1) / 2;
          if constexpr (G) {
#pragma unroll 1
            for (int y = lane; y < nz; y += 32) {
              const int z = S.vir[sz][y];
              const int cc = B.kind == 1 ? cb + (y > x ? y * (y - 1) / 2 + x : xx + y) : cb + y * cs;
              if (mask_bit<NINT>(Er, z) || !live(cc)) continue;
              const double ws = flip_sign(cjr * a2d(cc), mask_bit<NINT>(Mr, z));
              atomicAdd(&p.g_deri[eri_index(uo, q, uz, z)], ws);
              if (same) atomicAdd(&p.g_deri[eri_index(uz, q, uo, z)], -ws);
            }
            continue;
          }
          // two rounds of 32 cells at a time, their loads in flight together
#pragma unroll 1
          for (int y0 = lane; y0 < nz; y0 += 64) {
            int ca = -1, cn = -1;
            NT va = NT(0), vn = NT(0);
            auto fetch = [&](int y, int& c, NT& v) {
              if (y >= nz) return;
              const int z = S.vir[sz][y];
              int cc = cb + y * cs;
              if (B.kind == 1) cc = cb + (y > x ? y * (y - 1) / 2 + x : xx + y);
              if (mask_bit<NINT>(Er, z) || !live(cc)) return;
              c = cc;
              if constexpr (E4) {
                v = e1[z];
                if (same) v -= e2[z];
              } else {
                v = eri_n[eri_index(uo, q, uz, z)];
                if (same) v -= eri_n[eri_index(uz, q, uo, z)];
              }
              v = flip_sign(v, mask_bit<NINT>(Mr, z));
            };
            fetch(y0, ca, va);
            fetch(y0 + 32, cn, vn);
#pragma unroll 1
            for (int i = 0; i < 2; i++) {
              if (ca >= 0) add(ca, va, rj, cjr);
              ca = cn;
              va = vn;
            }
          }
        }
#pragma unroll 1
        for (unsigned m = __ballot_sync(kFull, sact); m; m &= m - 1) {
          const int src = __ffs((int)m) - 1;
          const uint32_t sc = __shfl_sync(kFull, scell, src), wq = __shfl_sync(kFull, sw, src);
          const int rj = __shfl_sync(kFull, r, src);
          const NT cjr = __shfl_sync(kFull, cj, src);
          const uint64_t hmr = __shfl_sync(kFull, hm, src), ptr_ = __shfl_sync(kFull, part, src);
          const int wo = wq & 0xFF, qo = (wq >> 8) & 0xFF, sq = (wq >> 16) & 1;
          if constexpr (G) {
            const double ws = flip_sign(cjr * a2d((int)(sc & 0x7fffffffu)), (sc >> 31) != 0u);
            if (lane < 2) atomicAdd(&p.g_dh[lane ? qo * norb + wo : wo * norb + qo], 0.5 * ws);
#pragma unroll 1
            for (int i = lane; i < nel; i += 32) {
              int mo = S.occ[i];
              if ((hmr >> i) & 1ull) mo = part_code(ptr_, __popcll(hmr & ((1ull << i) - 1)));
              const int sm = mo >= norb, o = mo - sm * norb;
              atomicAdd(&p.g_deri[eri_index(o, o, wo, qo)], ws);
              if (sm == sq) atomicAdd(&p.g_deri[eri_index(wo, o, o, qo)], -ws);
            }
            continue;
          }
          NT v = NT(0);
          if constexpr (sizeof(NT) == 8) {  // J's orbitals: I's, with particles in the place of its holes
#pragma unroll 1
            for (int i = lane; i < nel; i += 32) {
              int mo = S.occ[i];
              if ((hmr >> i) & 1ull) mo = part_code(ptr_, __popcll(hmr & ((1ull << i) - 1)));
              const int sm = mo >= norb, o = mo - sm * norb;
              v += eri_n[gidx<E4>(o, o, wo, qo, norb)];
              if (sm == sq) v -= eri_n[gidx<E4>(wo, o, o, qo, norb)];
            }
            v = warp_sum_nt<NT>(v) + h_n[wo * norb + qo];
          } else {
            // FP32: the sum keeps the ascending order of J's orbitals (its
            // rounding depends on it); the lanes load, one adds
            v = h_n[wo * norb + qo];
#pragma unroll
            for (int w = 0; w < 2 * NW; w++) {
              const int o = 32 * (w % (2 * NINT)) + lane;
              const bool sp = w / (2 * NINT) == sq;
              uint32_t bits = (uint32_t)(S.rw[(size_t)rj * NW + w / 2] >> (32 * (w & 1)));
              NT a = NT(0), b = NT(0);
              if ((bits >> lane) & 1u) {
                a = eri_n[gidx<E4>(o, o, wo, qo, norb)];
                if (sp) b = eri_n[gidx<E4>(wo, o, o, qo, norb)];
              }
              for (; bits; bits &= bits - 1) {
                const int src2 = __ffs((int)bits) - 1;
                v += __shfl_sync(kFull, a, src2);
                const NT bb = __shfl_sync(kFull, b, src2);
                if (sp) v -= bb;
              }
            }
          }
          if (lane == 0) add((int)(sc & 0x7fffffffu), flip_sign(v, (sc >> 31) != 0u), rj, cjr);
        }
      } else {
        const int j0 = (jd - ndraw) * 32;
        if (j0 >= n2) break;
        const int j = j0 + lane;
        if (j < n2) {
          // cells inside J's particles: J -> alpha moves the other two
          // entries of X to J's two holes outside the batch
          const int r = S.u.l.L12[kChunk - 1 - j];
          const uint64_t part = S.rpt[r];
          uint32_t X, T;
          int nx, nt;
          excitation_sets<NINT, NT>(B, S, part, S.rhm[r], &X, &nx, &T, &nt);
          const NT cj = (NT)S.rc[r];
          uint64_t Jw[NW];
#pragma unroll
          for (int w = 0; w < NW; w++) Jw[w] = S.rw[(size_t)r * NW + w];
#pragma unroll 1
          for (int k = 0; k < (B.h == 2 ? 6 : 4); k++) {
            // pairs (0, 1), (0, 2), (1, 2), (0, 3), (1, 3), (2, 3); one-hole batch: single particles
            const int k1 = B.h == 1 ? k : (k >= 3 ? 3 : k >= 1 ? 2 : 1), k0 = B.h == 1 ? k : (k >= 3 ? k - 3 : k >= 1 ? k - 1 : 0);
            const int e0 = part_code(part, k0), e1 = part_code(part, k1);
            if (e0 == kNoPart || e1 == kNoPart) continue;
            const int sx = e0 >= norb, sy = e1 >= norb;
            if (B.kind == 2 ? sx == sy : (sx != B.sa || sy != B.sa)) continue;
            const int vx = S.vidx[sx][e0 - sx * norb], vy = S.vidx[sy][e1 - sy * norb];
            const int cc = (B.kind == 0 ? vx : B.kind == 1 ? pair_cell(vx, vy) : (sx ? vy * S.nv[1] + vx : vx * S.nv[1] + vy)) - B.clo;
            if (!live(cc)) continue;
            if constexpr (G) {
              element_grad<NINT>(p.g_dh, p.g_deri, norb, Jw, X, nx, T, nt, e0, B.h == 2 ? e1 : -1, S.rc[r] * a2d(cc));
              continue;
            }
            int u0 = -1, u1 = -1;
#pragma unroll
            for (int i = 0; i < 4; i++) {
              const int xc = pk(X, i);
              if (i < nx && xc != e0 && xc != e1) {
                if (u0 < 0) u0 = xc;
                else u1 = xc;
              }
            }
            const NT v = double_element<NINT, NT, E4>(eri_n, norb, Jw, u0 < u1 ? u0 : u1, u0 < u1 ? u1 : u0, pk(T, 0), pk(T, 1));
            if constexpr (MS) {
#pragma unroll
              for (int st = 0; st < kMaxStates; st++)
                if (st < nst) atomicAdd(&A[st * mc + cc], S.rc[st * p.rc_stride + r] * (double)v);
            } else {
              unsigned long long l;
              int hh;
              fix_of(cj * v, F, l, hh);
              fix_atomic_add(A0, A1, A2, cc, l, hh);
            }
            con++;
          }
        }
      }
    }
  };

#pragma unroll 1
  for (int c0 = 0;; c0 += kChunk) {
    const int total = S.seg_s[3], c1 = min(c0 + kChunk, total);
    const bool last_round = c0 + kChunk >= total;
#pragma unroll 1
    for (int i = c0 + tid; i < c1; i += kThreads) {
      const int o = entry(i);
      const ulonglong2 en = i < kThreads ? en0 : S.ehp[o];
      const uint64_t hmr = en.x, part = en.y;
      if (part & kBeforeBit) continue;
      if (dup(i, hmr)) continue;
      if (B.h == 2 && hmr == 0ull) continue;  // J = I: added in the cells pass
      const int t = __popcll(hmr & ~B.hm);
      if (t > 2) continue;
      const int rec = (int)((i < kThreads ? rec0 : S.erec[o]) & 0x7FFFFFFFu);
      if (t == 0) S.u.l.L0[atomicAdd(&S.n0, 1)] = rec;
      else if (t == 1) {
        if (B.h == 1 || row_live<NINT, NT>(B, S, norb, part)) S.u.l.L12[atomicAdd(&S.n1, 1)] = rec;
      }
      else if (subset_live<NINT, NT>(B, S, norb, part, ban)) S.u.l.L12[kChunk - 1 - atomicAdd(&S.n2, 1)] = rec;
    }
    __syncthreads();
    const int n0 = S.n0;
    B = S.bt;
    if (!MS && c0 == 0) {
      // the list of the cells left, in cell order: every warp scans the ban
      // words, 32 at a time, and writes the cells of every eighth of them
      int base = 0;
#pragma unroll 1
      for (int w0 = 0; 32 * w0 < B.nct; w0 += 32) {
        const int n = B.nct - 32 * (w0 + lane);
        const unsigned left = n <= 0 ? 0u : ~ban[w0 + lane] & (n >= 32 ? ~0u : (1u << n) - 1u);
        int at = __popc(left);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(kFull, at, o);
          if (lane >= o) at += t;
        }
        const int sum = __shfl_sync(kFull, at, 31);
        at += base - __popc(left);
        base += sum;
#pragma unroll
        for (int k = 0; k < 32; k += kWarps) {
          const unsigned bits = __shfl_sync(kFull, left, warp + k);
          const int b0 = __shfl_sync(kFull, at, warp + k);
          if ((bits >> lane) & 1u)
            E.lst[b0 + __popc(bits & ((1u << lane) - 1u))] = (unsigned short)(32 * (w0 + warp + k) + lane);
        }
      }
      if (tid == 0) S.nlist = base;
    }
    row_pass(std::false_type{});
    __syncthreads();

    // ---- passes over the cells: the terms of the J reaching every cell, a
    // group of kGroup per pass; in the last pass the cells left are the
    // perturbers of I in this batch ----
    const int nt0 = B.h == 2 ? n0 : 0;
    bool done = false;
#pragma unroll 1
    for (int g0 = 0;; g0 += kGroup) {
      B = S.bt;
      const int m = max(0, min(kGroup, nt0 - g0));
      const bool fin = last_round && g0 + kGroup >= nt0;
      if (!fin && m == 0) break;
      if (g0 > 0 && m > 0) {  // the first group's tables came with the row pass
        __syncthreads();
#pragma unroll 1
        for (int j = warp; j < m; j += kWarps) build_table(j, S.u.l.L0[g0 + j]);
        __syncthreads();
      }
      if (fin) {
        if (p.k > 0 && tkcnt + B.nct > p.cap) compact_selection<NINT, NT>(p, S, buf_e(p), buf_a(p), buf_key<NINT>(p));
      }
      const unsigned long long tau = S.tau;
      double acc_e = 0.0, acc_s2 = 0.0;
      unsigned long long acc_d0 = 0, acc_d1 = 0, acc_min = ~0ull;  // acc_min: units of 2^-S (FP: bits of |D|)
      unsigned int acc_na = 0;  // multi-state form
      double acc_es[kMaxStates], acc_s2s[kMaxStates];  // multi-state form: sums per state
#pragma unroll
      for (int st = 0; st < kMaxStates; st++) acc_es[st] = acc_s2s[st] = 0.0;
      const int nleft = MS ? B.nct : S.nlist;
      // a copy per kind: without the tests of it and the values one kind alone
      // needs, two words per spin 63.0 -> 57.3 ms.  With one word and the kinds
      // mixed in time three copies are more code in flight than the caches
      // hold (150 determinants 415 -> 423 us): one copy for all kinds then.
      auto cells = [&](auto kd) {
        constexpr int KD = decltype(kd)::value;
        const int kind = KD >= 0 ? KD : B.kind;
#pragma unroll 1
        for (int i = tid; i < nleft; i += kThreads) {
          int cc = i, x, y, ro_, so_;
          if constexpr (MS) {
            if ((ban[cc >> 5] >> (cc & 31)) & 1u) continue;
          } else {
            cc = E.lst[i];
          }
          cell_orbitals<NINT, NT, KD>(B, S, B.clo + cc, &ro_, &so_, &x, &y);
          y = y < 0 ? 0 : y;
          const typename BatchShared<NINT, NT>::Side R = S.row[x], C = S.col[y];
          const int ro = R.orb, so = C.orb;
          // the generator's own integrals and the pair's term of D, loaded ahead
          // of the terms of the J reaching every cell
          NT own = NT(0), own2 = NT(0);
          long long dpair = 0;
          if (fin && kind > 0) {
            if constexpr (E4) {
              own = eri_n[(R.idx & 0x7fffffff) + (C.idx & 0x7fffffff)];
              if (kind == 1) own2 = eri_n[ibase + so * norb + ro];
            } else {
              own = eri_n[tri(R.idx & 0x7fffffff, C.idx & 0x7fffffff)];
              if (kind == 1) own2 = eri_n[tri(S.row[y].idx & 0x7fffffff, S.col[x].idx & 0x7fffffff)];
            }
            dpair = (kind == 2 ? p.Ji : p.Wi)[ro * norb + so];
          }
          unsigned long long lo = 0ull;  // exact sum
          int hi = 0;
          double accs[kMaxStates];  // multi-state form: one sum per state
#pragma unroll
          for (int st = 0; st < kMaxStates; st++) accs[st] = 0.0;
          if constexpr (!MS) {
            lo = A0[cc] | ((unsigned long long)A1[cc] << 32);
            hi = (int)A2[cc];
          }
#pragma unroll 1
          for (int j = 0; j < m; j++) {
            const int rt = S.gRow[j][x], ct = S.gCol[j][y], rc = (int)((unsigned)rt + (unsigned)ct);
            if ((rt | ct) & (3 << 29)) continue;
            NT v;
            bool neg = rc < 0;
            if constexpr (E4) {
              v = eri_n[rc & 0x7fffffff];
              if (kind == 1) v -= eri_n[S.gB[j] + so * norb + ro];
            } else {
              v = eri_n[tri(rt & 0x1fffffff, ct & 0x1fffffff)];
              if (kind == 1) v -= eri_n[tri(S.gRow[j][y] & 0x1fffffff, S.gCol[j][x] & 0x1fffffff)];
            }
            if (kind == 1) {
              const int x2 = S.gx2[j];
              neg ^= ro > (so < x2 ? so : x2) && ro < (so < x2 ? x2 : so);
            }
            v = flip_sign(v, neg);
            con++;
            if constexpr (MS) {
#pragma unroll
              for (int st = 0; st < kMaxStates; st++)
                if (st < nst) accs[st] = fma(ms_gc[j * kMaxStates + st], (double)v, accs[st]);
            } else {
              unsigned long long l;
              int hh;
              fix_of(S.gcj[j] * v, F, l, hh);
              fix_add(lo, hi, l, hh);
            }
          }
          if (!fin) {
            if constexpr (MS) {
#pragma unroll
              for (int st = 0; st < kMaxStates; st++)
                if (st < nst) A[st * mc + cc] += accs[st];
            } else {
              A0[cc] = (uint32_t)lo;
              A1[cc] = (uint32_t)(lo >> 32);
              A2[cc] = (uint32_t)hi;
            }
            continue;
          }
          if constexpr (MS) {
            double vI = 0.0;  // <I|H|alpha> for the generator's own term
            if (kind > 0) {
              NT t = own;
              bool neg = (R.idx ^ C.idx) < 0;
              if (kind == 1) t -= own2;
              if (kind == 1) neg ^= ro > (so < B.qb ? so : B.qb) && ro < (so < B.qb ? B.qb : so);
              t = flip_sign(t, neg);
              vI = (double)t;
              con++;
            }
            long long D0 = R.d;  // E0_0 - H_aa
            if (kind > 0) D0 -= C.d + dpair;
            double crit = 0.0, a0 = 0.0;
#pragma unroll
            for (int st = 0; st < kMaxStates; st++) {
              if (st >= nst) break;
              const double a = A[st * mc + cc] + accs[st] + ms_cI[st] * vI;
              long long D = D0 + ms_de[st];
              const double q = FP ? den64_quot(p, a, R, C, kind, p.st_e0[st] - p.st_e0[0], &D) : div_fix<MS>(a, D, E.dscale);
              const double e = a * q;
              acc_es[st] += e;
              acc_s2s[st] += q * q;
              crit += ms_w[st] * e;  // c_alpha,s A_s / max_I c_Is^2
              const unsigned long long db = D < 0 ? 0ull - (unsigned long long)D : (unsigned long long)D;
              acc_min = db < acc_min ? db : acc_min;
              if (st == 0) a0 = a;
            }
            acc_na++;
            if (abs_bits(a0) < 0x3D06849B86A12B9Bull) atomicAdd(&S.tiny, 1u);
            uint64_t key[NW];
            const int kwr = B.sa * NINT + (ro >> 6), kws = (kind > 0) ? B.sb * NINT + (so >> 6) : -1;
#pragma unroll
            for (int w = 0; w < NW; w++)
              key[w] = S.kbase[w] | (w == kwr ? 1ull << (ro & 63) : 0ull) | (w == kws ? 1ull << (so & 63) : 0ull);
            uint64_t hk = 0;
#pragma unroll
            for (int w = 0; w < NW; w++) hk = splitmix64(hk ^ key[w]);
            acc_d0 += hk;
            acc_d1 ^= splitmix64(hk ^ 0x243F6A8885A308D3ull);
            if (p.k > 0) {
              const unsigned long long eb = abs_bits(crit);
              if (eb >= tau) {
                atomicAdd(&p.sel_hist[sel_bin(eb)], 1u);
                const int pos = atomicAdd(&S.tkcnt, 1);
                buf_e(p)[pos] = crit;
                buf_a(p)[pos] = a0;
#pragma unroll
                for (int w = 0; w < NW; w++) buf_key<NINT>(p)[(size_t)pos * NW + w] = key[w];
              }
            }
          } else {
            double a = fix_to_double(lo, hi, F);
            // the generator's own term c_I <I|H|alpha>
            if (kind > 0) {
              NT t = own;
              bool neg = (R.idx ^ C.idx) < 0;
              if (kind == 1) t -= own2;
              if (kind == 1) neg ^= ro > (so < B.qb ? so : B.qb) && ro < (so < B.qb ? B.qb : so);
              t = flip_sign(t, neg);
              a += (double)(S.cI * t);
            }
            // D = E0 - H_aa from the row and column sums
            long long D = R.d;
            if (kind > 0) D -= C.d + dpair;
            const double q = FP ? den64_quot(p, a, R, C, kind, 0.0, &D) : div_fix<MS>(a, D, E.dscale);
            acc_e = fma(a, q, acc_e);  // e = A q
            acc_s2 += q * q;
            if (GRAD) {
              // numerator weight 2A/D for loop 3, here already for the
              // generator's own element; (A/D)^2 weights the diagonal
              const double w1 = 2.0 * q;
              const unsigned long long wb = (unsigned long long)__double_as_longlong(w1);
              A0[cc] = (uint32_t)wb;
              A1[cc] = (uint32_t)(wb >> 32);
              if (kind > 0) {
                w_grad(p, ro, B.sa, so, B.sb, q * q);
                bool neg = (R.idx ^ C.idx) < 0;
                if (kind == 1) neg ^= ro > (so < B.qb ? so : B.qb) && ro < (so < B.qb ? B.qb : so);
                const double ws = flip_sign((double)S.cI * w1, neg);
                atomicAdd(&p.g_deri[eri_index(B.qa, ro, B.qb, so)], ws);
                if (kind == 1) atomicAdd(&p.g_deri[eri_index(B.qa, so, B.qb, ro)], -ws);
              }
            }
            // |a| < 1e-14, compared on the bit pattern (no FP64 compare)
            if (abs_bits(a) < 0x3D06849B86A12B9Bull) atomicAdd(&S.tiny, 1u);
            const unsigned long long db = D < 0 ? 0ull - (unsigned long long)D : (unsigned long long)D;
            acc_min = db < acc_min ? db : acc_min;
            // alpha's word w: the batch's base with the cell's orbitals
            const int kwr = B.sa * NINT + (ro >> 6), kws = (kind > 0) ? B.sb * NINT + (so >> 6) : -1;
            auto key = [&](int w) {
              return S.kbase[w] | (w == kwr ? 1ull << (ro & 63) : 0ull) | (w == kws ? 1ull << (so & 63) : 0ull);
            };
            // digest: the fold over the spin-up words is the row's where they
            // depend on the row alone
            uint64_t hk = S.hk0[x];
            if (kind != 2 && B.sa == 0) {
              hk = 0;
#pragma unroll
              for (int w = 0; w < NINT; w++) hk = splitmix64(hk ^ key(w));
            }
#pragma unroll
            for (int w = NINT; w < NW; w++) hk = splitmix64(hk ^ key(w));
            acc_d0 += hk;
            acc_d1 ^= splitmix64(hk ^ 0x243F6A8885A308D3ull);
            // e = A q is formed only when it can reach the threshold: with biased
            // exponents ea, eq of A and q, |A q| < 2^(ea + eq - 2044), so
            // ea + eq <= et + 1021 (et: the exponent of tau) puts it below tau
            const int ea = (int)(abs_bits(a) >> 52), eqx = (int)(abs_bits(q) >> 52);
            if (p.k > 0 && (tau == 0ull || ea + eqx > (int)(tau >> 52) + 1021)) {
              const double e = a * q;
              const unsigned long long eb = abs_bits(e);
              if (eb >= tau) {
                atomicAdd(&p.sel_hist[sel_bin(eb)], 1u);
                const int pos = atomicAdd(&S.tkcnt, 1);
                buf_e(p)[pos] = e;
                buf_a(p)[pos] = a;
#pragma unroll
                for (int w = 0; w < NW; w++) buf_key<NINT>(p)[(size_t)pos * NW + w] = key(w);
              }
            }
          }
        }
      };
      if (FP || (NINT == 1 && !MS && !GRAD && !by_kind(p))) cells(std::integral_constant<int, -1>{});
      else if (B.kind == 2) cells(std::integral_constant<int, 2>{});
      else if (B.kind == 1) cells(std::integral_constant<int, 1>{});
      else cells(std::integral_constant<int, 0>{});
      if (!fin) continue;
      // ---- the item's sums.  The digest, min |D| and the tiny count are the
      // sweep's: this thread's shares stay in shared memory until the kernel
      // ends.  e and (A/D)^2 go to the item's own slot (the generator's eps_I and
      // sum A^2/D^2 are reduced from the slots in item order after the wave, so
      // they do not depend on which CTA finished first); the last warp to arrive
      // adds them, thread by thread in a fixed order ----
      S.td0[tid] += acc_d0;
      S.td1[tid] ^= acc_d1;
      if (acc_min < S.tmin[tid]) S.tmin[tid] = acc_min;
      double* its = p.it_sum + ((size_t)slot * nper + jitem) * p.it_stride;
      if constexpr (MS) acc_e = acc_es[0], acc_s2 = acc_s2s[0];
      add_con();
      const unsigned int wna = MS ? __reduce_add_sync(kFull, acc_na) : 0u;
      S.u.red_t[0][tid] = acc_e;
      S.u.red_t[1][tid] = acc_s2;
      __threadfence_block();
      __syncwarp();
      int order = 0;
      if (lane == 0) {
        S.red_na[warp] = wna;
        __threadfence_block();
        order = atomicAdd(&S.arrive, 1);
      }
      order = __shfl_sync(kFull, order, 0);
      if (order == kWarps - 1) {
        __threadfence_block();
        // lanes 0-15 add e, 16-31 (A/D)^2
        double v = 0.0;
        const double* src = S.u.red_t[lane >> 4];
#pragma unroll 4
        for (int i = lane & 15; i < kThreads; i += 16) v += src[i];
#pragma unroll
        for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        const double vs = __shfl_sync(kFull, v, 16);
        unsigned long long tn = lane < kWarps ? S.red_na[lane] : 0ull, tc = lane < kWarps ? S.red_con[lane] : 0ull;
        tn = warp_sum_u(tn);
        tc = warp_sum_u(tc);
        if constexpr (!MS) {  // every cell of the list, each with the generator's own term (two-hole batch)
          tn = (unsigned long long)S.nlist;
          if (B.h == 2) tc += tn;
        }
        if (lane == 0) {
          its[0] = v;
          its[1] = vs;
          S.sw2 = vs;
          S.arrive = 0;
          if (tn) {
            atomicAdd(&p.na[M->g], tn);
            atomicAdd(&p.ncon[M->g], tc);
          }
        }
      }
      if constexpr (MS) {  // the other states' eps and s2, one at a time
#pragma unroll
        for (int st = 1; st < kMaxStates; st++) {
          if (st >= nst) break;
          __syncthreads();
          S.u.red_t[0][tid] = acc_es[st];
          S.u.red_t[1][tid] = acc_s2s[st];
          __syncthreads();
          if (warp == 0) {
            double ue = 0.0, us = 0.0;
            for (int i = lane; i < kThreads; i += 32) {
              ue += S.u.red_t[0][i];
              us += S.u.red_t[1][i];
            }
            ue = warp_sum(ue);
            us = warp_sum(us);
            if (lane == 0) {
              its[2 * st] = ue;
              its[2 * st + 1] = us;
            }
          }
        }
      }
      done = true;
      break;
    }
    if (done) break;
    add_con();
    __syncthreads();
    if (tid == 0) S.n0 = S.n1 = S.n2 = S.cnext = 0;
    __syncthreads();
  }
  if (GRAD) {
    __syncthreads();
    // ---- loop 3: c_J (2A/D) d<J|H|alpha> over the same (J, cell) pairs, by
    // the same rows and pair tables ----
    for (int c0 = 0; c0 < S.seg_s[3]; c0 += kChunk) {
      if (tid == 0) S.n0 = S.n1 = S.n2 = S.cnext = 0;
      __syncthreads();
      const int c1 = min(c0 + kChunk, S.seg_s[3]);
#pragma unroll 1
      for (int i = c0 + tid; i < c1; i += kThreads) {
        const int o = entry(i);
        const ulonglong2 en = S.ehp[o];
        const uint64_t hmr = en.x, part = en.y;
        if ((part & kBeforeBit) || dup(i, hmr)) continue;
        if (B.h == 2 && hmr == 0ull) continue;  // J = I: in the cells pass
        const int t = __popcll(hmr & ~B.hm);
        if (t > 2) continue;
        const int rec = (int)(S.erec[o] & 0x7FFFFFFFu);
        if (t == 0) S.u.l.L0[atomicAdd(&S.n0, 1)] = rec;
        else if (t == 1) {
          if (B.h == 1 || row_live<NINT, NT>(B, S, norb, part)) S.u.l.L12[atomicAdd(&S.n1, 1)] = rec;
        }
        else if (subset_live<NINT, NT>(B, S, norb, part, ban)) S.u.l.L12[kChunk - 1 - atomicAdd(&S.n2, 1)] = rec;
      }
      __syncthreads();
      row_pass(std::true_type{});
      __syncthreads();
      const int nt0 = B.h == 2 ? S.n0 : 0;
#pragma unroll 1
      for (int g0 = 0; g0 < nt0; g0 += kGroup) {
        const int m = min(kGroup, nt0 - g0);
        if (g0 > 0) {
          __syncthreads();
#pragma unroll 1
          for (int j = warp; j < m; j += kWarps) build_table(j, S.u.l.L0[g0 + j]);
          __syncthreads();
        }
#pragma unroll 1
        for (int i = tid; i < S.nlist; i += kThreads) {
          const int cc = E.lst[i];
          int ro, so, x, y;
          cell_orbitals<NINT, NT>(B, S, B.clo + cc, &ro, &so, &x, &y);
          const double w = a2d(cc);
#pragma unroll 1
          for (int j = 0; j < m; j++) {
            const int rt = S.gRow[j][x], ct = S.gCol[j][y];
            if ((rt | ct) & (3 << 29)) continue;
            const int x1 = S.gx1[j], x2 = S.gx2[j];
            bool neg = (rt ^ ct) < 0;
            if (B.kind == 1) neg ^= ro > (so < x2 ? so : x2) && ro < (so < x2 ? x2 : so);
            const double ws = flip_sign((double)S.gcj[j] * w, neg);
            atomicAdd(&p.g_deri[eri_index(x1, ro, x2, so)], ws);
            if (B.kind == 1) atomicAdd(&p.g_deri[eri_index(x1, so, x2, ro)], -ws);
          }
        }
      }
      __syncthreads();
    }
    // ---- diagonal: H_aa = H_II - F(a) [- F(b) + W(a,b)] + F(r) [+ F(s)]
    //      - W(r,a) [- W(r,b) - W(s,a) - W(s,b) + W(r,s)]; the W(r,s) terms
    //      were scattered per cell, the rest goes by row sums ----
    const int g = M->g;
    double* wF = p.g_wF + (size_t)g * 2 * norb;
    // four lanes per row or column of cells: sums of (A/D)^2 (cells outside the
    // list are zero).  (Adding each cell's into shared memory was a
    // compare-and-swap loop of up to 32 lanes on one word.)
    const int nvc = S.nv[1], nrows = B.kind == 2 ? B.nct / nvc : S.nv[B.sa], x0 = B.kind == 2 ? B.clo / nvc : 0;
    const int nsum = nrows + (B.kind == 2 ? nvc : 0);
#pragma unroll 1
    for (int u0 = 0; u0 < nsum; u0 += kThreads / 4) {
      const int u = u0 + (tid >> 2), sub = tid & 3;
      const bool row = u < nrows;
      double w = 0.0;
      if (u < nsum) {
        const int len = B.kind == 0 ? 1 : B.kind == 2 && row ? nvc : nrows;
#pragma unroll 2
        for (int v = sub; v < len; v += 4) {
          if (B.kind == 1 && v == u) continue;
          const double a = a2d(B.kind == 0 ? u : B.kind == 1 ? pair_cell(u, v) : row ? u * nvc + v : v * nvc + u - nrows);
          w = fma(a, a, w);
        }
      }
      w += __shfl_xor_sync(kFull, w, 1);
      w += __shfl_xor_sync(kFull, w, 2);
      w *= 0.25;
      if (u >= nsum || w == 0.0) continue;
      const int sr = row ? B.sa : 1, r = S.vir[sr][row ? x0 + u : u - nrows];
      if (sub == 0) atomicAdd(&wF[sr * norb + r], w);
      if (sub == 1) w_grad(p, r, sr, B.qa, B.sa, -w);
      if (sub == 2 && B.h == 2) w_grad(p, r, sr, B.qb, B.sb, -w);
    }
    if (tid == 0 && S.sw2 != 0.0) {
      const double sw = S.sw2;
      atomicAdd(&p.g_wH[g], sw);
      atomicAdd(&wF[B.sa * norb + B.qa], -sw);
      if (B.h == 2) {
        atomicAdd(&wF[B.sb * norb + B.qb], -sw);
        w_grad(p, B.qa, B.sa, B.qb, B.sb, sw);
      }
    }
  }
}

// This CTA's digest, min |D| and tiny counts into the sweep's totals.
template <int NINT, typename NT, bool FP>
__device__ __forceinline__ void flush_totals(const SweepParams& p, BatchShared<NINT, NT>& S, int dscale) {
  const int tid = threadIdx.x, lane = tid & 31;
  const unsigned long long d0 = warp_sum_u(S.td0[tid]), d1 = warp_xor_u(S.td1[tid]), mn = warp_min_u(S.tmin[tid]);
  if (lane == 0 && mn != ~0ull) {
    atomicAdd(&p.digest[0], d0);
    atomicXor(&p.digest[1], d1);
    atomicMin(p.min_den_bits, FP ? mn : (unsigned long long)__double_as_longlong(den_double(mn, dscale)));
  }
  if (tid == 0 && S.tiny) atomicAdd(p.n_tiny, (unsigned long long)S.tiny);
}

// The shared state of a CTA for the sweep of p.
template <int NINT, typename NT>
__device__ __forceinline__ void begin_sweep(const SweepParams& p, BatchShared<NINT, NT>& S) {
  const int tid = threadIdx.x;
  S.td0[tid] = S.td1[tid] = 0ull;
  S.tmin[tid] = ~0ull;
  if (tid == 0) {
    S.tiny = 0u;
    S.tkcnt = p.tk_cnt[blockIdx.x];
    S.tau = p.tk_tau[blockIdx.x];
    S.arrive = 0;
    S.nv[0] = p.norb - p.nalpha;
    S.nv[1] = p.norb - p.nbeta;
    S.inv_nv1 = S.nv[1] > 0 ? 1.0f / (float)S.nv[1] : 0.0f;
  }
}

// Thread 0's draws from the queue of live items (prep_slot's list): an item
// is published one item ahead, its list entry loaded two ahead and its queue
// position drawn three ahead, so that no latency of the queue is waited for.
struct Drawer {
  int pos, nxt;  // the position drawn last; the next item to publish (-1: none)
  // take(n): the first of n queue positions
  template <typename BS, typename Fn>
  __device__ __forceinline__ void draw(BS& S, int chunk, Fn&& take) {
    if (S.inext >= S.iend) {
      const int b0 = take(chunk);
      S.inext = b0;
      S.iend = b0 + chunk;
    }
    pos = S.inext++;
  }
  template <typename BS>
  __device__ __forceinline__ int entry(const BS& S, const SweepParams& p) const {
    if ((unsigned)pos >= (unsigned)S.nlive) return -1;
    return (int)p.live[pos < S.nfirst ? pos : p.wave_slots * p.nper - 1 - (pos - S.nfirst)];
  }
  // The first item of the sweep of p.  FP: of the items listed for the FP64
  // form (den64), else of the others.
  template <bool FP, typename BS, typename Fn>
  __device__ __forceinline__ void begin(BS& S, const SweepParams& p, int chunk, Fn&& take) {
    S.nfirst = FP ? 0 : p.live_cnt[0];
    S.nlive = S.nfirst + (FP == (p.den64 != 0) ? p.live_cnt[1] : 0);
    S.inext = S.iend = 0;
    draw(S, chunk, take);
    S.item[0] = entry(S, p);
    draw(S, chunk, take);
    nxt = entry(S, p);
    draw(S, chunk, take);
  }
  // No further item is published (the watchdog).
  template <typename BS>
  __device__ __forceinline__ void stop(BS& S) {
    S.nlive = 0;
    nxt = -1;
  }
  template <typename BS, typename Fn>
  __device__ __forceinline__ void advance(BS& S, const SweepParams& p, int par, int chunk, Fn&& take) {
    S.item[par ^ 1] = nxt;
    nxt = entry(S, p);
    draw(S, chunk, take);
  }
};

// Three CTAs per SM for one word per spin; two words per spin come with
// larger accumulators (at most two CTAs fit in shared memory), so those
// kernels take the registers of two CTAs and do not spill; so does the
// gradient's, whose row pass is there twice (17.8 -> 17.5 ms).
//
// FP = true: the items of the generators whose denominators are in FP64
// (den_form), which another launch runs after the others' items; as a branch of
// one kernel that form took 2% of every sweep's time.
//
// MS = true: the multi-state form (several states at once, FP64 only).
// Each state s has its own accumulator A_s (dynamic shared memory, one
// stride of max_cells each); a (J, cell) element is formed once and added
// with c_Js to every A_s.  The cells pass forms e_s = A_s^2/(E0_s - H_aa)
// for every state, sums each into its own eps and s2, and offers the
// determinant to the selection with the criterion sum_s w_s e_s,
// w_s = 1/max_I c_Is^2 (Sec. "Selected CI", the criterion of Angeli et al.).
template <int NINT, typename NT, bool GRAD = false, bool MS = false, bool E4 = true, bool FP = false>
__global__ void __launch_bounds__(kThreads, (NINT == 1 && !GRAD) ? 3 : 2) batch_kernel(const __grid_constant__ SweepParams p) {
  static_assert(!(MS && GRAD), "the gradient is a one-state form");
  static_assert(!MS || sizeof(NT) == 8, "the multi-state form is FP64");
  __shared__ BatchShared<NINT, NT> S;
  const int tid = threadIdx.x;
  const ItemEnv E = item_env<MS>(p);
  const NT* eri_n = numer_eri<NT, E4>(p);
  const NT* h_n = numer_h<NT>(p);

  begin_sweep<NINT, NT>(p, S);
  const int F = MS ? 0 : fix_scale(p);  // fixed-point scale of A_alpha (units of 2^-F)
  auto take = [&](int n) { return atomicAdd(p.queue, n); };
  // watchdog: stop taking work, report the timeout
  auto expired = [&]() {
    if (!p.timeout_ns || global_ns() - *((volatile unsigned long long*)p.t_start) <= p.timeout_ns) return false;
    atomicOr(p.err, 128);
    return true;
  };
  Drawer D;
  if (tid == 0) {
    if (p.timeout_ns) atomicCAS(p.t_start, 0ull, global_ns());
    D.begin<FP>(S, p, p.chunk, take);
    if (S.item[0] >= 0 && expired()) {
      S.item[0] = -1;
      D.stop(S);
    }
  }
  for (int par = 0;; par ^= 1) {
    __syncthreads();
    const int item = S.item[par];
    if (item < 0) break;
    if (tid == 0) {
      if (D.nxt >= 0 && expired()) D.stop(S);
      D.advance(S, p, par, p.chunk, take);
    }
    batch_item<NINT, NT, GRAD, MS, E4, FP>(p, S, item, F, E, eri_n, h_n);
  }
  flush_totals<NINT, NT, FP>(p, S, E.dscale);
  if (p.k > 0 && p.last_wave) compact_selection<NINT, NT>(p, S, buf_e(p), buf_a(p), buf_key<NINT>(p));
  __syncthreads();
  if (tid == 0) {
    p.tk_cnt[blockIdx.x] = S.tkcnt;
    p.tk_tau[blockIdx.x] = S.tau;
  }
}

// The work items of one wave of several instances' sweeps (one word count
// and precision): the wave's pieces (instance, run of generator slots) one
// after another, each piece's items from its own queue, `m.chunk` per draw.
// A CTA moves to the next piece when the current one's queue is empty; it
// stores its selection state (candidate count and threshold) for the
// instance it leaves and loads the state of the one it enters.  The dynamic
// shared memory is sized for the largest accumulator of the instances.
// Every instance has its own candidate buffers for each CTA of the launch;
// they are compacted to k entries by compact_multi_kernel after the last
// wave.
template <int NINT, typename NT, bool FP = false>
__global__ void __launch_bounds__(kThreads, (NINT == 1) ? 3 : 2) batch_multi_kernel(const __grid_constant__ MultiWaveInline m) {
  __shared__ BatchShared<NINT, NT> S;
  const int tid = threadIdx.x;
  if (tid == 0 && m.timeout_ns) atomicCAS(m.t_start, 0ull, global_ns());
  // the pieces one after another, each from its own queue: the piece index
  // is the same in every thread, so its parameters are read like a single
  // sweep's
#pragma unroll 1
  for (int pc = 0; pc < m.n; pc++) {
    const SweepParams& p = m.ps[pc];
    __syncthreads();
    begin_sweep<NINT, NT>(p, S);
    const int F = fix_scale(p);
    const ItemEnv E = item_env<false>(p);
    auto take = [&](int n) { return (int)atomicAdd(m.queue + pc, (unsigned long long)n); };
    auto expired = [&]() {
      if (!m.timeout_ns || global_ns() - *((volatile unsigned long long*)m.t_start) <= m.timeout_ns) return false;
      atomicOr(m.err, 128);  // watchdog: stop taking work, report the timeout
      return true;
    };
    Drawer D;
    if (tid == 0) {
      D.begin<FP>(S, p, m.chunk, take);
      if (S.item[0] >= 0 && expired()) {
        S.item[0] = -1;
        D.stop(S);
      }
    }
    for (int par = 0;; par ^= 1) {
      __syncthreads();
      const int item = S.item[par];
      if (item < 0) break;
      if (tid == 0) {
        if (D.nxt >= 0 && expired()) D.stop(S);
        D.advance(S, p, par, m.chunk, take);
      }
      batch_item<NINT, NT, false, false, true, FP>(p, S, item, F, E, numer_eri<NT, true>(p), numer_h<NT>(p));
    }
    flush_totals<NINT, NT, FP>(p, S, E.dscale);
    __syncthreads();
    if (tid == 0) {
      p.tk_cnt[blockIdx.x] = S.tkcnt;
      p.tk_tau[blockIdx.x] = S.tau;
    }
  }
}

// After the last wave: CTA buffer blockIdx.x of instance blockIdx.y keeps its
// k best candidates (as the last wave of a single sweep does).
template <int NINT, typename NT>
__global__ void __launch_bounds__(kThreads) compact_multi_kernel(const SweepParams* __restrict__ ps) {
  constexpr int NW = 2 * NINT;
  __shared__ BatchShared<NINT, NT> S;
  const SweepParams& p = ps[blockIdx.y];
  if (p.k <= 0) return;
  if (threadIdx.x == 0) {
    S.tkcnt = p.tk_cnt[blockIdx.x];
    S.tau = p.tk_tau[blockIdx.x];
  }
  compact_selection<NINT, NT>(p, S, p.tk_e + (size_t)blockIdx.x * (size_t)p.cap,
                              p.tk_a + (size_t)blockIdx.x * (size_t)p.cap,
                              p.tk_key + (size_t)blockIdx.x * (size_t)p.cap * NW);
  __syncthreads();
  if (threadIdx.x == 0) {
    p.tk_cnt[blockIdx.x] = S.tkcnt;
    p.tk_tau[blockIdx.x] = S.tau;
  }
}

// The batch launches of one wave: with den64 the FP64 form's items after the
// others, from the queue again.
template <auto* K, typename P>
static cudaError_t launch_smem(const P& p, int grid, size_t smem, cudaStream_t st) {
  const cudaError_t e = allow_smem<K>();
  if (e != cudaSuccess) return e;
  K<<<grid, kThreads, smem, st>>>(p);
  return cudaGetLastError();
}
template <int NINT, typename NT, bool GRAD, bool MS, bool E4>
static cudaError_t batch_launch_nint(const SweepParams& p, int grid, size_t smem, cudaStream_t st) {
  cudaError_t e = launch_smem<batch_kernel<NINT, NT, GRAD, MS, E4, false>>(p, grid, smem, st);
  if (e != cudaSuccess || !p.den64) return e;
  if ((e = cudaMemsetAsync(p.queue, 0, sizeof(int), st)) != cudaSuccess) return e;
  return launch_smem<batch_kernel<NINT, NT, GRAD, MS, E4, true>>(p, grid, smem, st);
}
template <typename NT, bool GRAD = false, bool MS = false, bool E4 = true>
static cudaError_t batch_launch(int nint, const SweepParams& p, int grid, size_t smem, cudaStream_t st) {
  return nint == 1 ? batch_launch_nint<1, NT, GRAD, MS, E4>(p, grid, smem, st)
                   : batch_launch_nint<2, NT, GRAD, MS, E4>(p, grid, smem, st);
}

// Launch helpers of the multi-instance batch kernels, instantiated for FP64
// in sweep.cu and for the mixed form in sweep_mixed.cu (the prep kernel is
// launched from sweep.cu only).
template <int NINT, typename NT>
static cudaError_t multi_launch_nint(const MultiWaveInline& m, int grid, size_t smem, cudaStream_t st) {
  cudaError_t e = launch_smem<batch_multi_kernel<NINT, NT, false>>(m, grid, smem, st);
  bool den64 = false;
  for (int i = 0; i < m.n; i++) den64 |= m.ps[i].den64 != 0;
  if (e != cudaSuccess || !den64) return e;
  if ((e = cudaMemsetAsync(m.queue, 0, sizeof(unsigned long long) * m.n, st)) != cudaSuccess) return e;
  return launch_smem<batch_multi_kernel<NINT, NT, true>>(m, grid, smem, st);
}
template <typename NT>
static cudaError_t multi_wave_launch(int nint, const MultiWaveInline& m, int total_slots, int grid, size_t smem,
                                     cudaStream_t st) {
  if (total_slots <= 0) return cudaSuccess;
  return nint == 1 ? multi_launch_nint<1, NT>(m, grid, smem, st) : multi_launch_nint<2, NT>(m, grid, smem, st);
}

template <typename NT>
static cudaError_t multi_compact_launch(int nint, const SweepParams* ps, int n, int grid, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (nint == 1) compact_multi_kernel<1, NT><<<dim3(grid, n), kThreads, 0, st>>>(ps);
  else compact_multi_kernel<2, NT><<<dim3(grid, n), kThreads, 0, st>>>(ps);
  return cudaGetLastError();
}

template <typename NT>
static int multi_blocks_per_sm(int nint, size_t smem) {
  return nint == 1 ? blocks_per_sm<batch_multi_kernel<1, NT>>(kThreads, smem)
                   : blocks_per_sm<batch_multi_kernel<2, NT>>(kThreads, smem);
}

// Per generator: wH * dH_II + sum_{s,x} wF[s][x] * dF^I_s(x), with
// F^I_s(x) = h_xx + sum_{j in I} W(x, j) and H_II = sum_i h_ii + sum_{i<j} W(i, j).
template <int NINT>
__global__ void __launch_bounds__(kThreads) grad_gen_kernel(const __grid_constant__ SweepParams p) {
  constexpr int NW = 2 * NINT;
  __shared__ int s_occ[kMaxElec];
  const int g = blockIdx.x, tid = threadIdx.x, norb = p.norb, nel = p.nel;
  const double wH = p.g_wH[g];
  const double* wF = p.g_wF + (size_t)g * 2 * norb;
  const uint64_t* I = p.dets + (size_t)p.order[g] * NW;
  if (tid == 0) {
    int n = 0;
    for (int s = 0; s < 2; s++)
      for (int q = 0; q < norb; q++)
        if ((I[s * NINT + (q >> 6)] >> (q & 63)) & 1ull) s_occ[n++] = s * norb + q;
  }
  __syncthreads();
  if (wH != 0.0)
    for (int ij = tid; ij < nel * nel; ij += kThreads) {
      const int i = ij / nel, j = ij - i * nel;
      const int ci = s_occ[i], si = ci >= norb, qi = ci - si * norb;
      if (i == j) atomicAdd(&p.g_dh[qi * norb + qi], wH);
      else if (i < j) {
        const int cj = s_occ[j], sj = cj >= norb, qj = cj - sj * norb;
        w_grad(p, qi, si, qj, sj, wH);
      }
    }
  for (int x = tid; x < 2 * norb; x += kThreads) {
    const double w = wF[x];
    if (w == 0.0) continue;
    const int s = x / norb, q = x - s * norb;
    atomicAdd(&p.g_dh[q * norb + q], w);
    for (int i = 0; i < nel; i++) {
      const int c = s_occ[i], sj = c >= norb, j = c - sj * norb;
      atomicAdd(&p.g_deri[eri_index(q, q, j, j)], w);
      if (sj == s) atomicAdd(&p.g_deri[eri_index(q, j, j, q)], -w);
    }
  }
}

}  // namespace qp
