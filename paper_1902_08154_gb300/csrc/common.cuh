// common.cuh -- device helpers and launch parameters of the sm_103a EN-PT2
// sweep (Quantum Package 2.0, arXiv:1902.08154).  Internal to the library.
#pragma once
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

struct qp_pt2_ctx;

namespace qp {

constexpr int kMaxOrb = 128;
// bits of a sweep's error word (16 and 32: the no-allocation entry point's
// symmetry check, the selection's candidate space; 64: coefficients times
// integrals beyond the exact accumulator's range)
enum : int { kErrOcc = 1, kErrDup = 2, kErrCoef = 4, kErrBucket = 8, kErrRange = 64, kErrTimeout = 128 };
constexpr int kMaxElec = 64;   // per determinant (both spins); hole masks are uint64
constexpr int kMaxBatch = kMaxElec + kMaxElec * (kMaxElec - 1) / 2;
constexpr int kSelBins = 1024;  // |e| histogram: 128 binary exponents (2^-100 .. 2^27) x 8 sub-bins
constexpr int kMaxStates = 4;   // states of one multi-state sweep

// Fold of splitmix64 over the key words: the digest hash of a determinant.
// splitmix64 is the generator of Steele, Lea & Flood (2014); its finaliser
// constants are those of Vigna's public reference implementation.
__host__ __device__ inline uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

// Compound triangular index of Algorithm hash (0-based).
__device__ __forceinline__ int tri(int a, int b) {
  int hi = a > b ? a : b, lo = a > b ? b : a;
  return hi * (hi + 1) / 2 + lo;
}

__device__ __forceinline__ int eri_index(int p, int q, int r, int s) {
  return tri(tri(p, q), tri(r, s));
}

// Four-index layout of the integrals for the sweep's numerator gathers:
// (pq|rs) at ((p * norb + r) * norb + q) * norb + s, so that the integrals
// (pq|rs) of a fixed pair (p, r) form one norb x norb slab, row q, column s.
// The cells of a batch vary q and s over the virtual orbitals with (p, r)
// fixed (two holes, or a J's two particles), so a warp reads consecutive s
// of one row.  norb^4 entries (below 2^31 for norb <= 128).
__device__ __forceinline__ int eri4_index(int p, int q, int r, int s, int norb) {
  return ((p * norb + r) * norb + q) * norb + s;
}

// Number of set bits of the spin string sw (NINT words) strictly between
// orbitals lo < hi: the masked popcount that gives a single substitution's
// phase (Sec. "Internal representation of determinants").
template <int NINT>
__device__ __forceinline__ int count_between(const uint64_t* sw, int lo, int hi) {
  int a = lo + 1, b = hi, n = 0;
#pragma unroll
  for (int w = 0; w < NINT; w++) {
    int l = a - 64 * w, u = b - 64 * w;
    l = l < 0 ? 0 : l;
    u = u > 64 ? 64 : u;
    if (l < u) {
      uint64_t m = (u == 64 ? ~0ull : ((1ull << u) - 1)) & ~((1ull << l) - 1);
      n += __popcll(sw[w] & m);
    }
  }
  return n;
}

// What the Hamiltonian/Davidson unit needs of a context (filled by
// qp_pt2.cu, which owns the context), and the library's error reporter.
struct CtxView {
  int norb, nalpha, nbeta, nint, nel, device;
  const double *h, *eri, *Jm, *Km;  // device copies, [norb*norb] and packed
  cudaStream_t st;
  struct ::qp_pt2_ctx* ctx;
};
int ctx_view(struct ::qp_pt2_ctx* x, CtxView* v);
// The context's workspace for the Hamiltonian and Davidson unit: taken by one
// call at a time (false: another holds it), given back with the size wanted.
bool ctx_ws_take(struct ::qp_pt2_ctx* x, void** p, size_t* bytes);
void ctx_ws_give(struct ::qp_pt2_ctx* x, size_t bytes);
int report(int code, const char* msg);

// Bucket entries per coarse-filter record with holes Q of I (d = |Q|), at
// most: d = 1 the shared list and its hole's, d = 2 the shared list, two
// holes' and the pair's, d = 3 three holes' and three pairs', d = 4 six pairs'.
__host__ __device__ inline long long bucket_entries_per_record(int nel) {
  return nel >= 3 ? 6 : (nel == 2 ? 4 : 2);
}

// Bit masks of the cells that J ranked before I ban, per generator slot (see
// prep_slot).  Words of one set: a bit per cell of a spin-up pair batch (ca),
// a spin-down pair batch (cb) and an opposite-spin batch (cm).  A slot holds
// the base set [ca | cb | cm], then per hole of I [same spin | opposite spin]
// with stride hs.
struct MaskDims {
  int ca, cb, cm, hs;
};
__host__ __device__ inline MaskDims mask_dims(int norb, int na, int nb) {
  const int va = norb - na, vb = norb - nb;
  MaskDims m;
  m.ca = (va * (va - 1) / 2 + 31) / 32;
  m.cb = (vb * (vb - 1) / 2 + 31) / 32;
  m.cm = (va * vb + 31) / 32;
  m.hs = (m.ca > m.cb ? m.ca : m.cb) + m.cm;
  return m;
}
__host__ __device__ inline int mask_words(int norb, int na, int nb) {  // even: 64-bit masks follow
  const MaskDims m = mask_dims(norb, na, nb);
  return (m.ca + m.cb + m.cm + (na + nb) * m.hs + 1) & ~1;
}
// 64-bit orbital masks per slot: rows banned in every pair batch [2][nint],
// cells banned in every one-hole batch [2][nint], and per hole its rows
// [2][nint] and one-hole cells [nint].
__host__ __device__ inline int orb_mask_words(int nint, int nel) { return (4 + 3 * nel) * nint; }

// Cells of the largest work item when the opposite-spin batches are split
// into t tiles of rows.
inline int cells_for_tile(int norb, int n_alpha, int n_beta, int t) {
  const int va = norb - n_alpha, vb = norb - n_beta;
  int m = (n_alpha > 0 && n_beta > 0) ? ((va + t - 1) / t) * vb : 0;
  const int others[4] = {va, vb, va * (va - 1) / 2, vb * (vb - 1) / 2};
  for (int o : others) m = o > m ? o : m;
  return m < 1 ? 1 : m;
}

// Dynamic shared memory of the one-state batch kernel for mc cells: A_alpha
// as a 96-bit integer per cell (three 32-bit words; the exact accumulation in
// sweep_impl.cuh), one ban bit per cell and the list of the cells left (16 bits
// each).
__host__ __device__ inline size_t sweep_smem(int mc) {
  const size_t m = (size_t)(mc < 1 ? 1 : mc);
  return 8 * m + 4 * ((m + 1) & ~(size_t)1) + 4 * ((m + 31) / 32) + 2 * m;
}

// Lets kernel K have all the dynamic shared memory that its static part leaves
// of a block's.  The limit belongs to the process: a size per launch would let
// one thread's smaller launch lower it between another's call and launch.
template <auto* K>
inline cudaError_t allow_smem() {
  static std::atomic<int> room{0};
  if (!room) {
    int dev = 0, all = 0;
    cudaFuncAttributes a;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&all, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, K);
    if (e != cudaSuccess) return e;
    room = all - (int)a.sharedSizeBytes;
  }
  return cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, room);
}
// CTAs of kernel K per SM, 0 when one does not fit.
template <auto* K>
inline int blocks_per_sm(int threads, size_t smem) {
  int n = 0;
  if (allow_smem<K>() != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, K, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

struct GenMeta;
// Device bytes per generator slot of a wave: metadata, nd coarse-filter
// records (words, nst coefficients, hole mask, particles), bucket offsets,
// ent_cap self-contained entries (20 bytes), the ban masks, the live-item
// list and the nper items' FP64 sums (2 per state).
inline size_t wave_slot_bytes(size_t meta_bytes, int norb, int na, int nb, int nbat, size_t nd, int nst, int nper) {
  const int nint = (norb - 1) / 64 + 1, nw = 2 * nint, nel = na + nb;
  const size_t ent_cap = nd * (size_t)bucket_entries_per_record(nel);
  return meta_bytes + nd * (8 * (size_t)nw + 8 * (size_t)nst + 8 + 8) + 4 * (size_t)(nbat + 2) + 20 * ent_cap +
         4 * (size_t)mask_words(norb, na, nb) + 8 * (size_t)orb_mask_words(nint, nel) +
         4 * (size_t)nper + 16 * (size_t)nper * (size_t)nst;
}

// The fixed-point unit of a sweep's denominators is 2^-62 of a power of two at
// most the bound |E0| + n max|h| + n (n - 1) max|(pq|rs)|, n = n_el + 2; a
// generator has that form where this power is at most kDenRange times the
// magnitude of its energies (den_form in sweep_impl.cuh).  False: |E0| alone
// is large enough for that, so that all generators have it.
constexpr double kDenRange = 128.0;
inline bool den_maybe_fp64(double hmax, double emax, int nel, double e0_max, double e0_min) {
  const double n = (double)(nel + 2), bound = e0_max + n * hmax + n * (n - 1.0) * emax;
  if (!(bound < 0.99e300)) return true;
  int e;
  frexp(bound, &e);  // bound < 2^e
  return !(ldexp(1.0, e - 1 > -838 ? e - 1 : -838) <= kDenRange * e0_min);
}

// Per-generator data built by the prep kernel and read by the batch kernel.
struct GenMeta {
  uint64_t I[4];            // generator determinant (2*NINT words used)
  int g;                    // rank of the generator (-1: empty slot)
  int nrec;                 // coarse-filter records
  long long hii;            // <I|H|I>, fixed point or the bits of FP64 (den_form in sweep_impl.cuh)
  double cI;                // c_I
  int occ[kMaxElec];        // spin-orbital codes s*norb+q of I, ordered
  long long F[2][kMaxOrb];  // Fock diagonal of I, likewise
};

struct SweepParams {
  int norb, nalpha, nbeta, nel, nbat;
  // ntile > 1: every opposite-spin two-hole batch is split into ntile work
  // items over consecutive blocks of ceil(nv_up / ntile) rows (so that its
  // accumulator fits, or fits more than once, in an SM's shared memory);
  // nper = work items per generator = nbat + (ntile - 1) n_alpha n_beta
  int ntile, nper;
  // work items taken from the queue per draw (>= 1)
  int chunk;
  // watchdog: with timeout_ns > 0 a CTA stops taking work items once
  // timeout_ns nanoseconds (device global timer) have passed since *t_start,
  // the time the first CTA of the call started, and sets error flag 128
  unsigned long long timeout_ns;
  unsigned long long* t_start;
  int64_t ndet;
  const uint64_t* dets;   // [ndet][2][NINT]
  const double* coefs;    // [ndet]
  const int32_t* order;   // det index by rank
  const int32_t* rank_of; // rank by det index
  const double* h;        // [norb*norb]
  const double* eri;      // packed
  const float* h32;       // FP32 copies for the mixed-precision numerator (NULL in FP64 mode)
  const float* eri32;
  const double* eri4;     // [norb^4] four-index layout (eri4_index) of the batch kernel's gathers
  const float* eri4_32;   // its FP32 copy (mixed precision; NULL in FP64 mode)
  int mixed;              // 1: numerator gathers and products in FP32
  const double* Jm;       // [norb*norb] (pp|qq)
  const double* Km;       // [norb*norb] (pq|qp)
  long long *Ji, *Wi;     // [norb*norb] Jm and Jm - Km in fixed point (written by the prep kernel)
  double e0;
  int shard_index, shard_count;   // generators of rank shard_index + t*shard_count
  const int32_t* gen_list;        // if set: the generator of slot t has rank gen_list[t]
  // target space: alpha must hold every core spin orbital, no deleted one,
  // and (tgt_max_exc >= 0) at most tgt_max_exc electrons moved from tgt_ref
  int tgt_on, tgt_max_exc;
  uint64_t tgt_ref[4], tgt_core[4], tgt_del[4];
  // several states (nst > 1, multi-state batch kernel only): state s has its
  // coefficients at coefs + s*ndet, its records' coefficients at
  // r_coef + s*rc_stride, its E0 in st_e0[s], its per-generator sums at
  // eps + s*ndet and s2 + s*ndet; st_cmax[s] holds the bits of max_I |c_Is|
  int nst;
  int64_t rc_stride;
  double st_e0[kMaxStates];
  const unsigned long long* st_cmax;

  // wave of generator slots
  int wave_start;                 // first generator position (t) of this wave
  int wave_slots;                 // slots in this wave
  int last_wave;                  // 1 on the last wave: final selection compaction
  int* queue;                     // per-wave item counter

  // per-slot data (capacity ndet records, ent_cap bucket entries)
  GenMeta* meta;                  // [slots]
  uint64_t* r_words;              // [slots][ndet][2*NINT]
  double* r_coef;                 // [slots][ndet]
  uint64_t* r_hmask;              // [slots][ndet]  holes of I missing from J (occupied index bits)
  uint64_t* r_part;               // [slots][ndet]  up to 4 particle codes of J outside I, 16 bits each
  int* b_ofs;                     // [slots][nbat + 2]  bucket offsets (bucket nbat: the shared list)
  uint32_t* b_mask;               // [slots][mask_w]  cells banned by J ranked before I (MaskDims)
  uint64_t* o_mask;               // [slots][orb_w]   rows and one-hole cells banned (orb_mask_words)
  int mask_w, orb_w;
  // bucket entries, self-contained so that the batch kernel classifies a
  // bucket by streaming it: the record's hole mask and particle codes, and
  // its index with the rank flag (rank(J) < rank(I)) in bit 31
  ulonglong2* e_hp;               // [slots][ent_cap]: hole mask, particles (one 16-byte load)
  uint32_t* e_rec;                // [slots][ent_cap]
  // the wave's work items (slot * nper + item), without those of batches
  // banned as a whole, in the order the prep kernel finished the slots (den64:
  // those of generators with denominators in FP64 from the back)
  uint32_t* live;                 // [slots * nper]
  int* live_cnt;                  // per wave: items listed from the front, from the back; zero before the prep kernel
  int64_t ent_cap;

  // exact accumulation of A_alpha: bits of max_I |c_I| (written by the
  // validation) and of max |h_pq| and max |(pq|rs)| (the context's), from
  // which every CTA derives the same fixed-point scale
  const unsigned long long* cmax_bits;
  const unsigned long long* hmax_bits;  // [2]: max |h|, max |eri|

  // per-item sums of the wave, reduced per generator in a fixed order:
  // it_sum[(slot * nper + item) * it_stride + 2 s + {0, 1}] = (e, A^2/D^2)
  // of state s
  double* it_sum;
  int it_stride;

  // per-generator outputs, by rank
  double* eps;
  double* s2;
  unsigned long long* na;
  unsigned long long* ncon;
  // global accumulators
  unsigned long long* digest;       // [2]
  unsigned long long* min_den_bits; // bits of min |D| (non-negative double)
  unsigned long long* n_tiny;

  // selection
  int64_t k;
  int64_t cap;                   // per-CTA candidate capacity (>= k + max cells)
  double* tk_e;                  // [grid][cap]
  double* tk_a;                  // [grid][cap]
  uint64_t* tk_key;              // [grid][cap][2*NINT]
  int* tk_cnt;                   // [grid]
  unsigned long long* tk_tau;    // [grid] CTA thresholds (bits of |e|)
  unsigned long long* tau_bits;  // global selection threshold (bits of |e|)
  unsigned int* sel_hist;        // [kSelBins] counts of candidates offered to the buffers, by |e| bin

  int max_cells;
  int den64;                     // 1: generators with denominators in FP64 are possible (den_maybe_fp64)
  int* err;                      // device error flags (0 = fine)

  // gradient of E_PT2 (Psi0 and E0 fixed); used by the GRAD batch kernel
  double* g_dh;                  // [norb*norb]  symmetric halves off the diagonal
  double* g_deri;                // [P]          packed integrals
  double* g_wF;                  // [ndet][2][norb]  weights of dF^I_s(x) per generator rank
  double* g_wH;                  // [ndet]           weight of dH_II per generator rank
};

// The batch kernel's view of one wave of several instances: the pieces'
// parameters travel inside the kernel's parameters (constant bank, read-only
// and uncontended like a single sweep's), at most kMaxPieces per wave.
constexpr int kMaxPieces = 16;
struct MultiWaveInline {
  SweepParams ps[kMaxPieces];
  long long item_ofs[kMaxPieces + 1];
  int n;
  int chunk;                   // work items per draw from a piece's queue
  unsigned long long* queue;   // [n] the pieces' item counters
  unsigned long long timeout_ns;
  unsigned long long* t_start;
  int* err;                    // flag 128: the watchdog stopped the launch
};

// Slots a wave may hold for its work items to be numbered in 31 bits.
inline long long max_wave_slots(int nper) { return ((1ll << 31) - 1) / (nper > 0 ? nper : 1); }

// One wave of several instances' sweeps in one launch: ps[i] holds instance
// i's parameters for the wave; slot_ofs / item_ofs number the instances'
// generator slots / work items one instance after the other.
struct MultiWave {
  const SweepParams* ps;       // [n]
  const int* slot_ofs;         // [n + 1]
  const long long* item_ofs;   // [n + 1]
  int n;
  int chunk;                   // work items per draw (batch kernel)
  unsigned long long* queue;   // the pieces' item counters (batch kernel)
  unsigned long long timeout_ns;
  unsigned long long* t_start;
  int* err;                    // flag 128: the watchdog stopped the launch
};

}  // namespace qp
