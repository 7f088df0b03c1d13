// Budget, element threshold and filter of the NSF step (steps a4-a6).
//
// Budget (Eq. 1.18 with the fixed phase of Sec. 3.2 / Sec. 4): the RMS budget
// is c4 * tol_stage while r >= switch_resid, else 3/4 r^2 / (3x + x^3), with
// r = ||T - I||_F / sqrt(n) and x = ||X||_F / sqrt(n) of the current iterate;
// the filter's absolute Frobenius bound is b = sqrt(n) * beta.
//
// EXACT threshold: tau is the smallest magnitude v such that the squares of
// all entries with |x| <= v sum to more than b^2 (every |x| < tau is
// dropped, every |x| >= tau kept, so equal magnitudes share their fate); if
// all entries with |x| <= b fit, tau is the smallest magnitude above b
// (+inf if there is none). It is found by a radix select on the IEEE bit
// pattern of |x| (positive doubles order like unsigned integers): a histogram
// of the top 16 bits over the buckets that can hold the crossing, then 8-bit
// digits over the candidates of the crossing bucket. The crossing is never
// below b / sqrt(N), N the matrix's entries (N smaller squares fit b^2), so
// everything below that is one sum kept in registers and only the entries of
// [b / sqrt(N), b] go to a bucket. The squares are
// summed as exact 128-bit integers on a fixed grid of the matrix, q(x) =
// floor(x^2 / 2^(2e - 62)) with 2^e <= b < 2^(e+1), against Q = q(b): the
// decision does not depend on the order of the additions, and it is the exact
// one up to the flooring, less than one grid step (2^-62 b^2) per entry.
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"
#include "kernels.h"
#include "seg.cuh"

namespace cg = cooperative_groups;

namespace sgn {

namespace {

constexpr int NB0 = kSelBuckets;  // level-0 buckets: the sum below the pivot, then 16 per octave
constexpr int NDIG = 256;         // digit buckets

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__global__ void k_select_bound(int nb, const int *active, MatScalars *ms) {
  after_previous();
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= nb || !active[m]) return;
  int64_t c = ms[m].nnz_bar;
  ms[m].tau = c > 0 ? __ddiv_rn(ms[m].b, __dsqrt_rn(double(c))) : __longlong_as_double(0x7ff0000000000000LL);
}

// ------------------------------------------------------------ EXACT select
struct SelState {
  unsigned long long prefix;              // key bits known so far
  unsigned long long below_lo, below_hi;  // 128-bit sum of q strictly below the prefix range
  unsigned long long below0_lo, below0_hi;  // the same below the crossing level-0 bucket
  int found;                              // 1: a crossing exists; 0: everything <= b fits
  int pad;
};

// Scratch: 128-bit sums (lo, hi) per level-0 bucket, the smallest key above b
// per matrix, the select states, the candidate counts and the candidates
// (key, row of the values), each matrix's in a region of its own.
struct SelScratch {
  unsigned long long *hist0;     // nb * NB0 * 2
  unsigned long long *minabove;  // nb
  SelState *st;                  // nb
  unsigned long long *overflow;  // 1: set when a matrix has more candidates than room
  unsigned long long *redo;      // 1: the candidates are taken again, into exact regions
  unsigned long long *ncand;     // nb; may count past the room
  unsigned long long *cbase;     // nb: matrix m's candidates lie at [cbase, cbase + croom)
  unsigned long long *croom;     // nb
  unsigned long long *cand;      // cap
  int *cand_r;                   // cap
};

static_assert(sizeof(SelState) <= kSelStateBytes, "select state outgrew its scratch slot");

inline size_t align_up(size_t x) { return sel_align(x); }

SelScratch carve(void *base, int nb, int64_t cap) {
  char *p = static_cast<char *>(base);
  SelScratch s;
  s.hist0 = reinterpret_cast<unsigned long long *>(p);
  p += align_up(size_t(nb) * NB0 * 2 * 8);
  s.minabove = reinterpret_cast<unsigned long long *>(p);
  p += align_up(size_t(nb) * 8);
  s.st = reinterpret_cast<SelState *>(p);
  p += align_up(size_t(nb) * kSelStateBytes);
  s.overflow = reinterpret_cast<unsigned long long *>(p);
  s.redo = s.overflow + 1;
  s.ncand = s.overflow + 2;
  s.cbase = s.ncand + nb;
  s.croom = s.cbase + nb;
  p += align_up((3 * size_t(nb) + 2) * 8);
  s.cand = reinterpret_cast<unsigned long long *>(p);
  p += align_up(size_t(cap > 0 ? cap : 1) * 8);
  s.cand_r = reinterpret_cast<int *>(p);
  return s;
}

// Rows of the values to select over: row r holds entries [rs[r], re[r]) and
// belongs to matrix seg[r]; with rs == nullptr the values are one flat array
// of flat_nnz entries cut into rows of FLAT_ROW, all of matrix 0.
constexpr int64_t FLAT_ROW = kFlatRow;
constexpr int SEL_THREADS = 256;

__device__ __forceinline__ int row_mat(const SelRows &R, int64_t r) { return R.seg ? R.seg[r] : 0; }

constexpr unsigned long long INF_KEY = 0x7FF0000000000000ULL;

// The filter's rule on keys: x is kept when x != 0 and |x| >= tau, tau given
// by its bit pattern. For every |x| that is not NaN this is the comparison of
// the two doubles (non-negative doubles order like their bit patterns); NaN
// entries are dropped, as by the floating-point comparison. The count and
// the write of a filter both decide with this one function.
__device__ __forceinline__ bool keep_key(unsigned long long key, unsigned long long tkey) {
  return key != 0ULL && key <= INF_KEY && key >= tkey;
}

__device__ __forceinline__ void row_range(const SelRows &R, int64_t r, int64_t &b, int64_t &e) {
  if (R.rs) {
    b = R.rs[r];
    e = R.re[r];
  } else {
    b = r * FLAT_ROW;
    e = min(b + FLAT_ROW, R.flat_nnz);
  }
}

// Bit pattern of |x| as an FP64 number. For FP32 values of the normal range
// it is built with integer operations (exponent rebiased by 1023 - 127 = 896,
// mantissa widened by 29 bits): the same bits as the exact conversion, with
// no work for the FP64 pipe, which this GPU runs at 1/64 of its FP32 rate.
__device__ __forceinline__ unsigned long long key_f32(float x) {
  const uint32_t b = __float_as_uint(x) & 0x7FFFFFFFu, e = b >> 23;
  if (e != 0u && e != 0xFFu)
    return ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)(b & 0x7FFFFFu) << 29);
  if (b == 0u) return 0ULL;
  return (unsigned long long)__double_as_longlong(fabs(double(x)));  // subnormal, inf, NaN
}

__device__ __forceinline__ unsigned long long key_f64(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFULL;
}

template <typename T>
__device__ __forceinline__ unsigned long long key_t(T x);
template <>
__device__ __forceinline__ unsigned long long key_t<float>(float x) { return key_f32(x); }
template <>
__device__ __forceinline__ unsigned long long key_t<double>(double x) { return key_f64(x); }

// Keys in the width of the values: FP32 values are compared as 32-bit keys,
// with every bound converted once per row. ceil_key(k): the smallest key of
// the type whose magnitude is at least that of the 64-bit key k (all ones past
// infinity); floor_key(k): the largest whose magnitude is at most that.
template <typename T>
struct KeyT;
template <>
struct KeyT<float> {
  using K = uint32_t;
  static constexpr K kInf = 0x7F800000u;
  static __device__ __forceinline__ K of(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
  static __device__ __forceinline__ unsigned long long wide(K k) {
    return key_f32(__uint_as_float(k));
  }
  static __device__ __forceinline__ K ceil_key(unsigned long long k) {
    if (k > INF_KEY) return ~0u;
    return __float_as_uint(__double2float_ru(__longlong_as_double((long long)k)));
  }
  static __device__ __forceinline__ K floor_key(unsigned long long k) {
    if (k > INF_KEY) return 0x7FFFFFFFu;
    return __float_as_uint(__double2float_rd(__longlong_as_double((long long)k)));
  }
};
template <>
struct KeyT<double> {
  using K = unsigned long long;
  static constexpr K kInf = INF_KEY;
  static __device__ __forceinline__ K of(double x) { return key_f64(x); }
  static __device__ __forceinline__ unsigned long long wide(K k) { return k; }
  static __device__ __forceinline__ K ceil_key(unsigned long long k) { return k; }
  static __device__ __forceinline__ K floor_key(unsigned long long k) { return k; }
};

// (hi, lo) += x^2 for FP32 x, exactly: the square's rounding error comes from
// an FMA and the sum's from TwoSum; all in FP32, which this GPU runs at 64x
// its FP64 rate. Inputs are scaled by 2^48 (exact), so that squares of
// entries from 2^-111 to 2^16 stay normal FP32 numbers.
__device__ __forceinline__ void ff_add_sq48(float x, float &hi, float &lo) {
  const float y = __fmul_rn(x, 281474976710656.0f);  // 2^48
  const float p = __fmul_rn(y, y), e = __fmaf_rn(y, y, -p);
  const float s = __fadd_rn(hi, p), bb = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb)), e));
  hi = s;
}

__device__ __forceinline__ void ff_add(float &hi, float &lo, float h2, float l2) {
  const float s = __fadd_rn(hi, h2), bb = __fsub_rn(s, hi);
  const float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(h2, bb));
  lo = __fadd_rn(__fadd_rn(lo, l2), err);
  hi = s;
}

// q = floor(x^2 / 2^(2e - 62)) for 0 < |x| <= b, with |x| given by its FP64
// bit pattern (significand M, biased exponent E; a subnormal counts as E = 1)
// and e the biased exponent of b (likewise): x^2 / 2^(2e - 62) = M^2 2^-s with
// s = 42 + 2 (e - E) >= 42, so q is M^2 shifted right by s, exactly, in
// integers (q < 2^64 since |x| <= b). q >= 1 exactly when E >= e - 31.
// FP32 values have M = m 2^29 with m < 2^24, and q = m^2 2^(58 - s) needs one
// 32 x 32-bit product.
template <typename T>
__device__ __forceinline__ unsigned long long qval(unsigned long long key, int eb) {
  const int ex = int(key >> 52);
  const int s = 42 + 2 * (eb - (ex ? ex : 1));
  if (s >= 106) return 0ULL;
  const unsigned long long M = (key & 0xFFFFFFFFFFFFFULL) | (ex ? (1ULL << 52) : 0ULL);
  if constexpr (sizeof(T) == 4) {
    const unsigned m = unsigned(M >> 29);
    const unsigned long long m2 = (unsigned long long)m * m;  // < 2^48
    return s <= 58 ? m2 << (58 - s) : m2 >> (s - 58);
  } else {
    const unsigned long long lo = M * M, hi = __umul64hi(M, M);
    if (s >= 64) return hi >> (s - 64);
    return (lo >> s) | (hi << (64 - s));
  }
}

// q of a key of the values' own width, and its level-0 bucket (base: the top 16
// bits of the pivot). FP32 keys of the normal range need 32-bit operations and
// one 32 x 32-bit product.
template <typename T>
__device__ __forceinline__ unsigned long long q_bucket(typename KeyT<T>::K key, int eb, int base,
                                                       int &bk) {
  if constexpr (sizeof(T) == 4) {
    if (key >= 0x00800000u) {
      const int ex = int(key >> 23);
      const unsigned m = (key & 0x7FFFFFu) | 0x800000u;
      const unsigned long long m2 = (unsigned long long)m * m;  // < 2^48
      const int sh = 16 - 2 * (eb - 896 - ex);  // q = m^2 2^sh; above -48 since q >= 1
      bk = int(key >> 19) + (896 << 4) - base + 1;
      return sh >= 0 ? m2 << sh : m2 >> -sh;
    }
  }
  const unsigned long long wide = KeyT<T>::wide(key);
  bk = int(wide >> 48) - base + 1;
  return qval<T>(wide, eb);
}

// A matrix of `entries` stored values (row lists; a flat array's nnz_bar is set):
// nnz_bar, e (the biased exponent of b, 1 for a subnormal b), Q = q(b), the
// smallest key with q >= 1 (the key of 2^(e - 31 - 1023)) and the pivot's bucket: a
// power of two fraction below b / sqrt(nnz_bar), so that no rounding lifts it above.
// b = 0, +inf or NaN: no key is summed (tiny = all ones), every q counts as 0.
// Clears the matrix's minimum and candidate count, and sets its candidate region.
__device__ __forceinline__ void prepare_matrix(int m, const SelRows &R, unsigned long long entries,
                                               MatScalars *ms, const SelScratch &sc) {
  const unsigned long long bkey = (unsigned long long)__double_as_longlong(ms[m].b);
  const int64_t nnz = R.rs ? int64_t(entries) : ms[m].nnz_bar;
  sc.minabove[m] = ~0ULL;
  sc.ncand[m] = 0ULL;
  if (m == 0) *sc.overflow = *sc.redo = 0ULL;
  if (R.rs) ms[m].nnz_bar = nnz;
  // the candidate region: the matrix's range of slots, shifted right by cshift
  // when the room is a fraction of the slots, so the regions are disjoint
  sc.cbase[m] = R.rs ? (unsigned long long)(R.rs[R.moff[m]] >> R.cshift) : 0ULL;
  sc.croom[m] = (unsigned long long)(nnz >> R.cshift);
  const int e = int(bkey >> 52);
  if (bkey == 0ULL || e >= 0x7FF) {  // b <= 0 (sign bit) is caught here as well
    ms[m].sel_e = 0;
    ms[m].sel_q = 0ULL;
    ms[m].tiny = ~0ULL;
    ms[m].sel_base = int((bkey & 0x7FFFFFFFFFFFFFFFULL) >> 48);
    return;
  }
  const int eb = e ? e : 1;
  ms[m].sel_e = eb;
  ms[m].sel_q = qval<double>(bkey, eb);
  ms[m].tiny = eb > 32 ? (unsigned long long)(eb - 31) << 52 : 0ULL;
  const int64_t N = nnz > 1 ? nnz : 1;
  const double pivot = __longlong_as_double((long long)bkey) / sqrt(double(N)) * 0.999;
  const int base = int((unsigned long long)__double_as_longlong(pivot) >> 48);
  ms[m].sel_base = pivot < 0x1p-1000 && base > 0 ? base - 1 : base;  // rounding near underflow
}

// prepare_matrix of every matrix, its entries counted and its histogram cleared by a
// cluster or (many small matrices) by a CTA. A flat array is one matrix (R.moff null).
__global__ void __cluster_dims__(RED_C, 1, 1) __launch_bounds__(RED_T)
    k_sel_prepare(int nb, int per, SelRows R, MatScalars *ms, SelScratch sc) {
  after_previous();
  __shared__ unsigned long long s_cnt;  // the matrix's entries (joint: CTA 0's)
  cg::cluster_group cl = cg::this_cluster();
  const int q = int(cl.block_rank());
  auto clear = [&](int m, int first, int step) {
    for (int t = first; t < 2 * NB0; t += step) sc.hist0[size_t(m) * NB0 * 2 + t] = 0ULL;
  };
  auto solo = [&](int m) {
    if (threadIdx.x == 0) s_cnt = 0ULL;
    __syncthreads();
    clear(m, threadIdx.x, RED_T);
    const unsigned long long k =
        seg_entries(R.rs, R.re, R.moff[m], R.moff[m + 1], threadIdx.x, RED_T);
    if (lane_id() == 0 && k) atomicAdd(&s_cnt, k);
    __syncthreads();
    if (threadIdx.x == 0) prepare_matrix(m, R, s_cnt, ms, sc);
  };
  auto joint = [&](int m) {
    if (threadIdx.x == 0) s_cnt = 0ULL;
    cl.sync();
    clear(m, q * RED_T + threadIdx.x, RED_C * RED_T);
    if (R.rs) {
      const unsigned long long k = seg_entries(R.rs, R.re, R.moff[m], R.moff[m + 1],
                                               q * RED_T + threadIdx.x, RED_C * RED_T);
      if (lane_id() == 0 && k) atomicAdd(cl.map_shared_rank(&s_cnt, 0), k);
    }
    cl.sync();
    if (q == 0 && threadIdx.x == 0) prepare_matrix(m, R, s_cnt, ms, sc);
  };
  cluster_each(nb, per, R.moff, blockIdx.x / RED_C, q, solo, joint);
}

// (lo, hi) += (alo, ahi) atomically in memory; exact, order-independent.
__device__ __forceinline__ void add128(unsigned long long *lohi, unsigned long long alo,
                                       unsigned long long ahi) {
  unsigned long long old = atomicAdd(&lohi[0], alo);
  if (old + alo < old) ++ahi;
  if (ahi) atomicAdd(&lohi[1], ahi);
}

// A chunk of consecutive rows, their extents and matrices staged in shared
// memory by one thread per row, so that a warp's loop over the chunk's rows
// waits on the values only, not on the chain row -> matrix -> scalars.
// Rows of inactive matrices are staged empty.
constexpr int RPC = 64;  // most rows of a chunk

struct ChunkRows {
  int64_t b[RPC], e[RPC];
  int m[RPC];
};

// Stages rows [r0, r1) (r1 - r0 <= RPC) and returns the thread's row
// slot (-1 if none) with its matrix in m; the caller adds its own per-row
// scalars, then synchronises.
__device__ __forceinline__ int stage_rows(const SelRows &R, const int *active, int64_t r0,
                                          int64_t r1, ChunkRows &cr, int &m) {
  const int t = threadIdx.x;
  if (t >= r1 - r0) return -1;
  const int64_t r = r0 + t;
  m = row_mat(R, r);
  int64_t b, e;
  row_range(R, r, b, e);
  cr.b[t] = b;
  cr.e[t] = active[m] ? e : b;
  cr.m[t] = m;
  return t;
}

// How a pass over the rows is cut. LPR lanes per row: 8 for the short rows of
// many (four rows per warp at a time), 32 for long rows, and for few rows,
// where the chip is not full anyway and a row's latency counts. A chunk of
// rows is what one CTA stages at a time: 64 rows (two turns of its 8 warps'
// 8-lane groups), or 8 (a row per warp), so that 4096 rows of 4096 entries
// make 512 chunks; as 64 chunks of 8-lane rows the three passes of a filter
// over them took 690, 376 and 276 us, now 66, 43 and 47.
struct SelCut {
  int lpr, rpc;
};
SelCut sel_cut(int64_t nrows, int64_t nvals) {
  // 152 SMs x 8 warps x 8 rows: fewer rows leave warps without one
  const bool wide = nrows < 152 * 64 || nvals / (nrows > 0 ? nrows : 1) >= 512;
  return wide ? SelCut{32, 8} : SelCut{8, RPC};
}

// Adds q to bucket bk of a shared histogram of 96-bit sums kept as three
// 32-bit words: 32-bit shared atomics are native, 64-bit ones are loops.
__device__ __forceinline__ void add96(uint32_t (*h)[NB0], int bk, unsigned long long q) {
  const uint32_t l = uint32_t(q), old = atomicAdd(&h[0][bk], l);
  uint32_t c = old + l < old ? 1u : 0u;
  const uint32_t u = uint32_t(q >> 32), v = u + c;
  c = v < u ? 1u : 0u;
  if (v) {
    const uint32_t old1 = atomicAdd(&h[1][bk], v);
    c += old1 + v < old1 ? 1u : 0u;
  }
  if (c) atomicAdd(&h[2][bk], c);
}

// Level-0 histogram. A warp takes 32 / LPR rows of the CTA's chunk at a time,
// LPR lanes each, neighbouring lanes on neighbouring entries (which have
// similar magnitudes, so they mostly take the same way). Of each entry's key:
// above b, the smallest is kept; below the pivot's bucket, the squares are
// summed in the lane's registers; between, they go to the bucket, in shared
// memory for the chunk's first matrix (almost every row: matrices span many
// chunks), else in the global histogram. Bound by instruction issue.
template <typename T, int LPR>
__global__ void __launch_bounds__(SEL_THREADS)
    k_sel_hist0(SelRows R, int rpc, const int *active, const T *val, const MatScalars *ms,
                SelScratch sc) {
  after_previous();
  using K = typename KeyT<T>::K;
  __shared__ uint32_t s_h[3][NB0];
  __shared__ unsigned long long s_min, s_below[2];
  __shared__ ChunkRows cr;
  __shared__ K s_b[RPC], s_tiny[RPC], s_base[RPC];
  __shared__ int s_eb[RPC], s_top[RPC];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = SEL_THREADS / 32;
  constexpr int U = 4;  // loads in flight per lane
  const int64_t nchunks = (R.nrows + rpc - 1) / rpc;
  for (int64_t c = blockIdx.x; c < nchunks; c += gridDim.x) {
    const int64_t r0 = c * rpc, r1 = min(r0 + rpc, R.nrows);
    for (int t = threadIdx.x; t < 3 * NB0; t += SEL_THREADS) (&s_h[0][0])[t] = 0u;
    if (threadIdx.x == 0) {
      s_min = ~0ULL;
      s_below[0] = s_below[1] = 0ULL;
    }
    int mt = 0;
    const int t = stage_rows(R, active, r0, r1, cr, mt);
    if (t >= 0) {
      s_b[t] = KeyT<T>::floor_key((unsigned long long)__double_as_longlong(ms[mt].b));
      s_tiny[t] = KeyT<T>::ceil_key(ms[mt].tiny);
      s_base[t] = KeyT<T>::ceil_key((unsigned long long)ms[mt].sel_base << 48);
      s_eb[t] = ms[mt].sel_e;
      s_top[t] = ms[mt].sel_base;
    }
    __syncthreads();
    const int m0 = cr.m[0];
    const int g = lane / LPR, gl = lane % LPR;
    const int nr = int(r1 - r0);
    unsigned long long blo = 0, bhi = 0;  // squares below the pivot (matrix m0)
    K mymin = ~K(0);                      // smallest key above b (matrix m0)
    for (int i = warp * (32 / LPR) + g; i < nr; i += nw * (32 / LPR)) {
      const int64_t e1 = cr.e[i];
      const int m = cr.m[i];
      const K bk_ = s_b[i], tiny = s_tiny[i], base = s_base[i];
      const int eb = s_eb[i], top = s_top[i];
      for (int64_t p = cr.b[i] + gl; p < e1; p += U * LPR) {
        T x[U];
#pragma unroll
        for (int u = 0; u < U; ++u) x[u] = p + u * LPR < e1 ? val[p + u * LPR] : T(0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const K key = KeyT<T>::of(x[u]);
          if (key > bk_) {
            if (m == m0)
              mymin = key < mymin ? key : mymin;
            else
              atomicMin(&sc.minabove[m], KeyT<T>::wide(key));
          } else if (key >= tiny && key != 0) {
            int bk;
            const unsigned long long q = q_bucket<T>(key, eb, top, bk);
            if (m == m0) {
              if (key >= base) {
                add96(s_h, bk, q);
              } else {
                blo += q;
                bhi += blo < q ? 1ULL : 0ULL;
              }
            } else {
              add128(sc.hist0 + (size_t(m) * NB0 + (key >= base ? bk : 0)) * 2, q, 0ULL);
            }
          }
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const K y = __shfl_xor_sync(0xffffffffu, mymin, o);
      mymin = y < mymin ? y : mymin;
      const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, blo, o);
      const unsigned long long h2 = __shfl_xor_sync(0xffffffffu, bhi, o);
      blo += l2;
      bhi += h2 + (blo < l2 ? 1ULL : 0ULL);
    }
    if (lane == 0) {
      if (mymin != ~K(0)) atomicMin(&s_min, KeyT<T>::wide(mymin));
      if (blo | bhi) add128(s_below, blo, bhi);
    }
    __syncthreads();
    if (active[m0]) {
      unsigned long long *gh = sc.hist0 + size_t(m0) * NB0 * 2;
      for (int t2 = threadIdx.x; t2 < NB0; t2 += SEL_THREADS) {
        const unsigned long long lo = s_h[0][t2] | ((unsigned long long)s_h[1][t2] << 32);
        if (lo | s_h[2][t2]) add128(gh + 2 * t2, lo, s_h[2][t2]);
      }
      if (threadIdx.x == 0) {
        if (s_below[0] | s_below[1]) add128(gh, s_below[0], s_below[1]);
        if (s_min != ~0ULL) atomicMin(&sc.minabove[m0], s_min);
      }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void u128_add(unsigned long long &lo, unsigned long long &hi,
                                         unsigned long long alo, unsigned long long ahi) {
  unsigned long long o = lo;
  lo += alo;
  hi += ahi + (lo < o ? 1ULL : 0ULL);
}

// (hi, lo) > Q ?
__device__ __forceinline__ bool exceeds(unsigned long long lo, unsigned long long hi,
                                        unsigned long long Q) {
  return hi != 0ULL || lo > Q;
}

// The first of nbk buckets (128-bit sums h[2c], h[2c+1]) at which the running
// sum, started at (lo, hi), exceeds Q = q(b), found by one warp: 32 buckets at a
// time, lane c of a round holding bucket c and an inclusive prefix sum over
// the round by shuffles. The sums are exact integers, so the crossing is the
// one a serial walk finds. Returns the bucket (or -1, with (lo, hi) the total)
// and leaves in (lo, hi) the sum of the buckets below it.
__device__ __forceinline__ int warp_crossing(const unsigned long long *h, int nbk,
                                             unsigned long long Q, unsigned long long &lo,
                                             unsigned long long &hi) {
  const int lane = threadIdx.x & 31;
  for (int c0 = 0; c0 < nbk; c0 += 32) {
    const int c = c0 + lane;
    const unsigned long long blo = c < nbk ? h[2 * c] : 0ULL, bhi = c < nbk ? h[2 * c + 1] : 0ULL;
    unsigned long long plo = blo, phi = bhi;  // inclusive prefix of the round
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long ulo = __shfl_up_sync(0xffffffffu, plo, o);
      const unsigned long long uhi = __shfl_up_sync(0xffffffffu, phi, o);
      if (lane >= o) u128_add(plo, phi, ulo, uhi);
    }
    unsigned long long rlo = lo, rhi = hi;
    u128_add(rlo, rhi, plo, phi);
    const unsigned over = __ballot_sync(0xffffffffu, c < nbk && exceeds(rlo, rhi, Q));
    if (over) {
      const int f = __ffs(over) - 1;
      // the sum below bucket f: start + inclusive prefix of f - h[f]
      unsigned long long elo = rlo - blo, ehi = rhi - bhi - (rlo < blo ? 1ULL : 0ULL);
      lo = __shfl_sync(0xffffffffu, elo, f);
      hi = __shfl_sync(0xffffffffu, ehi, f);
      return c0 + f;
    }
    lo = __shfl_sync(0xffffffffu, rlo, 31);
    hi = __shfl_sync(0xffffffffu, rhi, 31);
  }
  return -1;
}

// One warp per matrix: the level-0 bucket where the exact sums cross Q (never
// the sum below the pivot, bucket 0).
__global__ void k_sel_find0(int nb, const int *active, const MatScalars *ms, SelScratch sc) {
  after_previous();
  const int m = int((int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (m >= nb) return;
  SelState st = {};
  if (active[m]) {
    const unsigned long long bkey = (unsigned long long)__double_as_longlong(ms[m].b);
    const int base = ms[m].sel_base;
    const int nbk = min(NB0, int(bkey >> 48) - base + 2);  // up to b's own bucket
    unsigned long long lo = 0, hi = 0;
    const int c = warp_crossing(sc.hist0 + size_t(m) * NB0 * 2, nbk, ms[m].sel_q, lo, hi);
    if (c >= 0) {
      st.found = 1;
      st.prefix = (unsigned long long)(base + c - 1) << 48;
      st.below_lo = st.below0_lo = lo;
      st.below_hi = st.below0_hi = hi;
    }
  }
  if (lane == 0) sc.st[m] = st;
}

// Square sums of a row's dropped entries: 32 partial sums, of every 32nd entry
// of the row, 32 / W on each of its W lanes (lane gl holds gl, gl + W, ..), added
// 16 apart, 8 apart and so on, the same additions for every W. FP32 values exactly in
// FP32 pairs (scaled by 2^96), FP64 values by FMA.
template <typename T, int W>
struct DropSum;
template <int W>
struct DropSum<float, W> {
  static constexpr int N = 32 / W;
  float hi[N] = {}, lo[N] = {};
  __device__ __forceinline__ void add(float x, int u) { ff_add_sq48(x, hi[u], lo[u]); }
  __device__ __forceinline__ double total() {  // valid in every lane of the W
    bool any = false;
#pragma unroll
    for (int u = 0; u < N; ++u) any = any || hi[u] != 0.0f;
    if (!__any_sync(0xffffffffu, any)) return 0.0;
#pragma unroll
    for (int h = N / 2; h > 0; h >>= 1)
#pragma unroll
      for (int u = 0; u < h; ++u) ff_add(hi[u], lo[u], hi[u + h], lo[u + h]);
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) {
      const float h2 = __shfl_xor_sync(0xffffffffu, hi[0], o, W);
      const float l2 = __shfl_xor_sync(0xffffffffu, lo[0], o, W);
      ff_add(hi[0], lo[0], h2, l2);
    }
    return (double(hi[0]) + double(lo[0])) * 0x1p-96;  // exact scaling, one rounding as ldexp
  }
};
template <int W>
struct DropSum<double, W> {
  static constexpr int N = 32 / W;
  double d[N] = {};
  __device__ __forceinline__ void add(double x, int u) { d[u] = __fma_rn(x, x, d[u]); }
  __device__ __forceinline__ double total() {
    bool any = false;
#pragma unroll
    for (int u = 0; u < N; ++u) any = any || d[u] != 0.0;
    if (!__any_sync(0xffffffffu, any)) return 0.0;  // FP64 adds only for rows that drop
#pragma unroll
    for (int h = N / 2; h > 0; h >>= 1)
#pragma unroll
      for (int u = 0; u < h; ++u) d[u] += d[u + h];
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) d[0] += __shfl_xor_sync(0xffffffffu, d[0], o, W);
    return d[0];
  }
};

constexpr int EX_U = 4;  // entries per lane of a row loaded at once

// Candidates: the entries of the crossing bucket (top 16 bits of the key equal
// to the prefix, 0 < key <= b), appended to the matrix's region with one atomic
// per row's lanes and load round.
// With cnt (the filter of a solve) the same pass also counts, per row, what
// does not depend on where tau falls inside the crossing bucket: entries
// above the bucket or above b are kept (cnt[r]); entries below it are
// dropped, their squares summed into dropped[r] as in k_filter_count. A
// matrix without a crossing already has its tau (the smallest key above b),
// so every entry is decided here. k_sel_digits adds the kept candidates
// once tau is final; the dropped candidates' squares come from the select's
// exact sums (k_drop_sums). Rows of inactive matrices get 0 and 0.
// Per row two bounds on the keys decide: below s_lo an entry is dropped, from
// s_up on it is kept, between it is a candidate (a NaN is dropped).
template <typename T, int LPR>
__global__ void __launch_bounds__(SEL_THREADS, 4)
    k_sel_extract(SelRows R, int rpc, const int *active, const T *val, const MatScalars *ms,
                  SelScratch sc, int64_t *cnt, double *dropped, const unsigned long long *run) {
  after_previous();
  if (run && *run == 0ULL) return;
  using K = typename KeyT<T>::K;
  __shared__ ChunkRows cr;
  __shared__ K s_lo[RPC], s_up[RPC];
  __shared__ int s_found[RPC];
  __shared__ unsigned long long s_cbase[RPC], s_room[RPC];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = SEL_THREADS / 32;
  const int64_t nchunks = (R.nrows + rpc - 1) / rpc;
  for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
    const int64_t r0 = ch * rpc, r1 = min(r0 + rpc, R.nrows);
    __syncthreads();  // the previous chunk's rows are read
    int mt = 0;
    const int t = stage_rows(R, active, r0, r1, cr, mt);
    if (t >= 0) {
      const bool found = active[mt] && sc.st[mt].found != 0;
      s_found[t] = found;
      if (found) {
        const unsigned long long lo = sc.st[mt].prefix, next = lo + (1ULL << 48);
        s_lo[t] = KeyT<T>::ceil_key(lo);
        const K top = KeyT<T>::ceil_key(next);
        const K above = KeyT<T>::floor_key((unsigned long long)__double_as_longlong(ms[mt].b)) + 1;
        s_up[t] = above < top ? above : top;
        s_cbase[t] = sc.cbase[mt];
        s_room[t] = sc.croom[mt];
      } else {
        const unsigned long long above = sc.minabove[mt];  // tau without a crossing
        s_lo[t] = s_up[t] = KeyT<T>::ceil_key(above == ~0ULL ? INF_KEY : above);
      }
    }
    __syncthreads();
    const int g = lane / LPR, gl = lane % LPR;
    const unsigned gmask = LPR == 32 ? 0xffffffffu : ((1u << (LPR & 31)) - 1u) << (g * LPR);
    const unsigned below = gmask & ((1u << lane) - 1u);
    const int nr = int(r1 - r0);
    for (int i0 = warp * (32 / LPR); i0 < nr; i0 += nw * (32 / LPR)) {
      const int i = i0 + g;
      const bool has = i < nr && (cnt || s_found[i] != 0);
      const int64_t r = r0 + i;
      // empty for inactive matrices: 0 and 0 written
      const int64_t e0 = has ? cr.b[i] : 0, e1 = has ? cr.e[i] : 0;
      const K lo = has ? s_lo[i] : K(0), up = has ? s_up[i] : K(0);
      int c = 0;
      DropSum<T, LPR> ds;
      static_assert(EX_U % (32 / LPR) == 0, "entry u of a lane belongs to partial sum u % N");
      for (int64_t p0 = e0;; p0 += LPR * EX_U) {
        // the warp's rows together (loops of their own would run one by one)
        if (!__any_sync(0xffffffffu, p0 < e1)) break;
        T x[EX_U];
#pragma unroll
        for (int u = 0; u < EX_U; ++u) {
          const int64_t p = p0 + LPR * u + gl;
          x[u] = p < e1 ? val[p] : T(0);  // a zero is neither counted nor dropped
        }
        unsigned take[EX_U];
        int n = 0;
#pragma unroll
        for (int u = 0; u < EX_U; ++u) {
          const K key = KeyT<T>::of(x[u]);
          const bool cand = key >= lo && key < up && key != 0;
          take[u] = __ballot_sync(0xffffffffu, cand) & gmask;
          n += __popc(take[u]);
          if (!cnt || cand || key == 0) continue;
          if (key >= up && key <= KeyT<T>::kInf)
            ++c;
          else
            ds.add(x[u], u % ds.N);
        }
        if (n) {  // the row's candidates of this round, in one reservation
          const int m = cr.m[i];
          unsigned long long at = 0;
          if (gl == 0) at = atomicAdd(&sc.ncand[m], (unsigned long long)n);
          at = __shfl_sync(gmask, at, g * LPR);
          const unsigned long long cb = s_cbase[i], room = s_room[i];
#pragma unroll
          for (int u = 0; u < EX_U; ++u) {
            if ((take[u] >> lane) & 1u) {
              const unsigned long long slot = at + __popc(take[u] & below);
              if (slot < room) {
                sc.cand[cb + slot] = KeyT<T>::wide(KeyT<T>::of(x[u]));
                sc.cand_r[cb + slot] = int(r);
              } else {  // past the room: the caller selects again with more
                *sc.overflow = 1ULL;
              }
            }
            at += __popc(take[u]);
          }
        }
      }
      if (!cnt) continue;
#pragma unroll
      for (int o = LPR / 2; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o, LPR);
      const double d = ds.total();
      if (gl == 0 && has) {
        cnt[r] = c;
        dropped[r] = d;
      }
    }
  }
}

// After a first pass with regions of a fraction of the entries (cshift > 0): if
// a matrix had more candidates than its region, the counts, which are complete,
// become the regions of a second pass, as long as they fit the room in all.
// One CTA; only stages above 2^28 slots come here.
constexpr int REG_T = 1024;
__global__ void __launch_bounds__(REG_T) k_sel_regions(int nb, unsigned long long cap,
                                                       SelScratch sc) {
  after_previous();
  __shared__ unsigned long long s[REG_T];
  if (*sc.overflow == 0ULL) return;
  const int t = threadIdx.x, per = (nb - 1) / REG_T + 1;
  const int m0 = min(nb, t * per), m1 = min(nb, m0 + per);
  unsigned long long sum = 0;
  for (int m = m0; m < m1; ++m) sum += sc.ncand[m];
  s[t] = sum;
  __syncthreads();
  for (int o = 1; o < REG_T; o <<= 1) {  // inclusive prefix sums
    const unsigned long long y = t >= o ? s[t - o] : 0ULL;
    __syncthreads();
    s[t] += y;
    __syncthreads();
  }
  if (s[REG_T - 1] > cap) return;  // the caller selects again with room for every value
  unsigned long long at = s[t] - sum;
  for (int m = m0; m < m1; ++m) {
    const unsigned long long k = sc.ncand[m];
    sc.cbase[m] = at;
    sc.croom[m] = k;
    sc.ncand[m] = 0ULL;
    at += k;
  }
  if (t == 0) {
    *sc.overflow = 0ULL;
    *sc.redo = 1ULL;
  }
}

// sums[m] = the dropped squares of matrix m's rows plus, with the select's
// scratch, those of the dropped candidates: the exact sum of their q
// (the select's sum below tau minus its sum below the crossing bucket) in
// grid steps 2^(2e - 62). A candidate's magnitude is at least b / sqrt(1.1
// nnz) (a bucket spans a factor 2^(1/16)), so its q is above 2^62 / (1.1 nnz)
// and its flooring to an integer is far below the FP64 rounding of the sum.
__device__ __forceinline__ double drop_sum(int m, double sum, const int *active, int exact,
                                           const SelScratch &sc, const MatScalars *ms) {
  if (!(exact && active[m] && sc.st[m].found)) return sum;
  const SelState st = sc.st[m];
  const unsigned long long lo = st.below_lo - st.below0_lo;
  const unsigned long long hi =
      st.below_hi - st.below0_hi - (st.below_lo < st.below0_lo ? 1ULL : 0ULL);
  const double qs = __fma_rn(double(hi), 18446744073709551616.0, double(lo));
  return __dadd_rn(sum, ldexp(qs, 2 * (ms[m].sel_e - 1023) - 62));
}

__global__ void __cluster_dims__(RED_C, 1, 1) __launch_bounds__(RED_LANES)
    k_drop_sums(int nb, int per, const int64_t *moff, const double *dropped, const int *active,
                int exact, SelScratch sc, const MatScalars *ms, double *sums) {
  after_previous();
  __shared__ double sm[RED_T];
  cg::cluster_group cl = cg::this_cluster();
  const int q = int(cl.block_rank()), t = q * RED_LANES + threadIdx.x;
  auto solo = [&](int m) {
    seg_sum_solo(sm, dropped, 1, 0, moff[m], moff[m + 1]);
    if (threadIdx.x == 0) sums[m] = drop_sum(m, sm[0], active, exact, sc, ms);
  };
  auto joint = [&](int m) {
    cl.sync();  // CTA 0 has started, and read its sums: its shared memory may be written
    *cl.map_shared_rank(&sm[t], 0) = seg_partial(dropped, 1, 0, moff[m], moff[m + 1], t);
    cl.sync();
    if (q != 0) return;
    seg_tree(sm);
    if (threadIdx.x == 0) sums[m] = drop_sum(m, sm[0], active, exact, sc, ms);
  };
  cluster_each(nb, per, moff, blockIdx.x / RED_C, q, solo, joint);
}

// The digits below the crossing bucket, tau and the kept candidates' counts of
// a matrix, in one cluster of DG_C CTAs: per digit every CTA sums its part of
// the candidates into a shared histogram, CTA 0 adds the histograms over
// distributed shared memory and finds the crossing. The candidates that match
// the first digit are kept in shared memory for the later ones when they fit.
// LEVELS: 6 digits cover the 48 bits of an FP64 key, 3 those of an FP32 value
// (its FP64 key's low 29 bits are zero). Up to DG_ONE candidates one CTA works
// alone, and up to DG_T it finds tau without digits, by every candidate's sum of
// the candidates up to its own key. Of many matrices a cluster has several (see
// seg.cuh): those that one CTA takes alone side by side, then the others one after
// another. Twelve launches over all candidates did this before: 6 x (5.0 + 5.2)
// us for one matrix of 500 rows, now 13 in all.
constexpr int DG_C = 8, DG_T = 512, DG_KEEP = 2048, DG_ONE = 4096;
static_assert(DG_C == RED_C, "clusters and groups of seg.cuh");
static_assert(DG_T <= 2 * NDIG && DG_T <= DG_KEEP && DG_T <= DG_ONE, "the short path's arrays");
struct DgShared {
  uint32_t h[3][NDIG];
  unsigned long long sum[NDIG * 2];
  unsigned long long keep[DG_KEEP];
  unsigned long long s_res[3];  // CTA 0: prefix and sum below it
  int s_nkeep;
};

// Matrix m, which has a crossing, by nc CTAs (1 or the cluster's DG_C). prefix, lo,
// hi: the key bits known so far and the sum below them; cb: the first of its `total`
// candidates.
template <int LEVELS>
__device__ __forceinline__ void digits_matrix(int m, int nc, int rank, unsigned long long prefix,
                                              unsigned long long lo, unsigned long long hi,
                                              unsigned long long cb, unsigned long long total,
                                              DgShared &sh, const SelScratch &sc, MatScalars *ms,
                                              int64_t *cnt) {
  auto &h = sh.h;
  auto &sum = sh.sum;
  auto &keep = sh.keep;
  auto &s_res = sh.s_res;
  int &s_nkeep = sh.s_nkeep;
  cg::cluster_group cl = cg::this_cluster();
  const int tid = threadIdx.x;
  const int eb = ms[m].sel_e;
  const unsigned long long Q = ms[m].sel_q;
  if (total <= DG_T) {  // one CTA alone: thread i sums the squares of the keys <= key i
    const int n = int(total);
    const unsigned long long key = tid < n ? sc.cand[cb + tid] : ~0ULL;
    keep[tid] = key;
    sum[tid] = tid < n ? qval<double>(key, eb) : 0ULL;
    if (tid == 0) s_res[0] = ~0ULL;
    __syncthreads();
    unsigned long long le_lo = lo, le_hi = hi, lt_lo = lo, lt_hi = hi;
    for (int i = 0; i < n; ++i) {
      const unsigned long long k = keep[i], q = sum[i];
      if (k <= key) u128_add(le_lo, le_hi, q, 0ULL);
      if (k < key) u128_add(lt_lo, lt_hi, q, 0ULL);
    }
    const bool over = tid < n && exceeds(le_lo, le_hi, Q);
    if (over) atomicMin(&s_res[0], key);
    __syncthreads();
    const unsigned long long tau = s_res[0];
    if (over && key == tau) {  // every thread of this key writes the same
      ms[m].tau = __longlong_as_double((long long)tau);
      sc.st[m].prefix = tau;
      sc.st[m].below_lo = lt_lo;
      sc.st[m].below_hi = lt_hi;
    }
    if (cnt && tid < n && keep_key(key, tau))
      atomicAdd(reinterpret_cast<unsigned long long *>(cnt + sc.cand_r[cb + tid]), 1ULL);
    return;
  }
  bool local = false;  // the survivors of the first digit are in keep
  for (int level = 0; level < LEVELS; ++level) {
    const int shift = 40 - 8 * level;
    for (int t = tid; t < 3 * NDIG; t += DG_T) (&h[0][0])[t] = 0u;
    if (level == 1 && tid == 0) s_nkeep = 0;
    __syncthreads();
    auto digit = [&](unsigned long long key) {
      if ((key >> (shift + 8)) != (prefix >> (shift + 8))) return false;
      const unsigned long long q = qval<double>(key, eb);
      const int d = int((key >> shift) & 255ULL);
      const uint32_t l = uint32_t(q), old = atomicAdd(&h[0][d], l);
      uint32_t c = old + l < old ? 1u : 0u;
      const uint32_t u = uint32_t(q >> 32), v = u + c;
      c = v < u ? 1u : 0u;
      if (v) {
        const uint32_t old1 = atomicAdd(&h[1][d], v);
        c += old1 + v < old1 ? 1u : 0u;
      }
      if (c) atomicAdd(&h[2][d], c);
      return true;
    };
    if (local) {
      for (int i = tid; i < s_nkeep; i += DG_T) digit(keep[i]);
    } else {
#pragma unroll 4
      for (unsigned long long i = (unsigned long long)rank * DG_T + tid; i < total;
           i += (unsigned long long)nc * DG_T) {
        const unsigned long long key = sc.cand[cb + i];
        if (digit(key) && level == 1) {
          const int at = atomicAdd(&s_nkeep, 1);
          if (at < DG_KEEP) keep[at] = key;
        }
      }
    }
    if (nc > 1) cl.sync(); else __syncthreads();
    if (level == 1) local = s_nkeep <= DG_KEEP;
    if (rank == 0) {
      if (tid < NDIG) {
        unsigned long long a = 0, b = 0;
        for (int q = 0; q < nc; ++q) {
          const uint32_t *hq = nc > 1 ? cl.map_shared_rank(&h[0][0], q) : &h[0][0];
          const unsigned long long w =
              hq[tid] | ((unsigned long long)hq[NDIG + tid] << 32);
          a += w;
          b += hq[2 * NDIG + tid] + (a < w ? 1ULL : 0ULL);
        }
        sum[2 * tid] = a;
        sum[2 * tid + 1] = b;
      }
      __syncthreads();
      if (tid < 32) {
        unsigned long long l2 = lo, h2 = hi;
        const int d = warp_crossing(sum, NDIG, Q, l2, h2);
        if (tid == 0) {
          s_res[0] = d >= 0 ? prefix | ((unsigned long long)d << shift) : prefix;
          s_res[1] = d >= 0 ? l2 : lo;
          s_res[2] = d >= 0 ? h2 : hi;
        }
      }
    }
    if (nc > 1) cl.sync(); else __syncthreads();
    const unsigned long long *res = nc > 1 ? cl.map_shared_rank(s_res, 0) : s_res;
    prefix = res[0];
    lo = res[1];
    hi = res[2];
  }
  if (rank == 0 && tid == 0) {
    ms[m].tau = __longlong_as_double((long long)prefix);
    sc.st[m].prefix = prefix;
    sc.st[m].below_lo = lo;
    sc.st[m].below_hi = hi;
  }
  // the kept candidates (key >= tau) into their rows' counts
  if (cnt) {
    for (unsigned long long i = (unsigned long long)rank * DG_T + tid; i < total;
         i += (unsigned long long)nc * DG_T)
      if (keep_key(sc.cand[cb + i], prefix))
        atomicAdd(reinterpret_cast<unsigned long long *>(cnt + sc.cand_r[cb + i]), 1ULL);
  }
  if (nc > 1) cl.sync();  // CTA 0's shared memory is read until here
}

// MANY: RED_C matrices per cluster (see seg.cuh), else one.
template <int LEVELS, bool MANY>
__global__ void __cluster_dims__(DG_C, 1, 1) __launch_bounds__(DG_T, 3)
    k_sel_digits(int nb, const int *active, SelScratch sc, MatScalars *ms, int64_t *cnt) {
  after_previous();
  __shared__ DgShared sh;
  const int rank = int(cg::this_cluster().block_rank()), cluster = blockIdx.x / DG_C;
  constexpr int PER = MANY ? RED_C : 1;
  // i = -1: this CTA's own matrix, if one CTA does; then those of the whole cluster, the
  // same m for all its CTAs. A lone matrix (i = 0) is either.
  for (int i = MANY ? -1 : 0; i < PER; ++i) {
    const int m = cluster * PER + (i < 0 ? rank : i);
    if (m >= nb) continue;
    // loaded together, before any of them is looked at
    const int act = active[m];
    const SelState st = sc.st[m];
    const unsigned long long total = min(sc.ncand[m], sc.croom[m]), cb = sc.cbase[m];
    if (!act) continue;
    const bool solo = total <= DG_ONE, mine = MANY ? i < 0 : rank == 0;
    if (!st.found) {
      if (mine && threadIdx.x == 0) {
        const unsigned long long k = sc.minabove[m];
        ms[m].tau = k == ~0ULL ? __longlong_as_double(0x7ff0000000000000LL)
                               : __longlong_as_double((long long)k);
      }
      continue;
    }
    if (solo ? !mine : i < 0) continue;
    if (MANY && i >= 0) __syncthreads();  // sh is free
    digits_matrix<LEVELS>(m, solo ? 1 : DG_C, solo ? 0 : rank, st.prefix, st.below_lo, st.below_hi,
                          cb, total, sh, sc, ms, cnt);
  }
}

// ------------------------------------------------------------ filter
__global__ void k_filter_count(int64_t n, const int32_t *seg, const int *active,
                               const int64_t *rs, const int64_t *re, const void *val, int f32,
                               const MatScalars *ms, int64_t *cnt, double *dropped) {
  after_previous();
  int lane = lane_id();
  int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = warp; r < n; r += nwarps) {
    int m = seg[r];
    const unsigned long long tkey = (unsigned long long)__double_as_longlong(ms[m].tau);
    int c = 0;
    double d2 = 0.0;
    if (active[m] && f32) {
      const float *v = static_cast<const float *>(val);
      float hi = 0.0f, lo = 0.0f;  // dropped squares, scaled by 2^96
      const int64_t pe = re[r];
#pragma unroll 4
      for (int64_t p = rs[r] + lane; p < pe; p += 32) {
        const float x = v[p];
        const unsigned long long key = key_f32(x);
        if (keep_key(key, tkey))
          ++c;
        else if (key != 0ULL)
          ff_add_sq48(x, hi, lo);
      }
      c = __reduce_add_sync(0xffffffffu, c);
      if (__any_sync(0xffffffffu, hi != 0.0f)) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
          const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
          ff_add(hi, lo, h2, l2);
        }
        if (lane == 0) d2 = (double(hi) + double(lo)) * 0x1p-96;  // exact scaling, one rounding as ldexp
      }
    } else if (active[m]) {
      const double *v = static_cast<const double *>(val);
      const int64_t pe = re[r];
#pragma unroll 4
      for (int64_t p = rs[r] + lane; p < pe; p += 32) {
        double x = v[p];
        if (keep_key(key_f64(x), tkey))
          ++c;
        else
          d2 = __fma_rn(x, x, d2);
      }
      c = __reduce_add_sync(0xffffffffu, c);
      if (__any_sync(0xffffffffu, d2 != 0.0)) {  // FP64 adds only for rows that drop
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
      }
    }
    if (lane == 0) {
      cnt[r] = c;
      dropped[r] = d2;
    }
  }
}

template <typename T, int LPR>
__global__ void __launch_bounds__(SEL_THREADS)
    k_filter_write(int64_t n, int rpc, const int32_t *seg, const int *active, const int64_t *rs,
                   const int64_t *re, const int32_t *col, const T *val, const MatScalars *ms,
                   const int64_t *orp, int32_t *ocol, T *oval) {
  after_previous();
  using K = typename KeyT<T>::K;
  __shared__ ChunkRows cr;
  __shared__ int64_t s_out[RPC], s_oend[RPC];
  __shared__ K s_tkey[RPC];
  const int lane = lane_id(), warp = threadIdx.x >> 5, nw = SEL_THREADS / 32;
  SelRows R{};
  R.nrows = n;
  R.seg = seg;
  R.rs = rs;
  R.re = re;
  const int64_t nchunks = (n + rpc - 1) / rpc;
  for (int64_t ch = blockIdx.x; ch < nchunks; ch += gridDim.x) {
    const int64_t r0 = ch * rpc, r1 = min(r0 + rpc, n);
    __syncthreads();  // the previous chunk's rows are read
    int mt = 0;
    const int t = stage_rows(R, active, r0, r1, cr, mt);
    if (t >= 0) {
      s_out[t] = orp[r0 + t];
      s_oend[t] = orp[r0 + t + 1];
      s_tkey[t] = KeyT<T>::ceil_key((unsigned long long)__double_as_longlong(ms[mt].tau));
    }
    __syncthreads();
    // LPR lanes per row, 32 / LPR rows of the chunk per warp at a time
    const int g = lane / LPR, gl = lane % LPR;
    const unsigned gmask = LPR == 32 ? 0xffffffffu : ((1u << (LPR & 31)) - 1u) << (g * LPR);
    const unsigned below = gmask & ((1u << lane) - 1u);
    const int nr = int(r1 - r0);
    for (int i0 = warp * (32 / LPR); i0 < nr; i0 += nw * (32 / LPR)) {
      const int i = i0 + g;
      const bool has = i < nr;
      // the row's room from the counts; the same rule decides both, and the
      // bound keeps a write inside the row whatever the values are
      const K tkey = has ? s_tkey[i] : ~K(0);
      int64_t out = has ? s_out[i] : 0;
      const int64_t oend = has ? s_oend[i] : 0, b = has ? cr.b[i] : 0, e = has ? cr.e[i] : 0;
      for (int64_t p0 = b;; p0 += LPR * EX_U) {
        if (!__any_sync(0xffffffffu, p0 < e)) break;  // every row of the warp done
        T x[EX_U];
        int32_t c[EX_U];
#pragma unroll
        for (int u = 0; u < EX_U; ++u) {
          const int64_t p = p0 + LPR * u + gl;
          x[u] = p < e ? val[p] : T(0);  // a zero is never kept
          c[u] = p < e ? col[p] : 0;
        }
#pragma unroll
        for (int u = 0; u < EX_U; ++u) {
          const K key = KeyT<T>::of(x[u]);
          const bool keep = key >= tkey && key != 0 && key <= KeyT<T>::kInf;
          const unsigned gm = __ballot_sync(0xffffffffu, keep) & gmask;
          const int64_t pos = out + __popc(gm & below);
          if (keep && pos < oend) {
            ocol[pos] = c[u];
            oval[pos] = x[u];
          }
          out += __popc(gm);
        }
      }
    }
  }
}

int grid_for(int64_t items, int per_block, int cap = 152 * 16) {
  int64_t g = (items + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return int(g);
}

__global__ void k_store_nnz_bar(int nb, const int64_t *nnz, MatScalars *ms) {
  after_previous();
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m < nb) ms[m].nnz_bar = nnz[m];
}

}  // namespace

void launch_store_nnz_bar(int nb, const int64_t *nnz, MatScalars *ms, cudaStream_t s) {
  launch_next(k_store_nnz_bar, (nb + 127) / 128, 128, 0, s, nb, nnz, ms);
}

void launch_select_bound(int nb, const int *active, MatScalars *ms, cudaStream_t s) {
  launch_next(k_select_bound, (nb + 127) / 128, 128, 0, s, nb, active, ms);
}

const unsigned long long *select_overflow(void *scratch, int nb) {
  return carve(scratch, nb, 1).overflow;
}

// f(lanes per row as a constant, rows per chunk, CTAs) of a pass over the rows
template <typename F>
static void sel_pass(int64_t nrows, int64_t nvals, F f) {
  if (nrows <= 0) return;
  const SelCut c = sel_cut(nrows, nvals);
  const int g = grid_for(nrows, c.rpc, 152 * 8);
  if (c.lpr == 32)
    f(std::integral_constant<int, 32>{}, c.rpc, g);
  else
    f(std::integral_constant<int, 8>{}, c.rpc, g);
}

template <typename T>
static void select_exact(int nb, const SelRows &R, int64_t nvals, int64_t cand_cap,
                         const int *active, const T *val, MatScalars *ms, const SelScratch &sc,
                         int64_t *cnt, double *dropped, cudaStream_t s) {
  {
    ProfScope ps(KC_SEL_HIST, s, 0.0, 0.0);
    launch_next(k_sel_prepare, cluster_ctas(nb), RED_T, 0, s, nb, cluster_matrices(nb), R, ms, sc);
    sel_pass(R.nrows, nvals, [&](auto lpr, int rpc, int g) {
      launch_next(k_sel_hist0<T, lpr.value>, g, SEL_THREADS, 0, s, R, rpc, active, val, ms, sc);
    });
    launch_next(k_sel_find0, (nb + 3) / 4, 128, 0, s, nb, active, ms, sc);
  }
  {
    ProfScope ps(KC_SEL_EXTRACT, s, 0.0, 0.0);
    auto extract = [&](const unsigned long long *run) {
      sel_pass(R.nrows, nvals, [&](auto lpr, int rpc, int g) {
        launch_next(k_sel_extract<T, lpr.value>, g, SEL_THREADS, 0, s, R, rpc, active, val, ms, sc,
                    cnt, dropped, run);
      });
    };
    extract(nullptr);
    if (R.cshift > 0) {
      launch_next(k_sel_regions, 1, REG_T, 0, s, nb, (unsigned long long)cand_cap, sc);
      extract(sc.redo);
    }
  }
  ProfScope ps(KC_SEL_DIGITS, s, 0.0, 0.0);
  constexpr int LEVELS = sizeof(T) == 4 ? 3 : 6;
  if (cluster_matrices(nb) > 1)
    launch_next(k_sel_digits<LEVELS, true>, cluster_ctas(nb), DG_T, 0, s, nb, active, sc, ms, cnt);
  else
    launch_next(k_sel_digits<LEVELS, false>, cluster_ctas(nb), DG_T, 0, s, nb, active, sc, ms, cnt);
}

void launch_select_exact(int nb, const SelRows &R, int64_t nvals, int64_t cand_cap,
                         const int *active, const void *val, int val_f32, MatScalars *ms,
                         void *scratch, int64_t *cnt, double *dropped, cudaStream_t s) {
  const SelScratch sc = carve(scratch, nb, cand_cap);
  if (val_f32)
    select_exact<float>(nb, R, nvals, cand_cap, active, static_cast<const float *>(val), ms, sc,
                        cnt, dropped, s);
  else
    select_exact<double>(nb, R, nvals, cand_cap, active, static_cast<const double *>(val), ms, sc,
                         cnt, dropped, s);
}

void launch_drop_sums(int nb, const int64_t *moff, const double *dropped, const int *active,
                      void *scratch, const MatScalars *ms, double *sums, cudaStream_t s) {
  if (nb == 0) return;
  const SelScratch sc = scratch ? carve(scratch, nb, 1) : SelScratch{};
  launch_next(k_drop_sums, cluster_ctas(nb), RED_LANES, 0, s, nb, cluster_matrices(nb), moff, dropped,
              active, scratch ? 1 : 0, sc, ms, sums);
}

void launch_filter_count(int64_t n, const int32_t *seg, const int *active, const int64_t *rs,
                         const int64_t *re, const void *val, int val_f32, const MatScalars *ms,
                         int64_t *cnt, double *dropped, cudaStream_t s) {
  if (n == 0) return;
  launch_next(k_filter_count, grid_for(n, 8), 256, 0, s, n, seg, active, rs, re, val, val_f32, ms,
              cnt, dropped);
}

void launch_filter_write(int64_t n, int64_t nvals, const int32_t *seg, const int *active,
                         const int64_t *rs, const int64_t *re, const int32_t *col, const void *val,
                         int val_f32, const MatScalars *ms, const int64_t *orp, int32_t *ocol,
                         void *oval, cudaStream_t s) {
  sel_pass(n, nvals, [&](auto lpr, int rpc, int g) {
    if (val_f32)
      launch_next(k_filter_write<float, lpr.value>, g, SEL_THREADS, 0, s, n, rpc, seg, active, rs,
                  re, col, static_cast<const float *>(val), ms, orp, ocol,
                  static_cast<float *>(oval));
    else
      launch_next(k_filter_write<double, lpr.value>, g, SEL_THREADS, 0, s, n, rpc, seg, active, rs,
                  re, col, static_cast<const double *>(val), ms, orp, ocol,
                  static_cast<double *>(oval));
  });
}

}  // namespace sgn
