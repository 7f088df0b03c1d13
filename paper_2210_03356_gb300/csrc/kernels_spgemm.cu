// Row-wise sparse products of the Newton-Schulz step (steps a2 and a3):
//   MODE_SQUARE:  T = X X, plus per-row partial sums for ||T - I||_F and ||X||_F
//   MODE_UPDATE:  Xbar = 1.5 X - 0.5 X T   (= 1/2 X (3I - X^2), Alg. 3.2.1 step 3)
//
// Operands are row ranges [rs[i], re[i]) into (col, val) with ascending
// columns, so both compact CSR (rs = rowptr, re = rowptr + 1) and the slotted
// outputs of earlier products can be read.
//
// Row i of C = A B is accumulated in shared memory over its column range
// [lo_i, lo_i + len_i) (union of the ranges of the rows B_k, k in A_i), indexed
// by column - lo_i, so the output comes out in ascending column order without
// hashing or sorting. Rows with len <= WARP_W go to one warp each; the columns
// of wider rows are split over the windows of one or several warps, each of
// which runs through all k on its own columns.
//
// No symbolic pass: each output row gets a slot of ub_i = min(len_i, work_i)
// entries (work_i = multiply-adds of the row, plus the row of A itself in
// MODE_UPDATE), which bounds its number of distinct columns; the numeric
// kernel writes the row at the start of its slot and records where it ends.
//
// Accumulation order: the k of A_i are visited in ascending order, one at a
// time; within one k the lanes (threads) stride over the entries of B_k,
// whose columns are distinct, so no two lanes touch the same slot, and a
// barrier separates consecutive k. Every slot therefore receives its
// products in ascending k with one fused multiply-add each, starting from
// +0: the result is the same bit for bit on every run and launch shape.
#include <climits>

#include "common.cuh"
#include "kernels.h"

namespace sgn {

namespace {

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }

// 1.5 x - 0.5 p with each product and the difference rounded once.
__device__ __forceinline__ double ns_combine(double x, double p) {
  return __dsub_rn(__dmul_rn(1.5, x), __dmul_rn(0.5, p));
}
__device__ __forceinline__ float ns_combine(float x, float p) {
  return __fsub_rn(__fmul_rn(1.5f, x), __fmul_rn(0.5f, p));
}

// Sum of squares of the values of one type, in FP64 precision. For float
// values it avoids FP64 arithmetic (1/64 rate on this part): v^2 = p + e
// exactly (p = v*v rounded, e = fma(v, v, -p)), accumulated as an unevaluated
// float pair with an error-free two-sum, so the sum carries ~48 bits.
template <typename T>
struct SqAcc;
template <>
struct SqAcc<double> {
  double s = 0.0;
  __device__ __forceinline__ void add_sq(double v) { s = __fma_rn(v, v, s); }
  __device__ __forceinline__ void merge(const SqAcc &o) { s += o.s; }
  __device__ __forceinline__ SqAcc from_lane_xor(unsigned mask, int o) const {
    return SqAcc{__shfl_xor_sync(mask, s, o)};
  }
  __device__ __forceinline__ double value() const { return s; }
};
template <>
struct SqAcc<float> {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float a) {
    float t = __fadd_rn(hi, a);
    float bb = __fsub_rn(t, hi);
    float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(t, bb)), __fsub_rn(a, bb));
    hi = t;
    lo = __fadd_rn(lo, err);
  }
  __device__ __forceinline__ void add_sq(float v) {
    float p = __fmul_rn(v, v);
    float e = __fmaf_rn(v, v, -p);
    add(p);
    lo = __fadd_rn(lo, e);
  }
  __device__ __forceinline__ void merge(const SqAcc &o) {  // the same with *this and o exchanged
    const float l = __fadd_rn(lo, o.lo);
    lo = 0.0f;
    add(o.hi);
    lo = __fadd_rn(l, lo);
  }
  __device__ __forceinline__ SqAcc from_lane_xor(unsigned mask, int o) const {
    return SqAcc{__shfl_xor_sync(mask, hi, o), __shfl_xor_sync(mask, lo, o)};
  }
  __device__ __forceinline__ double value() const { return double(hi) + double(lo); }
};

// (t_ii - 1)^2 of the diagonal entry v, 1 where none is stored.
__device__ __forceinline__ double diag_square(bool stored, double v) {
  const double d = stored ? v - 1.0 : -1.0;
  return d * d;
}

// The total of a row's 32 partial sums, 32 / G on each of the G lanes of mask
// (lane gl holds gl, gl + G, ..): added 16 apart, 8 apart and so on, the same
// additions for every G.
template <typename T, int G>
__device__ __forceinline__ double sum_of_32(SqAcc<T> (&p)[32 / G], unsigned mask) {
  constexpr int N = 32 / G;
  if constexpr (N == 1) {
    p[0].merge(p[0].from_lane_xor(mask, 16));
  } else {
#pragma unroll
    for (int u = 0; u < N / 2; ++u) p[u].merge(p[u + N / 2]);
  }
  double v = p[0].value();
  if constexpr (N == 4) v += p[1].value();
#pragma unroll
  for (int o = G < 16 ? G / 2 : 8; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, G);
  return v;
}

__device__ __forceinline__ int64_t lower_bound(const int32_t *a, int64_t lo, int64_t hi,
                                               int64_t v) {
  while (lo < hi) {
    int64_t mid = (lo + hi) >> 1;
    if (a[mid] < v)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

constexpr int BOUNDS_T = 256;  // threads of k_bounds
// A 16-row group goes to a band tile when its multiply-adds are at least a
// fraction band_min_eff (a schedule option, 0.08 by default) of the tile's
// estimated FMA slots: the band kernel spends about 2.5 instructions per slot,
// the row-wise product tens per multiply-add.

// Row grouping of k_bounds: GROUPS_NONE keeps every row on 32 lanes.
// GROUPS_THROUGHPUT (FP64 products, bound by the FP64 pipe) picks the group
// size that leaves the fewest lanes idle in a k-step. GROUPS_PAIRS (FP32
// products, bound by instruction issue and gather latency) sends every row
// that fits half a warp's accumulator to the pair kernel, where neighbouring
// rows share their passes over B (pair_rows).
enum { GROUPS_NONE = 0, GROUPS_THROUGHPUT = 1, GROUPS_PAIRS = 2 };

// Lane utilization of one k-step with g lanes and a B row of avg entries.
__device__ __forceinline__ float lane_use(float avg, int g) {
  float rounds = ceilf(avg / float(g));
  return avg / (rounds * float(g));
}

// B rows of at least this mean length keep their row on 32 lanes: below about
// 62 entries a banded row's head and tail overlap its neighbours' too much to
// be streamed.
constexpr float STREAM_AVG = 64.0f;

// The band layout of a row from its first and last column (last < first: empty).
__device__ __forceinline__ void put_span(const BandSpans &bs, int64_t r, int first, int last) {
  const int f = last < first ? 0 : first & ~3;
  const int w = last < first ? 0 : ((last + 4) & ~3) - f;
  bs.fc[r] = f;
  bs.nf[r] = w;
  bs.span[r] = w;
}

// Per row k of B: (first column, last column, entries, 0), so that k_bounds
// reads one 16-byte record per k instead of a chain of dependent loads. ends
// (nullable; FP64 products): of a row with at least 32 entries, the 31st
// column and the 31st from its end (see stream_rows). bs (fc nullable): the
// band layout of B's rows. Also clears the `words` of the product's head, which
// k_bounds adds to (a memset of its own would stand between the kernels).
__global__ void k_row_info(int64_t n, const int64_t *rs, const int64_t *re, const int32_t *col,
                           int4 *info, int2 *ends, BandSpans bs, unsigned long long *head,
                           int words) {
  after_previous();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < words; i += gridDim.x * blockDim.x)
    head[i] = 0ULL;
  for (int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < n;
       r += int64_t(gridDim.x) * blockDim.x) {
    const int64_t a = rs[r], b = re[r];
    const int4 x = b > a ? make_int4(col[a], col[b - 1], int(b - a), 0) : make_int4(0, -1, 0, 0);
    info[r] = x;
    if (ends && b - a >= 32) ends[r] = make_int2(col[a + 30], col[b - 31]);
    if (bs.fc) put_span(bs, r, x.x, x.y);
  }
}

// Rows of A with more entries than this are walked by a whole warp in k_bounds.
constexpr int64_t BOUNDS_LONG = 256;

// The bounds and class of one row of sparse work, from its k hull [kf, kl],
// its column hull [mn, mx] (mx < 0: no output) and its multiply-adds wk;
// writes lo, len, ub of row r and, for band tiles, the row's statistics.
__device__ __forceinline__ int bounds_row(int64_t r, int m, int64_t na, int32_t mn, int32_t mx,
                                          int32_t kf, int32_t kl, int64_t wk, int mode,
                                          int groups, float group_margin, int band, int32_t *lo,
                                          int32_t *len, int64_t *ub, int *sseg,
                                          int *slo, int *sL, int *skf, int *skl, int *sna,
                                          float *swk) {
  int cls = RC_NONE;
  if (mx < 0) {
    ub[r] = 0;
    len[r] = 0;
    lo[r] = 0;
  } else {
    const int32_t L = mx - mn + 1;
    const int64_t bound = wk + (mode == MODE_UPDATE ? na : 0);
    if (L > WARP_W) {
      cls = RC_CTA;
    } else if (!groups) {
      cls = RC_G32;
    } else if (groups == GROUPS_PAIRS) {
      cls = L <= WARP_W / 2 ? RC_G16 : RC_G32;
    } else {
      const float avg = float(wk) / float(na > 0 ? na : 1);
      // long B rows run one after another through full passes (stream_rows)
      const float u32 = avg >= STREAM_AVG ? 1.0f : lane_use(avg, 32), u16 = lane_use(avg, 16), u8 = lane_use(avg, 8);
      cls = RC_G32;
      if (L <= WARP_W / 2 && u16 > u32 + group_margin) cls = RC_G16;
      if (L <= WARP_W / 4 && u8 > (cls == RC_G16 ? u16 : u32) + group_margin) cls = RC_G8;
    }
    lo[r] = mn;
    len[r] = L;
    ub[r] = bound < L ? bound : L;
  }
  if (band) {
    *sseg = m;
    *slo = mx < 0 ? 0 : mn;
    *sL = mx < 0 ? 0 : mx - mn + 1;
    *skf = kf;
    *skl = kl;
    *sna = int(na);
    *swk = float(wk);
  }
  return cls;
}

// Whether a row of L > LONG_W columns goes to RC_LONG: it has many pairs of a window and
// 32 k, each a step of its warps, and the B rows (16 of them are looked at) fall into
// less than about a quarter of the windows. Scattered B rows do not: the FP32 squares of
// a matrix of order 20000 with 7 and 258 scattered entries a row take 15.4 ms that
// way, 12.9 with RC_CTA's rows.
__device__ __forceinline__ bool long_row(const int32_t *acol, const int4 *binfo, int64_t a0,
                                         int64_t a1, int L) {
  constexpr int SAMPLES = 16;
  if (int64_t(L / WARP_W) * ((a1 - a0) / 32) < 64) return false;  // a1 - a0 >= 32 from here on
  int64_t extent = 0;
#pragma unroll 4
  for (int i = 0; i < SAMPLES; ++i) {
    const int4 b = binfo[acol[a0 + i * ((a1 - a0) / SAMPLES)]];
    extent += b.z ? b.y - b.x + 1 : 0;
  }
  return (extent / SAMPLES + WARP_W) * 4 < L;
}

// Over the 16 lanes of a half warp.
__device__ __forceinline__ int half_min(unsigned hm, int v) { return __reduce_min_sync(hm, v); }
__device__ __forceinline__ int half_max(unsigned hm, int v) { return __reduce_max_sync(hm, v); }
__device__ __forceinline__ int half_sum(unsigned hm, int v) { return __reduce_add_sync(hm, v); }

// Bounds, class and lists of the rows of a product, TILE rows at a time per
// CTA, L lanes per row (its A entries L apart, four B records per lane in
// flight). Bound by the latency of row -> k -> record and, where rows are many
// and short, by atomics on single addresses (list lengths, multiply-adds),
// which are therefore made once per tile. With a lane per row throughout, an
// atomic per warp and the band decision by one lane per 16 rows, 16 products
// took 0.52 ms at 6001 rows and 0.79 at 262144, now 0.23 and 0.41 (with the
// rows' records and the band layouts' widths). cs (fc nullable): the band layout of
// the product's rows, whose first and last columns [lo, lo + len) are stored
// entries (each is the first or last column of some B_k).
// counters: [RC_*] list lengths, [RC_QUEUE + RC_*] work-queue heads of the numeric kernels.
template <int L, int TILE>
__global__ void __launch_bounds__(BOUNDS_T)
    k_bounds(int64_t n, const int64_t *ars, const int64_t *are, const int32_t *acol,
             const int4 *binfo, const int32_t *seg,
             const int *active, int mode, int groups, float group_margin, int band,
             float band_min_eff, const int *dslot,
             const int64_t *moff, int32_t *lo, int32_t *len, int64_t *ub, int32_t *lists,
             int *counters, unsigned long long *mults, double *band_work,
             unsigned char *bandrow, BandSpans cs) {
  after_previous();
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int ROWS = BOUNDS_T / L;  // rows of one pass
  constexpr int NW = (TILE + 31) / 32;  // warps with rows in the second part
  static_assert(TILE % ROWS == 0 && TILE <= BOUNDS_T, "whole passes, a thread per row");
  static_assert(TILE % 16 == 0, "band tiles are aligned groups of 16 rows");
  __shared__ unsigned char s_cls[TILE];
  __shared__ int s_cnt[NW][RC_N];
  __shared__ int s_base[RC_N];
  __shared__ unsigned long long s_mult, s_band_work;
  // per-row statistics of the band decision (rows of sparse work only)
  __shared__ int s_seg[TILE], s_lo[TILE], s_L[TILE];
  __shared__ int s_kf[TILE], s_kl[TILE], s_na[TILE];
  __shared__ float s_wk[TILE];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t ntiles = (n + TILE - 1) / TILE;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t t0 = tile * TILE;
    const int m0 = seg[t0];
    if (threadIdx.x == 0) s_mult = s_band_work = 0ULL;
    unsigned long long mywork = 0;  // multiply-adds of matrix m0 (leaders)
    auto add_work = [&](int m, unsigned long long w) {
      if (m == m0)
        mywork += w;
      else
        atomicAdd(&mults[m], w);
    };
#pragma unroll 1
    for (int i0 = 0; i0 < TILE; i0 += ROWS) {
      const int i = i0 + threadIdx.x / L, gl = threadIdx.x % L;
      const int64_t r = t0 + i;
      int cls = RC_NONE, m = 0;
      bool work = false, longrow = false;  // the row has sparse work; walked by the warp
      int64_t a0 = 0, a1 = 0;
      int32_t mn = INT_MAX, mx = -1, kf = INT_MAX, kl = -1;
      int64_t wk = 0;
      if (gl == 0) s_seg[i] = -1;  // not eligible for a band tile
      if (r < n) {
        m = seg[r];
        a0 = ars[r];
        a1 = are[r];
        if (!active[m] || (dslot && dslot[m] >= 0)) {
          // inactive, or on the dense path: no sparse work; a dense row of an
          // update gets a whole row of slots for 1.5 X - 0.5 X T
          if (gl == 0) {
            const bool dense = active[m] && dslot && dslot[m] >= 0;
            ub[r] = dense && mode == MODE_UPDATE ? moff[m + 1] - moff[m] : 0;
            len[r] = 0;
            lo[r] = 0;
            if (cs.fc) put_span(cs, r, 0, -1);
          }
        } else {
          work = true;
          // one lane per row: rows of more than BOUNDS_LONG entries are left to the warp
          longrow = L == 1 && a1 - a0 > BOUNDS_LONG;
          if (a1 > a0) {
            kf = acol[a0];
            kl = acol[a1 - 1];
          }
          if (!longrow) {
            for (int64_t p = a0 + gl; p < a1; p += 4 * L) {
              int32_t k[4];
              int4 b[4];
#pragma unroll
              for (int u = 0; u < 4; ++u) k[u] = p + u * L < a1 ? acol[p + u * L] : -1;
#pragma unroll
              for (int u = 0; u < 4; ++u) b[u] = k[u] >= 0 ? binfo[k[u]] : make_int4(0, -1, 0, 0);
#pragma unroll
              for (int u = 0; u < 4; ++u) {
                wk += b[u].z;
                // an empty B row has first column 0 and last -1: no effect on either
                mn = min(mn, b[u].z ? b[u].x : INT_MAX);
                mx = max(mx, b[u].y);
              }
            }
          }
        }
      }
#pragma unroll
      for (int o = L / 2; o > 0; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(FULL, mn, o));
        mx = max(mx, __shfl_xor_sync(FULL, mx, o));
        wk += __shfl_xor_sync(FULL, wk, o);
      }
      if constexpr (L == 1) {  // long rows: the warp walks each with its lanes striding over A_i
        unsigned lm = __ballot_sync(FULL, longrow);
        while (lm) {
          const int src = __ffs(lm) - 1;
          lm &= lm - 1;
          const int64_t la0 = __shfl_sync(FULL, a0, src), la1 = __shfl_sync(FULL, a1, src);
          int32_t lmn = INT_MAX, lmx = -1;
          int64_t lwk = 0;
          for (int64_t p = la0 + lane; p < la1; p += 32) {
            const int4 bi = binfo[acol[p]];
            lwk += bi.z;
            if (bi.z > 0) lmn = min(lmn, bi.x);
            lmx = max(lmx, bi.y);
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            lmn = min(lmn, __shfl_xor_sync(FULL, lmn, o));
            lmx = max(lmx, __shfl_xor_sync(FULL, lmx, o));
            lwk += __shfl_xor_sync(FULL, lwk, o);
          }
          if (lane == src) {
            mn = lmn;
            mx = lmx;
            wk = lwk;
          }
        }
      }
      if (work && gl == 0) {
        if (mode == MODE_UPDATE && a1 > a0) {  // the columns of X_i itself (ascending)
          mn = min(mn, kf);
          mx = max(mx, kl);
        }
        add_work(m, (unsigned long long)wk);
        cls = bounds_row(r, m, a1 - a0, mn, mx, kf, kl, wk, mode, groups, group_margin, band, lo,
                         len, ub, s_seg + i, s_lo + i, s_L + i, s_kf + i, s_kl + i, s_na + i,
                         s_wk + i);
        if (cs.fc) put_span(cs, r, mx < 0 ? 0 : mn, mx);
        if (cls == RC_CTA && mx - mn >= LONG_W && long_row(acol, binfo, a0, a1, mx - mn + 1))
          cls = RC_LONG;
      }
      if (gl == 0) s_cls[i] = (unsigned char)cls;
    }
    __syncthreads();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mywork += __shfl_xor_sync(FULL, mywork, o);
    if (lane == 0 && mywork) atomicAdd(&s_mult, mywork);
    // from here on a thread per row
    const int i = threadIdx.x;
    // band tiles: aligned groups of 16 rows of one matrix, all with sparse
    // work, whose estimated FMA slots the multiply-adds fill well enough
    bool inband = false;
    if (band && i < TILE) {
      const unsigned hm = 0xffffu << (lane & 16);
      const int sg = s_seg[i];
      if (__all_sync(hm, sg >= 0 && sg == s_seg[i & ~15])) {
        const bool some = s_L[i] > 0;
        const int jlo = half_min(hm, some ? s_lo[i] : INT_MAX);
        const int jhi = half_max(hm, some ? s_lo[i] + s_L[i] - 1 : -1);
        const int klo = half_min(hm, s_kf[i]), khi = half_max(hm, s_kl[i]);
        if (jhi >= 0 && khi >= 0 && khi - klo < BAND_KT - 3) {
          const int nwords = (jhi >> 5) - (jlo >> 5) + 1;
          if (nwords <= BAND_JW) {  // below 2^20 multiply-adds per row: sums exact in integers
            const int wsum = half_sum(hm, int(s_wk[i])), nsum = half_sum(hm, s_na[i]);
            const float bavg = float(wsum) / fmaxf(float(nsum), 1.0f);  // mean entries of a B row
            const float kc = fminf(float(khi - klo + 1), bavg + 35.0f);
            const float slots = 16.0f * 32.0f * float(nwords) * kc;
            inband = float(wsum) >= band_min_eff * slots;
            if (inband && (lane & 15) == 0 && band_work)
              atomicAdd(&s_band_work, (unsigned long long)wsum);
          }
        }
      }
    }
    // ordered compaction of the tile's rows into one list per class
    int my = i < TILE ? s_cls[i] : int(RC_NONE);
    const bool empty = i < TILE && t0 + i < n && my == RC_NONE;
    if (inband) my = (i & 15) == 0 ? RC_BAND : RC_NONE;
    if (bandrow && i < TILE && t0 + i < n) bandrow[t0 + i] = inband ? 1 : 0;
    unsigned bal[RC_N];
#pragma unroll
    for (int c = 0; c < RC_N; ++c) {
      bal[c] = __ballot_sync(FULL, my == c);
      if (lane == 0 && warp < NW) s_cnt[warp][c] = __popc(bal[c]);
    }
    const int nempty = __syncthreads_count(empty);
    if (i < RC_N) {
      int tot = 0;
      for (int w = 0; w < NW; ++w) tot += s_cnt[w][i];
      s_base[i] = tot ? atomicAdd(&counters[i], tot) : 0;
    } else if (i == 32) {
      if (s_mult) atomicAdd(&mults[m0], s_mult);
      if (s_band_work) atomicAdd(band_work, double(s_band_work));  // of the band tiles
      if (nempty) atomicAdd(&counters[RC_EMPTY], nempty);
    }
    __syncthreads();
    if (my < RC_N) {
      int off = s_base[my];
      for (int w = 0; w < warp; ++w) off += s_cnt[w][my];
      off += __popc(bal[my] & lt);
      lists[int64_t(my) * n + off] = int32_t(t0 + i);
    }
    __syncthreads();
  }
}

// Untouched slots are marked by their value, so that a product stores nothing
// but the sum (a flag byte per product was one of eight shared-memory
// wavefronts of an FP64 pass, whose kernels run that unit at 75%).
// FP32: an untouched slot holds -0.0; each product is fma(a, b, acc) + 0, and
// adding +0 turns a -0 result into +0 and leaves every other value as it is. A
// slot reads -0 only until its first product, and its values are those of an
// accumulation from +0 (which can never produce -0) bit for bit.
// FP64: an untouched slot holds a NaN of a payload that no operation produces;
// a product that finds it starts from +0.
constexpr int kEmptyHi = int(0xFFF85E17u);  // high word of the FP64 mark
__device__ __forceinline__ bool untouched(float v) { return __float_as_uint(v) == 0x80000000u; }
__device__ __forceinline__ bool untouched(double v) { return __double2hiint(v) == kEmptyHi; }
template <typename T>
__device__ __forceinline__ T empty_slot() {
  if constexpr (sizeof(T) == 4)
    return -0.0f;
  else
    return __hiloint2double(kEmptyHi, 0);
}
__device__ __forceinline__ void mac(float *acc, int j, float a, float v) {
  acc[j] = __fadd_rn(fma_rn(a, v, acc[j]), 0.0f);
}
__device__ __forceinline__ void mac(double *acc, int j, double a, double v) {
  const double c = acc[j];
  acc[j] = fma_rn(a, v, untouched(c) ? 0.0 : c);
}

// One k of the accumulation: lanes stride over B_k = [q0, q1) and add
// a * b_kj into acc[col - c0], up to four independent products per lane in
// flight. The columns of B_k are distinct, so the slots of one call never
// collide.
template <typename T, int STRIDE>
__device__ __forceinline__ void accumulate_k(T a, int64_t q0, int64_t q1, const int32_t *bcol,
                                             const T *bval, int64_t c0, T *acc, int tid) {
  if constexpr (sizeof(T) == 8) {
    // FP64 (DFMA-bound): passes of STRIDE entries taken four, then two, then
    // one at a time, the same for every lane of the group, so that only the
    // row's last pass is partly active. A DFMA costs the FP64 pipe the same
    // whatever its active lanes, and lanes running different unrollings
    // would issue the instructions of each. 64-bit positions (~1% faster
    // here than offsets).
    const int np = int((q1 - q0 + STRIDE - 1) / STRIDE);  // group-uniform
    int64_t q = q0 + tid;
    int pass = 0;
    for (; pass + 4 <= np; pass += 4, q += 4 * STRIDE) {
      const bool ok3 = q + 3 * STRIDE < q1;  // only the last pass can be partial
      const int j0 = int(bcol[q] - c0), j1 = int(bcol[q + STRIDE] - c0);
      const int j2 = int(bcol[q + 2 * STRIDE] - c0);
      const int j3 = ok3 ? int(bcol[q + 3 * STRIDE] - c0) : 0;
      const T v0 = bval[q], v1 = bval[q + STRIDE], v2 = bval[q + 2 * STRIDE];
      const T v3 = ok3 ? bval[q + 3 * STRIDE] : T(0);
      mac(acc, j0, a, v0);
      mac(acc, j1, a, v1);
      mac(acc, j2, a, v2);
      if (ok3) mac(acc, j3, a, v3);
    }
    if (pass + 2 <= np) {
      const bool ok1 = q + STRIDE < q1;
      const int j0 = int(bcol[q] - c0), j1 = ok1 ? int(bcol[q + STRIDE] - c0) : 0;
      const T v0 = bval[q], v1 = ok1 ? bval[q + STRIDE] : T(0);
      mac(acc, j0, a, v0);
      if (ok1) mac(acc, j1, a, v1);
      pass += 2;
      q += 2 * STRIDE;
    }
    if (pass < np && q < q1) mac(acc, int(bcol[q] - c0), a, bval[q]);
  } else {
    // FP32 (issue-bound): 32-bit offsets from the start of B_k, one 64-bit
    // address per k (~4% faster)
    const int n = int(q1 - q0);
    const int32_t *bc = bcol + q0;
    const T *bv = bval + q0;
    const int32_t cz = int32_t(c0);
    int i = tid;
    for (; i + 3 * STRIDE < n; i += 4 * STRIDE) {
      int j0 = bc[i] - cz, j1 = bc[i + STRIDE] - cz;
      int j2 = bc[i + 2 * STRIDE] - cz, j3 = bc[i + 3 * STRIDE] - cz;
      T v0 = bv[i], v1 = bv[i + STRIDE], v2 = bv[i + 2 * STRIDE], v3 = bv[i + 3 * STRIDE];
      mac(acc, j0, a, v0);
      mac(acc, j1, a, v1);
      mac(acc, j2, a, v2);
      mac(acc, j3, a, v3);
    }
    if (i + STRIDE < n) {
      int j0 = bc[i] - cz, j1 = bc[i + STRIDE] - cz;
      T v0 = bv[i], v1 = bv[i + STRIDE];
      mac(acc, j0, a, v0);
      mac(acc, j1, a, v1);
      i += 2 * STRIDE;
    }
    if (i < n) mac(acc, bc[i] - cz, a, bv[i]);
  }
}

// The products of up to 32 consecutive k (lane t < nk holds a_t and the B row
// [qs, qs + len)) as one stream of entries, 32 per pass, so that every pass but
// the last is full: a DFMA costs the FP64 pipe the same whatever its active
// lanes, and with a pass structure per k a B row of 145 entries left 10% of
// the lanes idle. A pass may hold the tail of B_t and the head of B_(t+1); it
// stays free of collisions, and every slot keeps its ascending k, when each
// row has at least 32 entries (so a pass meets at most two rows) and the last
// 31 columns of B_t all lie above the first 31 of B_(t+1) (ends). Returns false,
// doing nothing, when that does not hold for all nk rows. Up to eight passes'
// loads are in flight.
__device__ __forceinline__ bool stream_rows(int nk, double av, int64_t qs, int len, int2 ends,
                                            const int32_t *bcol, const double *bval, int32_t c0,
                                            double *acc, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  const int next_head = __shfl_down_sync(FULL, ends.x, 1);
  const bool ok = lane >= nk || (len >= 32 && (lane == nk - 1 || ends.y > next_head));
  if (!__all_sync(FULL, ok)) return false;
  int end = lane < nk ? len : 0;  // inclusive prefix: where row t ends in the stream
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(FULL, end, o);
    if (lane >= o) end += y;
  }
  const int total = __shfl_sync(FULL, end, 31);
  const int64_t off = qs - (end - len);  // stream position p of row t is entry off + p
  // row t of the pass's first entry (uniform) and row t + 1: where t ends, the
  // factors and the offsets, fetched from their lanes when t advances
  int t = 0, e = __shfl_sync(FULL, end, 0);
  double at = __shfl_sync(FULL, av, 0), an = __shfl_sync(FULL, av, 1);
  int64_t ot = __shfl_sync(FULL, off, 0), on = __shfl_sync(FULL, off, 1);
  int j[4], jn[4];
  double a[4], v[4], aw[4], vw[4];
  auto fetch = [&](int p0, int (&j)[4], double (&a)[4], double (&v)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int p = p0 + 32 * u + lane;
      const bool head = p >= e;  // of row t + 1
      a[u] = head ? an : at;
      const int64_t q = (head ? on : ot) + p;
      j[u] = -1;
      if (p < total) {
        j[u] = bcol[q] - c0;
        v[u] = bval[q];
      }
      if (p0 + 32 * (u + 1) >= e && t < 31) {
        ++t;
        e = __shfl_sync(FULL, end, t);
        at = an;
        ot = on;
        const int nx = min(t + 1, 31);
        an = __shfl_sync(FULL, av, nx);
        on = __shfl_sync(FULL, off, nx);
      }
    }
  };
  auto add = [&](const int (&j)[4], const double (&a)[4], const double (&v)[4]) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (j[u] >= 0) mac(acc, j[u], a[u], v[u]);
      __syncwarp();
    }
  };
  fetch(0, j, a, v);
  for (int p0 = 0; p0 < total; p0 += 256) {  // the next four passes load while four are added
    if (p0 + 128 < total) fetch(p0 + 128, jn, aw, vw);
    add(j, a, v);
    if (p0 + 128 >= total) break;
    if (p0 + 256 < total) fetch(p0 + 256, j, a, v);
    add(jn, aw, vw);
  }
  return true;
}

// The k-loop of one row by one warp when rows are few and latency counts: the
// B rows of 32 k are located together (the next 32 while these run), and the
// first 64 entries of four k are loaded while the four before them are added.
// The k still run one after another, one fused multiply-add per slot each.
template <typename T>
__device__ __forceinline__ void ahead_rows(int64_t a0, int64_t a1, const int32_t *acol,
                                           const T *aval, const int64_t *brs, const int64_t *bre,
                                           const int32_t *bcol, const T *bval, int32_t c0, T *acc,
                                           int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int D = 4;
  struct Four {
    T a[D], v0[D], v1[D];
    int64_t q[D];
    int n[D], j0[D], j1[D];
  };
  T av = T(0), nav = T(0);
  int64_t qs = 0, nqs = 0;
  int qn = 0, nqn = 0;
  auto locate = [&](int64_t p, T &a, int64_t &q, int &n) {
    n = 0;
    if (p < a1) {
      const int32_t k = acol[p];
      a = aval[p];
      q = brs[k];
      n = int(bre[k] - q);
    }
  };
  auto load = [&](Four &x, int t0) {
#pragma unroll
    for (int t = 0; t < D; ++t) {
      x.a[t] = __shfl_sync(FULL, av, t0 + t);
      x.q[t] = __shfl_sync(FULL, qs, t0 + t);
      x.n[t] = __shfl_sync(FULL, qn, t0 + t);
      if (lane < x.n[t]) {
        x.j0[t] = int(bcol[x.q[t] + lane] - c0);
        x.v0[t] = bval[x.q[t] + lane];
      }
      if (lane + 32 < x.n[t]) {
        x.j1[t] = int(bcol[x.q[t] + lane + 32] - c0);
        x.v1[t] = bval[x.q[t] + lane + 32];
      }
    }
  };
  auto add = [&](const Four &x) {
#pragma unroll
    for (int t = 0; t < D; ++t) {
      if (lane < x.n[t]) mac(acc, x.j0[t], x.a[t], x.v0[t]);
      if (lane + 32 < x.n[t]) mac(acc, x.j1[t], x.a[t], x.v1[t]);
      if (x.n[t] > 64)
        accumulate_k<T, 32>(x.a[t], x.q[t] + 64, x.q[t] + x.n[t], bcol, bval, c0, acc, lane);
      __syncwarp();
    }
  };
  locate(a0 + lane, av, qs, qn);
  Four x, y;
  for (int64_t pb = a0; pb < a1; pb += 32) {
    const int nk = int(min(int64_t(32), a1 - pb));
    locate(pb + 32 + lane, nav, nqs, nqn);
    load(x, 0);
    for (int t = 0; t < nk; t += 2 * D) {  // lanes past nk hold empty rows
      if (t + D < nk) load(y, t + D);
      add(x);
      if (t + D < nk) {
        if (t + 2 * D < nk) load(x, t + 2 * D);
        add(y);
      }
    }
    av = nav;
    qs = nqs;
    qn = nqn;
  }
}

// accumulate_k for one k shared by two rows (a_ik and a_i'k): every entry of
// B_k is loaded once and added into both rows' accumulators.
template <typename T>
__device__ __forceinline__ void accumulate_k2(T a, T b, int64_t q0, int64_t q1,
                                              const int32_t *bcol, const T *bval, int32_t ca,
                                              T *acca, int32_t cb, T *accb, int tid) {
  const int n = int(q1 - q0);
  const int32_t *bc = bcol + q0;
  const T *bv = bval + q0;
  int i = tid;
  for (; i + 96 < n; i += 128) {
    int32_t c0 = bc[i], c1 = bc[i + 32], c2 = bc[i + 64], c3 = bc[i + 96];
    T v0 = bv[i], v1 = bv[i + 32], v2 = bv[i + 64], v3 = bv[i + 96];
    mac(acca, c0 - ca, a, v0);
    mac(acca, c1 - ca, a, v1);
    mac(acca, c2 - ca, a, v2);
    mac(acca, c3 - ca, a, v3);
    mac(accb, c0 - cb, b, v0);
    mac(accb, c1 - cb, b, v1);
    mac(accb, c2 - cb, b, v2);
    mac(accb, c3 - cb, b, v3);
  }
  // at most three entries per lane are left: two loaded together, then one
  if (i + 32 < n) {
    int32_t c0 = bc[i], c1 = bc[i + 32];
    T v0 = bv[i], v1 = bv[i + 32];
    mac(acca, c0 - ca, a, v0);
    mac(acca, c1 - ca, a, v1);
    mac(accb, c0 - cb, b, v0);
    mac(accb, c1 - cb, b, v1);
    i += 64;
  }
  if (i < n) {
    int32_t c = bc[i];
    T v = bv[i];
    mac(acca, c - ca, a, v);
    mac(accb, c - cb, b, v);
  }
}

// The k-loop of two rows run by one warp (rows of the 16-lane pair class).
// Their k lists, each ascending, are merged: a k found in both rows is one
// step that feeds both accumulators from a single pass over B_k, a k of one
// row only is a step of that row alone. Each row thus still receives its k in
// ascending order, one FMA per slot per k, exactly as with a warp of its own.
// Rows of a banded iterate that are neighbours share almost all of their k,
// so the pair gathers B about half as often as two warps would.
// Row x has k entries [pa, ea) and accumulator acca for columns from
// ca; row y likewise (an absent row has pb == eb).
template <typename T>
__device__ __forceinline__ void pair_rows(int64_t pa, int64_t ea, int64_t pb, int64_t eb,
                                          const int32_t *acol, const T *aval,
                                          const int64_t *brs, const int64_t *bre,
                                          const int32_t *bcol, const T *bval, int32_t ca,
                                          T *acca, int32_t cb, T *accb, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  // lane l holds the (k, a_k, start, length) of the l-th k of each row's window
  int ka = INT_MAX, kb = INT_MAX, na = 0, nb = 0;
  T va = T(0), vb = T(0);
  int64_t qa = 0, qb = 0;
  {
    int64_t p = pa + lane;
    if (p < ea) {
      ka = acol[p];
      va = aval[p];
      qa = brs[ka];
      na = int(bre[ka] - qa);
    }
    p = pb + lane;
    if (p < eb) {
      kb = acol[p];
      vb = aval[p];
      qb = brs[kb];
      nb = int(bre[kb] - qb);
    }
  }
  int ia = 0, ib = 0;
  for (;;) {
    if (ia == 32) {  // window of row x used up: the next 32 k
      pa += 32;
      ia = 0;
      int64_t p = pa + lane;
      ka = INT_MAX;
      if (p < ea) {
        ka = acol[p];
        va = aval[p];
        qa = brs[ka];
        na = int(bre[ka] - qa);
      }
    }
    if (ib == 32) {
      pb += 32;
      ib = 0;
      int64_t p = pb + lane;
      kb = INT_MAX;
      if (p < eb) {
        kb = acol[p];
        vb = aval[p];
        qb = brs[kb];
        nb = int(bre[kb] - qb);
      }
    }
    const int ha = __shfl_sync(FULL, ka, ia), hb = __shfl_sync(FULL, kb, ib);
    if (ha == INT_MAX && hb == INT_MAX) break;
    if (ha == hb) {
      const T a = __shfl_sync(FULL, va, ia), b = __shfl_sync(FULL, vb, ib);
      const int64_t q0 = __shfl_sync(FULL, qa, ia);
      const int n = __shfl_sync(FULL, na, ia);
      accumulate_k2<T>(a, b, q0, q0 + n, bcol, bval, ca, acca, cb, accb, lane);
      ++ia;
      ++ib;
    } else if (ha < hb) {
      const T a = __shfl_sync(FULL, va, ia);
      const int64_t q0 = __shfl_sync(FULL, qa, ia);
      const int n = __shfl_sync(FULL, na, ia);
      accumulate_k<T, 32>(a, q0, q0 + n, bcol, bval, ca, acca, lane);
      ++ia;
    } else {
      const T b = __shfl_sync(FULL, vb, ib);
      const int64_t q0 = __shfl_sync(FULL, qb, ib);
      const int n = __shfl_sync(FULL, nb, ib);
      accumulate_k<T, 32>(b, q0, q0 + n, bcol, bval, cb, accb, lane);
      ++ib;
    }
    __syncwarp();
  }
}

constexpr int AHEAD_OCC = 4;  // CTAs per SM of the ahead_rows kernels (registers for loads in flight)
constexpr int PAIR_OCC = 8;  // CTAs per SM of the pair kernel: 64 registers, no spills
template <typename T>
struct WarpOcc;  // CTAs per SM of the warp kernel (shared memory and registers)
template <> struct WarpOcc<double> { static constexpr int value = 6; };
template <> struct WarpOcc<float> { static constexpr int value = 10; };

// G lanes per row, 32/G rows per warp; each group owns WARP_W*G/32 slots of
// its warp's accumulator and runs the ascending-k accumulation of its own row
// with group-wide barriers, so the result is the same as with a whole warp.
// A row's sums of squares are 32 partial sums, of the columns lo + p, lo + p + 32,
// ... (the diagonal's square is added last) and of every 32nd entry of X_i, in
// ascending order, then added by sum_of_32: whatever lanes a row runs on, which
// depends on the other rows of the launch too, its part of the residual is the same.
// LOOP: LOOP_PAIR (with G = 16): the two rows of a warp share its k-loop
// (pair_rows); the rest of the kernel is that of 16-lane groups. LOOP_AHEAD
// (with G = 32): the k-loop of ahead_rows.
enum { LOOP_ROW = 0, LOOP_PAIR = 1, LOOP_AHEAD = 2 };
template <typename T, int LOOP>
constexpr int group_occ() {
  return LOOP == LOOP_PAIR ? PAIR_OCC : LOOP == LOOP_AHEAD ? AHEAD_OCC : WarpOcc<T>::value;
}
template <typename T, int MODE, int G, int LOOP = LOOP_ROW>
__global__ void __launch_bounds__(WARPS_PER_CTA * 32, group_occ<T, LOOP>())
    k_num_group(const int64_t *ars, const int64_t *are, const int32_t *acol, const T *aval,
                const int64_t *brs, const int64_t *bre, const int32_t *bcol, const T *bval,
                const int2 *ends, const int32_t *lo, const int32_t *len, const int32_t *list,
                int *counters, int cls, const int64_t *cs, int64_t *ce, int32_t *ccol, T *cval,
                double *part) {
  after_previous();
  constexpr bool PAIR = LOOP == LOOP_PAIR;
  static_assert(!PAIR || G == 16, "pairs are two 16-lane groups");
  static_assert(LOOP != LOOP_AHEAD || G == 32, "a warp per row");
  constexpr int NG = 32 / G;
  constexpr int SLOTS = WARP_W / NG;
  // group bases staggered across shared-memory banks: without it the groups of
  // a warp (or of a half-warp, for 8-byte values) start on the same bank and
  // their lanes, which touch neighbouring slots, collide
  constexpr int PAD = G == 32 ? 0 : (sizeof(T) == 4 ? G : (G == 8 ? 8 : 0));
  __shared__ T acc_all[WARPS_PER_CTA][WARP_W + 3 * PAD];
  // MODE_UPDATE: slots that hold x_ij, written once per entry of X_i
  __shared__ unsigned char flags[WARPS_PER_CTA][MODE == MODE_UPDATE ? WARP_W + 3 * PAD : 1];
  const int lane = lane_id(), w = threadIdx.x >> 5;
  const int g = lane / G, gl = lane % G;
  const unsigned gbits = G == 32 ? 0xffffffffu : ((1u << G) - 1u);
  const unsigned gmask = gbits << (g * G);
  const unsigned lt = (1u << gl) - 1u;
  T *acc = acc_all[w] + g * (SLOTS + PAD);
  unsigned char *f = flags[w] + (MODE == MODE_UPDATE ? g * (SLOTS + PAD) : 0);
  const int total = counters[cls];
  for (;;) {
    int base = 0;
    if (lane == 0) base = atomicAdd(&counters[RC_QUEUE + cls], NG);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (base >= total) break;
    const int idx = base + g;
    if (PAIR || idx < total) {
      const bool has = idx < total;  // the second row of the last pair may be absent
      const int32_t r = has ? list[idx] : 0;
      const int L = has ? len[r] : 0;
      const int32_t c0 = has ? lo[r] : 0;
      for (int s = gl; s < L; s += G) {
        acc[s] = empty_slot<T>();
        if (MODE == MODE_UPDATE) f[s] = 0;
      }
      const int64_t a0 = has ? ars[r] : 0, a1 = has ? are[r] : 0;
      if constexpr (PAIR) {
        __syncwarp();
        constexpr unsigned FULL = 0xffffffffu;
        pair_rows<T>(__shfl_sync(FULL, a0, 0), __shfl_sync(FULL, a1, 0),
                     __shfl_sync(FULL, a0, G), __shfl_sync(FULL, a1, G), acol, aval, brs, bre,
                     bcol, bval, __shfl_sync(FULL, c0, 0), acc_all[w], __shfl_sync(FULL, c0, G),
                     acc_all[w] + (SLOTS + PAD), lane);
      } else if constexpr (LOOP == LOOP_AHEAD) {
        __syncwarp();
        ahead_rows<T>(a0, a1, acol, aval, brs, bre, bcol, bval, c0, acc, lane);
      } else {
        __syncwarp(gmask);
        // ascending k; the (a_ik, start, end) of G k at a time are fetched by
        // the group's lanes together and broadcast inside the group
        for (int64_t pb = a0; pb < a1; pb += G) {
          const int nk = int(min(int64_t(G), a1 - pb));
          T av = T(0);
          int64_t qs = 0, qe = 0;
          int2 be = make_int2(0, 0);
          if (gl < nk) {
            int32_t k = acol[pb + gl];
            av = aval[pb + gl];
            qs = brs[k];
            qe = bre[k];
            if constexpr (sizeof(T) == 8 && G == 32) be = ends[k];
          }
          if constexpr (sizeof(T) == 8 && G == 32) {
            if (stream_rows(nk, av, qs, int(qe - qs), be, bcol, bval, c0, acc, lane)) continue;
          }
          for (int t = 0; t < nk; ++t) {
            T a = __shfl_sync(gmask, av, t, G);
            int64_t q0 = __shfl_sync(gmask, qs, t, G);
            int64_t q1 = __shfl_sync(gmask, qe, t, G);
            accumulate_k<T, G>(a, q0, q1, bcol, bval, c0, acc, gl);
            __syncwarp(gmask);
          }
        }
      }
      if (has) {  // group-uniform
        if (MODE == MODE_UPDATE) {
          for (int64_t p = a0 + gl; p < a1; p += G) {
            int j = acol[p] - c0;
            T xt = acc[j];
            if (untouched(xt)) xt = T(0);
            acc[j] = ns_combine(aval[p], xt);
            f[j] = 2;
          }
          __syncwarp(gmask);
        }
        int64_t out = cs[r];
        SqAcc<T> racc[NG];  // 32 partial sums per row, NG to a lane
        T vdiag = T(0);     // t_ii, whose square is added last
        bool diag = false;
        for (int s32 = 0; s32 < L; s32 += 32) {
#pragma unroll
          for (int u = 0; u < NG; ++u) {
            const int s0 = s32 + u * G;
            if (u > 0 && s0 >= L) break;
            int s = s0 + gl;
            int fl = 0;
            if (s < L) {
              // touched: a product or, in an update, x_ij
              fl = MODE == MODE_UPDATE ? f[s] : 0;
              if (!fl && !untouched(acc[s])) fl = 1;
            }
            unsigned m = (__ballot_sync(gmask, fl != 0) >> (g * G)) & gbits;
            if (fl) {
              int64_t pos = out + __popc(m & lt);
              int32_t cj = c0 + s;
              T v = acc[s];
              if (MODE == MODE_UPDATE && !(fl & 2)) v = ns_combine(T(0), v);
              ccol[pos] = cj;
              cval[pos] = v;
              if (MODE == MODE_SQUARE) {
                if (cj == r) {
                  vdiag = v;
                  diag = true;
                } else {
                  racc[u].add_sq(v);
                }
              }
            }
            out += __popc(m);
          }
        }
        if (gl == 0) ce[r] = out;
        if (MODE == MODE_SQUARE) {
          SqAcc<T> xacc[NG];
          for (int64_t p = a0 + gl; p < a1; p += 4 * G) {  // four loads in flight
            T x[4];
#pragma unroll
            for (int t = 0; t < 4; ++t) x[t] = p + t * G < a1 ? aval[p + t * G] : T(0);
#pragma unroll
            for (int t = 0; t < 4; ++t)
              if (p + t * G < a1) xacc[t % NG].add_sq(x[t]);
          }
          const double rs = sum_of_32<T, G>(racc, gmask), xs = sum_of_32<T, G>(xacc, gmask);
          const unsigned dm = __ballot_sync(gmask, diag);
          const T vd = __shfl_sync(gmask, vdiag, dm ? __ffs(dm) - 1 : 0, G);
          if (gl == 0) {
            part[2 * int64_t(r)] = rs + diag_square(dm != 0, vd);
            part[2 * int64_t(r) + 1] = xs;
          }
        }
        __syncwarp(gmask);
      }
    }
    __syncwarp();
  }
}

// Column blocks of B's rows: off[k * stride + b] is the number of entries of
// row k in columns before block b (blocks of 1 << sh columns from the first
// column of the row's matrix), b = 0 .. stride - 1. A warp per row.
__global__ void k_col_blocks(int64_t n, const int64_t *rs, const int64_t *re, const int32_t *col,
                             const int32_t *seg, const int64_t *moff, int sh, int stride,
                             int *off) {
  after_previous();
  const int lane = lane_id();
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; r < n; r += nwarps) {
    const int64_t a = rs[r], e = re[r], base = moff[seg[r]];
    int *o = off + r * stride;
    int last = -1;  // block of the entry before the chunk
    for (int64_t p0 = a; p0 < e; p0 += 32) {
      const int64_t p = p0 + lane;
      const int b = p < e ? int((col[p] - base) >> sh) : stride - 1;
      int prev = __shfl_up_sync(0xffffffffu, b, 1);
      if (lane == 0) prev = last;
      if (p < e)
        for (int i = prev + 1; i <= b; ++i) o[i] = int(p - a);
      last = __shfl_sync(0xffffffffu, b, int(min(int64_t(31), e - 1 - p0)));
    }
    for (int i = last + 1 + lane; i < stride; i += 32) o[i] = int(e - a);
  }
}

// Rows of more than WARP_W columns. P warps (a power of two up to 8) take a row
// together, each a window of at most WARP_W columns of it at a time: the warp
// runs through the k of A_i in ascending order and adds the part of B_k that
// falls in its window, found in the column-block table (or, without one, by
// binary search), so no barrier separates the k; the warps of a row meet only
// to add up their entry counts before each writes its part. P follows the
// mean length of B's rows: enough entries of B_k per warp to fill its lanes
// (an FP64 instruction costs the pipe the same whatever its active lanes).
// A row's sums of squares are 256 partial sums, of every 256th column and of every
// 256th entry of X_i in ascending order, 256 / P to a warp, added 128 apart, 64
// apart and so on, the diagonal's last: the same for every P and window (and for every first column that
// the 256 are counted from, which is the window's). One warp adds its squares as it
// writes the row; several read each other's accumulators. Rows of the 32-lane class
// take that class's 32 sums.
// One CTA per row with a barrier per k took 12.0 and 6.0 ms for the update and
// the square of the 16^3 Laplacian's FP32 iterate just below the dense path's
// density, now 7.8 and 4.0.
// The rows of RC_LONG (WIDE_LONG) always take eight warps, and a warp looks through
// the k by the first and last columns of their B rows, 128 at a time, before it locates
// any: such a row has many windows and most k fall into few of them. With one warp that located every k in every window the FP64 products of a
// solve of a tridiagonal matrix of order 65536 with one full row took 3.5 s (1.1 s
// with one CTA per row before that), now 0.088.
constexpr int WIDE_WARPS = 8;
constexpr int WIDE_K = 4;  // k whose first 32 entries are loaded ahead
enum { WIDE_ROWS = 0, WIDE_NARROW = 1, WIDE_LONG = 2 };
// CTAs per SM: FP64 as many as the accumulators leave room for; FP32 four, with 64
// registers a thread (P = 2 and 4 spill up to 84 B). Five (48) spilled up to 300 B:
// squares and updates of the 16^3 Laplacian's solve 2.19 and 3.51 ms, with four 1.87
// and 3.21; of the 45^2 Laplacian's 1.77 and 2.52, with four 1.58 and 2.32.
template <typename T, int KIND>
constexpr int wide_occ() {
  return KIND == WIDE_LONG ? 2 : sizeof(T) == 8 ? 3 : 4;
}
template <typename T, int MODE>
constexpr size_t wide_smem() {
  return size_t(WIDE_WARPS) * WARP_W * (sizeof(T) + (MODE == MODE_UPDATE ? 1 : 0));
}

template <typename T, int MODE, int P, int KIND>
__global__ void __launch_bounds__(WIDE_WARPS * 32, wide_occ<T, KIND>())
    k_num_wide(const int64_t *ars, const int64_t *are, const int32_t *acol, const T *aval,
               const int64_t *brs, const int64_t *bre, const int32_t *bcol, const T *bval,
               const int4 *binfo, const int32_t *seg, const int64_t *moff, const int *off, int sh,
               int stride, const int32_t *lo, const int32_t *len, const int32_t *list,
               int *counters, int cls, const int64_t *cs, int64_t *ce, int32_t *ccol, T *cval, double *part) {
  after_previous();
  constexpr unsigned FULL = 0xffffffffu;
  constexpr bool NARROW = KIND == WIDE_NARROW;
  constexpr int NG = WIDE_WARPS / P;     // rows in flight per CTA
  extern __shared__ __align__(16) unsigned char wide_smem_raw[];
  constexpr int NQ = WIDE_WARPS / P;     // eighths of a row's sums per warp
  __shared__ int s_idx[NG], s_cnt[WIDE_WARPS];
  __shared__ double s_red[2][MODE == MODE_SQUARE && P > 1 ? WIDE_WARPS : 1][32];
  __shared__ int s_diag[WIDE_WARPS];
  __shared__ T s_vdiag[WIDE_WARPS];
  const int lane = lane_id(), w = threadIdx.x >> 5, g = w / P, wr = w % P;
  const unsigned lt = (1u << lane) - 1u;
  T *acc = reinterpret_cast<T *>(wide_smem_raw) + w * WARP_W;
  unsigned char *f = wide_smem_raw + size_t(WIDE_WARPS) * WARP_W * sizeof(T) + w * WARP_W;
  // the warps of one row
  auto row_sync = [&] {
    if constexpr (P == 1)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(P * 32) : "memory");
  };
  const int total = counters[cls];
  for (;;) {
    if (wr == 0 && lane == 0) s_idx[g] = atomicAdd(&counters[RC_QUEUE + cls], 1);
    row_sync();
    const int idx = s_idx[g];
    if (idx >= total) break;
    const int32_t r = list[idx];
    const int64_t base = moff[seg[r]], a0 = ars[r], a1 = are[r];
    const int b0 = int((lo[r] - base) >> sh), b1 = int((int64_t(lo[r]) + len[r] - 1 - base) >> sh);
    const int bpw = min(WARP_W >> sh, (b1 - b0 + P) / P);  // blocks per warp and window
    int64_t out = cs[r];
    SqAcc<T> racc[1];  // NARROW: the sums of k_num_group, by warp 0
    // FP64: indexed at run time and so kept in local memory. In registers through the
    // k loop they cost it its loads in flight (two squares of a matrix of order 20000
    // with 7 and 258 scattered entries a row: 13.0 ms, now 11.6); the FP32 words are better unrolled
    // (12.8 ms against 11.0).
    double rq[NQ] = {};
    T vdiag = T(0);  // t_ii, whose square is added last
    bool diag = false;
    for (int win = b0; win <= b1; win += P * bpw) {
      const int w0 = win + wr * bpw, w1 = min(w0 + bpw, b1 + 1);  // this warp's blocks
      const bool has = w0 < w1;
      const int64_t c0 = base + (int64_t(w0) << sh);
      const int W = has ? (w1 - w0) << sh : 0;  // its columns
      for (int s = lane; s < W; s += 32) {
        acc[s] = empty_slot<T>();
        if (MODE == MODE_UPDATE) f[s] = 0;
      }
      __syncwarp();
      if (has) {
        // lane t's k: the factor and the part of its B row in the window
        auto add_rows = [&](T av, int64_t qs, int qn) {
          unsigned todo = __ballot_sync(FULL, qn > 0);
          while (todo) {  // ascending k, WIDE_K at a time
            T a[WIDE_K], v[WIDE_K];
            int64_t q0[WIDE_K];
            int nn[WIDE_K], j[WIDE_K];
#pragma unroll
            for (int t = 0; t < WIDE_K; ++t) {
              const int src = todo ? __ffs(todo) - 1 : 0;
              const bool any = todo != 0;
              todo &= todo - 1;
              a[t] = __shfl_sync(FULL, av, src);
              q0[t] = __shfl_sync(FULL, qs, src);
              nn[t] = __shfl_sync(FULL, qn, src);
              if (!any) nn[t] = 0;
              if (lane < nn[t]) {
                j[t] = int(bcol[q0[t] + lane] - c0);
                v[t] = bval[q0[t] + lane];
              }
            }
#pragma unroll
            for (int t = 0; t < WIDE_K; ++t) {
              if (lane < nn[t]) mac(acc, j[t], a[t], v[t]);
              if (nn[t] > 32)
                accumulate_k<T, 32>(a[t], q0[t] + 32, q0[t] + nn[t], bcol, bval, c0, acc, lane);
              __syncwarp();
            }
          }
        };
        // the part of row k of B in the window
        auto locate = [&](int32_t k, int64_t &qs, int &qn) {
          qs = brs[k];
          if (off) {
            const int *o = off + int64_t(k) * stride;
            const int o0 = o[w0];
            qn = o[w1] - o0;
            qs += o0;
          } else {
            const int64_t e = bre[k];
            qs = lower_bound(bcol, qs, e, c0);
            qn = int(lower_bound(bcol, qs, e, c0 + W) - qs);
          }
        };
        if constexpr (KIND == WIDE_LONG) {
          constexpr int KB = 4;  // groups of 32 k looked at together
          for (int64_t pb = a0; pb < a1; pb += 32 * KB) {
            int32_t kk[KB];
            bool hit[KB];
            int4 bi[KB];
#pragma unroll
            for (int u = 0; u < KB; ++u) {
              hit[u] = pb + 32 * u + lane < a1;
              kk[u] = hit[u] ? acol[pb + 32 * u + lane] : 0;
            }
#pragma unroll
            for (int u = 0; u < KB; ++u) bi[u] = binfo[kk[u]];
#pragma unroll
            for (int u = 0; u < KB; ++u)
              hit[u] = hit[u] && bi[u].z > 0 && bi[u].x < c0 + W && bi[u].y >= c0;
#pragma unroll
            for (int u = 0; u < KB; ++u) {
              if (!__any_sync(FULL, hit[u])) continue;
              T av = T(0);
              int64_t qs = 0;
              int qn = 0;
              if (hit[u]) {
                av = aval[pb + 32 * u + lane];
                locate(kk[u], qs, qn);
              }
              add_rows(av, qs, qn);
            }
          }
        } else {
          for (int64_t pb = a0; pb < a1; pb += 32) {
            T av = T(0);
            int64_t qs = 0;
            int qn = 0;
            if (pb + lane < a1) {
              const int32_t k = acol[pb + lane];
              av = aval[pb + lane];
              locate(k, qs, qn);
            }
            add_rows(av, qs, qn);
          }
        }
        if (MODE == MODE_UPDATE) {  // x_ij of the window
          const int64_t x0 = lower_bound(acol, a0, a1, c0), x1 = lower_bound(acol, x0, a1, c0 + W);
          for (int64_t p = x0 + lane; p < x1; p += 32) {
            const int jx = int(acol[p] - c0);
            T xt = acc[jx];
            if (untouched(xt)) xt = T(0);
            acc[jx] = ns_combine(aval[p], xt);
            f[jx] = 2;
          }
          __syncwarp();
        }
      }
      auto touched = [&](int s) -> int {
        if (s >= W) return 0;
        int fl = MODE == MODE_UPDATE ? f[s] : 0;
        if (!fl && !untouched(acc[s])) fl = 1;
        return fl;
      };
      int64_t at = out;
      if constexpr (P > 1) {
        int cnt = 0;
        for (int s0 = 0; s0 < W; s0 += 32)
          cnt += __popc(__ballot_sync(FULL, touched(s0 + lane) != 0));
        if (lane == 0) s_cnt[w] = cnt;
        row_sync();
        for (int i = 0; i < P; ++i) {
          const int ci = s_cnt[g * P + i];
          if (i < wr) at += ci;
          out += ci;
        }
      }
      auto emit = [&](int s0, auto also) {
        const int s = s0 + lane, fl = touched(s);
        const unsigned mk = __ballot_sync(FULL, fl != 0);
        if (fl) {
          const int64_t pos = at + __popc(mk & lt);
          const int64_t cj = c0 + s;
          T v = acc[s];
          if (MODE == MODE_UPDATE && !(fl & 2)) v = ns_combine(T(0), v);
          ccol[pos] = int32_t(cj);
          cval[pos] = v;
          also(cj, v);
        }
        at += __popc(mk);
      };
      if constexpr (P == 1 && MODE == MODE_SQUARE) {
#pragma unroll 1
        for (int s0 = 0; s0 < W; s0 += 32)
          emit(s0, [&](int64_t cj, T v) {
            if (cj == r) {
              vdiag = v;
              diag = true;
            } else {
              double &sum = rq[s0 / 32 % NQ];
              sum = __fma_rn(double(v), double(v), sum);
            }
          });
      } else {
        for (int s0 = 0; s0 < W; s0 += 32) emit(s0, [](int64_t, T) {});
      }
      if constexpr (P == 1) out = at;
      if constexpr (MODE == MODE_SQUARE && P > 1) {
        // the squares of the window's columns, from the accumulators of all the row's
        // warps: words of 32 columns, each within one warp's (o, up to column oend)
        const int words = ((min(win + P * bpw, b1 + 1) - win) << sh) / 32;
        const int bcol = bpw << sh, idiag = int(r - base) - (win << sh);
        const T *const row = acc - wr * WARP_W + lane;
        int o = 0, oend = bcol;
        auto square = [&](int j, auto add) {
          while (32 * j >= oend) {
            ++o;
            oend += bcol;
          }
          const T v = row[o * (WARP_W - bcol) + 32 * j];
          if (untouched(v)) return;
          if (32 * j + lane == idiag) {
            vdiag = v;
            diag = true;
          } else {
            add(v);
          }
        };
        if constexpr (NARROW) {
          if (wr == 0)
            for (int j = 0; j < words; ++j) square(j, [&](T v) { racc[0].add_sq(v); });
        } else {
          auto add_to = [&](int j, double &sum) {
            square(j, [&](T v) { sum = __fma_rn(double(v), double(v), sum); });
          };
          if constexpr (sizeof(T) == 4 || NQ == 1) {
            for (int j8 = wr; j8 < words; j8 += 8)
#pragma unroll
              for (int q = 0; q < NQ; ++q)
                if (j8 + q * P < words) add_to(j8 + q * P, rq[q]);
          } else {
            int q = 0;
#pragma unroll 1
            for (int j = wr; j < words; j += P) {
              add_to(j, rq[q]);
              q = (q + 1) % NQ;
            }
          }
        }
      }
      row_sync();  // s_cnt and the accumulators are free again
    }
    if (wr == 0 && lane == 0) ce[r] = out;
    if constexpr (MODE == MODE_SQUARE) {
      const unsigned dm = __ballot_sync(FULL, diag);
      if constexpr (NARROW) {
        if (wr == 0) {
          SqAcc<T> xacc[1];
          for (int64_t p = a0 + lane; p < a1; p += 32) xacc[0].add_sq(aval[p]);
          const double rs = sum_of_32<T, 32>(racc, FULL), xs = sum_of_32<T, 32>(xacc, FULL);
          const T vd = __shfl_sync(FULL, vdiag, dm ? __ffs(dm) - 1 : 0);
          if (lane == 0) {
            part[2 * int64_t(r)] = rs + diag_square(dm != 0, vd);
            part[2 * int64_t(r) + 1] = xs;
          }
        }
      } else {
        double xq[NQ] = {};
        for (int64_t p = a0; p < a1; p += 256)
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            const int64_t i = p + 32 * (wr + q * P) + lane;
            if (i < a1) {
              const double x = double(aval[i]);
              xq[q] = __fma_rn(x, x, xq[q]);
            }
          }
#pragma unroll
        for (int h = NQ / 2; h > 0; h >>= 1)  // 128, 64, 32 apart: in this lane
#pragma unroll
          for (int q = 0; q < h; ++q) {
            rq[q] += rq[q + h];
            xq[q] += xq[q + h];
          }
        double rs = rq[0], xs = xq[0];
        bool any = dm != 0;
        T vd = __shfl_sync(FULL, vdiag, dm ? __ffs(dm) - 1 : 0);
        if constexpr (P > 1) {  // in those of the other warps
          s_red[0][w][lane] = rs;
          s_red[1][w][lane] = xs;
          if (lane == 0) {
            s_diag[w] = any;
            s_vdiag[w] = vd;
          }
          row_sync();
          if (wr == 0) {
            double a[P], b[P];
#pragma unroll
            for (int i = 0; i < P; ++i) {
              a[i] = s_red[0][w + i][lane];
              b[i] = s_red[1][w + i][lane];
              if (s_diag[w + i]) {
                any = true;
                vd = s_vdiag[w + i];
              }
            }
#pragma unroll
            for (int h = P / 2; h > 0; h >>= 1)
#pragma unroll
              for (int i = 0; i < h; ++i) {
                a[i] += a[i + h];
                b[i] += b[i + h];
              }
            rs = a[0];
            xs = b[0];
          }
        }
        if (wr == 0) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            rs += __shfl_xor_sync(FULL, rs, o);
            xs += __shfl_xor_sync(FULL, xs, o);
          }
          if (lane == 0) {
            part[2 * int64_t(r)] = rs + diag_square(any, vd);
            part[2 * int64_t(r) + 1] = xs;
          }
        }
      }
    }
    row_sync();  // s_idx and s_red are read
  }
}

// Rows with an empty column range, also those of a band tile whose other rows
// have output (k_band passes over them): their slot stays empty (ce = cs) and, in
// MODE_SQUARE, they still contribute (0 - 1)^2 = 1 for the missing diagonal
// and sum_k a_ik^2 to the norms. The rows of dense-path matrices (dslot[seg]
// >= 0) are empty here too, but their norms come from the dense blocks: their
// values are not read (4096 full rows of 4096 entries: 610 us -> 4 us).
template <typename T>
__global__ void k_rows_empty(int64_t n, const int64_t *ars, const int64_t *are, const T *aval,
                             const int32_t *len, const int32_t *seg, const int *dslot,
                             const int64_t *cs, int64_t *ce, double *part) {
  after_previous();
  int lane = lane_id();
  const int g = lane >> 3, gl = lane & 7;  // four groups of 8 lanes
  int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  // a lane per row finds the empty ones, 32 at a time; the warp's four groups
  // of 8 lanes serve them four at a time
  for (int64_t r0 = warp * 32; r0 < n; r0 += nwarps * 32) {
    unsigned empty = __ballot_sync(0xffffffffu, r0 + lane < n && len[r0 + lane] == 0);
    while (empty) {
      int my = -1;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (!empty) break;
        if (k == g) my = __ffs(empty) - 1;
        empty &= empty - 1;
      }
      const bool has = my >= 0;
      const int64_t r = r0 + (has ? my : 0);
      if (has && gl == 0) ce[r] = cs[r];
      if (!part) continue;
      double xs = 0.0;
      const bool norms = has && !(dslot && dslot[seg[r]] >= 0);
      if (norms)
        for (int64_t p = ars[r] + gl; p < are[r]; p += 8) {
          double x = double(aval[p]);
          xs += x * x;
        }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) xs += __shfl_xor_sync(0xffffffffu, xs, o, 8);
      if (norms && gl == 0) {
        part[2 * r] = 1.0;
        part[2 * r + 1] = xs;
      }
    }
  }
}

int sm_count() {
  static const int n = [] {  // once, thread-safe (server lanes launch from several threads)
    int dev = 0, v = 0;
    SGN_CUDA(cudaGetDevice(&dev));
    SGN_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev));
    return v;
  }();
  return n;
}

int grid_cap(int64_t items, int per_block, int per_sm) {
  int64_t g = (items + per_block - 1) / per_block;
  int64_t cap = int64_t(sm_count()) * per_sm;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return int(g);
}

}  // namespace

void launch_bounds(int64_t n, const Rows &A, int64_t nnzA, const Rows &B, const int32_t *seg,
                   const int *active,
                   int mode, int groups, float group_margin, int band, float band_min_eff,
                   const int *dslot, const int64_t *moff, int32_t *lo, int32_t *len,
                   int64_t *ub, int32_t *lists, int *counters, unsigned long long *mults,
                   double *band_work, unsigned char *bandrow, int4 *binfo, int2 *ends,
                   const BandSpans &bspans, const BandSpans &cspans, void *head,
                   size_t head_bytes, cudaStream_t s) {
  if (n == 0) {
    SGN_CUDA(cudaMemsetAsync(head, 0, head_bytes, s));
    return;
  }
  launch_next(k_row_info, grid_cap(n, 256, 8), 256, 0, s, n, B.rs, B.re, B.col, binfo, ends,
              bspans, static_cast<unsigned long long *>(head), int(head_bytes / 8));
  auto run = [&](auto kern, int tile) {
    launch_next(kern, grid_cap(n, tile, 8), BOUNDS_T, 0, s, n, A.rs, A.re, A.col, binfo, seg,
                active, mode, groups, group_margin, band, band_min_eff, dslot, moff, lo, len, ub,
                lists, counters, mults, band_work, bandrow, cspans);
  };
  // Few rows: 16 lanes each, for the latency of a row. Rows of many entries,
  // where a lane per row would not fill the chip: 8. Otherwise a lane per row,
  // whose chain of loads before the first entry serves the most rows at once
  // (the bounds of 24 products of a batch of 512 banded matrices: 3.5 ms, with 8 lanes 4.6)
  if (n < 152 * 64)
    run(k_bounds<16, 16>, 16);
  else if (n < 152 * 8 * 256 && nnzA / n >= 16)
    run(k_bounds<8, 64>, 64);
  else
    run(k_bounds<1, 256>, 256);
}

template <typename T, int MODE, int G, int LOOP = LOOP_ROW>
static void group_launch(int rows, int64_t n, const Rows &A, const T *aval, const Rows &B,
                         const T *bval, const int2 *ends, const int32_t *lo, const int32_t *len,
                         const int32_t *lists, int *ctr, int cls, const int64_t *cs, int64_t *ce,
                         int32_t *ccol, T *cval, double *part, cudaStream_t s) {
  if (rows <= 0) return;
  launch_next(k_num_group<T, MODE, G, LOOP>,
              grid_cap(rows, WARPS_PER_CTA * (32 / G), group_occ<T, LOOP>()), WARPS_PER_CTA * 32, 0,
              s, A.rs, A.re, A.col, aval, B.rs, B.re, B.col, bval, ends, lo, len,
              lists + int64_t(cls) * n, ctr, cls, cs, ce, ccol, cval, part);
}

template <typename T, int MODE>
static void num_launch(int64_t n, const int *rows, bool few, const Rows &A, const T *aval,
                       const Rows &B, const T *bval, const int2 *ends, const int32_t *lo,
                       const int32_t *len, const int32_t *lists, int *ctr, const int64_t *cs,
                       int64_t *ce, int32_t *ccol, T *cval, double *part, cudaStream_t s) {
  if (few) {
    group_launch<T, MODE, 32, LOOP_AHEAD>(rows[RC_G32], n, A, aval, B, bval, ends, lo, len, lists,
                                          ctr, RC_G32, cs, ce, ccol, cval, part, s);
    return;
  }
  group_launch<T, MODE, 32>(rows[RC_G32], n, A, aval, B, bval, ends, lo, len, lists, ctr, RC_G32,
                            cs, ce, ccol, cval, part, s);
  // FP32: the 16-lane class holds row pairs (GROUPS_PAIRS)
  group_launch<T, MODE, 16, sizeof(T) == 4 ? LOOP_PAIR : LOOP_ROW>(
      rows[RC_G16], n, A, aval, B, bval, ends, lo, len, lists, ctr, RC_G16, cs, ce, ccol, cval,
      part, s);
  if constexpr (sizeof(T) == 8)
    group_launch<T, MODE, 8>(rows[RC_G8], n, A, aval, B, bval, ends, lo, len, lists, ctr, RC_G8,
                             cs, ce, ccol, cval, part, s);
}

template <typename T, int MODE, int P, int KIND>
static void wide_launch(int rows, const Rows &A, const T *aval, const Rows &B, const T *bval,
                        const WideTable &wt, const int32_t *lo, const int32_t *len,
                        const int32_t *list, int *ctr, int cls, const int64_t *cs, int64_t *ce,
                        int32_t *ccol, T *cval, double *part, cudaStream_t s) {
  constexpr size_t sm = wide_smem<T, MODE>();
  static const bool attr = [] {  // once, thread-safe
    SGN_CUDA(cudaFuncSetAttribute(k_num_wide<T, MODE, P, KIND>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, int(sm)));
    return true;
  }();
  (void)attr;
  launch_next(k_num_wide<T, MODE, P, KIND>, grid_cap(rows, WIDE_WARPS / P, wide_occ<T, KIND>()),
              WIDE_WARPS * 32, sm, s, A.rs, A.re, A.col, aval, B.rs, B.re, B.col, bval, wt.binfo,
              wt.seg, wt.moff, wt.off, wt.sh, wt.stride, lo, len, list, ctr, cls, cs, ce, ccol,
              cval, part);
}

template <typename T, int MODE>
static void wide_launch_p(int rows, int p, const Rows &A, const T *aval, const Rows &B,
                          const T *bval, const WideTable &wt, const int32_t *lo,
                          const int32_t *len, const int32_t *list, int *ctr, int cls,
                          const int64_t *cs, int64_t *ce, int32_t *ccol, T *cval, double *part,
                          cudaStream_t s) {
#define SGN_WIDE(P, KIND) \
  wide_launch<T, MODE, P, KIND>(rows, A, aval, B, bval, wt, lo, len, list, ctr, cls, cs, ce, ccol, \
                                cval, part, s)
  if (cls == RC_LONG) {
    SGN_WIDE(8, WIDE_LONG);
  } else if (cls != RC_CTA) {  // rows of the 32-lane class
    if (p >= 8) SGN_WIDE(8, WIDE_NARROW);
    else SGN_WIDE(4, WIDE_NARROW);
  } else if (p >= 8) {
    SGN_WIDE(8, WIDE_ROWS);
  } else if (p >= 4) {
    SGN_WIDE(4, WIDE_ROWS);
  } else if (p >= 2) {
    SGN_WIDE(2, WIDE_ROWS);
  } else {
    SGN_WIDE(1, WIDE_ROWS);
  }
#undef SGN_WIDE
}

void launch_col_blocks(int64_t n, const Rows &B, const int32_t *seg, const int64_t *moff, int sh,
                       int stride, int *off, cudaStream_t s) {
  if (n == 0) return;
  launch_next(k_col_blocks, grid_cap(n, 8, 16), 256, 0, s, n, B.rs, B.re, B.col, seg, moff, sh,
              stride, off);
}

int wide_block_shift(int64_t max_n) {
  int sh = 5;
  while (sh < 9 && (max_n >> sh) >= 64) ++sh;
  return sh;
}

template <typename T>
void launch_numeric_wide(int64_t n, int cls, int rows, double mean_b, const Rows &A, const T *aval,
                         const Rows &B, const T *bval, int mode, const WideTable &wt,
                         const int32_t *lo, const int32_t *len, const int32_t *lists,
                         int *counters, const int64_t *cs, int64_t *ce, int32_t *ccol, T *cval,
                         double *part, cudaStream_t s) {
  if (rows <= 0) return;
  // warps per row: about 64 (FP32) or 128 (FP64) entries of a B row per warp, a
  // pass for each where rows are few
  const double per = cls != RC_CTA ? 32.0 : sizeof(T) == 8 ? 128.0 : 64.0;
  int p = mean_b >= 8 * per ? 8 : mean_b >= 4 * per ? 4 : mean_b >= 2 * per ? 2 : 1;
  // and all eight where the rows leave warps idle: beside one full row, the rows that
  // have it among their k are as wide, and the mean says nothing of them (the solve of
  // a tridiagonal matrix of order 65536 with one full row: 216 ms without, 171 with)
  while (p < 8 && int64_t(rows) * p < int64_t(sm_count()) * 16) p *= 2;
  const int32_t *list = lists + int64_t(cls) * n;
  if (mode == MODE_SQUARE)
    wide_launch_p<T, MODE_SQUARE>(rows, p, A, aval, B, bval, wt, lo, len, list, counters, cls, cs,
                                  ce, ccol, cval, part, s);
  else
    wide_launch_p<T, MODE_UPDATE>(rows, p, A, aval, B, bval, wt, lo, len, list, counters, cls, cs,
                                  ce, ccol, cval, part, s);
}
template void launch_numeric_wide<double>(int64_t, int, int, double, const Rows &, const double *,
                                          const Rows &, const double *, int, const WideTable &,
                                          const int32_t *, const int32_t *, const int32_t *, int *,
                                          const int64_t *, int64_t *, int32_t *, double *,
                                          double *, cudaStream_t);
template void launch_numeric_wide<float>(int64_t, int, int, double, const Rows &, const float *,
                                         const Rows &, const float *, int, const WideTable &,
                                         const int32_t *, const int32_t *, const int32_t *, int *,
                                         const int64_t *, int64_t *, int32_t *, float *, double *,
                                         cudaStream_t);

template <typename T>
void launch_numeric(int64_t n, const int *rows, int empty, bool shared, bool few, const Rows &A, const T *aval,
                    const Rows &B, const T *bval, int mode, const int2 *ends, const int32_t *lo,
                    const int32_t *len, const int32_t *seg, const int *dslot,
                    const int32_t *lists, int *counters, const int64_t *cs, int64_t *ce,
                    int32_t *ccol, T *cval, double *part, cudaStream_t s) {
  if (n == 0) return;
  if (empty > 0) {
    launch_next(k_rows_empty<T>, grid_cap(n, 8 * 32, 16), 256, 0, s, n, A.rs, A.re, aval, len, seg,
                dslot, cs, ce, mode == MODE_SQUARE ? part : nullptr);
  }
  if (shared) return;
  if (mode == MODE_SQUARE)
    num_launch<T, MODE_SQUARE>(n, rows, few, A, aval, B, bval, ends, lo, len, lists, counters, cs,
                               ce, ccol, cval, part, s);
  else
    num_launch<T, MODE_UPDATE>(n, rows, few, A, aval, B, bval, ends, lo, len, lists, counters, cs,
                               ce, ccol, cval, part, s);
}

template void launch_numeric<double>(int64_t, const int *, int, bool, bool, const Rows &, const double *,
                                     const Rows &, const double *, int, const int2 *,
                                     const int32_t *, const int32_t *, const int32_t *,
                                     const int *, const int32_t *, int *, const int64_t *,
                                     int64_t *, int32_t *, double *, double *, cudaStream_t);
template void launch_numeric<float>(int64_t, const int *, int, bool, bool, const Rows &, const float *,
                                    const Rows &, const float *, int, const int2 *,
                                    const int32_t *, const int32_t *, const int32_t *, const int *,
                                    const int32_t *, int *, const int64_t *, int64_t *, int32_t *,
                                    float *, double *, cudaStream_t);

}  // namespace sgn
