// CSR utilities of the sign solver: validation, the reproducible 1-norm and
// scaling of step a1, prefix scans, block-diagonal assembly of batches and
// deterministic per-matrix reductions.
#include <cooperative_groups.h>

#include <cfloat>

#include "common.cuh"
#include "kernels.h"
#include "seg.cuh"

namespace cg = cooperative_groups;

namespace sgn {

namespace {

__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }

template <typename F>
__device__ __forceinline__ void for_each_row_warp(int64_t n, F f) {
  int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = warp; r < n; r += nwarps) f(r);
}

// Rows taken by groups of 8 lanes, four rows per warp at a time: for short
// rows (an input A has a few to a few tens of entries per row). f(r, has, gl)
// is called by every lane of the warp, has = false for a group without a row.
template <typename F>
__device__ __forceinline__ void for_each_row_group8(int64_t n, F f) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r0 = warp * 4; r0 < n; r0 += nwarps * 4) {
    const int64_t r = r0 + (lane >> 3);
    f(r < n ? r : r0, r < n, lane & 7);
  }
}

int grid_for(int64_t items, int per_block, int cap = 152 * 16) {
  int64_t g = (items + per_block - 1) / per_block;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return int(g);
}

// ------------------------------------------------------------ validation
__global__ void k_validate(int64_t n, int64_t nnz, const int64_t *rp, const int32_t *col,
                           const double *val, int *flag) {
  after_previous();
  int lane = lane_id();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (rp[0] != 0 || rp[n] != nnz) atomicOr(flag, 1);
  }
  for_each_row_warp(n, [&](int64_t r) {
    int64_t b = rp[r], e = rp[r + 1];
    if (e < b || b < 0 || e > nnz) {
      if (lane == 0) atomicOr(flag, 1);
      return;
    }
    bool bad = false;
    for (int64_t p = b + lane; p < e; p += 32) {
      int32_t c = col[p];
      if (c < 0 || c >= n) bad = true;
      if (p > b && col[p - 1] >= c) bad = true;
      if (!isfinite(val[p])) bad = true;
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(flag, 1);
  });
}

// The same checks for a batch of matrices in one launch: 8 lanes per row of
// all of them (row_off: exclusive prefix of the row counts), the matrix
// found by binary search; thread m also checks matrix m's first and last
// row pointer.
__global__ void k_validate_batch(int count, const ValidateJob *jobs, const int64_t *row_off,
                                 int *flags) {
  after_previous();
  const int64_t tid = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (tid < count) {
    const ValidateJob &j = jobs[tid];
    if (j.rp[0] != 0 || j.rp[j.n] != j.nnz) atomicOr(flags + tid, 1);
  }
  for_each_row_group8(row_off[count], [&](int64_t g, bool has, int gl) {
    if (!has) return;
    int lo = 0, hi = count - 1;  // the last matrix whose first row is <= g
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (row_off[mid] <= g) lo = mid; else hi = mid - 1;
    }
    const ValidateJob &j = jobs[lo];
    const int64_t r = g - row_off[lo];
    const int64_t b = j.rp[r], e = j.rp[r + 1];
    if (e < b || b < 0 || e > j.nnz) {
      if (gl == 0) atomicOr(flags + lo, 1);
      return;
    }
    bool bad = false;
    for (int64_t p = b + gl; p < e; p += 8) {
      const int32_t c = j.col[p];
      if (c < 0 || c >= j.n) bad = true;
      if (p > b && j.col[p - 1] >= c) bad = true;
      if (!isfinite(j.val[p])) bad = true;
    }
    if (bad) atomicOr(flags + lo, 1);
  });
}

// ------------------------------------------------------------ gathered copies
// One CTA per chunk (grid-stride), 16-byte words with up to three 4-byte words
// before and after them (every chunk's length and address is a multiple of 4).
// Where the two sides are offset against each other, the far side (host memory,
// whose accesses should be whole lines: src of a chunk read from the host, else
// dst) is taken in aligned 16-byte words and the near one word by word. A
// batch's results go into arrays packed one after another, which are seldom
// aligned: 1.2 GB took 11.5 ms in 4-byte words, now 9.1 (8.9 where both start on
// a line).
__global__ void k_copy_chunks(int count, const CopyChunk *chunks) {
  constexpr int U = 4;  // 16-byte words per thread in flight
  const int T = blockDim.x, t = threadIdx.x;
  for (int c = blockIdx.x; c < count; c += gridDim.x) {
    const CopyChunk ch = chunks[c];
    const uint32_t *s1 = static_cast<const uint32_t *>(ch.src);
    uint32_t *d1 = static_cast<uint32_t *>(ch.dst);
    const int64_t n1 = ch.bytes >> 2;
    const uintptr_t a = reinterpret_cast<uintptr_t>(s1), b = reinterpret_cast<uintptr_t>(d1);
    const uintptr_t far = ch.host_src ? a : b;
    const int64_t head = min(n1, int64_t((16u - (far & 15u)) & 15u) >> 2);
    const int64_t n4 = (n1 - head) >> 2, tail = head + 4 * n4;
    if (t < head) d1[t] = s1[t];
    if (t < n1 - tail) d1[tail + t] = s1[tail + t];
    s1 += head;
    d1 += head;
    const bool same = ((a ^ b) & 15u) == 0;
    if (same) {
      const int4 *s4 = reinterpret_cast<const int4 *>(s1);
      int4 *d4 = reinterpret_cast<int4 *>(d1);
      for (int64_t i = t; i < n4; i += U * T) {
        int4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i + u * T < n4) v[u] = s4[i + u * T];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i + u * T < n4) d4[i + u * T] = v[u];
      }
    } else if (ch.host_src) {
      const int4 *s4 = reinterpret_cast<const int4 *>(s1);
      for (int64_t i = t; i < n4; i += U * T) {
        int4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i + u * T < n4) v[u] = s4[i + u * T];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i + u * T < n4) {
            uint32_t *d = d1 + 4 * (i + u * T);
            d[0] = uint32_t(v[u].x);
            d[1] = uint32_t(v[u].y);
            d[2] = uint32_t(v[u].z);
            d[3] = uint32_t(v[u].w);
          }
      }
    } else {
      int4 *d4 = reinterpret_cast<int4 *>(d1);
      for (int64_t i = t; i < n4; i += U * T) {
        int4 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i + u * T < n4) {
            const uint32_t *s = s1 + 4 * (i + u * T);
            v[u] = make_int4(int(s[0]), int(s[1]), int(s[2]), int(s[3]));
          }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (i + u * T < n4) d4[i + u * T] = v[u];
      }
    }
  }
}

// ------------------------------------------------------------ readback
// bytes (a multiple of 8) of src into mapped host memory, then the flag: the
// host polls it instead of a copy's completion.
constexpr int PUB_T = 1024;
__global__ void __launch_bounds__(PUB_T)
    k_publish(const unsigned long long *src, unsigned long long *dst, int64_t words,
              volatile unsigned *flag, unsigned seq) {
  after_previous();
  for (int64_t i = threadIdx.x; i < words; i += PUB_T) dst[i] = src[i];
  __threadfence_system();
  __syncthreads();
  if (threadIdx.x == 0) *flag = seq;
}

// ------------------------------------------------------------ footprint statistics
// Per row: diagonal magnitude, off-diagonal sum and farthest column, folded
// into the matrix-wide Gershgorin gap, row-sum bound and half-bandwidth.
__global__ void k_gersh(int64_t n, const int64_t *rp, const int32_t *col, const double *val,
                        GershStats *g) {
  after_previous();
  int lane = lane_id();
  for_each_row_warp(n, [&](int64_t r) {
    double diag = 0.0, off = 0.0;
    long long bw = 0;
    for (int64_t p = rp[r] + lane; p < rp[r + 1]; p += 32) {
      int64_t c = col[p];
      double a = fabs(val[p]);
      if (c == r) diag += a; else off += a;
      long long d = c > r ? c - r : r - c;
      bw = d > bw ? d : bw;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      diag += __shfl_xor_sync(0xffffffffu, diag, o);
      off += __shfl_xor_sync(0xffffffffu, off, o);
      long long b2 = __shfl_xor_sync(0xffffffffu, bw, o);
      bw = b2 > bw ? b2 : bw;
    }
    if (lane == 0) {
      double gap = diag - off, rowsum = diag + off;
      if (gap > 0.0)
        atomicMin(&g->min_gap_bits, (unsigned long long)__double_as_longlong(gap));
      else
        atomicOr(&g->nogap, 1);
      atomicMax(&g->max_rowsum_bits, (unsigned long long)__double_as_longlong(rowsum));
      atomicMax(&g->max_bw, bw);
    }
  });
}

// ------------------------------------------------------------ scan
constexpr int SCAN_T = 1024;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_TILE = SCAN_T * SCAN_ITEMS;

// Exclusive scan of v over the block (1024 threads); *total gets the sum.
__device__ int64_t block_excl_scan(int64_t v, int64_t *sm, int64_t *total) {
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sm[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int64_t t = sm[lane];
    int64_t u = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int64_t y = __shfl_up_sync(0xffffffffu, u, o);
      if (lane >= o) u += y;
    }
    sm[lane] = u - t;
    if (lane == 31) sm[32] = u;
  }
  __syncthreads();
  int64_t r = sm[warp] + x - v;
  if (total) *total = sm[32];
  __syncthreads();
  return r;
}

// blockIdx.y: the scan, its tile totals at tmp + blockIdx.y * tmp_stride.
__global__ void __launch_bounds__(SCAN_T)
    k_scan_reduce(int64_t n, ScanJobs J, int64_t *tmp, int64_t tmp_stride) {
  after_previous();
  __shared__ int64_t sm[33];
  const int64_t *cnt = blockIdx.y == 0 ? J.cnt[0] : blockIdx.y == 1 ? J.cnt[1] : J.cnt[2];
  int64_t base = int64_t(blockIdx.x) * SCAN_TILE + int64_t(threadIdx.x) * SCAN_ITEMS;
  int64_t v = 0;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i)
    if (base + i < n) v += cnt[base + i];
  int64_t total;
  block_excl_scan(v, sm, &total);
  if (threadIdx.x == 0) tmp[blockIdx.y * tmp_stride + blockIdx.x] = total;
}

// A tile's scan: the tiles before it are added from their totals in tmp (a
// single tile has none). seg, eoff (nullable): the scan's value at the end of
// each matrix; total (nullable): the sum of all.
__global__ void __launch_bounds__(SCAN_T)
    k_scan_final(int64_t n, ScanJobs J, const int64_t *tmp, int64_t tmp_stride,
                 const int32_t *seg, int64_t *eoff) {
  after_previous();
  __shared__ int64_t sm[33];
  const int y = blockIdx.y;  // picked by comparison: an indexed parameter is copied to local memory
  static_assert(SCAN_JOBS == 3, "three to pick from");
  const int64_t *cnt = y == 0 ? J.cnt[0] : y == 1 ? J.cnt[1] : J.cnt[2];
  int64_t *const out = y == 0 ? J.out[0] : y == 1 ? J.out[1] : J.out[2];
  int64_t *const total = y == 0 ? J.total[0] : y == 1 ? J.total[1] : J.total[2];
  tmp += blockIdx.y * tmp_stride;
  int64_t before = 0;
  if (blockIdx.x > 0) {
    int64_t v = 0;
    for (int64_t i = threadIdx.x; i < blockIdx.x; i += SCAN_T) v += tmp[i];
    block_excl_scan(v, sm, &before);
  }
  int64_t base = int64_t(blockIdx.x) * SCAN_TILE + int64_t(threadIdx.x) * SCAN_ITEMS;
  int64_t v[SCAN_ITEMS];
  int64_t s = 0;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    v[i] = base + i < n ? cnt[base + i] : 0;
    s += v[i];
  }
  int64_t ex = block_excl_scan(s, sm, nullptr) + before;
#pragma unroll
  for (int i = 0; i < SCAN_ITEMS; ++i) {
    ex += v[i];
    const int64_t r = base + i;
    if (r >= n) break;
    out[r + 1] = ex;
    if (eoff && (r + 1 == n || seg[r + 1] != seg[r])) eoff[seg[r] + 1] = ex;
    if (total && r + 1 == n) *total = ex;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    out[0] = 0;
    if (eoff) eoff[0] = 0;
  }
}

// ------------------------------------------------------------ assembly
__device__ __forceinline__ int find_block(const int64_t *off, int nb, int64_t r) {
  int lo = 0, hi = nb;  // off[lo] <= r < off[hi]
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (off[mid] <= r)
      lo = mid;
    else
      hi = mid;
  }
  return lo;
}

__global__ void k_asm_lens(int nblocks, const AsmBlock *blocks, const int64_t *boff, int64_t n,
                           int64_t *lens) {
  after_previous();
  for (int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < n;
       r += int64_t(gridDim.x) * blockDim.x) {
    int b = find_block(boff, nblocks, r);
    const AsmBlock &B = blocks[b];
    int64_t sr = B.row0 + (r - boff[b]);
    lens[r] = B.rp[sr + 1] - B.rp[sr];
  }
}

__global__ void k_asm_vals(int nblocks, const AsmBlock *blocks, const int64_t *boff, int64_t n,
                           const int64_t *drp, int32_t *dcol, void *dval, int dst_f32) {
  after_previous();
  // 8 lanes per row, four rows per warp at a time (rows are short)
  constexpr int L = 8;
  const int lane = lane_id(), gl = lane % L;
  const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = warp * (32 / L) + lane / L; r < n; r += nwarps * (32 / L)) {
    int b = find_block(boff, nblocks, r);
    const AsmBlock B = blocks[b];
    int64_t sr = B.row0 + (r - boff[b]);
    int64_t sb = B.rp[sr], se = B.rp[sr + 1], d = drp[r] - sb;
    if (B.val_f32 && dst_f32) {  // FP32 to FP32: the values as they are
      const float *sv = static_cast<const float *>(B.val);
      float *dv = static_cast<float *>(dval);
      for (int64_t p = sb + gl; p < se; p += L) {
        dcol[d + p] = int32_t(B.col[p] + B.col_shift);
        dv[d + p] = sv[p];
      }
    } else {
      for (int64_t p = sb + gl; p < se; p += L) {
        dcol[d + p] = int32_t(B.col[p] + B.col_shift);
        double v = B.val_f32 ? double(static_cast<const float *>(B.val)[p])
                             : static_cast<const double *>(B.val)[p];
        if (dst_f32)
          static_cast<float *>(dval)[d + p] = __double2float_rn(v);
        else
          static_cast<double *>(dval)[d + p] = v;
      }
    }
  }
}

__global__ void k_fill_seg(int nb, const int64_t *moff, int64_t n, int32_t *seg) {
  after_previous();
  for (int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < n;
       r += int64_t(gridDim.x) * blockDim.x)
    seg[r] = find_block(moff, nb, r);
}

// ------------------------------------------------------------ 1-norm (step a1)
// ||A||_1 = max_j sum_i |a_ij|, made independent of summation order: with
// M = max |a_ij| < 2^e every |a_ij| is put on the grid 2^(e-62) by one
// round-to-nearest-even conversion of the exact product |a| * 2^(62-e); the
// column sums are exact 128-bit integers (two 64-bit atomics with carry), and
// the largest one, hi * 2^64 + lo, comes back as
// ((double)hi * 2^64 + (double)lo) * 2^(e-62).

// p[m] = max(p[m], v) for every lane of the warp (v = 0: nothing to add). The
// lanes of one matrix are reduced first, and the value is read before the
// atomic: it only grows, so a maximum at or below it needs none. A large
// matrix's rows otherwise queue on one address (262144 rows: about 170 us for
// each of the three maxima, now 41, 4 and 12).
__device__ __forceinline__ void max_into(unsigned long long *p, int m, unsigned long long v) {
  const int m0 = __shfl_sync(0xffffffffu, m, 0);
  bool put = v != 0ULL;
  if (__all_sync(0xffffffffu, m == m0)) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
      v = w > v ? w : v;
    }
    put = v != 0ULL && lane_id() == 0;
  }
  if (put && *reinterpret_cast<volatile unsigned long long *>(p + m) < v) atomicMax(p + m, v);
}

__device__ __forceinline__ void add128(unsigned long long *lohi, unsigned long long q) {
  unsigned long long old = atomicAdd(&lohi[0], q);
  if (old + q < old) atomicAdd(&lohi[1], 1ULL);
}

__global__ void k_absmax(int64_t n, const int32_t *seg, const int64_t *rp, const double *val,
                         unsigned long long *mmax) {
  after_previous();
  for_each_row_group8(n, [&](int64_t r, bool has, int gl) {
    double m = 0.0;
    if (has)
      for (int64_t p = rp[r] + gl; p < rp[r + 1]; p += 8) m = fmax(m, fabs(val[p]));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o, 8));
    max_into(mmax, seg[r],
             has && gl == 0 && m > 0.0 ? (unsigned long long)__double_as_longlong(m) : 0ULL);
  });
}

__global__ void k_colsum(int64_t n, const int32_t *seg, const int64_t *rp, const int32_t *col,
                         const double *val, const unsigned long long *mmax,
                         unsigned long long *colsum) {
  after_previous();
  for_each_row_group8(n, [&](int64_t r, bool has, int gl) {
    if (!has) return;
    double M = __longlong_as_double((long long)mmax[seg[r]]);
    if (M == 0.0) return;
    int e;
    frexp(M, &e);
    for (int64_t p = rp[r] + gl; p < rp[r + 1]; p += 8) {
      unsigned long long q = __double2ull_rn(ldexp(fabs(val[p]), 62 - e));
      if (q) add128(&colsum[2 * int64_t(col[p])], q);
    }
  });
}

// A whole warp stays in the loop (max_into); its lanes past the end add nothing.
__global__ void k_colmax_hi(int64_t n, const int32_t *seg, const unsigned long long *colsum,
                            unsigned long long *maxhi) {
  after_previous();
  for (int64_t j0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x - lane_id(); j0 < n;
       j0 += int64_t(gridDim.x) * blockDim.x) {
    const int64_t j = j0 + lane_id() < n ? j0 + lane_id() : n - 1;
    max_into(maxhi, seg[j], colsum[2 * j + 1]);
  }
}

__global__ void k_colmax_lo(int64_t n, const int32_t *seg, const unsigned long long *colsum,
                            const unsigned long long *maxhi, unsigned long long *maxlo) {
  after_previous();
  for (int64_t j0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x - lane_id(); j0 < n;
       j0 += int64_t(gridDim.x) * blockDim.x) {
    const int64_t j = j0 + lane_id() < n ? j0 + lane_id() : n - 1;
    const int m = seg[j];
    max_into(maxlo, m, colsum[2 * j + 1] == maxhi[m] ? colsum[2 * j] : 0ULL);
  }
}

__global__ void k_norm_final(int nb, const unsigned long long *mmax,
                             const unsigned long long *maxhi, const unsigned long long *maxlo,
                             double *norm) {
  after_previous();
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= nb) return;
  double M = __longlong_as_double((long long)mmax[m]);
  if (M == 0.0) {
    norm[m] = 0.0;
    return;
  }
  int e;
  frexp(M, &e);
  double d = __dadd_rn(__dmul_rn(__ull2double_rn(maxhi[m]), 18446744073709551616.0),
                       __ull2double_rn(maxlo[m]));
  norm[m] = ldexp(d, e - 62);
}

__global__ void k_scale(int64_t n, const int32_t *seg, const int64_t *rp, double *val,
                        const double *norm) {
  after_previous();
  for_each_row_group8(n, [&](int64_t r, bool has, int gl) {
    if (!has) return;
    double s = norm[seg[r]];
    for (int64_t p = rp[r] + gl; p < rp[r + 1]; p += 8) val[p] = __ddiv_rn(val[p], s);
  });
}

__global__ void k_gather_offsets(int nb, const int64_t *moff, const int64_t *rp, int64_t *out) {
  after_previous();
  int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m <= nb) out[m] = rp[moff[m]];
}

// ------------------------------------------------------------ reductions
// Sums per matrix. A matrix is served by a cluster of RED_C CTAs: with one CTA
// a matrix of 262144 rows took 232 us per sum of two components and 267 us
// per count (one SM's FP64 pipe and load latency bound it). With the clusters
// and the 1-norm's maxima below, the mixed solve of the tridiagonal matrix of
// that order went from 16.3 to 11.9 ms, and to 11.0 with the rows prefetched
// and the maxima reduced per warp (GB300).

// out[m] = the sum of part over matrix m's rows.
__global__ void __cluster_dims__(RED_C, 1, 1) __launch_bounds__(RED_LANES)
    k_seg_reduce(int nb, int per, const int64_t *moff, const double *part, double *out) {
  after_previous();
  __shared__ double sm[RED_T];
  cg::cluster_group cl = cg::this_cluster();
  const int q = int(cl.block_rank()), t = q * RED_LANES + threadIdx.x;
  auto solo = [&](int m) {
    seg_sum_solo(sm, part, 1, 0, moff[m], moff[m + 1]);
    if (threadIdx.x == 0) out[m] = sm[0];
  };
  auto joint = [&](int m) {
    cl.sync();  // CTA 0 has started, and read its sums: its shared memory may be written
    *cl.map_shared_rank(&sm[t], 0) = seg_partial(part, 1, 0, moff[m], moff[m + 1], t);
    cl.sync();
    if (q != 0) return;
    seg_tree(sm);
    if (threadIdx.x == 0) out[m] = sm[0];
  };
  cluster_each(nb, per, moff, blockIdx.x / RED_C, q, solo, joint);
}

// r, x, beta and b of a matrix of n rows from its sums of squares, and its entries.
__device__ __forceinline__ void put_scalars(int64_t n, double rsum, double xsum, int64_t entries,
                                            double c4, double tol_stage, double switch_resid,
                                            MatScalars &ms, int64_t &nnz) {
  const double sn = __dsqrt_rn(double(n));
  const double r = __ddiv_rn(__dsqrt_rn(rsum), sn);
  const double x = __ddiv_rn(__dsqrt_rn(xsum), sn);
  double beta;
  if (r >= switch_resid)
    beta = __dmul_rn(c4, tol_stage);
  else
    beta = __ddiv_rn(__dmul_rn(__dmul_rn(0.75, r), r),
                     __dadd_rn(__dmul_rn(3.0, x), __dmul_rn(__dmul_rn(x, x), x)));
  ms.r = r;
  ms.x = x;
  ms.beta = beta;
  ms.b = __dmul_rn(sn, beta);
  nnz = entries;
}

// The check of a round in one launch: per matrix the sums of the two columns of
// part (warps 0 and 1 of each CTA), the entries of T (warp 2) and from them r,
// x, beta and b.
__global__ void __cluster_dims__(RED_C, 1, 1) __launch_bounds__(3 * RED_LANES)
    k_check_scalars(int nb, int per, const int64_t *moff, const double *part, const int64_t *rs,
                    const int64_t *re, double c4, double tol_stage, double switch_resid,
                    MatScalars *ms, int64_t *nnz) {
  after_previous();
  __shared__ double sm[2][RED_T];
  __shared__ unsigned long long s_cnt;
  cg::cluster_group cl = cg::this_cluster();
  const int q = int(cl.block_rank()), c = threadIdx.x / RED_LANES;
  const int t = q * RED_LANES + lane_id();
  auto put = [&](int m) {
    put_scalars(moff[m + 1] - moff[m], sm[0][0], sm[1][0], int64_t(s_cnt), c4, tol_stage,
                switch_resid, ms[m], nnz[m]);
  };
  auto solo = [&](int m) {
    const int64_t b = moff[m], e = moff[m + 1];
    if (c < 2) {
      seg_sum_solo(sm[c], part, 2, c, b, e);
    } else {
      const unsigned long long k = seg_entries(rs, re, b, e, lane_id(), 32);
      if (lane_id() == 0) s_cnt = k;
    }
    __syncthreads();
    if (threadIdx.x == 0) put(m);
  };
  auto joint = [&](int m) {
    if (threadIdx.x == 0) s_cnt = 0ULL;
    cl.sync();  // CTA 0 has started, and read its sums: its shared memory may be written
    const int64_t b = moff[m], e = moff[m + 1];
    if (c < 2) {
      *cl.map_shared_rank(&sm[c][t], 0) = seg_partial(part, 2, c, b, e, t);
    } else {
      const unsigned long long k = seg_entries(rs, re, b, e, t, RED_T);
      if (lane_id() == 0 && k) atomicAdd(cl.map_shared_rank(&s_cnt, 0), k);
    }
    cl.sync();
    if (q != 0) return;
    if (c < 2) seg_tree(sm[c]);
    __syncthreads();
    if (threadIdx.x == 0) put(m);
  };
  cluster_each(nb, per, moff, blockIdx.x / RED_C, q, solo, joint);
}

__global__ void __cluster_dims__(RED_C, 1, 1) __launch_bounds__(RED_T)
    k_seg_count(int nb, int per, const int64_t *moff, const int64_t *rs, const int64_t *re,
                int64_t *out) {
  after_previous();
  __shared__ unsigned long long sm;  // the matrix's count (joint: CTA 0's)
  cg::cluster_group cl = cg::this_cluster();
  const int q = int(cl.block_rank());
  auto solo = [&](int m) {
    if (threadIdx.x == 0) sm = 0ULL;
    __syncthreads();
    const unsigned long long k = seg_entries(rs, re, moff[m], moff[m + 1], threadIdx.x, RED_T);
    if (lane_id() == 0 && k) atomicAdd(&sm, k);
    __syncthreads();
    if (threadIdx.x == 0) out[m] = int64_t(sm);
  };
  auto joint = [&](int m) {
    if (threadIdx.x == 0) sm = 0ULL;
    cl.sync();
    const unsigned long long k = seg_entries(rs, re, moff[m], moff[m + 1], q * RED_T + threadIdx.x,
                                             RED_C * RED_T);
    if (lane_id() == 0 && k) atomicAdd(cl.map_shared_rank(&sm, 0), k);
    cl.sync();
    if (q == 0 && threadIdx.x == 0) out[m] = int64_t(sm);
  };
  cluster_each(nb, per, moff, blockIdx.x / RED_C, q, solo, joint);
}

// One CTA per extracted matrix: rebased row pointers, shifted columns,
// values widened to FP64.
// blockIdx.y walks the blocks; the gridDim.x CTAs of a block share its rows
// and entries, so that a large matrix is copied by many SMs.
__global__ void k_extract(int nblocks, const ExtractBlock *blocks) {
  after_previous();
  for (int b = blockIdx.y; b < nblocks; b += gridDim.y) {
    const ExtractBlock B = blocks[b];
    const int64_t t0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    const int64_t step = int64_t(gridDim.x) * blockDim.x;
    const int64_t e0 = B.rp[B.row0];
    for (int64_t i = t0; i <= B.nrows; i += step) B.drp[i] = B.rp[B.row0 + i] - e0;
    const int64_t ne = B.rp[B.row0 + B.nrows] - e0;
    for (int64_t p = t0; p < ne; p += step) {
      B.dcol[p] = int32_t(B.col[e0 + p] + B.col_shift);
      B.dval[p] = B.val_f32 ? double(static_cast<const float *>(B.val)[e0 + p])
                            : static_cast<const double *>(B.val)[e0 + p];
    }
  }
}

__global__ void k_row_lengths(int64_t n, const int64_t *rs, const int64_t *re, int64_t *out) {
  after_previous();
  for (int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; r < n;
       r += int64_t(gridDim.x) * blockDim.x)
    out[r] = re[r] - rs[r];
}

__global__ void k_compact_rows(int64_t n, const int64_t *rs, const int64_t *re,
                               const int32_t *col, const void *val, int vsize, const int64_t *orp,
                               int32_t *ocol, void *oval) {
  after_previous();
  int lane = lane_id();
  for_each_row_warp(n, [&](int64_t r) {
    int64_t b = rs[r], e = re[r], d = orp[r];
    for (int64_t p = b + lane; p < e; p += 32) {
      ocol[d + (p - b)] = col[p];
      if (vsize == 8)
        static_cast<double *>(oval)[d + (p - b)] = static_cast<const double *>(val)[p];
      else
        static_cast<float *>(oval)[d + (p - b)] = static_cast<const float *>(val)[p];
    }
  });
}

}  // namespace

void launch_row_lengths(int64_t n, const int64_t *rs, const int64_t *re, int64_t *out,
                        cudaStream_t s) {
  if (n == 0) return;
  launch_next(k_row_lengths, grid_for(n, 256), 256, 0, s, n, rs, re, out);
}

void launch_compact_rows(int64_t n, const int64_t *rs, const int64_t *re, const int32_t *col,
                         const void *val, int vsize, const int64_t *orp, int32_t *ocol,
                         void *oval, cudaStream_t s) {
  if (n == 0) return;
  launch_next(k_compact_rows, grid_for(n, 8), 256, 0, s, n, rs, re, col, val, vsize, orp, ocol,
              oval);
}

void launch_seg_count(int nb, const int64_t *moff, const int64_t *rs, const int64_t *re,
                      int64_t *out, cudaStream_t s) {
  if (nb == 0) return;
  launch_next(k_seg_count, cluster_ctas(nb), RED_T, 0, s, nb, cluster_matrices(nb), moff, rs, re,
              out);
}

void launch_extract(int nblocks, const ExtractBlock *blocks, int64_t max_entries, cudaStream_t s) {
  if (nblocks == 0) return;
  // about 8 entries per thread of a 512-thread CTA, at most 152 CTAs per block
  const int64_t per = (max_entries + 4095) / 4096;
  dim3 grid(unsigned(per < 1 ? 1 : (per > 152 ? 152 : per)), unsigned(nblocks < 65535 ? nblocks : 65535));
  launch_next(k_extract, grid, 512, 0, s, nblocks, blocks);
}

void launch_gersh(int64_t n, const int64_t *rp, const int32_t *col, const double *val,
                  GershStats *g, cudaStream_t s) {
  launch_next(k_gersh, grid_for(n, 8), 256, 0, s, n, rp, col, val, g);
}

void launch_validate(int64_t n, int64_t nnz, const int64_t *rp, const int32_t *col,
                     const double *val, int *flag, cudaStream_t s) {
  launch_next(k_validate, grid_for(n, 8), 256, 0, s, n, nnz, rp, col, val, flag);
}

void launch_validate_batch(int count, const ValidateJob *jobs, const int64_t *row_off,
                           int64_t total_rows, int *flags, cudaStream_t s) {
  if (count < 1) return;
  const int64_t items = total_rows > count ? total_rows : count;
  launch_next(k_validate_batch, grid_for(items, 32), 256, 0, s, count, jobs, row_off, flags);
}

void launch_copy_chunks(int count, const CopyChunk *chunks, cudaStream_t s) {
  if (count < 1) return;
  k_copy_chunks<<<count < 152 * 8 ? count : 152 * 8, 256, 0, s>>>(count, chunks);
  SGN_LAUNCH_CHECK();
}

void launch_publish(const void *src, void *dst, size_t bytes, unsigned *flag, unsigned seq,
                    cudaStream_t s) {
  launch_next(k_publish, 1, PUB_T, 0, s, static_cast<const unsigned long long *>(src),
              static_cast<unsigned long long *>(dst), int64_t(bytes / 8), flag, seq);
}

int64_t scan_tmp_elems(int64_t n) { return (n + SCAN_TILE - 1) / SCAN_TILE + 1; }

static void run_scans(int64_t n, int jobs, const ScanJobs &J, int64_t *tmp, const int32_t *seg,
                      int64_t *eoff, cudaStream_t s) {
  const int64_t nblocks = (n + SCAN_TILE - 1) / SCAN_TILE;
  if (nblocks == 0) {
    for (int j = 0; j < jobs; ++j) {
      SGN_CUDA(cudaMemsetAsync(J.out[j], 0, sizeof(int64_t), s));
      if (J.total[j]) SGN_CUDA(cudaMemsetAsync(J.total[j], 0, sizeof(int64_t), s));
    }
    if (eoff) SGN_CUDA(cudaMemsetAsync(eoff, 0, sizeof(int64_t), s));
    return;
  }
  const dim3 grid{unsigned(nblocks), unsigned(jobs)};
  const int64_t stride = scan_tmp_elems(n);
  if (nblocks > 1) {
    launch_next(k_scan_reduce, grid, SCAN_T, 0, s, n, J, tmp, stride);
  }
  launch_next(k_scan_final, grid, SCAN_T, 0, s, n, J, tmp, stride, seg, eoff);
}

void launch_scans(int64_t n, int jobs, const ScanJobs &J, int64_t *tmp, cudaStream_t s) {
  run_scans(n, jobs, J, tmp, nullptr, nullptr, s);
}

void launch_scan(int64_t n, const int64_t *cnt, int64_t *out, int64_t *tmp, cudaStream_t s,
                 const int32_t *seg, int64_t *eoff, int64_t *total) {
  ScanJobs J = {};
  J.cnt[0] = cnt;
  J.out[0] = out;
  J.total[0] = total;
  run_scans(n, 1, J, tmp, seg, eoff, s);
}

void launch_assemble_rows(int nblocks, const AsmBlock *blocks, const int64_t *boff, int64_t n_dst,
                          int64_t *lens, int64_t *dst_rp, int64_t *scan_tmp, cudaStream_t s) {
  if (n_dst > 0) {
    launch_next(k_asm_lens, grid_for(n_dst, 256), 256, 0, s, nblocks, blocks, boff, n_dst, lens);
  }
  launch_scan(n_dst, lens, dst_rp, scan_tmp, s);
}

void launch_assemble_vals(int nblocks, const AsmBlock *blocks, const int64_t *boff, int64_t n_dst,
                          const int64_t *dst_rp, int32_t *dst_col, void *dst_val, int dst_f32,
                          cudaStream_t s) {
  if (n_dst == 0) return;
  launch_next(k_asm_vals, grid_for(n_dst, 32), 256, 0, s, nblocks, blocks, boff, n_dst, dst_rp,
              dst_col, dst_val, dst_f32);
}

void launch_fill_seg(int nb, const int64_t *moff, int64_t n, int32_t *seg, cudaStream_t s) {
  if (n == 0) return;
  launch_next(k_fill_seg, grid_for(n, 256), 256, 0, s, nb, moff, n, seg);
}

void launch_onenorm(int nb, const int64_t *moff, const int32_t *seg, int64_t n, const int64_t *rp,
                    const int32_t *col, const double *val, unsigned long long *work, double *norm,
                    cudaStream_t s) {
  (void)moff;
  unsigned long long *colsum = work;            // 2n
  unsigned long long *mmax = work + 2 * n;      // nb
  unsigned long long *maxhi = mmax + nb;        // nb
  unsigned long long *maxlo = maxhi + nb;       // nb
  SGN_CUDA(cudaMemsetAsync(work, 0, sizeof(unsigned long long) * size_t(2 * n + 3 * nb), s));
  launch_next(k_absmax, grid_for(n, 32), 256, 0, s, n, seg, rp, val, mmax);
  launch_next(k_colsum, grid_for(n, 32), 256, 0, s, n, seg, rp, col, val, mmax, colsum);
  launch_next(k_colmax_hi, grid_for(n, 256), 256, 0, s, n, seg, colsum, maxhi);
  launch_next(k_colmax_lo, grid_for(n, 256), 256, 0, s, n, seg, colsum, maxhi, maxlo);
  launch_next(k_norm_final, (nb + 127) / 128, 128, 0, s, nb, mmax, maxhi, maxlo, norm);
}

void launch_scale(int64_t n, const int32_t *seg, const int64_t *rp, double *val,
                  const double *norm, cudaStream_t s) {
  launch_next(k_scale, grid_for(n, 32), 256, 0, s, n, seg, rp, val, norm);
}

void launch_gather_offsets(int nb, const int64_t *moff, const int64_t *rp, int64_t *out,
                           cudaStream_t s) {
  launch_next(k_gather_offsets, (nb + 1 + 127) / 128, 128, 0, s, nb, moff, rp, out);
}

void launch_seg_reduce(int nb, const int64_t *moff, const double *part, double *out,
                       cudaStream_t s) {
  if (nb == 0) return;
  launch_next(k_seg_reduce, cluster_ctas(nb), RED_LANES, 0, s, nb, cluster_matrices(nb), moff, part,
              out);
}

void launch_check_scalars(int nb, const int64_t *moff, const double *part, const int64_t *rs,
                          const int64_t *re, double c4, double tol_stage, double switch_resid,
                          MatScalars *ms, int64_t *nnz, cudaStream_t s) {
  if (nb == 0) return;
  launch_next(k_check_scalars, cluster_ctas(nb), 3 * RED_LANES, 0, s, nb, cluster_matrices(nb), moff,
              part, rs, re, c4, tol_stage, switch_resid, ms, nnz);
}

}  // namespace sgn
