// Newton's method with filtering (NMF, Alg. 3.1.1): the dense inverse of the
// current iterate and the Newton update Xbar = (X + X^-1) / 2.
//
// The inverse follows LU with partial pivoting (for each column c the first row
// of largest magnitude at or below c becomes the pivot, the rows below are
// reduced by l = a_rc / a_cc with one rounded product and one rounded
// subtraction per entry), the forward substitution L y = P e for each column
// e of the identity and the back substitution U x = y, both with their sums
// in ascending index order. Every operation is an explicitly rounded FP64
// operation and every entry takes its operations in that order (but for those
// with a zero that k_lu_trail leaves out), so the inverse is the same on every run
// and for every blocking.
//
// The forward substitution rides along with the elimination: the identity's
// rows are swapped and reduced like those of the matrix, [A | I] -> [U | y].
// Columns are taken in panels: k_lu_panel factors a panel in one CTA, and
// k_lu_trail applies its swaps and its reductions, in ascending column order,
// to every column right of it and to the identity, a strip of 4 columns per
// CTA. Four launches per column and one thread per column of the identity
// (a chain of n^2 dependent steps, each waiting on its loads) took 36 ms for
// n = 500; now 8 ms.
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "kernels.h"

namespace sgn {

namespace {

// Product and difference, each rounded once, as fused multiply-adds with an
// exact factor or addend: fma(a, b, -0) is a b rounded (and keeps the sign of
// a zero product), fma(b, -1, a) is a - b rounded. One FP64 warp instruction
// occupies its quarter of the SM for 64 cycles as a DFMA and 76 as a DADD
// (measured), and takes as long in a dependent chain.
// In inline PTX, so that the compiler does not see a product and a difference
// that it could contract into one rounding.
__device__ __forceinline__ double fma_ptx(double a, double b, double c) {
  double r;
  asm("fma.rn.f64 %0, %1, %2, %3;" : "=d"(r) : "d"(a), "d"(b), "d"(c));
  return r;
}
__device__ __forceinline__ double mul_rn(double a, double b) { return fma_ptx(a, b, -0.0); }
__device__ __forceinline__ double sub_rn(double a, double b) { return fma_ptx(b, -1.0, a); }

// |v| as an integer that orders like it; a NaN orders below everything, as in
// a scan with v > best.
__device__ __forceinline__ long long mag_key(double v) {
  const long long k = __double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFll;
  return k > 0x7FF0000000000000ll ? -1ll : k;
}

constexpr int PANEL_T = 1024;        // threads of the panel kernel
constexpr int PANEL_W = 8;           // most columns of a panel
constexpr size_t PANEL_SMEM = 200 * 1024;
constexpr int STRIP = 4;             // columns per CTA of the trailing update
constexpr int TRAIL_T = 256;

// Columns of a panel: as many as fit the panel kernel's shared memory; one,
// worked on in place, when even a column does not fit.
int panel_width(int n) {
  int w = PANEL_W;
  while (w > 1 && size_t(n) * w * sizeof(double) > PANEL_SMEM) w /= 2;
  return w;
}

// inv = I
__global__ void k_inv_init(int n, int ld, double *inv) {
  const int64_t total = int64_t(n) * n;
  for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < total;
       t += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = t / n, j = t - i * n;
    inv[i * ld + j] = i == j ? 1.0 : 0.0;
  }
}

// Factors the panel of columns [c0, c0 + w), rows c0 .. n - 1: one CTA, a
// thread per row (more for long columns), the panel in shared memory column
// by column unless in_place. The pivot of a column is its first row of
// largest magnitude (a NaN diagonal keeps its row, as a sequential scan from
// there would); a largest magnitude of 0 marks the matrix singular. swaps[c]
// is the row swapped with row c; *wild becomes 1 with a multiplier that is not
// finite. Bound by the FP64 pipe of one SM (the
// divisions) and the barriers: two per column.
__global__ void __launch_bounds__(PANEL_T)
    k_lu_panel(int n, int ld, double *lu, int c0, int w, int in_place, int *swaps,
               int *singular, int *wild) {
  after_previous();
  extern __shared__ double panel[];
  __shared__ long long sv[PANEL_T / 32];
  __shared__ int si[PANEL_T / 32], s_pivot;
  if (*singular) return;
  const int R = n - c0, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double *const G = lu + int64_t(c0) * ld + c0;
  // entry (row r, column k) of the panel at P[k * sk + r * sr]
  double *const P = in_place ? G : panel;
  const int64_t sk = in_place ? 1 : R, sr = in_place ? ld : 1;
  if (!in_place) {
    for (int t = tid; t < R * w; t += PANEL_T) panel[(t % w) * R + t / w] = G[int64_t(t / w) * ld + t % w];
    __syncthreads();
  }
  for (int k = 0; k < w; ++k) {
    long long best = -1;
    int bi = R;
    for (int r = k + tid; r < R; r += PANEL_T) {
      const long long v = mag_key(P[k * sk + r * sr]);
      if (v > best) {  // rows ascend within a thread: ties keep the first
        best = v;
        bi = r;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) {
        best = ov;
        bi = oi;
      }
    }
    if (lane == 0) {
      sv[warp] = best;
      si[warp] = bi;
    }
    __syncthreads();
    if (warp == 0) {
      best = sv[lane];
      bi = si[lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ov > best || (ov == best && oi < bi)) {
          best = ov;
          bi = oi;
        }
      }
      const double d = P[k * sk + k * sr];
      if (d != d) {  // NaN pivot candidate: kept
        best = 1;
        bi = k;
      }
      const int p = bi < R ? bi : k;
      __syncwarp();
      if (best == 0) {
        if (lane == 0) s_pivot = -1;
      } else {
        if (lane < w && p != k) {
          const double t = P[lane * sk + k * sr];
          P[lane * sk + k * sr] = P[lane * sk + p * sr];
          P[lane * sk + p * sr] = t;
        }
        if (lane == 0) {
          s_pivot = p;
          swaps[c0 + k] = c0 + p;
        }
      }
    }
    __syncthreads();
    if (s_pivot < 0) {
      if (tid == 0) *singular = 1;
      return;
    }
    const double piv = P[k * sk + k * sr];
    for (int r = k + 1 + tid; r < R; r += PANEL_T) {
      const double l = __ddiv_rn(P[k * sk + r * sr], piv);
      P[k * sk + r * sr] = l;
      if ((__double2hiint(l) & 0x7FF00000) == 0x7FF00000) *wild = 1;
      for (int j = k + 1; j < w; ++j)
        P[j * sk + r * sr] = sub_rn(P[j * sk + r * sr], mul_rn(l, P[j * sk + k * sr]));
    }
    __syncthreads();
  }
  if (!in_place)
    for (int t = tid; t < R * w; t += PANEL_T) G[int64_t(t / w) * ld + t % w] = panel[(t % w) * R + t / w];
}

// The panel's swaps and reductions on a strip of 4 columns: of lu right of the
// panel, then of inv. W: the panel's width. Bound by the FP64 pipe. A strip whose
// part of U is all +0 (columns of the identity whose row has not been a pivot
// yet: half of them on average) is left as it is after the swaps: a - l 0 = a
// for every finite l, but that -0 - l 0 is +0 for l < 0. So U may keep a zero of the
// other sign, which the inverse does not show: y never holds -0 (it starts from the
// identity), and s - (+-0) x = s for every other s. Strips of 8 columns took 21 us per launch for n = 500, as
// one CTA per SM bounded them; the whole solve went from 57.2 to 54.8 ms.
template <int W>
__global__ void __launch_bounds__(TRAIL_T)
    k_lu_trail(int n, int ld, double *lu, double *inv, int c0, const int *swaps,
               const int *singular, const int *wild) {
  after_previous();
  __shared__ int rows[2 * W], src[2 * W];
  __shared__ int nrows;
  __shared__ double moved[2 * W][STRIP], L[W][W], U[W][STRIP];
  if (*singular) return;
  const int c1 = c0 + W, lu_strips = (n - c1 + STRIP - 1) / STRIP;
  const bool in_lu = int(blockIdx.x) < lu_strips;
  const int j = threadIdx.x % STRIP, rr = threadIdx.x / STRIP;
  constexpr int RT = TRAIL_T / STRIP;  // rows at a time
  const int col = in_lu ? c1 + int(blockIdx.x) * STRIP + j
                        : (int(blockIdx.x) - lu_strips) * STRIP + j;
  double *const A = (in_lu ? lu : inv) + col;  // column col
  const bool has = col < n;
  // where the contents of the rows that the swaps touch come from
  if (threadIdx.x == 0) {
    int m = 0;
    auto slot = [&](int r) {
      for (int i = 0; i < m; ++i)
        if (rows[i] == r) return i;
      rows[m] = src[m] = r;
      return m++;
    };
    for (int k = 0; k < W; ++k) {
      const int a = slot(c0 + k), b = slot(swaps[c0 + k]);
      const int t = src[a];
      src[a] = src[b];
      src[b] = t;
    }
    nrows = m;
  }
  for (int t = threadIdx.x; t < W * W; t += TRAIL_T)
    L[t / W][t % W] = lu[int64_t(c0 + t / W) * ld + c0 + t % W];
  __syncthreads();
  for (int i = rr; i < nrows; i += RT)
    if (has) moved[i][j] = A[int64_t(src[i]) * ld];
  __syncthreads();
  // the panel's rows, reduced one after another (row c0 + k is slot k or was
  // listed before it): U
  for (int i = rr; i < nrows; i += RT)
    if (has && (rows[i] < c0 || rows[i] >= c1)) A[int64_t(rows[i]) * ld] = moved[i][j];
  if (rr == 0 && has) {
    double u[W];
    for (int i = 0; i < nrows; ++i)
      if (rows[i] < c1) U[rows[i] - c0][j] = moved[i][j];
#pragma unroll
    for (int k = 0; k < W; ++k) {
      double a = U[k][j];
#pragma unroll
      for (int i = 0; i < k; ++i) a = sub_rn(a, mul_rn(L[k][i], u[i]));
      u[k] = a;
      U[k][j] = a;
      A[int64_t(c0 + k) * ld] = a;
    }
  }
  __syncthreads();
  double u[W];
  bool some = false;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    u[k] = has ? U[k][j] : 0.0;
    some = some || __double_as_longlong(u[k]) != 0;
  }
  if (!__syncthreads_or(some) && *wild == 0) return;
  if (!has) return;
#pragma unroll 2
  for (int r = c1 + rr; r < n; r += RT) {
    const double *l = lu + int64_t(r) * ld + c0;
    double a = A[int64_t(r) * ld];
#pragma unroll
    for (int k = 0; k < W; ++k) a = sub_rn(a, mul_rn(l[k], u[k]));
    A[int64_t(r) * ld] = a;
  }
}

// U x = y for 32 columns of inv per CTA, in place: for i = n - 1 .. 0,
// x_i = (y_i - sum_{j > i, ascending} u_ij x_j) / u_ii. A sum starts with the
// x found last, so the n^2 / 2 subtractions of a column are one dependent
// chain of 64-cycle instructions, which bounds the kernel. Warp 0 runs the
// chain and nothing else; warps 1 .. 3, on the other quarters of the SM,
// prepare the products, BACK_C at a time, one chunk ahead, through shared
// memory. Only the product with the x found last is left to warp 0: the
// chunks of row i start at j = i + 2, whose x is known a row earlier. One warp
// doing both took 186 cycles per term (11.2 ms for n = 500), now 84 (5.5 ms).
constexpr int BACK_P = 32;          // products per producer warp and chunk
constexpr int BACK_C = 3 * BACK_P;  // products per chunk
__global__ void __launch_bounds__(128)
    k_back(int n, int ld, const double *lu, double *inv, const int *singular) {
  __shared__ double prod[2][BACK_C][32];
  if (*singular) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  const bool has = e < n;
  double *const x = inv + (has ? e : n - 1);  // lanes past the end repeat the last column
  // products of the chunk of row i that starts at column j0
  auto produce = [&](double (*p)[32], int i, int j0) {
    const double *ui = lu + int64_t(i) * ld;
    const int j1 = j0 + (warp - 1) * BACK_P;
    double u[BACK_P], v[BACK_P];
#pragma unroll
    for (int t = 0; t < BACK_P; ++t)
      if (j1 + t < n) {
        u[t] = ui[j1 + t];
        v[t] = x[int64_t(j1 + t) * ld];
      }
#pragma unroll
    for (int t = 0; t < BACK_P; ++t)
      if (j1 + t < n) p[(warp - 1) * BACK_P + t][lane] = mul_rn(u[t], v[t]);
  };
  // the chunks in order: row i, columns from j0; every row has at least one
  int i = n - 1, j0 = n + 1, buf = 0;
  if (warp > 0) produce(prod[0], i, j0);
  __syncthreads();
  double s = 0.0, xl = 0.0;  // the row's sum, the x found last
  double y = 0.0, d = 0.0, u1 = 0.0;
  if (warp == 0) {
    y = x[int64_t(i) * ld];
    d = lu[int64_t(i) * ld + i];
  }
  for (bool first = true; i >= 0;) {
    const bool last = j0 + BACK_C >= n;  // the row's last chunk
    const int ni = last ? i - 1 : i, nj0 = last ? i + 1 : j0 + BACK_C;
    if (warp > 0) {
      if (ni >= 0) produce(prod[buf ^ 1], ni, nj0);
    } else {
      if (first) s = i + 1 < n ? sub_rn(y, mul_rn(u1, xl)) : y;
      double yn = 0.0, dn = 0.0, un = 0.0;
      if (last && i > 0) {  // the next row's start
        yn = x[int64_t(i - 1) * ld];
        dn = lu[int64_t(i - 1) * ld + i - 1];
        un = lu[int64_t(i - 1) * ld + i];
      }
      const int m = min(BACK_C, n - j0);
      if (m == BACK_C) {  // the next BACK_P products load while these are subtracted
        double p[2][BACK_P];
#pragma unroll
        for (int t = 0; t < BACK_P; ++t) p[0][t] = prod[buf][t][lane];
#pragma unroll
        for (int h = 0; h < BACK_C / BACK_P; ++h) {
#pragma unroll
          for (int t = 0; t < BACK_P; ++t)
            if (h + 1 < BACK_C / BACK_P)
              p[(h + 1) & 1][t] = prod[buf][(h + 1) * BACK_P + t][lane];
#pragma unroll
          for (int t = 0; t < BACK_P; ++t) s = sub_rn(s, p[h & 1][t]);
        }
      } else {
#pragma unroll 4
        for (int t = 0; t < m; ++t) s = sub_rn(s, prod[buf][t][lane]);
      }
      if (last) {
        xl = __ddiv_rn(s, d);
        if (has) x[int64_t(i) * ld] = xl;
        y = yn;
        d = dn;
        u1 = un;
      }
    }
    __syncthreads();
    first = last;
    i = ni;
    j0 = nj0;
    buf ^= 1;
  }
}

// part[i] = sum_j inv_ij^2 (warp per row, fixed order)
__global__ void k_inv_rowsq(int n, int ld, const double *inv, double *part) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; i < n; i += nw) {
    double a = 0.0;
    for (int j = lane; j < n; j += 32) a = __fma_rn(inv[i * ld + j], inv[i * ld + j], a);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a = __dadd_rn(a, __shfl_xor_sync(0xffffffffu, a, o));
    if (lane == 0) part[i] = a;
  }
}

// *out = sqrt(sum_i part[i]) / sqrt(n), the rows added in order (one warp: 32
// rows loaded at once, the next ones while these are added)
__global__ void k_inv_norm(int n, const double *part, double *out) {
  const int lane = threadIdx.x;
  double s = 0.0, v = lane < n ? part[lane] : 0.0;
  for (int i0 = 0; i0 < n; i0 += 32) {
    const double w = i0 + 32 + lane < n ? part[i0 + 32 + lane] : 0.0;
    const int m = min(32, n - i0);
    for (int t = 0; t < m; ++t) s = __dadd_rn(s, __shfl_sync(0xffffffffu, v, t));
    v = w;
  }
  if (lane == 0) *out = __ddiv_rn(__dsqrt_rn(s), __dsqrt_rn(double(n)));
}

__global__ void k_nmf_densify(int n, int ld, const int64_t *rp, const int32_t *col,
                              const double *val, int64_t row0, double *dx) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; i < n; i += nw)
    for (int64_t p = rp[row0 + i] + lane; p < rp[row0 + i + 1]; p += 32)
      dx[i * ld + (col[p] - row0)] = val[p];
}

// Xbar = (X + X^-1) / 2 as n full rows of slots from slot0 (global columns
// from row0), every entry kept (the filter drops the exact zeros)
__global__ void k_nmf_combine(int n, int ld, const double *dx, const double *inv, int64_t row0,
                              int64_t slot0, int64_t *rs, int64_t *re, int32_t *ccol,
                              double *cval) {
  const int64_t total = int64_t(n) * n;
  for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < total;
       t += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = t / n, j = t - i * n;
    ccol[slot0 + t] = int32_t(row0 + j);
    cval[slot0 + t] = __dmul_rn(0.5, __dadd_rn(dx[i * ld + j], inv[i * ld + j]));
    if (j == 0) {
      rs[row0 + i] = slot0 + i * n;
      re[row0 + i] = slot0 + (i + 1) * n;
    }
  }
}

// Eq. (1.13): c4 tol while r >= switch_resid, else r^2 / (x + ||X^-1||)
__global__ void k_nmf_budget(int m, int64_t n, const double *xinv, double c4, double tol,
                             double switch_resid, MatScalars *ms) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double r = ms[m].r, x = ms[m].x;
  const double beta = r >= switch_resid ? __dmul_rn(c4, tol)
                                        : __ddiv_rn(__dmul_rn(r, r), __dadd_rn(x, *xinv));
  ms[m].beta = beta;
  ms[m].b = __dmul_rn(__dsqrt_rn(double(n)), beta);
}

int blocks_for(int64_t items, int per) {
  int64_t g = (items + per - 1) / per;
  return int(g < 1 ? 1 : (g > 152 * 32 ? 152 * 32 : g));
}

}  // namespace

void launch_dense_inverse(int n, int ld, double *lu, int *swaps, int *singular, int *wild,
                          double *inv, cudaStream_t s) {
  if (n <= 0) return;
  static const bool attr = [] {  // once, thread-safe
    SGN_CUDA(cudaFuncSetAttribute(k_lu_panel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  int(PANEL_SMEM)));
    return true;
  }();
  (void)attr;
  SGN_CUDA(cudaMemsetAsync(singular, 0, sizeof(int), s));
  SGN_CUDA(cudaMemsetAsync(wild, 0, sizeof(int), s));
  k_inv_init<<<blocks_for(int64_t(n) * n, 256), 256, 0, s>>>(n, ld, inv);
  SGN_LAUNCH_CHECK();
  const int width = panel_width(n);
  for (int c0 = 0; c0 < n;) {
    int w = width;
    while (w > n - c0) w /= 2;  // the last columns: widths are powers of two
    const size_t smem = size_t(n - c0) * w * sizeof(double);
    const int in_place = smem > PANEL_SMEM ? 1 : 0;
    launch_next(k_lu_panel, 1, PANEL_T, in_place ? 0 : smem, s, n, ld, lu, c0, w, in_place, swaps,
                singular, wild);
    const unsigned strips =
        unsigned((n - c0 - w + STRIP - 1) / STRIP + (n + STRIP - 1) / STRIP);
    auto trail = [&](auto kernel) {
      launch_next(kernel, strips, TRAIL_T, 0, s, n, ld, lu, inv, c0, swaps, singular, wild);
    };
    if (w == 8) trail(k_lu_trail<8>);
    else if (w == 4) trail(k_lu_trail<4>);
    else if (w == 2) trail(k_lu_trail<2>);
    else trail(k_lu_trail<1>);
    c0 += w;
  }
  k_back<<<(n + 31) / 32, 128, 0, s>>>(n, ld, lu, inv, singular);
  SGN_LAUNCH_CHECK();
}

void launch_inv_norm(int n, int ld, const double *inv, double *part, double *out,
                     cudaStream_t s) {
  if (n <= 0) return;
  k_inv_rowsq<<<blocks_for(n, 8), 256, 0, s>>>(n, ld, inv, part);
  SGN_LAUNCH_CHECK();
  k_inv_norm<<<1, 32, 0, s>>>(n, part, out);
  SGN_LAUNCH_CHECK();
}

void launch_nmf_densify(int n, int ld, const int64_t *rp, const int32_t *col, const double *val,
                        int64_t row0, double *dx, cudaStream_t s) {
  if (n <= 0) return;
  k_nmf_densify<<<blocks_for(n, 8), 256, 0, s>>>(n, ld, rp, col, val, row0, dx);
  SGN_LAUNCH_CHECK();
}

void launch_nmf_combine(int n, int ld, const double *dx, const double *inv, int64_t row0,
                        int64_t slot0, int64_t *rs, int64_t *re, int32_t *col, double *val,
                        cudaStream_t s) {
  if (n <= 0) return;
  k_nmf_combine<<<blocks_for(int64_t(n) * n, 256), 256, 0, s>>>(n, ld, dx, inv, row0, slot0, rs,
                                                                 re, col, val);
  SGN_LAUNCH_CHECK();
}

void launch_nmf_budget(int m, int64_t n, const double *xinv, double c4, double tol,
                       double switch_resid, MatScalars *ms, cudaStream_t s) {
  k_nmf_budget<<<1, 32, 0, s>>>(m, n, xinv, c4, tol, switch_resid, ms);
  SGN_LAUNCH_CHECK();
}

}  // namespace sgn
