// Sums over the rows of a matrix by a cluster of RED_C CTAs, one warp of each
// per summed component; or, of many small matrices, by one CTA each.
#pragma once

#include <cooperative_groups.h>
#include <stdint.h>

namespace sgn {

constexpr int RED_T = 256;  // partial sums per component; their order is fixed
constexpr int RED_C = 8;    // CTAs per matrix (the portable cluster size)
constexpr int RED_LANES = RED_T / RED_C;
constexpr int RED_U = 32;   // rows loaded at once, the next ones while these are added
static_assert(RED_LANES == 32, "one warp of each CTA per component");

// Matrices per cluster in a launch over nb matrices: one, or from GROUP_NB on
// (every SM then has CTAs enough) RED_C. Of these, each CTA takes one of its own if
// that is small (solo); the larger ones are then taken by the whole cluster, one
// after another (joint), as a lone one is. The sums are the same either way. A
// cluster for each of 32768 matrices of order 16 took 1.20 ms per check, 0.82 for the
// select's preparation and histogram, 0.71 per digit search and 49 ms per solve,
// now 0.28, 0.27, 0.41 and 35; 1024 such matrices 2.30 ms, now 1.90.
constexpr int GROUP_NB = 1024;
constexpr int64_t SOLO_ROWS = 2048;
inline int cluster_matrices(int nb) { return nb >= GROUP_NB ? RED_C : 1; }
inline unsigned cluster_ctas(int nb) {
  const int per = cluster_matrices(nb);
  return unsigned((nb + per - 1) / per) * RED_C;
}
// solo(m) and joint(m) for the matrices of cluster `cluster`, by CTA q of it.
template <typename S, typename J>
__device__ __forceinline__ void cluster_each(int nb, int per, const int64_t *moff, int cluster,
                                             int q, S solo, J joint) {
  if (per == 1) {
    joint(cluster);
    return;
  }
  const int g0 = cluster * per, g1 = min(nb, g0 + per);
  auto small = [&](int m) { return moff[m + 1] - moff[m] <= SOLO_ROWS; };
  if (g0 + q < g1 && small(g0 + q)) solo(g0 + q);
  for (int m = g0; m < g1; ++m)
    if (!small(m)) joint(m);
}

// acc + v as a fused multiply-add (v * 1 is exact): in a chain of dependent FP64
// additions a DFMA takes 64 cycles, a DADD 76. In PTX, so that it stays one.
__device__ __forceinline__ double chain_add(double acc, double v) {
  double r;
  asm("fma.rn.f64 %0, %1, %2, %3;" : "=d"(r) : "d"(v), "d"(1.0), "d"(acc));
  return r;
}

// Partial sum t of component c: rows b + t, b + t + RED_T, ... below e, one after
// another.
__device__ __forceinline__ double seg_partial(const double *part, int ncomp, int c, int64_t b,
                                              int64_t e, int t) {
  double acc = 0.0;
  int64_t r = b + t;
  double v[RED_U], w[RED_U];  // absent rows are loaded as -0, which adds nothing
  auto fetch = [&](double (&d)[RED_U]) {
#pragma unroll
    for (int u = 0; u < RED_U; ++u, r += RED_T) d[u] = r < e ? part[r * ncomp + c] : -0.0;
  };
  auto add = [&](const double (&d)[RED_U]) {
#pragma unroll
    for (int u = 0; u < RED_U; ++u) acc = chain_add(acc, d[u]);
  };
  if (e - b <= 8 * RED_T) {  // short matrices: no rows to load ahead
    for (; r < e; r += RED_T) acc = chain_add(acc, part[r * ncomp + c]);
    return acc;
  }
  fetch(v);
  for (;;) {
    if (r >= e) {
      add(v);
      break;
    }
    fetch(w);
    add(v);
    if (r >= e) {
      add(w);
      break;
    }
    fetch(v);
    add(w);
  }
  return acc;
}

// One warp: the partial sums sm[0 .. RED_T) added pairwise, t + s into t for
// s = RED_T / 2 .. 1, into sm[0].
__device__ __forceinline__ void seg_tree(double *sm) {
  const int lane = threadIdx.x & 31;
  for (int s = RED_T / 2; s > 0; s >>= 1) {
    for (int i = lane; i < s; i += 32) sm[i] += sm[i + s];
    __syncwarp();
  }
}

// The partial sums of component c of the rows [b, e), all by one warp, then their sum
// in sm[0].
__device__ __forceinline__ void seg_sum_solo(double *sm, const double *part, int ncomp, int c,
                                             int64_t b, int64_t e) {
  const int lane = threadIdx.x & 31;
  for (int t = lane; t < RED_T; t += 32) sm[t] = seg_partial(part, ncomp, c, b, e, t);
  __syncwarp();
  seg_tree(sm);
}

// Warp q of a matrix's cluster: its share of the entries of the rows [b, e).
__device__ __forceinline__ unsigned long long seg_entries(const int64_t *rs, const int64_t *re,
                                                          int64_t b, int64_t e, int first,
                                                          int step) {
  long long acc = 0;
#pragma unroll 16
  for (int64_t r = b + first; r < e; r += step) acc += re[r] - rs[r];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return (unsigned long long)acc;
}

}  // namespace sgn
