// FP64-accurate dense products on the BF16 tensor cores, from exact integer
// slices (the error-free splitting of matrix products published by Ozaki,
// Ogita, Oishi and Rump, 2012), for matrices on the dense path in the FP64
// stage. GB300 runs FP64 at about 1/64 of its FP32 rate; this path moves the
// FP64 products of filled-in iterates to the tensor cores.
//
// Splitting. Row i of A (M x K) is scaled by its power of two 2^e_i >
// max_k |a_ik| and rounded to the grid 2^(e_i - 55); the integer q_ik
// (|q| < 2^55) is written as eight balanced base-128 digits,
//   a_ik ~= 2^(e_i + 1) * sum_{s=1..8} d_ik^(s) 2^(-7 s),   |d| <= 64,
// and likewise the rows of Bt (N x K) with 2^(f_j + 1). Every digit is a
// small integer, exact in BF16.
//
// Products. For a digit pair (s, t) the tensor cores form the integer matrix
// D_s E_t^T with FP32 accumulation: each product is at most 64 * 64 = 2^12 in
// magnitude, so an accumulator that takes at most 4096 products per entry, of
// one pair or of several of the same level s + t, only ever holds integers of
// magnitude at most 2^24 and is exact in any order. The pairs with s + t <= 9
// (36 of the 64) are kept; the dropped ones and the rounding of the inputs to
// the 2^-55 grid stay below 2^-41 * 2^(e_i + f_j) * K / 4096 in the worst case
// (digits of equal sign), about the error bound of an FP64 dot product.
// The levels 9 .. 4 of a K block are added as 64-bit integers,
//   L = sum_{l=4..9} 2^(7 (9 - l)) sum_{s+t=l} D_s E_t^T   (|L| < 2^62),
// the levels 3 and 2 likewise as H, and the block's product is
//   2^(e_i + f_j + 2) (2^-63 L + 2^-21 H),
// two integers converted to FP64 and one or two FP64 additions per entry;
// later blocks are added in FP64.
//
// Kernel: persistent, one CTA per SM, 320 threads, laid out as the
// split-TF32 kernel but with eight epilogue warps (two per 32 TMEM lanes,
// one per half of the columns). A work unit is one 128 x 256 tile of C. Its
// pairs are taken two levels at a time, (8, 9), (6, 7), (4, 5), (2, 3): step t
// of the levels (l, l + 1) multiplies the digit planes A_(l-t) and A_(l+1-t)
// by the same B_t into the two 256-column TMEM accumulators, one per level.
// The producer thread streams 32-wide K slices of the three planes with TMA
// into a six-stage ring (64-byte swizzle); the MMA thread issues two kind::f16
// (BF16) MMAs per accumulator and stage. Steps share an accumulator while its
// products stay within 4096 per entry (all of a level for K <= 512, one step
// for K > 2048); then the epilogue warps drain both accumulators into the
// CTA's tiles of integers (global scratch, 2 x 256 KB, stay in L2), the last
// run of a whole tile into C.
// What bounds it: the tensor pipe and, behind it, the L2 reads of the operand
// planes, 16 KB per pair and slice here against 24 KB when every pair loads
// its own two planes, and the FP64 pipe (16 cycles per warp instruction) when
// every pair is added into C in FP64, as an earlier form did: 6.07 ms at
// 4096^3 and 3.69 ms at 2744^3 (GB300), now 3.47 and 1.91 ms (1.43 PFLOP/s on
// the tensor pipe at 4096^3).
// Tiles of a last, partial wave are cut into S parts of about equal pairs, each
// a work unit of its own that leaves its integers in scratch; k_slices_finish
// adds them up (exactly, in any order) and writes C. 2744^3 has 242 tiles: two
// waves of 152 become 1 2/3 (2.31 -> 1.98 ms when it came), 1024^3 has 32: 0.29 ->
// 0.087 ms.
// Every wait has a clock budget, as in the split-TF32 kernel.
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "../../include/sign.h"
#include "common.cuh"
#include "kernels.h"
#include "tc.cuh"

namespace sgn {

namespace {

using namespace tc;

constexpr int XM = 128;    // tile rows (UMMA M)
constexpr int XN = 256;    // tile columns (UMMA N)
constexpr int XK = 32;     // K slice per stage: 32 BF16 = 64 bytes = one swizzle span
constexpr int XSTAGE = 6;  // ring of stages
constexpr int XSPAN = XK * 2;
constexpr int XA_BYTES = XM * XK * 2;  // 8 KB
constexpr int XB_BYTES = XN * XK * 2;  // 16 KB
constexpr int XSTAGE_BYTES = 2 * XA_BYTES + XB_BYTES;  // A_(l-t), A_(l+1-t), B_t
constexpr int XTHREADS = 320;  // producer, MMA, eight epilogue warps
constexpr uint32_t XTMEM_COLS = 2 * XN;
constexpr int XSMEM = XSTAGE * XSTAGE_BYTES + 1024;  // ring and alignment slack
constexpr int DIGIT_BITS = 7;
constexpr int KBLK = F64X_MAX_K / XK;       // K stages per exact block (integer sums <= 2^24)
// Level pairs (l, l + 1), l = 8, 6, 4, 2: the pairs with s + t <= 9 and 8 digits.
constexpr int XLP = 4;
static_assert(F64X_DIGITS == 8 && DIGIT_BITS == 7, "level pairs (8, 9) .. (2, 3) of 8 digits");
__host__ __device__ constexpr int lower_level(int lp) { return 8 - 2 * lp; }
// The steps (level pair, t) of a tile in the order in which a unit takes them: a
// whole tile from the smallest weight up, the levels 3 and 2 last; for parts
// the level pairs ordered so that halves, thirds and sixths of the pairs end
// between steps.
constexpr int XSTEPS = 20, XMAX_PARTS = 6;
struct StepList {
  unsigned char lp[2][XSTEPS], t[2][XSTEPS];  // [0] whole tiles, [1] parts
};
constexpr StepList make_steps() {
  StepList s{};
  const int order[2][XLP] = {{0, 1, 2, 3}, {0, 3, 1, 2}};
  for (int k = 0; k < 2; ++k) {
    int n = 0;
    for (int i = 0; i < XLP; ++i)
      for (int t = 1; t <= lower_level(order[k][i]); ++t, ++n) {
        s.lp[k][n] = (unsigned char)order[k][i];
        s.t[k][n] = (unsigned char)t;
      }
  }
  return s;
}
constexpr StepList kSteps = make_steps();
__constant__ StepList c_steps = kSteps;
constexpr int step_pairs(int i) {  // of the parts' order
  return kSteps.t[1][i] < lower_level(kSteps.lp[1][i]) ? 2 : 1;
}
// The units of a launch: nfull whole tiles, then S parts of each tile after them;
// part p takes the steps bound[p] .. bound[p + 1] - 1.
struct XPlan {
  int nfull, ntail, parts;
  int bound[XMAX_PARTS + 1];
  __host__ __device__ int units() const { return nfull + ntail * parts; }
};
constexpr int XPAIRS = 36;  // sum over the level pairs of (l - 1) + l
// an integer tile: 32-column chunks of a warp, column by column
constexpr size_t XTILE_BYTES = size_t(XM) * XN * sizeof(long long);

// Unit u -> its tile and steps [s0, s1) of the list k.
struct XUnit {
  int tile, k, s0, s1;
};
__device__ __forceinline__ XUnit unit_at(int u, const XPlan &pl) {
  if (u < pl.nfull) return XUnit{u, 0, 0, XSTEPS};
  const int v = u - pl.nfull, p = v % pl.parts;
  return XUnit{pl.nfull + v / pl.parts, 1, pl.bound[p], pl.bound[p + 1]};
}
// The end of the run of steps from i that share an accumulator: one level pair,
// at most `group` of them.
__device__ __forceinline__ int run_end(const XUnit &un, int i, int group) {
  int e = i + 1;
  while (e < un.s1 && e - i < group && c_steps.lp[un.k][e] == c_steps.lp[un.k][i]) ++e;
  return e;
}

// v 2^sc as an FP64 value, rounded to nearest: built with integer operations,
// the FP64 pipe being the scarce unit. Falls back to ldexp outside the
// normal range.
__device__ __forceinline__ double scaled_int(long long v, int sc) {
  if (v == 0) return 0.0;
  const unsigned long long a = v < 0 ? 0ULL - (unsigned long long)v : (unsigned long long)v;
  const int z = __clzll((long long)a);
  const unsigned long long m = a << z;  // top bit set
  const int e = 63 - z + sc + 1022;     // biased exponent less one (the top bit adds one)
  if (e < 0 || e >= 2045) return ldexp(double(v), sc);
  const unsigned long long mant = (m >> 11) + ((m >> 10) & 1ULL);
  return __longlong_as_double(
      (long long)((((unsigned long long)e << 52) + mant) | (v < 0 ? 1ULL << 63 : 0ULL)));
}

// The exact integers of an FP32 accumulator.
__device__ __forceinline__ long long acc_int(uint32_t bits) {
  return (long long)__float2int_rn(__uint_as_float(bits));
}

// Tile t of the launch -> job and tile origin (m0, n0); M blocks run fastest.
__device__ __forceinline__ void xtile_of(int t, const SliceJob *jobs, const int *tile_start,
                                         int njobs, int &j, int &m0, int &n0) {
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (tile_start[mid] <= t) lo = mid; else hi = mid - 1;
  }
  j = lo;
  const int local = t - tile_start[j];
  const int tm = (jobs[j].M + XM - 1) / XM;
  m0 = (local % tm) * XM;
  n0 = (local / tm) * XN;
}

// maps[2 j]: the digits of A of job j as one (8 M) x K array, maps[2 j + 1]
// those of Bt as (8 N) x K; digit s of row r is row (s - 1) rows + r. tiles and
// parts: two integer tiles (levels 9 .. 4, levels 3 and 2) per CTA and per part.
__global__ void __launch_bounds__(XTHREADS, 1)
    k_gemm_slices(const SliceJob *jobs, const CUtensorMap *maps, const int *tile_start,
                  int njobs, XPlan pl, long long *tiles, long long *parts, int *err) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[XSTAGE], empty[XSTAGE], tfull, tempty, done;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort, s_consumed;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  volatile int *abort = &s_abort;
  const int nunits = pl.units();
  if (tid == 0) {
    for (int i = 0; i < XSTAGE; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(&tfull, 1);
    mbar_init(&tempty, 8);
    mbar_init(&done, 1);
    s_abort = 0;
    s_consumed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(&tmem_slot, XTMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  int issued = 0;

  if (warp == 0) {
    if (lane == 0) {
      for (int u = blockIdx.x; u < nunits && !*abort; u += gridDim.x) {
        const XUnit un = unit_at(u, pl);
        int j, m0, n0;
        xtile_of(un.tile, jobs, tile_start, njobs, j, m0, n0);
        const SliceJob &J = jobs[j];
        const CUtensorMap *mp = maps + 2 * j;
        const int nk = (J.K + XK - 1) / XK;
        for (int k0 = 0; k0 < nk && !*abort; k0 += KBLK) {
          const int k1 = min(nk, k0 + KBLK);
          for (int i = un.s0; i < un.s1 && !*abort; ++i) {
            const int l = lower_level(c_steps.lp[un.k][i]), t = c_steps.t[un.k][i];
            const bool both = t < l;  // step l has no pair of level l
            const int y0 = (l - t - 1) * J.M + m0, y1 = (l - t) * J.M + m0;
            const int yb = (t - 1) * J.N + n0;
            for (int kb = k0; kb < k1; ++kb, ++issued) {
              const int st = issued % XSTAGE;
              if (!bounded_wait(&empty[st], ((issued / XSTAGE) & 1) ^ 1, abort)) break;
              const uint32_t d = sbase + uint32_t(st * XSTAGE_BYTES);
              mbar_expect_tx(&full[st], both ? XSTAGE_BYTES : XSTAGE_BYTES - XA_BYTES);
              if (both) tma_load_2d(d, mp + 0, kb * XK, y0, &full[st]);
              tma_load_2d(d + XA_BYTES, mp + 0, kb * XK, y1, &full[st]);
              tma_load_2d(d + 2 * XA_BYTES, mp + 1, kb * XK, yb, &full[st]);
            }
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16(XM, XN);
      int it = 0, uc = 0;  // stages consumed, accumulations (both accumulators) done
      bool any = false, ok = true;
      for (int u = blockIdx.x; u < nunits && ok && !*abort; u += gridDim.x) {
        const XUnit un = unit_at(u, pl);
        int j, m0, n0;
        xtile_of(un.tile, jobs, tile_start, njobs, j, m0, n0);
        const int nk = (jobs[j].K + XK - 1) / XK;
        for (int k0 = 0; k0 < nk && ok; k0 += KBLK) {
          const int k1 = min(nk, k0 + KBLK), group = KBLK / (k1 - k0);
          for (int i = un.s0; i < un.s1 && ok; ++uc) {
            const int e = run_end(un, i, group);  // steps i .. e - 1 accumulate together
            const int l = lower_level(c_steps.lp[un.k][i]);
            if (!bounded_wait(&tempty, (uc & 1) ^ 1, abort)) {
              ok = false;
              break;
            }
            tc_fence_after();
            for (int q = i; q < e && ok; ++q) {
              const bool both = c_steps.t[un.k][q] < l;
              for (int kb = k0; kb < k1; ++kb, ++it) {
                const int st = it % XSTAGE;
                if (!bounded_wait(&full[st], (it / XSTAGE) & 1, abort)) {
                  ok = false;
                  break;
                }
                tc_fence_after();
                const uint32_t d = sbase + uint32_t(st * XSTAGE_BYTES);
                const uint32_t more = q > i || kb > k0 ? 1u : 0u;
#pragma unroll
                for (int s = 0; s < XK / 16; ++s) {
                  const uint32_t ko = uint32_t(s) * 32u;
                  const uint64_t bd = smem_desc_sw<XSPAN>(d + 2 * XA_BYTES + ko);
                  if (both)
                    mma_bf16(tmem, smem_desc_sw<XSPAN>(d + ko), bd, idesc, s ? 1u : more);
                  mma_bf16(tmem + XN, smem_desc_sw<XSPAN>(d + XA_BYTES + ko), bd, idesc,
                           s ? 1u : more);
                }
                any = true;
                mma_commit(&empty[st]);
              }
            }
            if (!ok) break;
            mma_commit(&tfull);
            i = e;
          }
        }
      }
      s_consumed = it;
      if (any) {
        mma_commit(&done);
        if (!drain_wait(&done, 0, WAIT_BUDGET)) *abort = 1;
      }
    }
  } else {
    const int q = warp & 3;           // this warp's 32 TMEM lanes (rows)
    const int half = (warp - 2) >> 2;  // and its half of the tile's columns
    const uint32_t trow = tmem + (uint32_t(q * 32) << 16);
    int uc = 0;
    bool stop = false;
    for (int u = blockIdx.x; u < nunits && !stop; u += gridDim.x) {
      const XUnit un = unit_at(u, pl);
      const bool part = un.k != 0;
      int j, m0, n0;
      xtile_of(un.tile, jobs, tile_start, njobs, j, m0, n0);
      const SliceJob J = jobs[j];
      // this warp's part of the integer tiles, [chunk][column][lane]: one for the
      // levels 9 .. 4 and one for 3 and 2
      long long *const low = (part ? parts + size_t(u - pl.nfull) * (2 * XM * XN)
                                   : tiles + size_t(blockIdx.x) * (2 * XM * XN)) +
                             size_t(warp - 2) * (XM * XN / 8) + lane;
      const int gr = m0 + q * 32 + lane;
      const int ea = gr < J.M ? J.ea[gr] : 0;
      const int nk = (J.K + XK - 1) / XK;
      for (int k0 = 0; k0 < nk && !stop; k0 += KBLK) {
        const int group = KBLK / (min(nk, k0 + KBLK) - k0);
        bool first_low = true, first_high = true;
        {
          for (int i = un.s0; i < un.s1; ++uc) {
            const int e = run_end(un, i, group);
            const int lp = c_steps.lp[un.k][i], ta = c_steps.t[un.k][i], l = lower_level(lp);
            i = e;
            if (!bounded_wait(&tfull, uc & 1, abort)) {
              stop = true;
              break;
            }
            tc_fence_after();
            const bool both = ta < l;  // the lower level's accumulator was written
            const bool high = lp == XLP - 1;
            const bool first = high ? first_high : first_low;
            // a whole tile's last run: its sums are complete and go into C
            const bool into_c = high && !part && e == un.s1;
#pragma unroll 1
            for (int c = 0; c < XN / 64; ++c) {
              uint32_t v0[32], v1[32];
              const int col = half * (XN / 2) + c * 32;  // this warp's columns of the tile
              __syncwarp();
              if (both) tmem_ld_32x32(trow + uint32_t(col), v0);
              tmem_ld_32x32(trow + uint32_t(XN + col), v1);
              tmem_wait_ld();
              if (!both) {
#pragma unroll
                for (int i = 0; i < 32; ++i) v0[i] = 0u;
              }
              long long *const lc = low + c * 32 * 32 + (high ? XM * XN : 0);
              if (!into_c) {  // into an integer tile
                const int sh = high ? 0 : 2 * DIGIT_BITS * lp;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  long long o[16];
#pragma unroll
                  for (int i = 0; i < 16; ++i) o[i] = first ? 0ll : lc[(16 * h + i) * 32];
#pragma unroll
                  for (int i = 0; i < 16; ++i) {
                    const int x = 16 * h + i;
                    lc[x * 32] =
                        o[i] + (acc_int(v0[x]) * (1 << DIGIT_BITS) + acc_int(v1[x])) * (1ll << sh);
                  }
                }
                continue;
              }
              // C = [C +] 2^(e_i + f_j - 63) L + 2^(e_i + f_j - 21) H, H and L exact as
              // where the tile is cut into parts: the same bits either way
              const int gc = n0 + col;
              if (gr >= J.M) continue;
              double *const crow = J.C + int64_t(gr) * J.ldc + gc;
              const long long *const ll = lc - XM * XN;
              const bool add = k0 > 0 || J.accum;  // C holds earlier K blocks
#pragma unroll
              for (int h = 0; h < 4; ++h) {
                // eight columns: all loads in flight before any store (N and ldc even,
                // C 16-byte aligned: column pairs)
                long long hs[8], ls[8];
                double2 o[4];
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                  hs[i] = first ? 0ll : lc[(8 * h + i) * 32];
                  ls[i] = ll[(8 * h + i) * 32];
                }
                if (add) {
#pragma unroll
                  for (int i = 0; i < 4; ++i)
                    if (gc + 8 * h + 2 * i < J.N)
                      o[i] = reinterpret_cast<const double2 *>(crow)[4 * h + i];
                }
#pragma unroll
                for (int i = 0; i < 8; i += 2) {
                  const int x = 8 * h + i;
                  if (gc + x >= J.N) break;
                  const int2 eb = *reinterpret_cast<const int2 *>(J.eb + gc + x);
                  double r[2];
#pragma unroll
                  for (int p = 0; p < 2; ++p) {
                    const int sc = ea + (p ? eb.y : eb.x);
                    r[p] = scaled_int(hs[i + p] + acc_int(v0[x + p]) * (1 << DIGIT_BITS) +
                                          acc_int(v1[x + p]),
                                      sc - 3 * DIGIT_BITS);
                    r[p] += scaled_int(ls[i + p], sc - 9 * DIGIT_BITS);
                    if (add) r[p] += p ? o[i / 2].y : o[i / 2].x;
                  }
                  reinterpret_cast<double2 *>(crow)[x / 2] = make_double2(r[0], r[1]);
                }
              }
            }
            if (high) first_high = false; else first_low = false;
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty);
          }
        }
      }
    }
  }

  __syncthreads();
  if (warp == 0 && lane == 0) {
    for (int i = s_consumed; i < issued; ++i)
      if (!drain_wait(&full[i % XSTAGE], (i / XSTAGE) & 1, WAIT_BUDGET)) {
        *abort = 1;
        break;
      }
  }
  if (tid == 0 && *abort) atomicOr(err, 1);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem, XTMEM_COLS);
}

// C of the tiles that were cut into parts: the parts' integers added, then as in
// k_gemm_slices. low, high: bit p set if part p has steps of the levels 9 .. 4,
// or of 3 and 2. A CTA per 32 x 32 block of a tile; a thread writes 32 B.
__global__ void __launch_bounds__(256)
    k_slices_finish(const SliceJob *jobs, const int *tile_start, int njobs, XPlan pl,
                    const long long *parts, unsigned low, unsigned high) {
  const int tt = blockIdx.x / 32, blk = blockIdx.x % 32;
  int j, m0, n0;
  xtile_of(pl.nfull + tt, jobs, tile_start, njobs, j, m0, n0);
  const SliceJob J = jobs[j];
  const int w = blk / 4, c = blk % 4, lane = threadIdx.x & 31, i0 = (threadIdx.x >> 5) * 4;
  const int gr = m0 + ((w + 2) & 3) * 32 + lane;  // the layout of epilogue warp w + 2
  const int gc = n0 + (w >> 2) * (XN / 2) + c * 32 + i0;
  if (gr >= J.M || gc >= J.N) return;
  const long long *t = parts + size_t(tt) * pl.parts * (2 * XM * XN) + size_t(w) * (XM * XN / 8) +
                       c * 32 * 32 + lane;
  long long L[4] = {0, 0, 0, 0}, H[4] = {0, 0, 0, 0};
  for (int p = 0; p < pl.parts; ++p, t += 2 * XM * XN)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if ((low >> p) & 1u) L[i] += t[(i0 + i) * 32];
      if ((high >> p) & 1u) H[i] += t[XM * XN + (i0 + i) * 32];
    }
  const int ea = J.ea[gr];
  double *const crow = J.C + int64_t(gr) * J.ldc + gc;
#pragma unroll
  for (int i = 0; i < 4; i += 2) {
    if (gc + i >= J.N) break;  // N is even
    const int2 eb = *reinterpret_cast<const int2 *>(J.eb + gc + i);
    double2 v;
    v.x = scaled_int(H[i], ea + eb.x - 3 * DIGIT_BITS) + scaled_int(L[i], ea + eb.x - 9 * DIGIT_BITS);
    v.y = scaled_int(H[i + 1], ea + eb.y - 3 * DIGIT_BITS) +
          scaled_int(L[i + 1], ea + eb.y - 9 * DIGIT_BITS);
    double2 *const cp = reinterpret_cast<double2 *>(crow + i);
    if (J.accum) {
      const double2 o = *cp;
      v.x += o.x;
      v.y += o.y;
    }
    *cp = v;
  }
}

// Digit planes. HBM-bound: an entry is read as 8 B (twice: row maximum, then
// digits; the second read mostly hits L2) and written as 16 B. All arithmetic
// is on integers (an FP64 instruction costs 16 cycles per warp), every lane
// cuts two neighbouring entries and writes 4 B per plane, and the columns of x
// go through shared memory so that both sides are read and written in whole
// 128-byte lines. 4096 x 4096: rows 511 -> 130 us, columns 548 -> 160 us.

// |x| for the row maximum, by its bits: a NaN counts as 0 (as fmax skips it).
__device__ __forceinline__ unsigned long long max_key(double x) {
  const unsigned long long k = (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFULL;
  return k > 0x7FF0000000000000ULL ? 0ULL : k;
}

// e of 2^e > max (0 for a zero row)
__device__ __forceinline__ int row_exponent(unsigned long long key) {
  int e = 0;
  frexp(__longlong_as_double((long long)key), &e);
  return e;
}

// x 2^(55 - e) rounded to nearest even, |x| < 2^e: the significand shifted by
// integer operations; what is not finite goes through the conversion.
__device__ __forceinline__ long long grid_int(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int ex = int((unsigned long long)b >> 52) & 0x7FF;
  if (ex == 0x7FF) return __double2ll_rn(ldexp(x, 55 - e));
  const long long m = (b & 0xFFFFFFFFFFFFFll) | (ex ? 1ll << 52 : 0ll);
  const int sh = (ex ? ex : 1) - 1020 - e;  // at most 2
  long long q;
  if (sh >= 0) {
    q = m << sh;
  } else if (sh <= -54) {
    q = 0;
  } else {
    const int r = -sh;
    q = m >> r;
    const long long rem = m & ((1ll << r) - 1), half = 1ll << (r - 1);
    if (rem > half || (rem == half && (q & 1))) ++q;
  }
  return b < 0 ? -q : q;
}

// Writes the digits of two neighbouring entries (out: plane 1, 4-byte aligned).
// Digits 2 .. 8 lie in [-64, 63] and digit 1 takes the rest: with 64 added to
// each of them they are the base-128 digits of q + 64 sum_{i<7} 128^i.
__device__ __forceinline__ void put_digits(long long q0, long long q1, uint32_t *out,
                                           int64_t plane2) {
  constexpr long long kBias = 64ll * ((1ll << 49) - 1) / 127;
  q0 += kBias;
  q1 += kBias;
  // an integer |d| <= 64 has at most 7 significant bits: its BF16 bits are the
  // top half of its FP32 bits, exactly; 2^23 + u is the FP32 number of bits 0x4B000000 + u
  auto bf16 = [](int u) {
    return __float_as_uint(__fsub_rn(__uint_as_float(0x4B000000u + uint32_t(u)), 8388672.0f)) >> 16;
  };
#pragma unroll
  for (int s = 1; s <= F64X_DIGITS; ++s) {
    const int shift = DIGIT_BITS * (F64X_DIGITS - s);
    // digit 1 is not biased: 64 is added here to share the conversion
    const int u0 = s == 1 ? int(q0 >> shift) + 64 : int(q0 >> shift) & 127;
    const int u1 = s == 1 ? int(q1 >> shift) + 64 : int(q1 >> shift) & 127;
    out[(s - 1) * plane2] = bf16(u0) | (bf16(u1) << 16);
  }
}

// Digits of the rows of x (rows x K, leading dimension ldx): digit s of row r
// at out[(s - 1) rows ld + r ld + k], zero for K <= k < ld; w[r] = e_r + 1 with
// 2^e_r > max_k |x_rk|. A warp per row.
__global__ void __launch_bounds__(256)
    k_slices_rows(int rows, int K, const double *x, int ldx, uint16_t *out, int ld, int *w) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  const int64_t plane2 = int64_t(rows) * ld / 2;
  for (int64_t r = warp; r < rows; r += nwarps) {
    const double *xr = x + r * ldx;
    unsigned long long mx = 0;
#pragma unroll 8
    for (int k = lane; k < K; k += 32) {
      const unsigned long long key = max_key(xr[k]);
      mx = key > mx ? key : mx;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, mx, o);
      mx = y > mx ? y : mx;
    }
    const int e = row_exponent(mx);
    if (lane == 0) w[r] = e + 1;
    uint32_t *o = reinterpret_cast<uint32_t *>(out + r * ld);
#pragma unroll 2
    for (int k = 2 * lane; k < ld; k += 64) {
      const double x0 = k < K ? xr[k] : 0.0, x1 = k + 1 < K ? xr[k + 1] : 0.0;
      put_digits(grid_int(x0, e), grid_int(x1, e), o + k / 2, plane2);
    }
  }
}

// The same of the columns of x (K x rows): column r of x is row r of the planes.
// A CTA takes SC_C columns; their entries pass through shared memory SC_K at a
// time.
constexpr int SC_C = 16, SC_K = 128;
__global__ void __launch_bounds__(256)
    k_slices_cols(int rows, int K, const double *x, int ldx, uint16_t *out, int ld, int *w) {
  __shared__ double tile[SC_C][SC_K + 1];
  __shared__ unsigned long long s_mx[SC_C][256 / SC_C];
  __shared__ int s_e[SC_C];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = threadIdx.x % SC_C, kk = threadIdx.x / SC_C;
  constexpr int KT = 256 / SC_C;  // rows of x read at once
  const int r0 = blockIdx.x * SC_C;
  const bool has = r0 + c < rows;
  const double *xc = x + r0 + c;
  const int64_t plane2 = int64_t(rows) * ld / 2;
  unsigned long long mx = 0;
  if (has) {
#pragma unroll 8
    for (int k = kk; k < K; k += KT) {
      const unsigned long long key = max_key(xc[int64_t(k) * ldx]);
      mx = key > mx ? key : mx;
    }
  }
  s_mx[c][kk] = mx;
  __syncthreads();
  if (threadIdx.x < SC_C) {
    unsigned long long m = 0;
    for (int i = 0; i < KT; ++i) m = s_mx[threadIdx.x][i] > m ? s_mx[threadIdx.x][i] : m;
    const int e = row_exponent(m);
    s_e[threadIdx.x] = e;
    if (r0 + int(threadIdx.x) < rows) w[r0 + threadIdx.x] = e + 1;
  }
  for (int k0 = 0; k0 < ld; k0 += SC_K) {
    __syncthreads();  // the exponents are written, the tile is read
    double v[SC_K / KT];
#pragma unroll
    for (int u = 0; u < SC_K / KT; ++u) {
      const int k = k0 + kk + u * KT;
      v[u] = has && k < K ? xc[int64_t(k) * ldx] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < SC_K / KT; ++u) tile[c][kk + u * KT] = v[u];
    __syncthreads();
#pragma unroll
    for (int h = 0; h < SC_C / 8; ++h) {  // two columns per warp
      const int cc = warp * (SC_C / 8) + h, r = r0 + cc;
      if (r >= rows) break;
      const int e = s_e[cc];
      uint32_t *o = reinterpret_cast<uint32_t *>(out + int64_t(r) * ld);
#pragma unroll
      for (int u = 0; u < SC_K; u += 64) {
        const int k = u + 2 * lane;
        if (k0 + k >= ld) break;
        put_digits(grid_int(tile[cc][k], e), grid_int(tile[cc][k + 1], e), o + (k0 + k) / 2,
                   plane2);
      }
    }
  }
}

// Warp-per-row helpers of the FP64 dense path (same row loop as the FP32 one).
template <typename F>
__device__ __forceinline__ void dense_rows(int64_t n, F f) {
  const int64_t warp = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = (int64_t(gridDim.x) * blockDim.x) >> 5;
  for (int64_t r = warp; r < n; r += nwarps) f(r);
}

__global__ void k_densify64(int64_t n, const int32_t *seg, const int *dslot, const int64_t *moff,
                            const int64_t *rp, const int32_t *col, const double *val,
                            const DenseBuf64 *bufs) {
  const int lane = threadIdx.x & 31;
  dense_rows(n, [&](int64_t r) {
    const int m = seg[r], d = dslot[m];
    if (d < 0) return;
    const DenseBuf64 B = bufs[d];
    const int64_t r0 = moff[m], i = r - r0;
    for (int64_t p = rp[r] + lane; p < rp[r + 1]; p += 32) B.X[i * B.ld + (col[p] - r0)] = val[p];
  });
}

__global__ void k_dense_resid64(int64_t n, const int32_t *seg, const int *dslot,
                                const int64_t *moff, const DenseBuf64 *bufs, double *part,
                                unsigned long long *tcount) {
  const int lane = threadIdx.x & 31;
  dense_rows(n, [&](int64_t r) {
    const int m = seg[r], d = dslot[m];
    if (d < 0) return;
    const DenseBuf64 B = bufs[d];
    const int64_t i = r - moff[m];
    double rs = 0.0, xs = 0.0;
    unsigned cnt = 0;
    for (int j = lane; j < B.n; j += 32) {
      const double t = B.TT[i * B.ld + j], x = B.X[i * B.ld + j];
      const double e = j == i ? t - 1.0 : t;
      rs = fma(e, e, rs);
      xs = fma(x, x, xs);
      cnt += t != 0.0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      rs += __shfl_xor_sync(0xffffffffu, rs, o);
      xs += __shfl_xor_sync(0xffffffffu, xs, o);
      cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    }
    if (lane == 0) {
      part[2 * r] = rs;
      part[2 * r + 1] = xs;
      atomicAdd(&tcount[d], (unsigned long long)cnt);
    }
  });
}

__global__ void k_dense_emit64(int64_t n, const int32_t *seg, const int *dslot,
                               const int64_t *moff, const int *active, const DenseBuf64 *bufs,
                               const int64_t *cs, int64_t *ce, int32_t *ccol, double *cval) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  dense_rows(n, [&](int64_t r) {
    const int m = seg[r], d = dslot[m];
    if (d < 0 || !active[m]) return;
    const DenseBuf64 B = bufs[d];
    const int64_t r0 = moff[m], i = r - r0;
    int64_t out = cs[r];
    for (int j0 = 0; j0 < B.n; j0 += 32) {
      const int j = j0 + lane;
      double v = 0.0;
      if (j < B.n)
        v = __dsub_rn(__dmul_rn(1.5, B.X[i * B.ld + j]), __dmul_rn(0.5, B.P[i * B.ld + j]));
      const bool keep = v != 0.0;
      const unsigned mk = __ballot_sync(0xffffffffu, keep);
      if (keep) {
        const int64_t pos = out + __popc(mk & lt);
        ccol[pos] = int32_t(r0 + j);
        cval[pos] = v;
      }
      out += __popc(mk);
    }
    if (lane == 0) ce[r] = out;
  });
}

int rows_grid(int64_t n) {
  int64_t g = (n + 7) / 8;
  return int(g < 1 ? 1 : (g > 152 * 16 ? 152 * 16 : g));
}

size_t scratch_maps_x(int njobs) {
  return size_t(njobs) * 2 + (size_t(njobs + 1) * sizeof(int) + sizeof(CUtensorMap) - 1) /
                                 sizeof(CUtensorMap);
}
// the maps and tile offsets, then the CTAs' integer tiles
size_t scratch_maps_bytes_x(int njobs) {
  return (scratch_maps_x(njobs) * sizeof(CUtensorMap) + 255) & ~size_t(255);
}

// SMs of the device: the CTAs of k_gemm_slices.
int slice_ctas() {
  static const int nsm = [] {  // once, thread-safe
    int dev = 0, n = 0;
    SGN_CUDA(cudaGetDevice(&dev));
    SGN_CUDA(cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev));
    SGN_CUDA(cudaFuncSetAttribute(k_gemm_slices, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  XSMEM));
    return n;
  }();
  return nsm;
}

}  // namespace

int f64x_pairs() { return XPAIRS; }

void launch_densify64(int64_t n, const int32_t *seg, const int *dslot, const int64_t *moff,
                      const int64_t *rp, const int32_t *col, const double *val,
                      const DenseBuf64 *bufs, cudaStream_t s) {
  if (n == 0) return;
  k_densify64<<<rows_grid(n), 256, 0, s>>>(n, seg, dslot, moff, rp, col, val, bufs);
  SGN_LAUNCH_CHECK();
}

void launch_dense_resid64(int64_t n, const int32_t *seg, const int *dslot, const int64_t *moff,
                          const DenseBuf64 *bufs, double *part, unsigned long long *tcount,
                          cudaStream_t s) {
  if (n == 0) return;
  k_dense_resid64<<<rows_grid(n), 256, 0, s>>>(n, seg, dslot, moff, bufs, part, tcount);
  SGN_LAUNCH_CHECK();
}

void launch_dense_emit64(int64_t n, const int32_t *seg, const int *dslot, const int64_t *moff,
                         const int *active, const DenseBuf64 *bufs, const int64_t *cs,
                         int64_t *ce, int32_t *ccol, double *cval, cudaStream_t s) {
  if (n == 0) return;
  k_dense_emit64<<<rows_grid(n), 256, 0, s>>>(n, seg, dslot, moff, active, bufs, cs, ce, ccol,
                                              cval);
  SGN_LAUNCH_CHECK();
}

size_t f64x_digits_bytes(int rows, int ld) {
  return size_t(F64X_DIGITS) * size_t(rows) * size_t(ld) * sizeof(uint16_t);
}

int slice_tiles(int M, int N) { return ((M + XM - 1) / XM) * ((N + XN - 1) / XN); }

// Parts for the tiles of a partial last wave: the number that ends soonest, by
// the most pairs of a part, each part's drain costing about a hundredth of a
// tile; at most two units per CTA. Tiles of several K blocks stay whole.
static XPlan slice_plan(int ntiles, bool one_block) {
  const int nsm = slice_ctas();
  XPlan best{};
  best.nfull = ntiles;
  best.parts = 1;
  const int tail = ntiles % nsm;
  if (!one_block || tail == 0) return best;
  double cost = 1.0;
  for (int S = 2; S <= XMAX_PARTS; ++S) {
    if (tail * S > 2 * nsm) break;
    XPlan pl{};
    pl.nfull = ntiles - tail;
    pl.ntail = tail;
    pl.parts = S;
    int most = 0, sum = 0, at = 0, prev = 0;
    for (int i = 0; i < XSTEPS; ++i) {
      sum += step_pairs(i);
      if (at + 1 < S && sum * S >= XPAIRS * (at + 1)) {
        pl.bound[++at] = i + 1;
        most = std::max(most, sum - prev);
        prev = sum;
      }
    }
    most = std::max(most, XPAIRS - prev);
    pl.bound[S] = XSTEPS;
    const int waves = (tail * S + nsm - 1) / nsm;
    const double c = waves * (double(most) / XPAIRS + 0.01) + 0.04;
    if (at == S - 1 && c < cost) {
      cost = c;
      best = pl;
    }
  }
  return best;
}

size_t slice_jobs_scratch_bytes(int njobs, int ntiles) {
  const XPlan pl = slice_plan(ntiles, true);
  return scratch_maps_bytes_x(njobs) +
         2 * XTILE_BYTES * (size_t(std::min(ntiles, slice_ctas())) + size_t(pl.ntail) * pl.parts);
}

void launch_slices(int rows, int K, const double *x, int ldx, int transpose, uint16_t *digits,
                   int ld, int *w, cudaStream_t s) {
  if (rows <= 0) return;
  if (transpose) {
    k_slices_cols<<<unsigned((rows + SC_C - 1) / SC_C), 256, 0, s>>>(rows, K, x, ldx, digits, ld,
                                                                    w);
  } else {
    const int64_t g = (int64_t(rows) + 7) / 8;
    k_slices_rows<<<unsigned(std::min<int64_t>(g, 152 * 16)), 256, 0, s>>>(rows, K, x, ldx, digits,
                                                                          ld, w);
  }
  SGN_LAUNCH_CHECK();
}

void launch_slice_jobs(int njobs, const SliceJob *jobs_host, SliceJob *jobs_dev, void *scratch,
                       int *err, cudaStream_t s) {
  if (njobs <= 0) return;
  thread_local std::vector<CUtensorMap> host;
  host.resize(scratch_maps_x(njobs));
  CUtensorMap *maps = host.data();
  int *tile_start = reinterpret_cast<int *>(host.data() + size_t(njobs) * 2);
  int ntiles = 0;
  for (int j = 0; j < njobs; ++j) {
    const SliceJob &J = jobs_host[j];
    if (J.M <= 0 || J.N <= 0 || J.K <= 0 || J.lda % 8 || J.ldb % 8 ||
        J.ldc % 2 || J.N % 2)
      throw Error(SIGN_EINVAL, "slice job with bad shape");
    const CUtensorMapDataType bf = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
    maps[2 * j + 0] = tc::operand_map(J.A, bf, 2, F64X_DIGITS * J.M, J.K, J.lda, XK, XM);
    maps[2 * j + 1] = tc::operand_map(J.B, bf, 2, F64X_DIGITS * J.N, J.K, J.ldb, XK, XN);
    tile_start[j] = ntiles;
    ntiles += ((J.M + XM - 1) / XM) * ((J.N + XN - 1) / XN);
  }
  tile_start[njobs] = ntiles;
  bool one_block = true;
  for (int j = 0; j < njobs; ++j) one_block = one_block && jobs_host[j].K <= F64X_MAX_K;
  const XPlan pl = slice_plan(ntiles, one_block);
  SGN_CUDA(cudaMemcpyAsync(scratch, host.data(), host.size() * sizeof(CUtensorMap),
                           cudaMemcpyHostToDevice, s));
  SGN_CUDA(cudaMemcpyAsync(jobs_dev, jobs_host, sizeof(SliceJob) * size_t(njobs),
                           cudaMemcpyHostToDevice, s));
  unsigned char *sc = static_cast<unsigned char *>(scratch);
  const int *starts = reinterpret_cast<const int *>(sc + size_t(njobs) * 2 * sizeof(CUtensorMap));
  long long *tiles = reinterpret_cast<long long *>(sc + scratch_maps_bytes_x(njobs));
  long long *parts = tiles + size_t(std::min(ntiles, slice_ctas())) * (2 * XM * XN);
  k_gemm_slices<<<std::min(pl.units(), slice_ctas()), XTHREADS, XSMEM, s>>>(
      jobs_dev, reinterpret_cast<const CUtensorMap *>(sc), starts, njobs, pl, tiles, parts, err);
  SGN_LAUNCH_CHECK();
  if (pl.ntail > 0) {
    unsigned low = 0, high = 0;
    for (int p = 0; p < pl.parts; ++p)
      for (int i = pl.bound[p]; i < pl.bound[p + 1]; ++i)
        (kSteps.lp[1][i] == XLP - 1 ? high : low) |= 1u << p;
    k_slices_finish<<<unsigned(pl.ntail) * 32, 256, 0, s>>>(jobs_dev, starts, njobs, pl, parts, low,
                                                          high);
    SGN_LAUNCH_CHECK();
  }
}

}  // namespace sgn

// ---------------------------------------------------------------------------
namespace sgn {
void set_last_error(const std::string &msg);
}

extern "C" sign_status sign_dense_product_f64(int M, int N, int K, const double *A, int lda,
                                              const double *B, int ldb, double *C, int ldc,
                                              void *cuda_stream) {
  using namespace sgn;
  set_last_error("");
  if (M < 0 || N < 0 || K < 0 || !A || !B || !C || lda < K || ldb < N || ldc < N)
    return set_last_error("bad dimensions or NULL pointer"), SIGN_EINVAL;
  if (N % 2 || ldc % 2 || (reinterpret_cast<uintptr_t>(C) & 15u))
    return set_last_error("need N and ldc even, C 16-byte aligned"), SIGN_EINVAL;
  if (M == 0 || N == 0) return SIGN_OK;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  try {
    if (K == 0) {
      SGN_CUDA(cudaMemset2DAsync(C, sizeof(double) * size_t(ldc), 0, sizeof(double) * size_t(N),
                                 size_t(M), s));
      SGN_CUDA(cudaStreamSynchronize(s));
      return SIGN_OK;
    }
    const int kp = (K + 7) / 8 * 8;
    DevBuf dig, wts, err, job, scratch;
    uint16_t *da = static_cast<uint16_t *>(
        dig.ensure(f64x_digits_bytes(M, kp) + f64x_digits_bytes(N, kp) + 256, s));
    uint16_t *db = da + f64x_digits_bytes(M, kp) / sizeof(uint16_t);
    int *wa = static_cast<int *>(wts.ensure(sizeof(int) * size_t(M + N + 4), s));
    int *wb = wa + ((M + 3) / 4 * 4);  // 16-byte aligned
    launch_slices(M, K, A, lda, 0, da, kp, wa, s);
    launch_slices(N, K, B, ldb, 1, db, kp, wb, s);  // Bt = B^T: the columns of B
    SliceJob J{M, N, kp, da, kp, db, kp, wa, wb, C, ldc};  // digits are zero for K <= k < kp
    job.ensure(sizeof(SliceJob), s);
    scratch.ensure(slice_jobs_scratch_bytes(1, slice_tiles(M, N)), s);
    err.ensure(sizeof(int), s);
    SGN_CUDA(cudaMemsetAsync(err.p, 0, sizeof(int), s));
    {
      ProfScope ps(KC_DENSE64, s, 2.0 * XPAIRS * double(M) * double(N) * double(kp), 0.0);
      launch_slice_jobs(1, &J, job.as<SliceJob>(), scratch.p, err.as<int>(), s);
    }
    int herr = 0;
    SGN_CUDA(cudaMemcpyAsync(&herr, err.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    SGN_CUDA(cudaStreamSynchronize(s));
    if (herr) return set_last_error("tensor-core wait gave up"), SIGN_ETIMEOUT;
  } catch (const Error &e) {
    set_last_error(e.what());
    return sign_status(e.status);
  } catch (const std::bad_alloc &) {
    set_last_error("host allocation failed");
    return SIGN_ENOMEM;
  } catch (const std::exception &e) {
    set_last_error(e.what());
    return SIGN_ECUDA;
  }
  return SIGN_OK;
}
