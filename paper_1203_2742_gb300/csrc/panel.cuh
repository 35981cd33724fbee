// Cholesky panel building blocks of the dense and the grouped tier: the
// factorisation of a 32 x 32 block and the row solve against it.
//
// Both are chains of dependent FP64 operations (64 clocks each on GB300, the
// reciprocal square root 350), and a warp issues at most one FP64 instruction
// per 64 clocks whatever the number of active lanes, so what counts is the
// number of FP64 warp instructions on the chain:
//   chol32: four warps, warp w holding columns w mod 4 in registers, lane =
//     row.  Per column: update of the next column, its pivot, scaling, one
//     barrier (about 600 clocks); the warp that owned the pivot catches up on
//     its other columns in the next phase, beside the next pivot.
//   solve_rows: four lanes per row, each holding every fourth column: 32
//     scalings and 124 updates per row group instead of the 528 operations of
//     one lane per row.
// 32 x 32 factor and solve of 32 rows in one launch of mk_potrf_panel: 17 us;
// the earlier form (all threads sweep each column behind three barriers,
// 16 lanes per row) took 44 us.
#pragma once
#include <cstdint>

#include "front_views.cuh"

namespace chd {
namespace panel {

constexpr int PB = 32;    // panel width
constexpr int PTH = 128;  // threads of chol32

// Cholesky of the pb x pb block in Ls (lower; identity beyond pb), in place;
// rinv: reciprocal pivots.  128 threads (tid 0..127) of a CTA whose barrier is
// bar.sync(id, 128); col: 3 x 32 doubles of scratch.  A non-positive pivot is
// recorded and replaced by 1.  The block must be visible to the threads.
__device__ __forceinline__ void bar128(int id) { asm volatile("bar.sync %0, 128;\n" ::"r"(id) : "memory"); }
__device__ __forceinline__ void chol32(double (*Ls)[PB + 1], double* rinv, double (*col)[PB], int pb, int tid, int id,
                                       int64_t* st, int64_t code, int64_t snode, int64_t col0) {
  const int w = tid >> 5, lane = tid & 31;
  double a[9];  // a[t]: column 4 (g + t) + w of column group g
#pragma unroll
  for (int t = 0; t < 8; ++t) a[t] = Ls[lane][4 * t + w];
  a[8] = 0.0;
  bar128(id);
  // pivot of column j by its owner: scaled column to Ls and to col[j % 3]
  auto pivot = [&](int j, double v, double* cj) {
    double d = __shfl_sync(0xffffffffu, v, j);
    if (!(d > 0.0)) {
      if (lane == 0) record_error(st, code, snode, col0 < 0 ? -1 : col0 + j);
      d = 1.0;
    }
    const double r = rsqrt(d);
    const double l = lane == j ? d * r : v * r;
    cj[lane] = l;
    if (lane >= j) Ls[lane][j] = l;
    if (lane == 0) rinv[j] = r;
  };
  if (w == 0) pivot(0, a[0], col[0]);
  bar128(id);
  double *cp = col[2], *cj = col[0], *cn = col[1];  // columns j - 1, j, j + 1
#pragma unroll 1
  for (int g = 0; 4 * g + 1 < pb; ++g) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int j = 4 * g + i;
      if (j + 1 < pb) {  // the same for all threads
        const double lj = cj[lane];
        if (w == ((i + 1) & 3)) {
          const int t = (i + 1) >> 2;  // column j + 1
          a[t] = fma(-lj, cj[j + 1], a[t]);
          pivot(j + 1, a[t], cn);
        } else {
          const bool late = j > 0 && w == i;  // owned pivot j: column j - 1 is still to be applied
          const double lp = late ? cp[lane] : 0.0;
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            const int k = 4 * (g + t) + w;
            if (k < pb && k > j) {
              if (late) a[t] = fma(-lp, cp[k], a[t]);
              a[t] = fma(-lj, cj[k], a[t]);
            }
          }
        }
        bar128(id);
        double* x = cp;
        cp = cj;
        cj = cn;
        cn = x;
      }
    }
#pragma unroll
    for (int t = 0; t < 8; ++t) a[t] = a[t + 1];
  }
}

// Row group of four lanes (q = lane & 3): b[u] holds entry q + 4 u of the row;
// b := b L^{-T} for the pb x pb lower block Ls (rinv: reciprocal pivots).  Rolled
// over groups of four columns, the registers shifted after each: fully
// unrolled, a launch spends more on fetching the code once than on running it.
// g0: the entries before column 4 g0 are zero in all rows of the warp.
__device__ __forceinline__ void solve_row(double (&b)[8], const double (*Ls)[PB + 1], const double* rinv, int pb,
                                          int lane, int g0 = 0) {
  const int q = lane & 3;
#pragma unroll 1
  for (int g = 0; g < PB / 4; ++g) {
    if (g >= g0 && 4 * g < pb) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int c = 4 * g + i;
        if (c < pb) {
          double x = b[0] * rinv[c];
          x = __shfl_sync(0xffffffffu, x, (lane & 28) | i);
          if (q == i) b[0] = x;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int t = 4 * (g + u) + q;
            if (4 * (g + u) < pb && (u > 0 || i < 3)) {
              const double l = t > c && t < pb ? Ls[t][c] : 0.0;
              b[u] = fma(-l, x, b[u]);
            }
          }
        }
      }
    }
    // the finished entry goes to the back: after eight shifts all are in place
    const double f = b[0];
#pragma unroll
    for (int u = 0; u < 7; ++u) b[u] = b[u + 1];
    b[7] = f;
  }
}
// b := b L^{-1}: the same backwards
__device__ __forceinline__ void solve_row_back(double (&b)[8], const double (*Ls)[PB + 1], const double* rinv, int pb,
                                               int lane) {
  const int q = lane & 3;
#pragma unroll 1
  for (int g = PB / 4 - 1; g >= 0; --g) {
    // b[7] is group g here
    if (4 * g < pb) {
#pragma unroll
      for (int i = 3; i >= 0; --i) {
        const int c = 4 * g + i;
        if (c < pb) {
          double x = b[7] * rinv[c];
          x = __shfl_sync(0xffffffffu, x, (lane & 28) | i);
          if (q == i) b[7] = x;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int t = 4 * (g - 7 + u) + q;  // group g - 7 + u
            if (g - 7 + u >= 0 && (u < 7 || i > 0)) {
              const double l = t < c ? Ls[c][t] : 0.0;
              b[u] = fma(-l, x, b[u]);
            }
          }
        }
      }
    }
    const double f = b[7];
#pragma unroll
    for (int u = 7; u > 0; --u) b[u] = b[u - 1];
    b[0] = f;
  }
}

}  // namespace panel
}  // namespace chd
