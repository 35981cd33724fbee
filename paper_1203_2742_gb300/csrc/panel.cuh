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
  double a[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) a[t] = Ls[lane][4 * t + w];
  bar128(id);
  // pivot of column j by its owner: scaled column to Ls and to col[j % 3]
  auto pivot = [&](int j, double v) {
    double d = __shfl_sync(0xffffffffu, v, j);
    if (!(d > 0.0)) {
      if (lane == 0) record_error(st, code, snode, col0 < 0 ? -1 : col0 + j);
      d = 1.0;
    }
    const double r = rsqrt(d);
    const double l = lane == j ? d * r : v * r;
    col[j % 3][lane] = l;
    if (lane >= j) Ls[lane][j] = l;
    if (lane == 0) rinv[j] = r;
  };
  if (w == 0) pivot(0, a[0]);
  bar128(id);
#pragma unroll
  for (int j = 0; j < PB; ++j) {
    if (j + 1 < pb) {
      const double* cj = col[j % 3];
      const double lj = cj[lane];
      if (w == ((j + 1) & 3)) {
        a[(j + 1) >> 2] = fma(-lj, cj[j + 1], a[(j + 1) >> 2]);
        pivot(j + 1, a[(j + 1) >> 2]);
      } else {
        if (j > 0 && w == (j & 3)) {  // owned pivot j in the last phase: column j - 1 is still to be applied
          const double* cp = col[(j + 2) % 3];
          const double lp = cp[lane];
#pragma unroll
          for (int t = (j >> 2) + 1; t < 8; ++t)
            if (4 * t + w < pb) a[t] = fma(-lp, cp[4 * t + w], a[t]);
        }
#pragma unroll
        for (int t = 0; t < 8; ++t)
          if (4 * t + w > j && 4 * t + w < pb) a[t] = fma(-lj, cj[4 * t + w], a[t]);
      }
      bar128(id);
    }
  }
}

// Row group of four lanes (q = lane & 3): b[u] holds entry q + 4 u of the row;
// b := b L^{-T} for the pb x pb lower block Ls (rinv: reciprocal pivots)
__device__ __forceinline__ void solve_row(double (&b)[8], const double (*Ls)[PB + 1], const double* rinv, int pb,
                                          int lane) {
  const int q = lane & 3;
#pragma unroll
  for (int c = 0; c < PB; ++c) {
    if (c < pb) {
      double x = b[c >> 2] * rinv[c];
      x = __shfl_sync(0xffffffffu, x, (lane & 28) | (c & 3));
      if (q == (c & 3)) b[c >> 2] = x;
#pragma unroll
      for (int u = c >> 2; u < 8; ++u) {
        const int t = 4 * u + q;
        if (4 * u + 3 > c) {
          const double l = t > c ? Ls[t][c] : 0.0;
          b[u] = fma(-l, x, b[u]);
        }
      }
    }
  }
}

}  // namespace panel
}  // namespace chd
