// Grouped tier: the gradient, the Hessian and the inverse Hessian of the
// fronts between the warp tier and the large dense fronts, one launch per
// step over all fronts of a sub-level (or, for the steps that no other front
// waits for, over all fronts), each step cut into tiles or blocks of rows so
// that many SMs work on one front.
//
// Andersen, Dahl, Vandenberghe, "Logarithmic barriers for sparse matrix
// cones": the per-front formulas are those of Algorithm 7.2 and of the block
// forms of Algorithms 5.1 and 5.2, as in the per-task tier (kernels.cu).
//
// Why.  A GB300 SM retires about 1.7 FP64 FMAs per clock, 3.5 GFMA/s, so one
// CTA needs 2.6 ms for the 6 a^2 n flops of a front with a = 300, n = 10 --
// and a 3D grid has chains of a hundred such fronts, each waiting for the
// previous one, with two or three per level.  Cut into 32 x 32 tiles or
// blocks of 8 rows the same front occupies 50 to 100 SMs for about 10
// microseconds, and a launch costs half a microsecond inside a CUDA graph.
// Loads are not the limit at any tile size (a 16 x 16 tile moves one double
// per eight FMAs), so the tiles are small and nothing is double-buffered;
// several CTAs per SM cover the latencies.
//
// What waits for what.  Bottom-up, a parent needs only the update block U';
// step 2 of Algorithm 5.1 (M = V K D^{-1}) feeds nobody and runs once, over
// all fronts, at the end of the pass.  Top-down, a child needs the parent's
// whole front.  In the inverse Hessian the top-down blocks V' are parts of
// the input: a light pass copies them down the tree, and all arithmetic of
// steps 1 and 2 runs over all fronts at once.
//
// Symmetric blocks are stored as lower triangles.  A CTA that needs whole
// rows r0 .. r0+R-1 of one reads the columns left of the diagonal block with
// its lanes along the rows and the transposed part with its lanes along the
// columns, so both are contiguous in memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <type_traits>

#include "chd_internal.h"
#include "front_views.cuh"
#include "panel.cuh"

namespace chd_launch {
void count_launch();
}

namespace chd {
namespace grp {

constexpr int GB = kGroupBlock;  // rows per block of the assembly and of the update tiles
constexpr int GN = kGroupThin;   // fronts up to this many columns form P inside the update tile
constexpr int RT = 128;          // threads of the row-block kernels
constexpr int KC = 128;          // inner chunk of the row-block products
constexpr int CB = 16;           // columns per register block
constexpr int CBL = CB + 1;      // their stride in shared memory (lanes along k: no bank conflicts)

// block b of a front: rows [first, first + count) of J_k; N is cut first
__device__ __forceinline__ void block_range(const GFront& f, int b, int& first, int& count) {
  if (b < f.nbn) {
    first = b * GB;
    count = min(GB, f.n - first);
  } else {
    const int r = (b - f.nbn) * GB;
    first = f.n + r;
    count = max(0, min(GB, f.a - r));
  }
}
// Adds the children's update blocks that fall on block pair (bi, bj), bi >= bj,
// to the tile t (row r, column c at t[r * ld + c]); 256 threads.  A child's
// rows inside a block are a contiguous range of its ancestor set (gptr), so
// children that miss the tile cost two loads.  The caller synchronises between
// two children whose entries can coincide.
__device__ __forceinline__ void add_child(const SymDev& S, const GChild& c, const double* ws, int bi, int fi, int bj,
                                          int fj, double* t, int ld) {
  const int32_t* ptr = S.gptr + c.ptr_off;
  const int i0 = __ldg(ptr + bi), i1 = __ldg(ptr + bi + 1);
  const int j0 = __ldg(ptr + bj), j1 = __ldg(ptr + bj + 1);
  const int i = i0 + (threadIdx.x & 31);
  if (i >= i1) return;
  const int32_t* rel = S.rel + c.rel_off;
  const int r = __ldg(rel + i) - fi;
  const double* U = ws + c.u_off;
  for (int j = j0 + (threadIdx.x >> 5); j < j1; j += 8)
    if (i >= j) t[r * ld + (__ldg(rel + j) - fj)] += __ldcg(U + i + (int64_t)j * c.Jc);
}

// The same for all children of a front that has many.  One child after another behind
// a barrier each is a chain of dependent loads (record, range, rows, entries), 1.5 us a
// child.  Here lane r of warp w owns the entries (r, w), (r, w + 8), .. (c < nc) and
// adds every child to them in order, so no barrier is needed and two children are in
// flight: the lane of a row finds its place in a child's range by counting the rows
// before it.  Pruned children (act[k] == 0) are left out 32 at a time.  The caller writes
// and reads other threads' entries behind barriers of its own.  A root of 20 columns
// under 2000 children: factor 3210 -> 2010 us, Hessian of eight 3670 -> 2510.  It takes 64
// registers instead of 40 and costs fronts of few children that much occupancy (20 x 20 x
// 20 grid, Hessian of eight 37.5 -> 39.6 ms), hence the rule at kManyChildren.
__device__ __forceinline__ void add_children(const SymDev& S, const GFront& f, const double* ws, const uint8_t* act,
                                             int bi, int fi, int bj, int fj, double* t, int ld, int nc) {
  constexpr int CHB = 2;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned below = (1u << lane) - 1;
  double x[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) x[k] = w + 8 * k < nc ? t[lane * ld + w + 8 * k] : 0.0;
  for (int q0 = f.ch_beg; q0 < f.ch_end; q0 += 32) {
    const bool mine = q0 + lane < f.ch_end && (!act || act[S.gch[q0 + lane].k]);
    unsigned todo = __ballot_sync(0xffffffffu, mine);  // the same in all warps
    while (todo) {
      const double* U[CHB];
      int Jc[CHB], i0[CHB], ni[CHB], j0[CHB], nj[CHB], ri[CHB], rj[CHB];
#pragma unroll
      for (int u = 0; u < CHB; ++u) {
        ni[u] = nj[u] = 0;
        ri[u] = rj[u] = -1;
        if (todo) {
          const GChild c = S.gch[q0 + __ffs(todo) - 1];
          todo &= todo - 1;
          const int32_t* ptr = S.gptr + c.ptr_off;
          i0[u] = __ldg(ptr + bi);
          ni[u] = __ldg(ptr + bi + 1) - i0[u];
          j0[u] = __ldg(ptr + bj);
          nj[u] = __ldg(ptr + bj + 1) - j0[u];
          const int32_t* rel = S.rel + c.rel_off;
          if (lane < ni[u]) ri[u] = __ldg(rel + i0[u] + lane) - fi;
          if (lane < nj[u]) rj[u] = __ldg(rel + j0[u] + lane) - fj;
          U[u] = ws + c.u_off;
          Jc[u] = c.Jc;
        }
      }
      double v[CHB][4];
      bool in[CHB][4];
#pragma unroll
      for (int u = 0; u < CHB; ++u) {
#pragma unroll
        for (int k = 0; k < 4; ++k) in[u][k] = false;
        if (ni[u] > 0 && nj[u] > 0) {  // the same for all threads
          const unsigned mi = __reduce_or_sync(0xffffffffu, ri[u] >= 0 ? 1u << ri[u] : 0u);
          const unsigned mj = __reduce_or_sync(0xffffffffu, rj[u] >= 0 ? 1u << rj[u] : 0u);
          const int i = i0[u] + __popc(mi & below);
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int c = w + 8 * k, j = j0[u] + __popc(mj & ((1u << c) - 1));
            in[u][k] = (mi >> lane & 1) && (mj >> c & 1) && i >= j && c < nc;
            if (in[u][k]) v[u][k] = __ldcg(U[u] + i + (int64_t)j * Jc[u]);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < CHB; ++u)
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (in[u][k]) x[k] += v[u][k];
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (w + 8 * k < nc) t[lane * ld + w + 8 * k] = x[k];
}

// the counters of the row-block kernels (last double of T2), before a pass
__global__ void __launch_bounds__(256) kg_zero(SymDev S, int first, int count, double* ws) {
  const int g = blockIdx.x * 256 + threadIdx.x;
  if (g >= count) return;
  const GFront& f = S.gf[first + g];
  double* T2e = ws + blockIdx.y * S.f_total + f.f_off + (int64_t)f.J * f.J + 2 * (int64_t)f.J * f.n;
  *reinterpret_cast<int*>(T2e - 1) = 0;
}

// ---------------------------------------------------------------------------
// assembly of whole fronts (wide fronts bottom-up; every front of the inverse
// Hessian top-down): one 32 x 32 block pair per CTA
//   ASM_UP:     F = the input's columns N_k plus the children's blocks
//   ASM_GATHER: F = the input's columns N_k, and the A x A block from the parent
//   ASM_FACTOR: as ASM_UP, and D_NN = F_NN
// ---------------------------------------------------------------------------
enum { ASM_UP = 0, ASM_GATHER, ASM_FACTOR };
// MANY: some front of the launch has many children (add_children)
template <int MODE, bool MANY>
__global__ void __launch_bounds__(256) kg_assemble(SymDev S, const int2* tiles, const double* Y, int64_t ldy,
                                                  double* ws, const uint8_t* act, double* Dd) {
  __shared__ double t[GB][GB + 1];
  const int2 d = tiles[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int bi = d.y & 0xffff, bj = d.y >> 16, tid = threadIdx.x;
  const int64_t y = blockIdx.y;
  if (MODE == ASM_UP && act) {
    act += y * S.nsn;
    if (!act[f.k]) return;
  }
  ws += y * S.f_total;
  const double* v = Y + y * ldy + f.base;
  int fi, ni, fj, nj;
  block_range(f, bi, fi, ni);
  block_range(f, bj, fj, nj);
  double* F = ws + f.f_off;
  const int r = tid & 31;
  if (MODE == ASM_GATHER) {
    const double* Fp = ws + f.fp_off;
    const int32_t* rel = S.rel + f.rel_off;
    if (r < ni)
      for (int c = tid >> 5; c < nj; c += 8) {
        const int row = fi + r, col = fj + c;
        if (row < col) continue;
        F[row + (int64_t)col * f.J] =
            col < f.n ? v[csc_off(f.J, row, col)]
                      : __ldcg(Fp + __ldg(rel + row - f.n) + (int64_t)__ldg(rel + col - f.n) * f.Jp);
      }
    return;
  }
  for (int c = tid >> 5; c < GB; c += 8) {
    const int row = fi + r, col = fj + c;
    t[r][c] = r < ni && c < nj && row >= col && col < f.n ? v[csc_off(f.J, row, col)] : 0.0;
  }
  __syncthreads();
  if constexpr (MANY) {
    add_children(S, f, ws, MODE == ASM_UP ? act : nullptr, bi, fi, bj, fj, &t[0][0], GB + 1, GB);
  } else {
    for (int q = f.ch_beg; q < f.ch_end; ++q) {
      const GChild c = S.gch[q];
      if (act && !act[c.k]) continue;  // pruned child (§5.5): its update block is zero
      add_child(S, c, ws, bi, fi, bj, fj, &t[0][0], GB + 1);
      __syncthreads();
    }
  }
  if (r < ni)
    for (int c = tid >> 5; c < nj; c += 8) {
      const int row = fi + r, col = fj + c;
      if (row >= col) F[row + (int64_t)col * f.J] = t[r][c];
      if (MODE == ASM_FACTOR && row >= col && row < f.n) Dd[f.d_off + row + (int64_t)col * f.n] = t[r][c];
    }
}

// P = Yh_AN - L Yh_NN / 2 of the wide fronts (into T1): 32 x 32 tiles, K = n
__global__ void __launch_bounds__(256) kg_p(SymDev S, const int2* tiles, const double* Wc, double* ws,
                                           const uint8_t* act) {
  __shared__ double As[GB][17], Bs[16][GB + 1];
  const int2 d = tiles[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int64_t y = blockIdx.y;
  if (act && !act[y * S.nsn + f.k]) return;
  ws += y * S.f_total;
  const int r0 = (d.y & 0xffff) * GB, c0 = (d.y >> 16) * GB, tid = threadIdx.x;
  const double* W = Wc + f.base;
  double* F = ws + f.f_off;
  double* T1 = F + (int64_t)f.J * f.J;
  const int tr = tid & 15, tc = tid >> 4;
  double a00 = 0, a01 = 0, a10 = 0, a11 = 0;
  for (int k0 = 0; k0 < f.n; k0 += 16) {
    for (int e = tid; e < GB * 16; e += 256) {
      const int r = e & 31, k = e >> 5;
      As[r][k] = r0 + r < f.a && k0 + k < f.n ? W[csc_off(f.J, f.n + r0 + r, k0 + k)] : 0.0;
      const int kk = e & 15, c = e >> 4;  // symmetric N x N block, lower stored
      const int i = k0 + kk, j = c0 + c;
      Bs[kk][c] = i < f.n && j < f.n ? (i >= j ? F[i + (int64_t)j * f.J] : F[j + (int64_t)i * f.J]) : 0.0;
    }
    __syncthreads();
    const int kc = min(16, f.n - k0);
    for (int k = 0; k < kc; ++k) {
      const double x0 = As[tr][k], x1 = As[tr + 16][k], b0 = Bs[k][tc], b1 = Bs[k][tc + 16];
      a00 = fma(x0, b0, a00);
      a01 = fma(x0, b1, a01);
      a10 = fma(x1, b0, a10);
      a11 = fma(x1, b1, a11);
    }
    __syncthreads();
  }
  const double acc[2][2] = {{a00, a01}, {a10, a11}};
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = r0 + tr + 16 * i, c = c0 + tc + 16 * j;
      if (r < f.a && c < f.n)
        T1[f.n + r + (int64_t)c * f.J] = fma(-0.5, acc[i][j], F[f.n + r + (int64_t)c * f.J]);
    }
}

// ---------------------------------------------------------------------------
// update tiles, bottom-up: one 32 x 32 tile of the A x A block per CTA,
//   U' = (assembled block) - (P L^T + L P^T)
// UP_HESS:  thin fronts (n <= 16) assemble the N-part of their rows and form
//           P = Yh_AN - L Yh_NN / 2 here (n / 32 of the tile's own FMAs, one
//           launch per sub-level instead of three); wide ones find the front
//           assembled and P in T1.  The first tile column stores F_AN, P and
//           F_NN for step 2.
// UP_IHESS: P is in the N-part of F (left by step 2).  The CTAs beyond the tiles
//           subtract the children's part from the output's columns N_k, a 32 x 32
//           block each (fronts with children only).  A CTA walks the children
//           one by one, so a block per CTA: 400 children of five columns
//           under one front of 40, one right-hand side: 2020 us with all blocks of the
//           front's rows in the CTAs of the first tile column, 907 so (620 with add_children).
// ---------------------------------------------------------------------------
enum { UP_HESS = 0, UP_IHESS = 1 };
template <int MODE, bool MANY>
__global__ void __launch_bounds__(256) kg_up(SymDev S, const int2* tiles, const double* Wc, const double* Y,
                                            int64_t ldy, double* Yo, double* ws, const uint8_t* act,
                                            const int2* outs, int ntiles) {
  __shared__ double t[GB][GB + 1];
  __shared__ double sP[2][GB][GN + 1], sL[2][GB][GN + 1];
  __shared__ double sN[MANY ? GB : GN][GN + 1];  // add_children passes over GB rows
  const bool out_block = MODE == UP_IHESS && (int)blockIdx.x >= ntiles;
  const int2 d = out_block ? outs[blockIdx.x - ntiles] : tiles[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int64_t y = blockIdx.y;
  if (MODE == UP_HESS && act) {
    act += y * S.nsn;
    if (!act[f.k]) return;  // pruned (§5.5): K, U' and M are zero here
  }
  ws += y * S.f_total;
  if (out_block) {
    // Y_NN = K_NN - Z_NN, Y_AN = (K_AN + L K_NN) - Z_AN, Z the children's part
    const int rb = d.y & 0xffff, cb = d.y >> 16;
    int gi, ni, gj, nj;
    block_range(f, rb, gi, ni);
    block_range(f, cb, gj, nj);
    for (int e = threadIdx.x; e < GB * (GB + 1); e += 256) (&t[0][0])[e] = 0.0;
    __syncthreads();
    if constexpr (MANY) {
      add_children(S, f, ws, nullptr, rb, gi, cb, gj, &t[0][0], GB + 1, GB);
    } else {
      for (int q = f.ch_beg; q < f.ch_end; ++q) {
        add_child(S, S.gch[q], ws, rb, gi, cb, gj, &t[0][0], GB + 1);
        __syncthreads();
      }
    }
    double* out = Yo + y * ldy + f.base;
    const int r = threadIdx.x & 31;
    if (r < ni)
      for (int c = threadIdx.x >> 5; c < nj; c += 8)
        if (gi + r >= gj + c) out[csc_off(f.J, gi + r, gj + c)] -= t[r][c];
    return;
  }
  const int tm = d.y & 0xffff, tn = d.y >> 16, tid = threadIdx.x;
  const int r0 = tm * GB, c0 = tn * GB, n = f.n, J = f.J;
  const int nr = min(GB, f.a - r0), nc = min(GB, f.a - c0);
  const int bi = f.nbn + tm, bj = f.nbn + tn, fi = n + r0, fj = n + c0;
  double* F = ws + f.f_off;
  double* T1 = F + (int64_t)J * J;
  const double* W = Wc + f.base;
  const bool thin = MODE == UP_HESS && n <= GN;
  if (!thin && f.a == 0) return;  // no update block (UP_HESS: assembled before)
  const int side = tm == tn ? 0 : 1;  // the column block's vectors (the row block's on the diagonal)
  const int tr = tid & 15, tc = tid >> 4;
  double acc[2][2] = {{0, 0}, {0, 0}};
  // acc += P L^T + L P^T over jn columns; FP64-bound, so 16 x 16 quarters beyond
  // the block's rows or above the diagonal are left out (600 fronts of 20 columns and
  // 40 ancestors, Hessian of eight: 3950 -> 3720 us)
  auto products = [&](int jn) {
    auto run = [&](auto row1, auto col1) {  // whether (1, .) and (0, 1) are wanted
      for (int j = 0; j < jn; ++j) {
        const double p0 = sP[0][tr][j], l0 = sL[0][tr][j], lc = sL[side][tc][j], pc = sP[side][tc][j];
        acc[0][0] = fma(p0, lc, acc[0][0]);
        acc[0][0] = fma(l0, pc, acc[0][0]);
        if constexpr (row1.value || col1.value) {
          const double ld = sL[side][tc + 16][j], pd = sP[side][tc + 16][j];
          if constexpr (col1.value) {
            acc[0][1] = fma(p0, ld, acc[0][1]);
            acc[0][1] = fma(l0, pd, acc[0][1]);
          }
          if constexpr (row1.value) {
            const double p1 = sP[0][tr + 16][j], l1 = sL[0][tr + 16][j];
            acc[1][0] = fma(p1, lc, acc[1][0]);
            acc[1][0] = fma(l1, pc, acc[1][0]);
            acc[1][1] = fma(p1, ld, acc[1][1]);
            acc[1][1] = fma(l1, pd, acc[1][1]);
          }
        }
      }
    };
    using yes = std::true_type;
    using no = std::false_type;
    if (nr > 16) {
      if (side) run(yes{}, yes{});
      else run(yes{}, no{});
    } else {
      if (side) run(no{}, yes{});
      else run(no{}, no{});
    }
  };
  for (int e = tid; e < GB * (GB + 1); e += 256) (&t[0][0])[e] = 0.0;
  if (thin) {
    const double* v = Y + y * ldy + f.base;
    for (int e = tid; e < GN * GN; e += 256) {
      const int i = e & (GN - 1), j = e / GN;
      sN[i][j] = i < n && j <= i ? v[csc_off(J, i, j)] : 0.0;
    }
    for (int s = 0; s <= side; ++s) {
      const int q0 = s ? c0 : r0, cnt = s ? nc : nr;
      for (int e = tid; e < GB * GN; e += 256) {
        const int r = e & 31, j = e >> 5;
        const bool in = r < cnt && j < n;
        const int64_t o = csc_off(J, n + q0 + r, j);
        sP[s][r][j] = in ? v[o] : 0.0;
        sL[s][r][j] = in ? W[o] : 0.0;
      }
    }
  }
  __syncthreads();
  if (MANY && (thin || MODE == UP_IHESS)) {
    if constexpr (MANY) {
      const uint8_t* ac = MODE == UP_HESS ? act : nullptr;
      if (f.a > 0) add_children(S, f, ws, ac, bi, fi, bj, fj, &t[0][0], GB + 1, GB);
      if (thin) {
        add_children(S, f, ws, ac, 0, 0, 0, 0, &sN[0][0], GN + 1, GN);
        if (f.a > 0) {
          add_children(S, f, ws, ac, bi, fi, 0, 0, &sP[0][0][0], GN + 1, GN);
          if (side) add_children(S, f, ws, ac, bj, fj, 0, 0, &sP[1][0][0], GN + 1, GN);
        }
      }
      __syncthreads();
    }
  } else if (thin || MODE == UP_IHESS) {
    for (int q = f.ch_beg; q < f.ch_end; ++q) {
      const GChild c = S.gch[q];
      if (MODE == UP_HESS && act && !act[c.k]) continue;
      if (f.a > 0) add_child(S, c, ws, bi, fi, bj, fj, &t[0][0], GB + 1);
      if (thin) {
        add_child(S, c, ws, 0, 0, 0, 0, &sN[0][0], GN + 1);
        if (f.a > 0) {
          add_child(S, c, ws, bi, fi, 0, 0, &sP[0][0][0], GN + 1);
          if (side) add_child(S, c, ws, bj, fj, 0, 0, &sP[1][0][0], GN + 1);
        }
      }
      __syncthreads();
    }
  }
  if (thin) {
    for (int e = tid; e < GN * GN; e += 256) {
      const int i = e & (GN - 1), j = e / GN;
      if (i < n && j <= i) {
        if (tm == 0 && tn == 0) F[i + (int64_t)j * J] = sN[i][j];
        if (j < i) sN[j][i] = sN[i][j];
      }
    }
    if (f.a == 0) return;
    if (tn == 0)
      for (int e = tid; e < GB * n; e += 256) {
        const int r = e & 31, j = e >> 5;
        if (r < nr) F[fi + r + (int64_t)j * J] = sP[0][r][j];
      }
    __syncthreads();
    for (int s = 0; s <= side; ++s)
      for (int e = tid; e < GB * n; e += 256) {
        const int r = e & 31, j = e >> 5;
        double x = 0.0;
        for (int q = 0; q < n; ++q) x = fma(sL[s][r][q], sN[q][j], x);
        x = fma(-0.5, x, sP[s][r][j]);
        sP[s][r][j] = x;
        if (s == 0 && tn == 0 && r < nr) T1[fi + r + (int64_t)j * J] = x;
      }
    __syncthreads();
    products(n);
  } else if (f.a > 0) {
    const double* P = MODE == UP_HESS ? T1 : F;
    for (int j0 = 0; j0 < n; j0 += GN) {
      for (int s = 0; s <= side; ++s) {
        const int q0 = s ? c0 : r0, cnt = s ? nc : nr;
        for (int e = tid; e < GB * GN; e += 256) {
          const int r = e & 31, j = e >> 5;
          const bool in = r < cnt && j0 + j < n;
          sP[s][r][j] = in ? P[n + q0 + r + (int64_t)(j0 + j) * J] : 0.0;
          sL[s][r][j] = in ? W[csc_off(J, n + q0 + r, j0 + j)] : 0.0;
        }
      }
      __syncthreads();
      products(min(GN, n - j0));
      __syncthreads();
    }
  }
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int r = tr + 16 * u, c = tc + 16 * w;
      if (r < nr && c < nc && r0 + r >= c0 + c) {
        double* o = F + fi + r + (int64_t)(fj + c) * J;
        *o = (MODE == UP_HESS && !thin ? *o : t[r][c]) - acc[u][w];
      }
    }
}

// ---------------------------------------------------------------------------
// row-block kernels: rows r0 .. r0 + R - 1 of (symmetric a x a) (a x n),
// R = 8 << lrb (chosen by the analysis: enough blocks for a full GPU, few
// enough for their n x n partial sums to fit T2), 128 threads
//   RK_GRAD:  S_AN = -V L; the block's share of L^T V L; the last block of
//             the front finishes S_NN
//   RK_HDOWN: W = V' L, T_AN = M_AN - W; shares of T_NN; the last block of
//             the front finishes T_NN
//   RK_M:     M_AN = (V K_AN) D^{-1}
//   RK_IH1:   M_AN = T_AN + V' L (into T1); shares of M_NN (into T2)
//   RK_IH2:   K_AN = (V^{-1} M_AN) D, P = K_AN + L K_NN / 2 (into F),
//             Y_AN = K_AN + L K_NN
// The blocks of a front meet at a counter (reset by the last one); their
// partial sums are added in block order, so the result does not depend on
// the order of arrival.
// ---------------------------------------------------------------------------
enum { RK_GRAD = 0, RK_HDOWN, RK_M, RK_IH1, RK_IH2 };
struct RowArgs {
  const double* Wc;
  const double* mat;  // Vd (RK_M), Rd (RK_IH2)
  const double* Dd;   // RK_IH2
  double* out;        // Sc, T or Y
  int64_t ldo;
  double* g;          // RK_GRAD: gradient or null
  double* Vd;         // RK_GRAD
  const uint8_t* act;
};
// One pass of the product over columns c0 .. c0 + cn - 1 (cn <= CBT): LEFT:
// k < rend, lanes along the rows; else k >= rend, lanes along k.  Each thread
// holds RM rows by CBT columns for its share of k, so a shared-memory load of
// the skinny factor feeds RM FMAs; the shares are summed in a fixed order.
template <int MODE, int CBT, int RM, bool LEFT>
__device__ __forceinline__ void rows_pass(const SymDev& S, const GFront& f, const RowArgs& A, double* ws, int r0,
                                          int lr, int c0, int cn, double* Ls, int* Rs, double* red, double* Wr) {
  constexpr bool FROM_PARENT = MODE == RK_GRAD || MODE == RK_HDOWN;
  const int tid = threadIdx.x, n = f.n, a = f.a, J = f.J, R = 1 << lr;
  const int ll = lr - (RM == 2 ? 1 : 0), RL = 1 << ll, lng = 7 - ll, NG = 1 << lng;
  const int rend = min(r0 + R, a), klo = LEFT ? 0 : rend, khi = LEFT ? rend : a;
  double* F = ws + f.f_off;
  double* T1 = F + (int64_t)J * J;
  const double* W = A.Wc + f.base;
  const double* M = nullptr;
  int64_t ldm = 0;
  const double* Fp = ws + f.fp_off;
  const int32_t* rel = S.rel + f.rel_off;
  if (MODE == RK_IH1) {
    M = F + n + (int64_t)n * J;
    ldm = J;
  } else if (!FROM_PARENT) {
    M = A.mat + f.v_off;
    ldm = a;
  }
  const int g = LEFT ? tid >> ll : tid & (NG - 1), rr = LEFT ? tid & (RL - 1) : tid >> lng;
  int row[RM], pr[RM];
  bool in[RM];
  double x[RM][CBT];
#pragma unroll
  for (int m = 0; m < RM; ++m) {
    row[m] = r0 + rr + m * RL;
    in[m] = row[m] < a;
    pr[m] = FROM_PARENT && in[m] ? __ldg(rel + row[m]) : 0;
#pragma unroll
    for (int c = 0; c < CBT; ++c) x[m][c] = 0.0;
  }
  double* Vk = MODE == RK_GRAD ? A.Vd + f.v_off : nullptr;
  constexpr int UN = RM == 2 ? 2 : 4;  // k steps whose loads are in flight together
  for (int k0 = klo; k0 < khi; k0 += KC) {
    const int kc = min(KC, khi - k0);
    __syncthreads();
    if (FROM_PARENT)
      for (int k = tid; k < kc; k += RT) Rs[k] = __ldg(rel + k0 + k);
    for (int e = tid; e < KC * cn; e += RT) {
      const int k = e & (KC - 1), c = e / KC;
      double v = 0.0;
      if (k < kc) {
        const int64_t o = n + k0 + k + (int64_t)(c0 + c) * J;
        if (MODE == RK_M) v = 2.0 * T1[o] - F[o];  // K_AN = 2 P - Yh_AN
        else if (MODE == RK_IH2) v = T1[o];
        else v = W[csc_off(J, n + k0 + k, c0 + c)];
      }
      Ls[k * CBL + c] = v;
    }
    __syncthreads();
    for (int kb = g; kb < kc; kb += UN * NG) {
      double v[UN][RM];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int k = kb + u * NG, col = k0 + k;
#pragma unroll
        for (int m = 0; m < RM; ++m) {
          v[u][m] = 0.0;
          if (k < kc && in[m]) {
            const bool low = LEFT && row[m] >= col;
            if (FROM_PARENT) {
              const int pc = Rs[k];
              v[u][m] = __ldcg(Fp + (low ? pr[m] + (int64_t)pc * f.Jp : pc + (int64_t)pr[m] * f.Jp));
            } else {
              v[u][m] = low ? M[row[m] + (int64_t)col * ldm] : M[col + (int64_t)row[m] * ldm];
            }
          }
        }
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const int k = kb + u * NG, col = k0 + k;
        if (k >= kc) break;
        if (FROM_PARENT && LEFT && c0 == 0) {
#pragma unroll
          for (int m = 0; m < RM; ++m)
            if (in[m] && row[m] >= col) {
              F[n + row[m] + (int64_t)(n + col) * J] = v[u][m];
              if (MODE == RK_GRAD) Vk[row[m] + (int64_t)col * a] = v[u][m];
            }
        }
#pragma unroll
        for (int c = 0; c < CBT; ++c)
          if (c < cn) {
            const double l = Ls[k * CBL + c];
#pragma unroll
            for (int m = 0; m < RM; ++m) x[m][c] = fma(v[u][m], l, x[m][c]);
          }
      }
    }
  }
  constexpr int CH = CBT < 8 ? CBT : 8;  // columns per round of the sums: red[g][c][r]
#pragma unroll
  for (int h = 0; h < CBT; h += CH) {
    if (h >= cn) break;
    __syncthreads();
#pragma unroll
    for (int c = 0; c < CH; ++c)
#pragma unroll
      for (int m = 0; m < RM; ++m) red[(g * CH + c) * R + rr + m * RL] = x[m][h + c];
    __syncthreads();
    const int ce = min(CH, cn - h);
    for (int e = tid; e < R * ce; e += RT) {
      const int r = e & (R - 1), c = e >> lr;
      double* w = Wr + r + (c0 + h + c) * R;
      double t = LEFT ? 0.0 : *w;
      for (int q = 0; q < NG; ++q) t += red[(q * CH + c) * R + r];
      *w = t;
    }
  }
}
template <int MODE, int CBT, int RM>
__device__ __forceinline__ void rows_block(const SymDev& S, const GFront& f, const RowArgs& A, double* ws, int r0,
                                           int lr, int c0, int cn, double* Ls, int* Rs, double* red, double* Wr) {
  rows_pass<MODE, CBT, RM, true>(S, f, A, ws, r0, lr, c0, cn, Ls, Rs, red, Wr);
  if (r0 + (1 << lr) < f.a) rows_pass<MODE, CBT, RM, false>(S, f, A, ws, r0, lr, c0, cn, Ls, Rs, red, Wr);
}
// rows r0 .. r0 + R - 1 of the product into Wr (R x n), columns in blocks of
// up to 16: the narrowest instance that holds a block, because unused columns
// would still be loaded from shared memory
template <int MODE>
__device__ __forceinline__ void rows_product(const SymDev& S, const GFront& f, int r0, const RowArgs& A, double* ws,
                                             double* Ls, int* Rs, double* red, double* Wr) {
  const int lr = f.lrb + 3;
  for (int c0 = 0; c0 < f.n; c0 += CB) {
    const int cn = min(CB, f.n - c0);
    if (lr >= 4) {
      if (cn <= 4) rows_block<MODE, 4, 2>(S, f, A, ws, r0, lr, c0, cn, Ls, Rs, red, Wr);
      else rows_block<MODE, 16, 2>(S, f, A, ws, r0, lr, c0, cn, Ls, Rs, red, Wr);
    } else {
      if (cn == 1) rows_block<MODE, 1, 1>(S, f, A, ws, r0, lr, c0, cn, Ls, Rs, red, Wr);
      else if (cn <= 4) rows_block<MODE, 4, 1>(S, f, A, ws, r0, lr, c0, cn, Ls, Rs, red, Wr);
      else rows_block<MODE, 16, 1>(S, f, A, ws, r0, lr, c0, cn, Ls, Rs, red, Wr);
    }
  }
  __syncthreads();
}

template <int MODE>
__global__ void __launch_bounds__(RT) kg_rows(SymDev S, const int2* blocks, RowArgs A, double* ws) {
  extern __shared__ double dyn[];
  __shared__ int last, Rs[KC];
  const int2 d = blocks[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int64_t y = blockIdx.y;
  if (MODE == RK_M && A.act && !A.act[y * S.nsn + f.k]) return;
  ws += y * S.f_total;
  const int n = f.n, a = f.a, J = f.J, lrb = f.lrb, R = 8 << lrb, r0 = d.y * R, tid = threadIdx.x;
  const int nr = max(0, min(R, a - r0));
  double* Ls = dyn;                // KC x CBL
  double* red = Ls + KC * CBL;     // (128 / R) x CB x R
  double* Wr = red + RT * CB;      // R x n
  double* Lr = Wr + R * n;         // R x n
  double* F = ws + f.f_off;
  double* T1 = F + (int64_t)J * J;
  double* T2 = T1 + (int64_t)J * n;
  const double* W = A.Wc + f.base;
  double* out = A.out + y * A.ldo + f.base;
  if (a > 0) rows_product<MODE>(S, f, r0, A, ws, Ls, Rs, red, Wr);
  if (MODE == RK_M) {
    // M_AN = W D^{-1}
    for (int e = tid; e < R * n; e += RT) {
      const int r = e & (R - 1), c = e >> (lrb + 3);
      if (r >= nr) continue;
      double s = 0.0;
      for (int q = 0; q < n; ++q) s = fma(Wr[r + q * R], W[q >= c ? csc_off(J, q, c) : csc_off(J, c, q)], s);
      out[csc_off(J, n + r0 + r, c)] = s;
    }
    return;
  }
  if (MODE == RK_IH2) {
    const double* D = A.Dd + f.d_off;
    double* Kr = Lr;
    for (int e = tid; e < R * n; e += RT) {
      const int r = e & (R - 1), c = e >> (lrb + 3);
      double s = 0.0;
      for (int q = 0; q < n; ++q) s = fma(Wr[r + q * R], D[q >= c ? q + (int64_t)c * n : c + (int64_t)q * n], s);
      Kr[r + c * R] = s;
    }
    __syncthreads();
    for (int e = tid; e < R * n; e += RT) {
      const int r = e & (R - 1), c = e >> (lrb + 3);
      if (r >= nr) continue;
      double s = 0.0;
      for (int q = 0; q < n; ++q)
        s = fma(W[csc_off(J, n + r0 + r, q)], out[q >= c ? csc_off(J, q, c) : csc_off(J, c, q)], s);
      const double k = Kr[r + c * R], p = fma(0.5, s, k);
      F[n + r0 + r + (int64_t)c * J] = p;
      out[csc_off(J, n + r0 + r, c)] = 2.0 * p - k;
    }
    return;
  }
  // RK_GRAD, RK_HDOWN, RK_IH1: the block's rows, then its share of the N x N block
  for (int e = tid; e < R * n; e += RT) {
    const int r = e & (R - 1), c = e >> (lrb + 3);
    double l = 0.0, w = 0.0;
    if (r < nr) {
      const int row = n + r0 + r;
      const int64_t o = csc_off(J, row, c);
      l = W[o];
      w = Wr[r + c * R];
      if (MODE == RK_GRAD) {
        out[o] = -w;
        if (A.g) A.g[f.base + o] = w;
        F[row + (int64_t)c * J] = -w;
      } else if (MODE == RK_HDOWN) {
        const double m = out[o], t = m - w;
        out[o] = t;
        F[row + (int64_t)c * J] = t;
        w = m + t;  // 2 Q = 2 M_AN - W
      } else {
        const double t = F[row + (int64_t)c * J];
        T1[row + (int64_t)c * J] = t + w;
        w = 2.0 * t + w;  // T_AN^T L + L^T M_AN = sym(L^T (2 T_AN + V' L))
      }
    }
    Wr[r + c * R] = w;
    Lr[r + c * R] = l;
  }
  __syncthreads();
  const int np = n * (n + 1) / 2;
  if (a > 0) {
    double* part = T2 + (int64_t)d.y * np;
    for (int e = tid; e < np; e += RT) {
      int i = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
      while (i * (i + 1) / 2 > e) --i;
      while ((i + 1) * (i + 2) / 2 <= e) ++i;
      const int j = e - i * (i + 1) / 2;
      double s = 0.0;
      if (MODE == RK_GRAD) {
        for (int r = 0; r < nr; ++r) s = fma(Wr[r + i * R], Lr[r + j * R], s);
      } else {
        for (int r = 0; r < nr; ++r) {
          s = fma(Wr[r + i * R], Lr[r + j * R], s);
          s = fma(Lr[r + i * R], Wr[r + j * R], s);
        }
        s *= 0.5;
      }
      __stcg(part + e, s);
    }
  }
  if (MODE == RK_IH1) return;  // kg_nn adds the shares
  int* ctr = reinterpret_cast<int*>(T2 + (int64_t)J * n - 1);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(ctr, 1) == f.nb - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid == 0) *ctr = 0;
  for (int e = tid; e < np; e += RT) {
    int i = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
    while (i * (i + 1) / 2 > e) --i;
    while ((i + 1) * (i + 2) / 2 <= e) ++i;
    const int j = e - i * (i + 1) / 2;
    double s = 0.0;
    if (a > 0)
      for (int b = 0; b < f.nb; ++b) s += __ldcg(T2 + (int64_t)b * np + e);
    const int64_t o = csc_off(J, i, j);
    double v;
    if (MODE == RK_GRAD) {
      v = W[o] + s;
      if (A.g) A.g[f.base + o] = -v;
    } else {
      v = out[o] - s;
    }
    out[o] = v;
    F[i + (int64_t)j * J] = v;
  }
}

// N x N products of 16 rows: (B K) B for symmetric B, K (n x n)
//   NN_M:  M_NN = D^{-1} K_NN D^{-1} (K_NN in F, output T)
//   NN_IH: K_NN = D M_NN D, M_NN = T_NN + the shares of RK_IH1 (T_NN in F, output Y)
enum { NN_M = 0, NN_IH = 1 };
template <int MODE>
__global__ void __launch_bounds__(RT) kg_nn(SymDev S, const int2* blocks, const double* Wc, const double* Dd,
                                           double* Out, int64_t ldo, double* ws, const uint8_t* act) {
  extern __shared__ double dyn[];
  const int2 d = blocks[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int64_t y = blockIdx.y;
  if (act && !act[y * S.nsn + f.k]) return;
  ws += y * S.f_total;
  const int n = f.n, J = f.J, tid = threadIdx.x, i0 = d.y * 16, ld = n | 1;
  double* Br = dyn;               // 16 x n: rows i0 .. of B
  double* X = Br + 16 * ld;       // 16 x n: B K
  double* Cs = X + 16 * ld;       // n x 32: columns of K, then of B
  const double* F = ws + f.f_off;
  const double* T2 = F + (int64_t)J * J + (int64_t)J * n;
  const double* W = Wc + f.base;
  const double* D = MODE == NN_IH ? Dd + f.d_off : nullptr;
  const int np = n * (n + 1) / 2, rows = min(16, n - i0);
  auto B = [&](int r, int c) {
    return MODE == NN_M ? W[r >= c ? csc_off(J, r, c) : csc_off(J, c, r)]
                        : D[r >= c ? r + (int64_t)c * n : c + (int64_t)r * n];
  };
  auto K = [&](int r, int c) {
    const int i = max(r, c), j = min(r, c);
    double v = F[i + (int64_t)j * J];
    if (MODE == NN_IH && f.a > 0) {
      double t = 0.0;
      const double* part = T2 + i * (i + 1) / 2 + j;
      for (int b = 0; b < f.nb; ++b) t += part[(int64_t)b * np];
      v += t;
    }
    return v;
  };
  for (int e = tid; e < 16 * n; e += RT) {
    const int q = e % n, r = e / n;
    Br[r * ld + q] = r < rows ? B(i0 + r, q) : 0.0;
  }
  // 16 x 32 outputs at a time, four per thread
  const int r = tid & 15, cq = tid >> 4;
  double* out = Out + y * ldo + f.base;
  for (int half = 0; half < 2; ++half) {
    const double* A = (half ? X : Br) + r * ld;
    for (int c0 = 0; c0 < (half ? i0 + rows : n); c0 += 32) {
      const int cn = min(32, n - c0);
      __syncthreads();
      for (int e = tid; e < n * 32; e += RT) {
        const int q = e % n, c = e / n;
        Cs[q * 33 + c] = c < cn ? (half ? B(q, c0 + c) : K(q, c0 + c)) : 0.0;
      }
      __syncthreads();
      double x[4] = {0.0, 0.0, 0.0, 0.0};
      for (int q = 0; q < n; ++q) {
        const double av = A[q];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = fma(av, Cs[q * 33 + cq + 8 * u], x[u]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + cq + 8 * u;
        if (c >= n) continue;
        if (half == 0) X[r * ld + c] = x[u];
        else if (r < rows && c <= i0 + r) out[csc_off(J, i0 + r, c)] = x[u];
      }
    }
  }
}

// ---------------------------------------------------------------------------
// V_k^{-1} of many fronts at once (inverse Hessian, §5.3): Cholesky of the
// matrix [V; I] by panels of 32 columns, which turns I into L^{-T}, and
// V^{-1} = L^{-T} L^{-1}.  L overwrites V in Rd, L^{-T} (upper triangular)
// grows in the front's workspace.  Panel p touches the rows of V below it and
// the first p + 1 row blocks of I, so every panel has about a rows of work.
// Fronts come in order of decreasing a: those that still have a panel p are
// the first ones of the list.  Two launches per panel: the row solve, and the
// trailing update, whose CTA on the next diagonal block factors it at once.
// A 17 x 20 x 13 grid (474 fronts with 64 < a <= 350, 0.9 G FP64 FMA): 9000
// launches of per-front sequences took 110 ms, these 22 take 5 ms.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void factor_diag(double (*T)[GB + 1], double* rinv, double (*col)[GB], const GJob& J, int p,
                                            double* R, int64_t* st) {
  // 256 threads call; the first four warps factor
  const int pb = min(GB, J.a - p * GB), tid = threadIdx.x;
  __syncthreads();
  if (tid < panel::PTH) panel::chol32(T, rinv, col, pb, tid, 1, st, CHD_ERR_NOT_PD, J.k, -1);
  __syncthreads();
  double* D = R + (int64_t)p * GB * (J.a + 1);
  const int r = tid & 31;
  for (int c = tid >> 5; c < pb; c += 8)
    if (r < pb && r >= c) D[r + (int64_t)c * J.a] = T[r][c];
}
// fronts of one block (a <= 32): everything in one CTA, V^{-1} to R
__global__ void __launch_bounds__(128) kv_small(SymDev S, const int32_t* list, const double* Vd, double* Rd,
                                               int64_t* st) {
  __shared__ double T[GB][GB + 1], X[GB][GB + 1], rinv[GB], col[3][GB];
  const int k = list[blockIdx.x], tid = threadIdx.x;
  const int n = (int)(S.sn_ptr[k + 1] - S.sn_ptr[k]), a = (int)(S.rows_ptr[k + 1] - S.rows_ptr[k]) - n;
  const double* V = Vd + S.v_off[k];
  double* R = Rd + S.v_off[k];
  for (int e = tid; e < GB * GB; e += 128) {
    const int i = e & 31, j = e >> 5;
    T[i][j] = i < a && j <= i ? V[i + (int64_t)j * a] : (i == j ? 1.0 : 0.0);
  }
  __syncthreads();
  panel::chol32(T, rinv, col, a, tid, 1, st, CHD_ERR_NOT_PD, k, -1);
  __syncthreads();
  const int row = tid >> 2, q = tid & 3;
  if ((tid & ~31) / 4 < a) {  // X = L^{-T}, rows of the identity
    double b[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) b[u] = row == q + 4 * u ? 1.0 : 0.0;
    panel::solve_row(b, T, rinv, a, tid & 31, 2 * (tid >> 5));
#pragma unroll
    for (int u = 0; u < 8; ++u) X[row][q + 4 * u] = b[u];
  }
  __syncthreads();
  for (int e = tid; e < a * GB; e += 128) {
    const int i = e & 31, j = e >> 5;
    if (i >= a || j > i) continue;
    double v = 0.0;
    for (int c = i; c < a; ++c) v = fma(X[i][c], X[j][c], v);
    R[i + (int64_t)j * a] = v;
  }
}
// V into R, I into X (upper block triangle), and the first diagonal block's factor
__global__ void __launch_bounds__(256) kv_init(SymDev S, const int2* tiles, const double* Vd, double* Rd, double* ws,
                                              int64_t* st) {
  __shared__ double T[GB][GB + 1], rinv[GB], col[3][GB];
  const int2 d = tiles[blockIdx.x];
  const GJob J = S.gj[d.x];
  const int i = d.y & 1023, j = (d.y >> 10) & 1023, tid = threadIdx.x, r = tid & 31, a = J.a;
  const double* V = Vd + J.v_off;
  double* R = Rd + J.v_off;
  double* X = ws + J.w_off;
  for (int c = tid >> 5; c < GB; c += 8) {
    const int row = i * GB + r, cc = j * GB + c;
    const bool in = row < a && cc < a && row >= cc;
    const double v = in ? V[row + (int64_t)cc * a] : 0.0;
    T[r][c] = in ? v : (i == j && r == c ? 1.0 : 0.0);
    if (in && (i > 0 || j > 0)) R[row + (int64_t)cc * a] = v;
    // block (j, i) of X: row block j, column block i
    if (j * GB + r < a && i * GB + c < a) X[(j * GB + r) + (int64_t)(i * GB + c) * a] = (i == j && r == c) ? 1.0 : 0.0;
  }
  if (i == 0 && j == 0) factor_diag(T, rinv, col, J, 0, R, st);
}
// rows of one block against panel p: B := B L_pp^{-T}
__global__ void __launch_bounds__(128) kv_solve(SymDev S, const int2* tiles, int p, double* Rd, double* ws) {
  __shared__ double Ls[GB][GB + 1], rinv[GB];
  const int2 d = tiles[blockIdx.x];
  const GJob J = S.gj[d.x];
  const int blk = d.y & 1023, tid = threadIdx.x, a = J.a, pb = min(GB, a - p * GB);
  const bool isx = d.y >> 20;
  double* R = Rd + J.v_off;
  double* M = isx ? ws + J.w_off : R;
  const double* D = R + (int64_t)p * GB * (a + 1);
  for (int e = tid; e < GB * GB; e += 128) {
    const int i = e & 31, c = e >> 5;
    Ls[i][c] = i < pb && c < pb && i >= c ? D[i + (int64_t)c * a] : 0.0;
  }
  // thread -> (row, lane of the group): rows along the lanes of a warp in
  // memory order would need a transpose; four lanes read four columns instead
  const int row = blk * GB + (tid >> 2), q = tid & 3;
  const bool ok = row < a;
  double* B = M + (ok ? row : 0) + (int64_t)p * GB * a;
  double b[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) b[u] = ok && q + 4 * u < pb ? B[(int64_t)(q + 4 * u) * a] : 0.0;
  __syncthreads();
  if (tid < GB) rinv[tid] = tid < pb ? 1.0 / Ls[tid][tid] : 0.0;
  __syncthreads();
  // the diagonal block of X starts as the identity: rows 8 w.. of warp w are
  // zero before column 8 w
  panel::solve_row(b, Ls, rinv, pb, tid & 31, isx && blk == p ? 2 * (tid >> 5) : 0);
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (ok && q + 4 * u < pb) B[(int64_t)(q + 4 * u) * a] = b[u];
}
// C -= A B^T over one 32 x 32 x 32 block product, 256 threads, 2 x 2 outputs
struct Acc2 {
  double v[2][2];
};
__device__ __forceinline__ void stage_block(double (*B)[GB + 1], const double* M, int64_t ld, int r0, int c0, int rmax,
                                           int cmax) {
  const int r = threadIdx.x & 31;
  for (int c = threadIdx.x >> 5; c < GB; c += 8)
    B[c][r] = r0 + r < rmax && c0 + c < cmax ? M[(r0 + r) + (int64_t)(c0 + c) * ld] : 0.0;
}
// FP64-bound, so halves of the tile that are zero or not wanted are left out:
// low: a diagonal tile, of which only the lower triangle is stored; tri: A is
// upper triangular, its rows 16.. start at k = 16.  (12000 fronts of a = 61:
// the product 2.36 -> 1.44 ms, the update 1.87 -> 1.56)
__device__ __forceinline__ void block_product(Acc2& s, const double (*A)[GB + 1], const double (*B)[GB + 1], int kn,
                                             bool low = false, bool tri = false) {
  const int tr = threadIdx.x & 15, tc = threadIdx.x >> 4;
  auto run = [&](int k0, int k1, auto lower, auto upper_rows) {
    for (int k = k0; k < k1; ++k) {
      const double x0 = A[k][tr], y0 = B[k][tc];
      s.v[0][0] = fma(x0, y0, s.v[0][0]);
      if constexpr (!lower.value) s.v[0][1] = fma(x0, B[k][tc + 16], s.v[0][1]);
      if constexpr (!upper_rows.value) {
        const double x1 = A[k][tr + 16];
        s.v[1][0] = fma(x1, y0, s.v[1][0]);
        s.v[1][1] = fma(x1, B[k][tc + 16], s.v[1][1]);
      }
    }
  };
  using yes = std::true_type;
  using no = std::false_type;
  const int kt = tri ? min(16, kn) : 0;
  if (low) {
    run(0, kt, yes{}, yes{});
    run(kt, kn, yes{}, no{});
  } else {
    run(0, kt, no{}, yes{});
    run(kt, kn, no{}, no{});
  }
}
// trailing update by panel p; the CTA on block (p + 1, p + 1) of V factors it
__global__ void __launch_bounds__(256) kv_update(SymDev S, const int2* tiles, int p, double* Rd, double* ws,
                                                int64_t* st) {
  __shared__ double A[GB][GB + 1], B[GB][GB + 1], rinv[GB], col[3][GB];
  const int2 d = tiles[blockIdx.x];
  const GJob J = S.gj[d.x];
  const int i = d.y & 1023, j = (d.y >> 10) & 1023, tid = threadIdx.x, a = J.a;
  const bool isx = d.y >> 20, diag = !isx && i == p + 1 && j == p + 1;
  double* R = Rd + J.v_off;
  double* M = isx ? ws + J.w_off : R;
  const int pe = min(a, (p + 1) * GB);
  stage_block(A, M, a, i * GB, p * GB, a, pe);
  const bool same = !isx && i == j;
  if (!same) stage_block(B, R, a, j * GB, p * GB, a, pe);
  __syncthreads();
  Acc2 s{};
  block_product(s, A, same ? A : B, pe - p * GB, same, isx && i == p);
  const int tr = tid & 15, tc = tid >> 4;
  if (diag) __syncthreads();  // A is reused for the block to factor
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int r = tr + 16 * u, c = tc + 16 * w, row = i * GB + r, cc = j * GB + c;
      const bool in = row < a && cc < a && (isx || row >= cc);
      double v = r == c ? 1.0 : 0.0;
      if (in) {
        double* o = M + row + (int64_t)cc * a;
        v = *o - s.v[u][w];
        if (!diag) *o = v;
      } else if (row < a && cc < a) {
        v = 0.0;
      }
      if (diag) A[r][c] = v;
    }
  if (diag) factor_diag(A, rinv, col, J, p + 1, R, st);
}
// V^{-1} = X X^T with X = L^{-T} upper triangular: lower tile (i, j)
__global__ void __launch_bounds__(256) kv_product(SymDev S, const int2* tiles, double* Rd, const double* ws) {
  __shared__ double A[GB][GB + 1], B[GB][GB + 1];
  const int2 d = tiles[blockIdx.x];
  const GJob J = S.gj[d.x];
  const int i = d.y & 1023, j = (d.y >> 10) & 1023, tid = threadIdx.x, a = J.a;
  const double* X = ws + J.w_off;
  Acc2 s{};
  for (int k0 = i * GB; k0 < a; k0 += GB) {
    // within the diagonal block of X only the upper triangle counts: the
    // entries below it are zero already (solved from the identity)
    stage_block(A, X, a, i * GB, k0, a, a);
    if (i != j) stage_block(B, X, a, j * GB, k0, a, a);
    __syncthreads();
    block_product(s, A, i == j ? A : B, min(GB, a - k0), i == j, k0 == i * GB);
    __syncthreads();
  }
  const int tr = tid & 15, tc = tid >> 4;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int row = i * GB + tr + 16 * u, cc = j * GB + tc + 16 * w;
      if (row < a && cc <= row) Rd[J.v_off + row + (int64_t)cc * a] = s.v[u][w];
    }
}

// ---------------------------------------------------------------------------
// factorisation (Algorithm 7.1).  A parent needs the update block only, so
// the sub-levels compute C, B and U; D_NN^{-1} and L_AN = B C^{-1} of all
// fronts follow at the end.
//   kg_factor: fronts of up to 32 columns, one launch per sub-level; a 32 x 32
//     tile of U per CTA, which assembles the N-part of its rows, factors F_NN
//     (every tile the same bits) and solves its 64 rows itself: about 9 us a
//     front whatever its size, against 2.4 ms of one CTA per front and level
//     of a 17 x 20 x 13 grid's planes.
//   kf_panel, kf_update: wider fronts, assembled first, in panels of 32
//     columns: each CTA factors the diagonal block and solves one block of
//     rows; then the trailing tiles.
// ---------------------------------------------------------------------------
constexpr int GF = kGroupFactor;
template <bool MANY>
__global__ void __launch_bounds__(256) kg_factor(SymDev S, const int2* tiles, const double* X, double* Lc, double* Dd,
                                                double* ws, int64_t* st) {
  __shared__ double t[GB][GB + 1], Ns[GB][GB + 1], Bs[2][GB][GB + 1], rinv[GB], col[3][GB];
  const int2 d = tiles[blockIdx.x];
  const GFront f = S.gf[d.x];
  if (f.n > GF) return;
  const int tm = d.y & 0xffff, tn = d.y >> 16, tid = threadIdx.x;
  const int r0 = tm * GB, c0 = tn * GB, n = f.n, J = f.J;
  const int nr = min(GB, f.a - r0), nc = min(GB, f.a - c0);
  const int bi = f.nbn + tm, bj = f.nbn + tn, fi = n + r0, fj = n + c0;
  const int side = tm == tn ? 0 : 1;
  const double* v = X + f.base;
  double* F = ws + f.f_off;
  double* L = Lc + f.base;
  for (int e = tid; e < GB * (GB + 1); e += 256) (&t[0][0])[e] = 0.0;
  for (int e = tid; e < GB * GB; e += 256) {
    const int i = e & 31, j = e >> 5;
    Ns[i][j] = i < n && j <= i ? v[csc_off(J, i, j)] : (i == j ? 1.0 : 0.0);
    for (int s = 0; s <= side; ++s) {
      const int q0 = s ? c0 : r0, cnt = s ? nc : nr;
      Bs[s][i][j] = i < cnt && j < n ? v[csc_off(J, n + q0 + i, j)] : 0.0;
    }
  }
  __syncthreads();
  if constexpr (MANY) {
    add_children(S, f, ws, nullptr, 0, 0, 0, 0, &Ns[0][0], GB + 1, GB);
    if (f.a > 0) {
      add_children(S, f, ws, nullptr, bi, fi, bj, fj, &t[0][0], GB + 1, GB);
      add_children(S, f, ws, nullptr, bi, fi, 0, 0, &Bs[0][0][0], GB + 1, GB);
      if (side) add_children(S, f, ws, nullptr, bj, fj, 0, 0, &Bs[1][0][0], GB + 1, GB);
    }
    __syncthreads();
  } else {
    for (int q = f.ch_beg; q < f.ch_end; ++q) {
      const GChild c = S.gch[q];
      add_child(S, c, ws, 0, 0, 0, 0, &Ns[0][0], GB + 1);
      if (f.a > 0) {
        add_child(S, c, ws, bi, fi, bj, fj, &t[0][0], GB + 1);
        add_child(S, c, ws, bi, fi, 0, 0, &Bs[0][0][0], GB + 1);
        if (side) add_child(S, c, ws, bj, fj, 0, 0, &Bs[1][0][0], GB + 1);
      }
      __syncthreads();
    }
  }
  const bool first = tm == 0 && tn == 0;
  if (first)
    for (int e = tid; e < n * GB; e += 256) {
      const int i = e & 31, j = e >> 5;
      if (i < n && j <= i) Dd[f.d_off + i + (int64_t)j * n] = Ns[i][j];
    }
  __syncthreads();
  if (tid < panel::PTH) panel::chol32(Ns, rinv, col, n, tid, 1, st, CHD_ERR_NOT_PD, f.k, S.sn_ptr[f.k]);
  __syncthreads();
  if (first)
    for (int e = tid; e < n * GB; e += 256) {
      const int i = e & 31, j = e >> 5;
      if (i < n && j <= i) L[csc_off(J, i, j)] = Ns[i][j];
    }
  if (f.a == 0) return;
  const int s = tid >> 7, row = (tid & 127) >> 2, q = tid & 3;
  if (s <= side) {
    double b[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) b[u] = Bs[s][row][q + 4 * u];
    panel::solve_row(b, Ns, rinv, n, tid & 31);
#pragma unroll
    for (int u = 0; u < 8; ++u) Bs[s][row][q + 4 * u] = b[u];
  }
  __syncthreads();
  const int tr = tid & 15, tc = tid >> 4;
  double acc[2][2] = {{0, 0}, {0, 0}};
  for (int j = 0; j < n; ++j)
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int w = 0; w < 2; ++w) acc[u][w] = fma(Bs[0][tr + 16 * u][j], Bs[side][tc + 16 * w][j], acc[u][w]);
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int r = tr + 16 * u, c = tc + 16 * w;
      if (r < nr && c < nc && r0 + r >= c0 + c) F[fi + r + (int64_t)(fj + c) * J] = t[r][c] - acc[u][w];
    }
  if (tn == 0)
    for (int e = tid; e < n * GB; e += 256) {
      const int r = e & 31, j = e >> 5;
      if (r < nr) L[csc_off(J, fi + r, j)] = Bs[0][r][j];
    }
}
// panel p of the wide fronts: (front, block) pairs; block p stores the factor
// of the diagonal block in Lc (F keeps the unfactored one, which the other
// CTAs read), blocks below it their solved rows in F and Lc
__global__ void __launch_bounds__(128) kf_panel(SymDev S, const int2* blocks, int p, double* Lc, double* ws,
                                               int64_t* st) {
  __shared__ double Ns[GB][GB + 1], rinv[GB], col[3][GB];
  const int2 d = blocks[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int blk = d.y, tid = threadIdx.x;
  if (p >= f.nbn || blk < p) return;
  int fp, pb, fr, nr;
  block_range(f, p, fp, pb);
  block_range(f, blk, fr, nr);
  const int J = f.J;
  double* F = ws + f.f_off;
  double* L = Lc + f.base;
  for (int e = tid; e < GB * GB; e += 128) {
    const int i = e & 31, j = e >> 5;
    Ns[i][j] = i < pb && j <= i ? F[(fp + i) + (int64_t)(fp + j) * J] : (i == j ? 1.0 : 0.0);
  }
  const int row = tid >> 2, q = tid & 3;
  const bool ok = blk > p && row < nr;
  double* B = F + fr + (ok ? row : 0) + (int64_t)fp * J;
  double b[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) b[u] = ok && q + 4 * u < pb ? B[(int64_t)(q + 4 * u) * J] : 0.0;
  __syncthreads();
  panel::chol32(Ns, rinv, col, pb, tid, 1, st, CHD_ERR_NOT_PD, f.k, S.sn_ptr[f.k] + fp);
  __syncthreads();
  if (blk == p) {
    for (int e = tid; e < GB * GB; e += 128) {
      const int i = e & 31, j = e >> 5;
      if (i < pb && j <= i) L[csc_off(J, fp + i, fp + j)] = Ns[i][j];
    }
    return;
  }
  panel::solve_row(b, Ns, rinv, pb, tid & 31);
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (ok && q + 4 * u < pb) {
      B[(int64_t)(q + 4 * u) * J] = b[u];
      L[csc_off(J, fr + row, fp + q + 4 * u)] = b[u];
    }
}
// trailing tiles of panel p: F_ij -= B_i B_j^T, blocks i >= j > p
__global__ void __launch_bounds__(256) kf_update(SymDev S, const int2* tiles, int p, double* ws) {
  __shared__ double A[GB][GB + 1], B[GB][GB + 1];
  const int2 d = tiles[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int bi = d.y & 0xffff, bj = d.y >> 16, tid = threadIdx.x, J = f.J;
  if (p >= f.nbn || bj <= p) return;
  int fp, pb, fi, ni, fj, nj;
  block_range(f, p, fp, pb);
  block_range(f, bi, fi, ni);
  block_range(f, bj, fj, nj);
  double* F = ws + f.f_off;
  stage_block(A, F, J, fi, fp, fi + ni, fp + pb);
  if (bi != bj) stage_block(B, F, J, fj, fp, fj + nj, fp + pb);
  __syncthreads();
  Acc2 s{};
  block_product(s, A, bi == bj ? A : B, pb, bi == bj);
  const int tr = tid & 15, tc = tid >> 4;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int r = tr + 16 * u, c = tc + 16 * w;
      if (r < ni && c < nj && fi + r >= fj + c) F[(fi + r) + (int64_t)(fj + c) * J] -= s.v[u][w];
    }
}
// Rows of L_AN = B C^{-1} (into Wc) and of C^{-T} (into T1), 32 rows per CTA:
// back substitution through the panels of C for the rows of A_k, forward
// substitution from the identity for the rows beyond them
__global__ void __launch_bounds__(128) kg_factor_rows(SymDev S, const int2* blocks, const double* Lc, double* Wc,
                                                     double* ws) {
  extern __shared__ double dyn[];
  __shared__ double Cs[GB][GB + 1], rinv[GB];
  const int2 d = blocks[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int n = f.n, J = f.J, tid = threadIdx.x, lane = tid & 31, ld = n + 1;
  const int nba = (f.a + GB - 1) / GB;
  const bool ident = d.y >= nba;
  const int blk = ident ? d.y - nba : d.y, r0 = blk * GB, cnt = min(GB, (ident ? n : f.a) - r0);
  const double* L = Lc + f.base;
  double* rows = dyn;  // 32 x n
  for (int e = tid; e < GB * n; e += 128) {
    const int r = e & 31, c = e >> 5;
    rows[r * ld + c] = ident ? (r0 + r == c ? 1.0 : 0.0) : (r < cnt ? L[csc_off(J, n + r0 + r, c)] : 0.0);
  }
  const int row = tid >> 2, q = tid & 3;
  auto stage = [&](int i0, int j0) {  // block (i0, j0) of C, lower part
    __syncthreads();
    for (int e = tid; e < GB * GB; e += 128) {
      const int i = e & 31, j = e >> 5;
      Cs[i][j] = i0 + i < n && j0 + j <= i0 + i ? L[csc_off(J, i0 + i, j0 + j)] : 0.0;
    }
    __syncthreads();
  };
  const int np = f.nbn;
  for (int s = 0; s < np; ++s) {
    const int p = ident ? s : np - 1 - s, p0 = p * GB, pb = min(GB, n - p0);
    if (ident && p < blk) continue;  // zeros left of the row's own block
    stage(p0, p0);
    if (tid < GB) rinv[tid] = tid < pb ? 1.0 / Cs[tid][tid] : 0.0;
    __syncthreads();
    double b[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) b[u] = q + 4 * u < pb ? rows[row * ld + p0 + q + 4 * u] : 0.0;
    if (ident) {
      panel::solve_row(b, Cs, rinv, pb, lane);
    } else {
      panel::solve_row_back(b, Cs, rinv, pb, lane);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (q + 4 * u < pb) rows[row * ld + p0 + q + 4 * u] = b[u];
    // the other panels' columns: b_o -= x_p C_po (back), x_p C_op^T (forward)
    for (int o = ident ? p + 1 : 0; o < (ident ? np : p); ++o) {
      const int o0 = o * GB, ob = min(GB, n - o0);
      stage(ident ? o0 : p0, ident ? p0 : o0);
      for (int u = 0; u < 8; ++u) {
        const int c = q + 4 * u;
        if (4 * u >= ob) break;
        if (c < ob) {
          double acc = 0.0;
          for (int k = 0; k < pb; ++k) acc = fma(rows[row * ld + p0 + k], ident ? Cs[c][k] : Cs[k][c], acc);
          rows[row * ld + o0 + c] -= acc;
        }
      }
    }
    __syncthreads();
  }
  __syncthreads();
  double* T1 = ws + f.f_off + (int64_t)J * J;
  for (int e = tid; e < GB * n; e += 128) {
    const int r = e & 31, c = e >> 5;
    if (r >= cnt) continue;
    if (ident) T1[r0 + r + (int64_t)c * J] = rows[r * ld + c];
    else Wc[f.base + csc_off(J, n + r0 + r, c)] = rows[r * ld + c];
  }
}
// D_NN^{-1} = C^{-T} C^{-1} (16 rows per CTA), and the front's log det
__global__ void __launch_bounds__(RT) kg_factor_nn(SymDev S, const int2* blocks, const double* Lc, double* Wc,
                                                  const double* ws, double* ldet) {
  const int2 d = blocks[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int n = f.n, J = f.J, tid = threadIdx.x, i0 = d.y * 16, rows = min(16, n - i0);
  const double* X = ws + f.f_off + (int64_t)J * J;
  for (int e = tid; e < 16 * (i0 + rows); e += RT) {
    const int i = i0 + (e & 15), j = e >> 4;
    if (i >= n || j > i) continue;
    double s = 0.0;
    for (int k = i; k < n; ++k) s = fma(X[i + (int64_t)k * J], X[j + (int64_t)k * J], s);
    Wc[f.base + csc_off(J, i, j)] = s;
  }
  if (d.y == 0 && tid < 32) {
    double s = 0.0;
    for (int i = tid; i < n; i += 32) s += 2.0 * log(Lc[f.base + csc_off(J, i, i)]);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tid == 0) ldet[f.k] = s;
  }
}

// ---------------------------------------------------------------------------
// Cholesky product (Algorithm 3.2): block pair (bi, bj) of the front =
// children's blocks + G G^T, G = [C; B] (Lc); N columns to the output, the
// A x A block to F for the parent.  Only the additions wait for the children,
// so the product G G^T comes first in each CTA.  17 x 20 x 13 grid: 23.1 ms
// (one CTA per front) before.
// ---------------------------------------------------------------------------
template <bool MANY>
__global__ void __launch_bounds__(256) kg_product(SymDev S, const int2* tiles, const double* Lc, double* Xo,
                                                 double* ws) {
  __shared__ double t[GB][GB + 1], A[GB][GB + 1], B[GB][GB + 1];
  const int2 d = tiles[blockIdx.x];
  const GFront f = S.gf[d.x];
  const int bi = d.y & 0xffff, bj = d.y >> 16, tid = threadIdx.x, n = f.n, J = f.J;
  int fi, ni, fj, nj;
  block_range(f, bi, fi, ni);
  block_range(f, bj, fj, nj);
  const double* L = Lc + f.base;
  Acc2 s{};
  const int kmax = min(n, fj + nj);  // G(c, k) = 0 for k > c
  const int r = tid & 31;
  for (int k0 = 0; k0 < kmax; k0 += GB) {
    const int kc = min(GB, kmax - k0);
    for (int k = tid >> 5; k < GB; k += 8) {
      const int kk = k0 + k;
      A[k][r] = k < kc && r < ni && fi + r >= kk ? L[csc_off(J, fi + r, kk)] : 0.0;
      if (bi != bj) B[k][r] = k < kc && r < nj && fj + r >= kk ? L[csc_off(J, fj + r, kk)] : 0.0;
    }
    __syncthreads();
    block_product(s, A, bi == bj ? A : B, kc, bi == bj);
    __syncthreads();
  }
  const int tr = tid & 15, tc = tid >> 4;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) t[tr + 16 * u][tc + 16 * w] = s.v[u][w];
  __syncthreads();
  if constexpr (MANY) {
    add_children(S, f, ws, nullptr, bi, fi, bj, fj, &t[0][0], GB + 1, GB);
  } else {
    for (int q = f.ch_beg; q < f.ch_end; ++q) {
      add_child(S, S.gch[q], ws, bi, fi, bj, fj, &t[0][0], GB + 1);
      __syncthreads();
    }
  }
  double* F = ws + f.f_off;
  if (r < ni)
    for (int c = tid >> 5; c < nj; c += 8) {
      const int row = fi + r, col = fj + c;
      if (row < col) continue;
      if (col < n) Xo[f.base + csc_off(J, row, col)] = t[r][c];
      else F[row + (int64_t)col * J] = t[r][c];
    }
}

// ---------------------------------------------------------------------------
// Completion (Algorithm 7.3) of all the tier's fronts at once: the S-front in
// the order (A_k, N_k) goes through a partial Cholesky factorisation of its A
// columns in panels of 32, which leaves R = chol(V_k), Z^T = (R^{-1} S_AN)^T
// in the N rows and P = S_NN - Z^T Z = D_NN^{-1} in the N block; then
// L_AN^T = -Z^T R^{-1} by back substitution, D_NN = P^{-1}, C = chol(D_NN) and
// B = L_AN C.  No front waits for another, so a panel step is one launch over
// every front that still has one (fronts come by decreasing a), as in the
// grouped inverse; one CTA per front took 4.0 ms on er5000 and left 40 dense
// fronts to 5000 launches, 6.7 ms on a 17 x 20 x 13 grid.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void comp_block(const GComp& f, int b, int& first, int& count) {
  if (b < f.nA) {
    first = b * GB;
    count = min(GB, f.a - first);
  } else {
    first = f.a + (b - f.nA) * GB;
    count = min(GB, f.J - first);
  }
}
__device__ __forceinline__ void comp_diag(double (*T)[GB + 1], double* rinv, double (*col)[GB], const GComp& f, int p,
                                          double* F, int64_t* st) {
  const int pb = min(GB, f.a - p * GB), tid = threadIdx.x;
  __syncthreads();
  if (tid < panel::PTH) panel::chol32(T, rinv, col, pb, tid, 1, st, CHD_ERR_NOT_COMPLETABLE, f.k, -1);
  __syncthreads();
  double* D = F + (int64_t)p * GB * (f.J + 1);
  const int r = tid & 31;
  for (int c = tid >> 5; c < pb; c += 8)
    if (r < pb && r >= c) D[r + (int64_t)c * f.J] = T[r][c];
}
__global__ void __launch_bounds__(256) kp_init(SymDev S, const int2* tiles, const double* Sin, double* Vd, double* ws,
                                              int64_t* st) {
  __shared__ double T[GB][GB + 1], rinv[GB], col[3][GB];
  const int2 d = tiles[blockIdx.x];
  const GComp f = S.gc[d.x];
  const int i = d.y & 1023, j = (d.y >> 10) & 1023, r = threadIdx.x & 31;
  int fi, ni, fj, nj;
  comp_block(f, i, fi, ni);
  comp_block(f, j, fj, nj);
  double* F = ws + f.f_off;
  const int32_t* A = S.rows + f.rows_off + f.n;
  for (int c = threadIdx.x >> 5; c < GB; c += 8) {
    const int row = fi + r, cc = fj + c;
    const bool in = r < ni && c < nj && row >= cc;
    double v = i == j && r == c ? 1.0 : 0.0;
    if (in) {
      if (cc >= f.a) v = Sin[f.base + csc_off(f.J, row - f.a, cc - f.a)];         // N x N
      else if (row >= f.a) v = Sin[f.base + csc_off(f.J, f.n + cc, row - f.a)];   // N x A
      else {
        v = Sin[csc_find(S, __ldg(A + row), __ldg(A + cc))];
        Vd[f.v_off + row + (int64_t)cc * f.a] = v;
      }
      if (i > 0 || j > 0 || f.a == 0) F[row + (int64_t)cc * f.J] = v;
    }
    T[r][c] = v;
  }
  if (i == 0 && j == 0 && f.a > 0) comp_diag(T, rinv, col, f, 0, F, st);
}
__global__ void __launch_bounds__(128) kp_solve(SymDev S, const int2* blocks, int p, double* ws) {
  __shared__ double Ls[GB][GB + 1], rinv[GB];
  const int2 d = blocks[blockIdx.x];
  const GComp f = S.gc[d.x];
  const int tid = threadIdx.x, J = f.J, pb = min(GB, f.a - p * GB);
  int fi, ni;
  comp_block(f, d.y & 1023, fi, ni);
  double* F = ws + f.f_off;
  const double* D = F + (int64_t)p * GB * (J + 1);
  for (int e = tid; e < GB * GB; e += 128) {
    const int i = e & 31, c = e >> 5;
    Ls[i][c] = i < pb && c < pb && i >= c ? D[i + (int64_t)c * J] : 0.0;
  }
  const int row = tid >> 2, q = tid & 3;
  const bool ok = row < ni;
  double* B = F + fi + (ok ? row : 0) + (int64_t)p * GB * J;
  double b[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) b[u] = ok && q + 4 * u < pb ? B[(int64_t)(q + 4 * u) * J] : 0.0;
  __syncthreads();
  if (tid < GB) rinv[tid] = tid < pb ? 1.0 / Ls[tid][tid] : 0.0;
  __syncthreads();
  if ((tid & ~31) / 4 >= ni) return;  // whole warps beyond the block's rows
  panel::solve_row(b, Ls, rinv, pb, tid & 31);
#pragma unroll
  for (int u = 0; u < 8; ++u)
    if (ok && q + 4 * u < pb) B[(int64_t)(q + 4 * u) * J] = b[u];
}
__global__ void __launch_bounds__(256) kp_update(SymDev S, const int2* tiles, int p, double* ws, int64_t* st) {
  __shared__ double A[GB][GB + 1], B[GB][GB + 1], rinv[GB], col[3][GB];
  const int2 d = tiles[blockIdx.x];
  const GComp f = S.gc[d.x];
  const int i = d.y & 1023, j = (d.y >> 10) & 1023, tid = threadIdx.x, J = f.J;
  const bool diag = i == p + 1 && j == p + 1 && p + 1 < f.nA;
  int fi, ni, fj, nj;
  comp_block(f, i, fi, ni);
  comp_block(f, j, fj, nj);
  double* F = ws + f.f_off;
  const int p0 = p * GB, pe = min(f.a, p0 + GB);
  stage_block(A, F, J, fi, p0, fi + ni, pe);
  if (i != j) stage_block(B, F, J, fj, p0, fj + nj, pe);
  __syncthreads();
  Acc2 s{};
  block_product(s, A, i == j ? A : B, pe - p0, i == j);
  if (diag) __syncthreads();  // A is reused for the block to factor
  const int tr = tid & 15, tc = tid >> 4;
#pragma unroll
  for (int u = 0; u < 2; ++u)
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      const int r = tr + 16 * u, c = tc + 16 * w;
      double v = r == c ? 1.0 : 0.0;
      if (r < ni && c < nj) {
        v = 0.0;
        if (fi + r >= fj + c) {
          double* o = F + (fi + r) + (int64_t)(fj + c) * J;
          v = *o - s.v[u][w];
          if (!diag) *o = v;
        }
      }
      if (diag) A[r][c] = v;
    }
  if (diag) comp_diag(A, rinv, col, f, p + 1, F, st);
}
// L_AN^T = -Z^T R^{-1}, eight rows (columns of N_k) per CTA, through all panels
constexpr int BR = 8;
__global__ void __launch_bounds__(128) kp_back(SymDev S, const int2* blocks, double* Wc, const double* ws) {
  extern __shared__ double rows[];  // BR x (a + 1)
  __shared__ double Ls[GB][GB + 1], rinv[GB];
  const int2 d = blocks[blockIdx.x];
  const GComp f = S.gc[d.x];
  const int tid = threadIdx.x, lane = tid & 31, J = f.J, a = f.a, ld = a + 1;
  const int r0 = d.y * BR, nr = min(BR, f.n - r0);
  const double* F = ws + f.f_off;
  for (int c = tid / BR; c < a; c += 128 / BR) {
    const int r = tid & (BR - 1);
    if (r < nr) rows[r * ld + c] = -F[a + r0 + r + (int64_t)c * J];
  }
  for (int p = f.nA - 1; p >= 0; --p) {
    const int p0 = p * GB, pb = min(GB, a - p0);
    __syncthreads();
    for (int e = tid; e < GB * GB; e += 128) {
      const int i = e & 31, c = e >> 5;
      Ls[i][c] = i < pb && c <= i ? F[(p0 + i) + (int64_t)(p0 + c) * J] : 0.0;
    }
    __syncthreads();
    if (tid < 32) {
      rinv[lane] = lane < pb ? 1.0 / Ls[lane][lane] : 0.0;
      __syncwarp();
      const int row = lane >> 2, q = lane & 3;
      double b[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) b[u] = row < nr && q + 4 * u < pb ? rows[row * ld + p0 + q + 4 * u] : 0.0;
      panel::solve_row_back(b, Ls, rinv, pb, lane);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (row < nr && q + 4 * u < pb) rows[row * ld + p0 + q + 4 * u] = b[u];
    }
    __syncthreads();
    // the columns left of the panel: b_c -= x_p R_pc
    for (int e = tid; e < nr * p0; e += 128) {
      const int r = e % nr, c = e / nr;
      const double* R = F + p0 + (int64_t)c * J;
      double acc = 0.0;
      for (int k = 0; k < pb; ++k) acc = fma(rows[r * ld + p0 + k], __ldg(R + k), acc);
      rows[r * ld + c] -= acc;
    }
  }
  __syncthreads();
  for (int r = 0; r < nr; ++r)
    for (int c = tid; c < a; c += 128) Wc[f.base + csc_off(J, f.n + c, r0 + r)] = rows[r * ld + c];
}
// fronts of up to 32 columns: P to Wc, D_NN = P^{-1}, C = chol(D_NN), log det
__global__ void __launch_bounds__(128) kp_nn(SymDev S, const int32_t* list, double* Lc, double* Wc, double* Dd,
                                            const double* ws, double* ldet, int64_t* st) {
  __shared__ double P[GB][GB + 1], X[GB][GB + 1], rinv[GB], col[3][GB];
  const GComp f = S.gc[list[blockIdx.x]];
  const int tid = threadIdx.x, n = f.n, a = f.a, J = f.J;
  const double* F = ws + f.f_off;
  for (int e = tid; e < GB * GB; e += 128) {
    const int i = e & 31, j = e >> 5;
    double v = i == j ? 1.0 : 0.0;
    if (i < n && j <= i) {
      v = F[(a + i) + (int64_t)(a + j) * J];
      Wc[f.base + csc_off(J, i, j)] = v;
    }
    P[i][j] = v;
  }
  __syncthreads();
  panel::chol32(P, rinv, col, n, tid, 1, st, CHD_ERR_NOT_COMPLETABLE, f.k, S.sn_ptr[f.k]);
  __syncthreads();
  {  // X = Q^{-T} (rows of the identity)
    const int row = tid >> 2, q = tid & 3;
    double b[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) b[u] = row == q + 4 * u ? 1.0 : 0.0;
    panel::solve_row(b, P, rinv, n, tid & 31);
#pragma unroll
    for (int u = 0; u < 8; ++u) X[row][q + 4 * u] = b[u];
  }
  __syncthreads();
  for (int e = tid; e < GB * GB; e += 128) {
    const int i = e & 31, j = e >> 5;
    double v = i == j ? 1.0 : 0.0;
    if (i < n && j <= i) {
      v = 0.0;
      for (int k = i; k < n; ++k) v = fma(X[i][k], X[j][k], v);
      Dd[f.d_off + i + (int64_t)j * n] = v;
    } else if (j > i) {
      v = 0.0;
    }
    P[i][j] = v;
  }
  __syncthreads();
  panel::chol32(P, rinv, col, n, tid, 1, st, CHD_ERR_NOT_COMPLETABLE, f.k, S.sn_ptr[f.k]);
  __syncthreads();
  for (int e = tid; e < GB * GB; e += 128) {
    const int i = e & 31, j = e >> 5;
    if (i < n && j <= i) Lc[f.base + csc_off(J, i, j)] = P[i][j];
  }
  if (tid < 32) {
    double s = tid < n ? 2.0 * log(P[tid][tid]) : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (tid == 0) ldet[f.k] = s;
  }
}
// B = L_AN C, 32 rows per CTA
__global__ void __launch_bounds__(128) kp_b(SymDev S, const int2* blocks, double* Lc, const double* Wc) {
  const int2 d = blocks[blockIdx.x];
  const GComp f = S.gc[d.x];
  const int n = f.n, J = f.J, r0 = d.y * GB, nr = min(GB, f.a - r0);
  const int r = threadIdx.x & 31;
  if (r >= nr) return;
  const int row = n + r0 + r;
  for (int c = threadIdx.x >> 5; c < n; c += 4) {
    double s = 0.0;
    for (int k = c; k < n; ++k) s = fma(Wc[f.base + csc_off(J, row, k)], Lc[f.base + csc_off(J, k, c)], s);
    Lc[f.base + csc_off(J, row, c)] = s;
  }
}

}  // namespace grp
}  // namespace chd

namespace chd_launch {
using namespace chd;
using namespace chd::grp;

namespace {
size_t rows_smem(int rn) { return (size_t)(KC * CBL + RT * CB + 2 * rn) * 8; }
size_t nn_smem(int n) { return (size_t)(32 * (n | 1) + 33 * n) * 8; }
template <class K>
void allow_smem(K kernel) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGroupSmem);
}
// the kernels' shared-memory limit, once per device
void init() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  const uint64_t bit = uint64_t(1) << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return;
  allow_smem(kg_rows<RK_GRAD>);
  allow_smem(kg_rows<RK_HDOWN>);
  allow_smem(kg_rows<RK_M>);
  allow_smem(kg_rows<RK_IH1>);
  allow_smem(kg_rows<RK_IH2>);
  allow_smem(kg_nn<NN_M>);
  allow_smem(kg_nn<NN_IH>);
  allow_smem(kg_factor_rows);
  done.fetch_or(bit, std::memory_order_release);
}
}  // namespace

// gradient and Hessian top-down step of sub-level q
void group_zero(const chd_symbolic* s, cudaStream_t st, int m, double* ws) {
  const int nf = (int)s->gf.size();
  if (nf == 0) return;
  kg_zero<<<dim3((nf + 255) / 256, m), 256, 0, st>>>(s->dev, 0, nf, ws);
  count_launch();
}
void group_gradient(const chd_symbolic* s, cudaStream_t st, int q, const double* Wc, double* Sc, double* g, double* Vd,
                    double* ws) {
  init();
  const int b0 = s->gs_row[q], nb = s->gs_row[q + 1] - b0;
  if (nb == 0) return;
  RowArgs A{Wc, nullptr, nullptr, Sc, 0, g, Vd, nullptr};
  kg_rows<RK_GRAD><<<nb, RT, rows_smem(s->gs_rn[q]), st>>>(s->dev, s->dev.gt_row + b0, A, ws);
  count_launch();
}
void group_hess_down(const chd_symbolic* s, cudaStream_t st, int q, int m, const double* Wc, double* T, int64_t ldt,
                     double* ws) {
  init();
  const int b0 = s->gs_row[q], nb = s->gs_row[q + 1] - b0;
  if (nb == 0) return;
  RowArgs A{Wc, nullptr, nullptr, T, ldt, nullptr, nullptr, nullptr};
  kg_rows<RK_HDOWN><<<dim3(nb, m), RT, rows_smem(s->gs_rn[q]), st>>>(s->dev, s->dev.gt_row + b0, A, ws);
  count_launch();
}
void group_hess_up(const chd_symbolic* s, cudaStream_t st, int q, int m, const double* Wc, const double* Y,
                   int64_t ldy, double* ws, const uint8_t* act) {
  const int a0 = s->gs_asm[q], na = s->gs_asm[q + 1] - a0;
  if (na > 0) {
    const auto assemble = s->gs_many[q] ? kg_assemble<ASM_UP, true> : kg_assemble<ASM_UP, false>;
    assemble<<<dim3(na, m), 256, 0, st>>>(s->dev, s->dev.gt_asm + a0, Y, ldy, ws, act, nullptr);
    count_launch();
  }
  const int p0 = s->gs_p[q], np = s->gs_p[q + 1] - p0;
  if (np > 0) {
    kg_p<<<dim3(np, m), 256, 0, st>>>(s->dev, s->dev.gt_p + p0, Wc, ws, act);
    count_launch();
  }
  const int u0 = s->gs_up[q], nu = s->gs_up[q + 1] - u0;
  if (nu > 0) {
    const auto up = s->gs_many[q] ? kg_up<UP_HESS, true> : kg_up<UP_HESS, false>;
    up<<<dim3(nu, m), 256, 0, st>>>(s->dev, s->dev.gt_up + u0, Wc, Y, ldy, nullptr, ws, act, nullptr, nu);
    count_launch();
  }
}
// step 2 of Algorithm 5.1 over all fronts: M_NN, M_AN into T.  Where no front has
// ancestors (independent dense matrices in one object) there is no M_AN.
void group_hess_m(const chd_symbolic* s, cudaStream_t st, int m, const double* Wc, const double* Vd, double* T,
                  int64_t ldt, double* ws, const uint8_t* act) {
  init();
  const int nn = (int)s->gt_nn.size() / 2, nb = (int)s->gt_row.size() / 2;
  if (nn > 0) {
    kg_nn<NN_M><<<dim3(nn, m), RT, nn_smem(s->g_nmax), st>>>(s->dev, s->dev.gt_nn, Wc, nullptr, T, ldt, ws, act);
    count_launch();
  }
  if (s->g_amax > 0) {
    RowArgs A{Wc, Vd, nullptr, T, ldt, nullptr, nullptr, act};
    kg_rows<RK_M><<<dim3(nb, m), RT, rows_smem(s->g_rnmax), st>>>(s->dev, s->dev.gt_row, A, ws);
    count_launch();
  }
}
// inverse Hessian: V' and T_k of sub-level q into the fronts (top-down)
void group_ihess_gather(const chd_symbolic* s, cudaStream_t st, int q, int m, const double* T, int64_t ldt,
                        double* ws) {
  const int t0 = s->gs_gat[q], nt = s->gs_gat[q + 1] - t0;
  if (nt == 0) return;
  kg_assemble<ASM_GATHER, false><<<dim3(nt, m), 256, 0, st>>>(s->dev, s->dev.gt_gat + t0, T, ldt, ws, nullptr, nullptr);
  count_launch();
}
// steps 1 and 2 of Algorithm 5.2 over all fronts (K_NN only where none has
// ancestors: 300 blocks of 30 columns, eight right-hand sides, 338 us with the
// empty row products, 271 without)
void group_ihess_k(const chd_symbolic* s, cudaStream_t st, int m, const double* Wc, const double* Dd, const double* Rd,
                   double* Y, int64_t ldy, double* ws) {
  init();
  const int nn = (int)s->gt_nn.size() / 2, nb = (int)s->gt_row.size() / 2;
  if (nb == 0) return;
  const bool rows = s->g_amax > 0;
  RowArgs A{Wc, nullptr, nullptr, Y, ldy, nullptr, nullptr, nullptr};
  if (rows) {
    kg_rows<RK_IH1><<<dim3(nb, m), RT, rows_smem(s->g_rnmax), st>>>(s->dev, s->dev.gt_row, A, ws);
    count_launch();
  }
  kg_nn<NN_IH><<<dim3(nn, m), RT, nn_smem(s->g_nmax), st>>>(s->dev, s->dev.gt_nn, Wc, Dd, Y, ldy, ws, nullptr);
  count_launch();
  if (!rows) return;
  A.mat = Rd;
  A.Dd = Dd;
  kg_rows<RK_IH2><<<dim3(nb, m), RT, rows_smem(s->g_rnmax), st>>>(s->dev, s->dev.gt_row, A, ws);
  count_launch();
}
void group_ihess_up(const chd_symbolic* s, cudaStream_t st, int q, int m, const double* Wc, double* Y, int64_t ldy,
                    double* ws) {
  const int u0 = s->gs_up[q], nu = s->gs_up[q + 1] - u0;
  const int o0 = s->gs_out[q], no = s->gs_out[q + 1] - o0;
  if (nu == 0) return;
  const auto up = s->gs_many[q] ? kg_up<UP_IHESS, true> : kg_up<UP_IHESS, false>;
  up<<<dim3(nu + no, m), 256, 0, st>>>(s->dev, s->dev.gt_up + u0, Wc, nullptr, ldy, Y, ws, nullptr, s->dev.gt_out + o0,
                                       nu);
  count_launch();
}
// V_k^{-1} of the fronts of the grouped inverse (gj), into Rd
void group_inv_v(const chd_symbolic* s, cudaStream_t st, const double* Vd, double* Rd, double* ws, int64_t* status) {
  if (!s->gv_small.empty()) {
    kv_small<<<(unsigned)s->gv_small.size(), 128, 0, st>>>(s->dev, s->dev.gv_small, Vd, Rd, status);
    count_launch();
  }
  if (s->gj.empty()) return;
  const int nt = (int)s->gv_all.size() / 2;
  kv_init<<<nt, 256, 0, st>>>(s->dev, s->dev.gv_all, Vd, Rd, ws, status);
  count_launch();
  const int np = (int)s->gv_sol_ptr.size() - 1;
  for (int p = 0; p < np; ++p) {
    const int s0 = s->gv_sol_ptr[p], s1 = s->gv_sol_ptr[p + 1];
    kv_solve<<<s1 - s0, 128, 0, st>>>(s->dev, s->dev.gv_sol + s0, p, Rd, ws);
    count_launch();
    const int u0 = s->gv_upd_ptr[p], u1 = s->gv_upd_ptr[p + 1];
    if (u1 > u0) {
      kv_update<<<u1 - u0, 256, 0, st>>>(s->dev, s->dev.gv_upd + u0, p, Rd, ws, status);
      count_launch();
    }
  }
  kv_product<<<nt, 256, 0, st>>>(s->dev, s->dev.gv_all, Rd, ws);
  count_launch();
}
// factor: C, B, U of sub-level q
void group_factor(const chd_symbolic* s, cudaStream_t st, int q, const double* X, double* Lc, double* Dd, double* ws,
                  int64_t* status) {
  const int a0 = s->gs_asmf[q], na = s->gs_asmf[q + 1] - a0;
  if (na > 0) {
    const auto assemble = s->gs_many[q] ? kg_assemble<ASM_FACTOR, true> : kg_assemble<ASM_FACTOR, false>;
    assemble<<<na, 256, 0, st>>>(s->dev, s->dev.gt_asmf + a0, X, 0, ws, nullptr, Dd);
    count_launch();
    const int b0 = s->gs_wb[q], nb = s->gs_wb[q + 1] - b0;
    for (int p = 0; p < s->gs_np[q]; ++p) {
      kf_panel<<<nb, 128, 0, st>>>(s->dev, s->dev.gt_wb + b0, p, Lc, ws, status);
      count_launch();
      kf_update<<<na, 256, 0, st>>>(s->dev, s->dev.gt_asmf + a0, p, ws);
      count_launch();
    }
  }
  const int u0 = s->gs_up[q], nu = s->gs_up[q + 1] - u0;
  if (nu > 0 && s->gs_thin[q]) {
    const auto factor = s->gs_many[q] ? kg_factor<true> : kg_factor<false>;
    factor<<<nu, 256, 0, st>>>(s->dev, s->dev.gt_up + u0, X, Lc, Dd, ws, status);
    count_launch();
  }
}
// D_NN^{-1}, L_AN and the log dets of all fronts
void group_factor_post(const chd_symbolic* s, cudaStream_t st, const double* Lc, double* Wc, double* ws,
                       double* ldet) {
  if (s->gf.empty()) return;
  init();
  const int nr = (int)s->gt_fr.size() / 2, nn = (int)s->gt_nn.size() / 2;
  kg_factor_rows<<<nr, 128, (size_t)GB * (s->g_nmax + 1) * 8, st>>>(s->dev, s->dev.gt_fr, Lc, Wc, ws);
  count_launch();
  kg_factor_nn<<<nn, RT, 0, st>>>(s->dev, s->dev.gt_nn, Lc, Wc, ws, ldet);
  count_launch();
}
// Cholesky product of sub-level q
void group_product(const chd_symbolic* s, cudaStream_t st, int q, const double* Lc, double* X, double* ws) {
  const int t0 = s->gs_gat[q], nt = s->gs_gat[q + 1] - t0;
  if (nt == 0) return;
  const auto product = s->gs_many[q] ? kg_product<true> : kg_product<false>;
  product<<<nt, 256, 0, st>>>(s->dev, s->dev.gt_gat + t0, Lc, X, ws);
  count_launch();
}
// completion of the tier's fronts up to L_AN, and of those of at most 32
// columns to the end
void group_complete(const chd_symbolic* s, cudaStream_t st, const double* Sin, double* Lc, double* Wc, double* Dd,
                    double* Vd, double* ws, double* ldet, int64_t* status) {
  if (s->gc.empty()) return;
  kp_init<<<(unsigned)(s->gc_all.size() / 2), 256, 0, st>>>(s->dev, s->dev.gc_all, Sin, Vd, ws, status);
  count_launch();
  for (size_t p = 0; p + 1 < s->gc_sol_ptr.size(); ++p) {
    const int s0 = s->gc_sol_ptr[p], s1 = s->gc_sol_ptr[p + 1];
    if (s1 > s0) {
      kp_solve<<<s1 - s0, 128, 0, st>>>(s->dev, s->dev.gc_sol + s0, (int)p, ws);
      count_launch();
    }
    const int u0 = s->gc_upd_ptr[p], u1 = s->gc_upd_ptr[p + 1];
    if (u1 > u0) {
      kp_update<<<u1 - u0, 256, 0, st>>>(s->dev, s->dev.gc_upd + u0, (int)p, ws, status);
      count_launch();
    }
  }
  if (!s->gc_back.empty()) {
    kp_back<<<(unsigned)(s->gc_back.size() / 2), 128, (size_t)BR * (s->gc_amax + 1) * 8, st>>>(
        s->dev, s->dev.gc_back, Wc, ws);
    count_launch();
  }
  if (!s->gc_thin.empty()) {
    kp_nn<<<(unsigned)s->gc_thin.size(), 128, 0, st>>>(s->dev, s->dev.gc_thin, Lc, Wc, Dd, ws, ldet, status);
    count_launch();
  }
  if (!s->gc_b.empty()) {
    kp_b<<<(unsigned)(s->gc_b.size() / 2), 128, 0, st>>>(s->dev, s->dev.gc_b, Lc, Wc);
    count_launch();
  }
}
}  // namespace chd_launch
