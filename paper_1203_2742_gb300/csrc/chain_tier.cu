// Chain tier: runs of one-column fronts whose rows are contiguous and whose
// ancestor count a is the same along the run (the elimination chains of band
// patterns in natural order).
//
// Andersen, Dahl, Vandenberghe, "Logarithmic barriers for sparse matrix
// cones": for one-column fronts the supernodal Algorithms 7.1 and 7.2 and the
// block forms of Algorithm 5.1 reduce to the scalar recursions of Algorithms
// 3.1, 4.1 and 5.1.  Along such a run, front j has rows j .. j+a, its child
// is front j-1, and the child's update matrix (bottom-up) or the parent's
// front (top-down) covers rows j+1 .. j+a-1 of it.  So the a x a block that
// passes from front to front is a window that slides by one row per column.
// The run hands over to the rest of the tree through the workspace fronts
// exactly like the other tiers: its top front writes its update block
// (bottom-up) or reads the parent's front (top-down) there.
//
// What bounds it.  A GB300 SM retires one FP64 warp instruction per 19
// clocks, whatever the number of active lanes, and one warp at most one per
// 64 clocks (dependent or not); a reciprocal is 350 clocks, a barrier of 256
// threads 29.  So the cost of a column is the number of FP64 warp
// instructions that must run one column after another, and the design keeps
// only those in the serial kernels:
//   * what the next column does not need runs afterwards, over all columns
//     in parallel: the Cholesky scaling and log det of the factor, the
//     stored V_j of the gradient, M_A = V K_A / D of the Hessian;
//   * both passes of the inverse Hessian and the Cholesky product have no
//     recursion along the run at all (the windows are parts of the input, and
//     the update blocks only add up), so they run over all columns at once;
//   * the serial kernels hold the window in registers, one copy of every
//     entry (bottom-up) or whole rows (top-down), and address it modulo its
//     size, so nothing moves as it slides.
// Measured (band n = 12000, half-bandwidth 61, one matrix; before: window in
// shared memory, both triangles updated, log and sqrt in the chain): factor
// 49.4 -> 9.4 ms, gradient 53.0 -> 1.8 ms (in segments: transfer matrices 0.28,
// scan 0.80, segments 0.73), both passes of the inverse Hessian with two
// right-hand sides 112.6 -> 0.95 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "chd_internal.h"
#include "front_views.cuh"

namespace chd_launch {
void count_launch();
}

namespace chd {
namespace chain {

constexpr int AMAX = 64;    // largest a
constexpr int WP = 72;      // row of a window vector in shared memory
constexpr int RING = 8;     // columns of inputs kept in shared memory
constexpr int AHEAD = 6;    // columns loaded ahead of the one in work

// run of task t: its first front's record, the run length and a
struct Run {
  int L, a;
  int k0;                         // first supernode (the others follow)
  int64_t base0, col0, d0, v0, vstride, f0, fstride;
};
// ... from the record of its i-th front
__device__ __forceinline__ Run run_with(const WMeta& w, int i, int L) {
  Run r;
  r.L = L;
  r.a = w.J - 1;
  // per-front offsets of one-column fronts (the symbolic phase rounds each
  // block up to a multiple of four doubles)
  r.vstride = ((int64_t)r.a * r.a + 3) & ~int64_t(3);
  const int64_t J = r.a + 1;
  r.fstride = (J * J + 2 * J + 3) & ~int64_t(3);
  r.k0 = w.k - i;
  r.base0 = w.base - i * J;
  r.col0 = w.col0 - i;
  r.d0 = w.d_off - 4 * (int64_t)i;
  r.v0 = w.v_off - i * r.vstride;
  r.f0 = w.f_off - i * r.fstride;
  return r;
}
__device__ __forceinline__ Run run_of(const SymDev& S, int t) {
  const int q0 = S.task_ptr[t], q1 = S.task_ptr[t + 1];
  return run_with(S.tmeta[q0], 0, q1 - q0);
}
// Kernels over all columns of the launch's runs.  A grid of runs x longest run is
// empty nearly everywhere when one run is long and many are short (30000 runs of ten
// columns beside one of 1275: 24.6 ms for a gradient, 1.2 without the empty
// CTAs), so such runs' columns are taken one after another over all runs (LIST),
// each through its own record.  An empty CTA costs about 0.55 ns, the record,
// which neighbours in a run do not share, 0.4: the grid while it adds less than three
// quarters of the columns.
struct Columns {
  int task0;
  int q0, n;  // LIST: task positions q0 .. q0 + n - 1
};
// The run of the CTA's columns (its sub-th, `per` of them a CTA); they are i, i + step,
// .. while below R.L
template <bool LIST>
__device__ __forceinline__ Run run_of_columns(const SymDev& S, const Columns& c, int per, int sub, int& i, int& step) {
  if (!LIST) {
    i = blockIdx.y * per + sub;
    step = gridDim.y * per;
    return run_of(S, c.task0 + blockIdx.x);
  }
  const int q = blockIdx.x * per + sub;
  step = 1 << 30;
  if (q >= c.n) {
    Run none{};
    i = 0;
    return none;
  }
  const WMeta w = S.tmeta[c.q0 + q];
  i = w.place;
  return run_with(w, i, S.task_ptr[w.task + 1] - (c.q0 + q - i));
}

__device__ __forceinline__ void cp_async8(double* dst, const double* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}
// barrier of the first `n` threads of the CTA (the rest has returned)
__device__ __forceinline__ void bar(int n) { asm volatile("bar.sync 1, %0;\n" ::"r"(n) : "memory"); }

// ---------------------------------------------------------------------------
// bottom-up serial kernels (factor, Hessian step 1)
//
// The window covers the a + 1 rows i .. i+a while column i is in work; row
// rho lives in slot rho mod (a + 1), so the row that leaves (i) and the row
// that enters (i + 1 + a) share a slot.  Every unordered pair of slots is one
// entry, held in a register of one update thread for the whole run.  Per
// column, after one barrier:
//   warp 0 finishes column i+1: its window entries (published one column
//     earlier by their owners, with the updates through column i-1), its
//     input values and the update by column i; then the pivot, and the two
//     vectors the next update needs, into the other of two buffers;
//   the other warps update their pairs by column i and publish column i+2.
// So the pivot's latency (about 700 clocks) runs beside the update of
// the window (a = 61: 61 FP64 warp instructions, 1160 clocks; twice that in
// the Hessian).  Inputs arrive by cp.async, AHEAD columns early.
// ---------------------------------------------------------------------------
struct UpSmem {
  double ring[2][RING][WP];
  double f[2][WP], g[2][WP], uc[2][WP];
};
enum { UP_FACTOR = 0, UP_HESS = 1 };
struct UpArgs {
  const double* src;  // X or Y, the run's first column
  const double* wc;   // UP_HESS: Wc; the run's first column
  double* o0;         // Lc (raw column: F_11, F_21) or T (h_0, K_A)
  double* o1;         // UP_FACTOR: Wc
  double* dd;         // UP_FACTOR: Dd of the first column
  int64_t* st;
};
// Columns i0 .. L - 1 of the run.  in: the window before column i0 (a x a,
// lower, ld a) or null for zeros; outs: whether the columns' outputs are
// stored; the window after column L - 1 goes to G[p + q ldg], p >= q (or
// nowhere, G null).
struct Span {
  int i0, L;
  const double* in;
  bool outs;
  double* G;
  int64_t ldg;
};
template <int NT, int PP, int MODE>
__device__ void up_run(const Run& R, const Span& sp_, const UpArgs& A, UpSmem& sm) {
  constexpr int EL = NT <= 32 ? 1 : NT <= 96 ? 1 : 3;  // slots per lane of warp 0
  const int a = R.a, W = a + 1, tid = threadIdx.x, L = sp_.L, i0 = sp_.i0;
  const bool outs = sp_.outs;
  if (tid >= NT + 32) return;
  for (int e = tid; e < 2 * WP; e += NT + 32) (&sm.uc[0][0])[e] = 0.0;
  bar(NT + 32);
  if (tid < 32) {
    // ---- warp 0: inputs, pivots, outputs ----
    const int lane = tid;
    // slots of the column being loaded and of the column being finished
    int sload = i0 % W, scol = i0 % W;
    auto prefetch = [&](int c) {
      if (c < L) {
        const int s0 = sload;
        sload = sload + 1 == W ? 0 : sload + 1;
        for (int p = lane; p <= a; p += 32) {
          int s = s0 + p;
          if (s >= W) s -= W;
          cp_async8(&sm.ring[0][c % RING][s], A.src + (int64_t)c * W + p);
          if (MODE == UP_HESS) cp_async8(&sm.ring[1][c % RING][s], A.wc + (int64_t)c * W + p);
        }
      }
      cp_async_commit();
    };
    auto column = [&](int c) {
      const int s0 = scol, sp = s0 == 0 ? W - 1 : s0 - 1, cur = c & 1, prv = cur ^ 1;
      scol = scol + 1 == W ? 0 : scol + 1;
      double val[EL], l[EL];
      const double gs = c > i0 ? sm.g[prv][s0] : 0.0, fs = c > i0 ? sm.f[prv][s0] : 0.0;
#pragma unroll
      for (int e = 0; e < EL; ++e) {
        const int o = lane + 32 * e;
        val[e] = 0.0;
        l[e] = 0.0;
        if (o < W) {
          val[e] = sm.ring[0][c % RING][o];
          if (MODE == UP_HESS) l[e] = sm.ring[1][c % RING][o];
          if (o != sp) {  // slot sp: the row that enters, untouched so far
            val[e] += sm.uc[cur][o];
            if (c > i0) {
              val[e] = fma(-sm.f[prv][o], gs, val[e]);
              if (MODE == UP_HESS) val[e] = fma(-sm.g[prv][o], fs, val[e]);
            }
          }
        }
      }
      double d = val[0];
#pragma unroll
      for (int e = 1; e < EL; ++e)
        if (s0 / 32 == e) d = val[e];
      d = __shfl_sync(0xffffffffu, d, s0 & 31);
      if (MODE == UP_FACTOR) {
        if (!(d > 0.0)) {
          if (lane == 0) record_error(A.st, CHD_ERR_NOT_PD, R.k0 + c, R.col0 + c);
          d = 1.0;
        }
        const double r2 = 1.0 / d;
#pragma unroll
        for (int e = 0; e < EL; ++e) {
          const int o = lane + 32 * e;
          if (o < W) {
            const double gv = val[e] * r2;
            sm.f[cur][o] = val[e];
            sm.g[cur][o] = gv;
            int p = o - s0;
            if (p < 0) p += W;
            if (outs) {
              A.o0[(int64_t)c * W + p] = p == 0 ? d : val[e];
              A.o1[(int64_t)c * W + p] = p == 0 ? r2 : gv;
            }
          }
        }
        if (outs && lane == 0) A.dd[4 * (int64_t)c] = d;
      } else {
        // P = h_A - L h_0 / 2: U' = Yh_AA - (P L^T + L P^T); K_A = P - L h_0 / 2
        const double hh = 0.5 * d;
#pragma unroll
        for (int e = 0; e < EL; ++e) {
          const int o = lane + 32 * e;
          if (o < W) {
            const double pv = fma(-l[e], hh, val[e]);
            sm.f[cur][o] = pv;
            sm.g[cur][o] = l[e];
            int p = o - s0;
            if (p < 0) p += W;
            if (outs) A.o0[(int64_t)c * W + p] = p == 0 ? d : fma(-l[e], hh, pv);
          }
        }
      }
    };
    for (int c = i0; c < i0 + AHEAD; ++c) prefetch(c);
    cp_async_wait<AHEAD - 1>();
    bar(NT + 32);  // the window's columns i0 and i0 + 1 are in uc
    column(i0);
    bar(NT + 32);
    for (int i = i0; i < L; ++i) {
      if (i + 1 < L) {
        cp_async_wait<AHEAD - 2>();  // column i + 1
        __syncwarp();
        column(i + 1);
      }
      bar(NT + 32);
      prefetch(i + AHEAD);
    }
  } else {
    // ---- update warps: pairs (u, v), u >= v, of slots ----
    const int ut = tid - 32, np = W * (W + 1) / 2;
    int pu[PP], pv[PP];
    double U[PP];
#pragma unroll
    for (int t = 0; t < PP; ++t) {
      const int e = ut + NT * t;
      int u = 0, v = 0;
      if (e < np) {
        u = (int)((sqrtf(8.0f * e + 1.0f) - 1.0f) * 0.5f);
        while (u * (u + 1) / 2 > e) --u;
        while ((u + 1) * (u + 2) / 2 <= e) ++u;
        v = e - u * (u + 1) / 2;
      }
      pu[t] = u;
      pv[t] = v;
      U[t] = 0.0;
    }
    int s0 = i0 % W;
    if (sp_.in) {
      const int t1 = s0 + 1 == W ? 0 : s0 + 1;
#pragma unroll
      for (int t = 0; t < PP; ++t) {
        if (ut + NT * t >= np) break;
        const int u = pu[t], v = pv[t];
        const int p = u >= s0 ? u - s0 : u - s0 + W, q = v >= s0 ? v - s0 : v - s0 + W;
        const double x = p < a && q < a ? sp_.in[max(p, q) + (int64_t)min(p, q) * a] : 0.0;
        if (u == s0 || v == s0) sm.uc[i0 & 1][u == s0 ? v : u] = x;
        else if (i0 + 1 < L && (u == t1 || v == t1)) sm.uc[(i0 + 1) & 1][u == t1 ? v : u] = x;
        else U[t] = x;
      }
    }
    bar(NT + 32);
    bar(NT + 32);
    for (int i = i0; i < L; ++i) {
      const int s1 = i + 1 < L ? (s0 + 1 == W ? 0 : s0 + 1) : s0;
      int s2 = s0 + 2;
      if (s2 >= W) s2 -= W;
      const bool pub = i + 2 < L;
      const double* f = sm.f[i & 1];
      const double* g = sm.g[i & 1];
      double* uc = sm.uc[i & 1];
#pragma unroll
      for (int t = 0; t < PP; ++t) {
        if (ut + NT * t >= np) break;
        const int u = pu[t], v = pv[t];
        if (u != s0 && v != s0 && u != s1 && v != s1) {
          U[t] = fma(-f[u], g[v], U[t]);
          if (MODE == UP_HESS) U[t] = fma(-g[u], f[v], U[t]);
        }
        if (pub && (u == s2 || v == s2)) {
          uc[u == s2 ? v : u] = U[t];
          U[t] = 0.0;
        }
      }
      bar(NT + 32);
      s0 = s0 + 1 == W ? 0 : s0 + 1;
    }
    if (!sp_.G) return;
    // rows L .. L + a - 1, i.e. every slot but that of row L - 1
    const int sL = L % W, out = sL == 0 ? W - 1 : sL - 1;
#pragma unroll
    for (int t = 0; t < PP; ++t) {
      if (ut + NT * t >= np) break;
      const int u = pu[t], v = pv[t];
      if (u == out || v == out) continue;
      int p = u - sL, q = v - sL;
      if (p < 0) p += W;
      if (q < 0) q += W;
      sp_.G[max(p, q) + (int64_t)min(p, q) * sp_.ldg] = U[t];
    }
  }
}
// Threads by window size: the smallest set of update warps whose registers
// hold the pairs, so that short windows pay for few barriers and few FP64
// instructions (one warp up to a = 9, three up to a = 31, seven up to 64).
constexpr int UPT = 256;
template <int MODE>
__device__ __forceinline__ void up_dispatch(const Run& R, const Span& sp, const UpArgs& A, UpSmem& sm) {
  if (R.a <= 9) up_run<32, 2, MODE>(R, sp, A, sm);
  else if (R.a <= 31) up_run<96, 6, MODE>(R, sp, A, sm);
  else up_run<224, 10, MODE>(R, sp, A, sm);
}
// the top front's update block for the parent (its A x A part, ld J = a + 1)
__device__ __forceinline__ double* update_block(const Run& R, double* ws) {
  return ws + R.f0 + (int64_t)(R.L - 1) * R.fstride + R.a + 2;
}
// window handed over at the lower end of segment [s, ..): a x a, ld a, in the
// workspace front of its first column; the second column's holds a temporary
__device__ __forceinline__ double* seg_window(const Run& R, int s, double* ws) {
  return ws + R.f0 + (int64_t)s * R.fstride;
}

// Algorithm 7.1 for one-column fronts (Algorithm 3.1): D = F_11, L_AN =
// F_21 / D, U = F_22 - F_21 F_21^T / D.  Lc receives F_11 and F_21;
// kc_factor_post scales them to C = sqrt(D), B = F_21 / C.
__global__ void __launch_bounds__(UPT) kc_factor(SymDev S, int task0, const double* X, double* Lc, double* Wc,
                                                double* Dd, double* ws, int64_t* st) {
  __shared__ UpSmem sm;
  const Run R = run_of(S, task0 + blockIdx.x);
  UpArgs A{X + R.base0, nullptr, Lc + R.base0, Wc + R.base0, Dd + R.d0, st};
  up_dispatch<UP_FACTOR>(R, Span{0, R.L, nullptr, true, update_block(R, ws), R.a + 1}, A, sm);
}
// C, B and log D of every column of every run, one warp per column
template <bool LIST>
__global__ void __launch_bounds__(128) kc_factor_post(SymDev S, Columns cols, double* Lc, const double* Dd,
                                                     double* ldet) {
  int i, step;
  const Run R = run_of_columns<LIST>(S, cols, 4, threadIdx.x >> 5, i, step);
  const int lane = threadIdx.x & 31;
  for (; i < R.L; i += step) {
    const double d = Dd[R.d0 + 4 * (int64_t)i], r = rsqrt(d);
    double* c = Lc + R.base0 + (int64_t)i * (R.a + 1);
    for (int p = lane; p <= R.a; p += 32) c[p] *= r;
    if (lane == 0) ldet[R.k0 + i] = log(d);
  }
}

// Algorithm 5.1 step 1 for one-column fronts: with Yh the front's values
// plus the child's U', K_jj = Yh_jj, K_A = Yh_A - L_A Yh_jj,
// U' = Yh_AA - K_A L_A^T - L_A Yh_A^T; K goes to T, kc_hess_m applies step 2.
// act (pruned R(Y), §5.5): a front with act == 0 has Y zero in its subtree,
// so K, U' and M are zero; along a run these are its first columns.
__global__ void __launch_bounds__(UPT) kc_hess_up(SymDev S, int task0, const double* Wc, const double* Y, int64_t ldy,
                                                 double* T, int64_t ldt, double* ws, const uint8_t* act) {
  __shared__ UpSmem sm;
  const Run R = run_of(S, task0 + blockIdx.x);
  const int64_t y = blockIdx.y;
  int i0 = 0;
  if (act) {
    const uint8_t* ay = act + y * S.nsn + R.k0;
    if (!ay[R.L - 1]) return;  // nothing reaches the run; its parent skips its block
    int lo = 0, hi = R.L - 1;  // the first active column
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (ay[mid]) hi = mid;
      else lo = mid + 1;
    }
    i0 = lo;
  }
  UpArgs A{Y + y * ldy + R.base0, Wc + R.base0, T + y * ldt + R.base0, nullptr, nullptr, nullptr};
  up_dispatch<UP_HESS>(R, Span{i0, R.L, nullptr, true, update_block(R, ws + y * S.f_total), R.a + 1}, A, sm);
}
// the same by segments (phase 1: every segment but the last from a zero
// window, the first one for good; phase 2: the others from their windows)
__global__ void __launch_bounds__(UPT) kc_hess_up_seg(SymDev S, int task0, int phase, const double* Wc,
                                                     const double* Y, int64_t ldy, double* T, int64_t ldt,
                                                     double* ws) {
  __shared__ UpSmem sm;
  const ChainSeg g = S.cseg[blockIdx.x];
  if (phase == 1 ? g.p == g.P - 1 && g.P > 1 : g.p == 0) return;
  const Run R = run_of(S, task0 + g.run);
  const int64_t y = blockIdx.y;
  ws += y * S.f_total;
  UpArgs A{Y + y * ldy + R.base0, Wc + R.base0, T + y * ldt + R.base0, nullptr, nullptr, nullptr};
  const bool last = g.p == g.P - 1;
  const double* in = phase == 2 ? seg_window(R, S.cseg[blockIdx.x - 1].s, ws) : nullptr;
  double* win = last ? update_block(R, ws) : phase == 1 ? seg_window(R, g.s, ws) : nullptr;
  const Span sp{g.s, g.e, in, phase == 2 || g.p == 0, win, last ? R.a + 1 : R.a};
  up_dispatch<UP_HESS>(R, sp, A, sm);
}

// ---------------------------------------------------------------------------
// products with a symmetric a x a block per column, over all columns at once
// ---------------------------------------------------------------------------
constexpr int MT = 128;      // threads per column
constexpr int BLD = AMAX + 1;  // leading dimension of a staged block

// the symmetric block stored lower column-major (ld a) into both triangles of B
__device__ __forceinline__ void stage_sym(double (*B)[BLD], const double* M, int a) {
  const int lane = threadIdx.x & 31;
  for (int c = threadIdx.x >> 5; c < a; c += MT / 32)
    for (int r = c + lane; r < a; r += 32) {
      const double v = M[r + (int64_t)c * a];
      B[r][c] = v;
      B[c][r] = v;
    }
}
// y[r] = sum_s B(r, s) x[s], r < a; two threads per row, y written by the even one
__device__ __forceinline__ void sym_dot(const double (*B)[BLD], const double* x, int a, double* y) {
  const int r = threadIdx.x >> 1, h = threadIdx.x & 1;
  if ((threadIdx.x & ~31) / 2 < a) {  // whole warps beyond the block are idle
    double a0 = 0.0, a1 = 0.0;
    if (r < a) {
      int s = h;
      for (; s + 2 < a; s += 4) {
        a0 = fma(B[r][s], x[s], a0);
        a1 = fma(B[r][s + 2], x[s + 2], a1);
      }
      if (s < a) a0 = fma(B[r][s], x[s], a0);
    }
    a0 += a1;
    a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
    if (r < a && h == 0) y[r] = a0;
  }
}
// rows j+1 .. j+a of the matrix v (values of the run's columns, and the
// parent's front Fp beyond the run) as a full symmetric block
__device__ __forceinline__ void stage_window(const SymDev& S, const Run& R, int j, const double* v, const double* Fp,
                                            int Jp, const int32_t* rel, double (*B)[BLD]) {
  const int lane = threadIdx.x & 31, a = R.a;
  for (int c = threadIdx.x >> 5; c < a; c += MT / 32) {
    const int col = j + 1 + c;
    for (int r = c + lane; r < a; r += 32) {
      double x;
      if (col < R.L) {
        x = v[(int64_t)col * (a + 1) + (r - c)];
      } else {  // rows col .. of the run's top front lie in the parent
        const int pr = __ldg(rel + (j + 1 + r - R.L)), pc = __ldg(rel + (col - R.L));
        x = __ldcg(Fp + (pr >= pc ? pr + (int64_t)pc * Jp : pc + (int64_t)pr * Jp));
      }
      B[r][c] = x;
      B[c][r] = x;
    }
  }
}
struct Parent {
  const double* F;
  int J;
  const int32_t* rel;
};
__device__ __forceinline__ Parent parent_of(const SymDev& S, const Run& R, const double* ws) {
  Parent P;
  const int k1 = R.k0 + R.L - 1;
  const int64_t p = S.sn_par[k1];
  P.J = (int)(S.rows_ptr[p + 1] - S.rows_ptr[p]);
  P.F = ws + S.f_off[p];
  P.rel = S.rel + S.rows_ptr[k1] + 1;
  return P;
}

// Algorithm 5.1 step 2: M_jj = K_jj / D^2, M_A = V K_A / D (K in T, in place)
template <bool LIST>
__global__ void __launch_bounds__(MT) kc_hess_m(SymDev S, Columns cols, const double* Wc, const double* Vd, double* T,
                                               int64_t ldt, const uint8_t* act) {
  __shared__ double B[AMAX][BLD];
  __shared__ double x[AMAX], yv[AMAX];
  int i, step;
  const Run R = run_of_columns<LIST>(S, cols, 1, 0, i, step);
  const int a = R.a, tid = threadIdx.x;
  const int64_t y = blockIdx.z;
  for (; i < R.L; i += step) {
    if (act && !act[y * S.nsn + R.k0 + i]) continue;
    double* t = T + y * ldt + R.base0 + (int64_t)i * (a + 1);
    const double dinv = Wc[R.base0 + (int64_t)i * (a + 1)];
    stage_sym(B, Vd + R.v0 + (int64_t)i * R.vstride, a);
    if (tid < a) x[tid] = t[1 + tid] * dinv;
    __syncthreads();
    sym_dot(B, x, a, yv);
    __syncthreads();
    if (tid < a) t[1 + tid] = yv[tid];
    if (tid == MT - 1) t[0] = dinv * t[0] * dinv;
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// top-down serial kernels (gradient, Hessian step 3)
//
// The window covers the a rows c+1 .. c+a while column c is in work, row rho
// in slot rho mod a (row c takes the slot of row c + a).  Four threads hold
// a row each, entries v = part, part + 4, ..  Per column:
//   phase 1: they multiply the window with L_A (a = 61: 128 FP64 warp
//     instructions) and reduce over the four;
//   barrier; phase 2: T_A = M_A - w, once per entry; barrier; the new row
//     goes into the registers.
// The new diagonal entry, T_cc = (M_cc - 2 L_A^T M_A) + L_A^T w, needs a dot
// product over all rows: warp 0 takes w after the first barrier, passes the
// second without waiting and has until the next column's phase 2, where the
// one product that the missing entry enters is corrected.  (The bracket does
// not depend on the recursion: kc_down_pre forms it for all columns.)  Warp 0
// also loads the inputs.
// ---------------------------------------------------------------------------
struct DownSmem {
  double ring[2][RING][WP];  // L_A (slots), and M_A; [.][WP - 1]: the diagonal's part known beforehand
  double wv[WP], tv[2][WP], dg[2];
};
enum { DOWN_GRAD = 0, DOWN_HESS = 1 };
// second barrier of a column: the window threads wait, warp 0 only arrives
__device__ __forceinline__ void bar2_sync(int n) { asm volatile("bar.sync 2, %0;\n" ::"r"(n) : "memory"); }
__device__ __forceinline__ void bar2_arrive(int n) { asm volatile("bar.arrive 2, %0;\n" ::"r"(n) : "memory"); }
// Columns hi .. lo (downwards).  in: the window above column hi (rows hi + 1
// .. hi + a; a x a, lower, ld a), or the parent's front where it is null and
// `top`, or zeros; outs: whether outputs are stored; win: receives the window
// after column lo (rows lo .. lo + a - 1), or null.
struct DownSpan {
  int hi, lo;
  const double* in;
  bool top, outs;
  double* win;
};
template <int NT, int CP, int TP, int MODE>
__device__ void down_run(const SymDev& S, const Run& R, const DownSpan& sp, const double* wc, const double* src,
                         double* out, const double* ws, DownSmem& sm) {
  const int a = R.a, W = a + 1, tid = threadIdx.x, L = sp.hi + 1, lo = sp.lo;
  const bool outs = sp.outs;
  if (tid >= NT + 32) return;
  // slots past the window are multiplied by zeros: they must hold numbers
  for (int e = tid; e < 2 * RING * WP; e += NT + 32) (&sm.ring[0][0][0])[e] = 0.0;
  bar(NT + 32);
  if (tid < 32) {
    const int lane = tid;
    int sload = (L - 1) % a;
    auto prefetch = [&](int c) {
      if (c >= lo) {
        const int sc = sload;
        sload = sload == 0 ? a - 1 : sload - 1;
        for (int p = lane; p <= a; p += 32) {
          int s = sc + p;
          while (s >= a) s -= a;
          if (p == 0) s = WP - 1;
          cp_async8(&sm.ring[0][c % RING][s], wc + (int64_t)c * W + p);
          if (MODE == DOWN_HESS) cp_async8(&sm.ring[1][c % RING][s], src + (int64_t)c * W + p);
        }
      }
      cp_async_commit();
    };
    int steps = 1;
    while (steps < 32 && steps < a) steps <<= 1;
    for (int c = L - 1; c > L - 1 - AHEAD; --c) prefetch(c);
    cp_async_wait<AHEAD - 1>();
    bar(NT + 32);
    int s1 = -1;  // slot of row c + 1, whose diagonal entry d the window lacks
    double d = 0.0;
    for (int c = L - 1; c >= lo; --c) {
      cp_async_wait<AHEAD - 2>();  // column c - 1 has arrived
      bar(NT + 32);
      const double* l = sm.ring[0][c % RING];
      const double q = MODE == DOWN_HESS ? sm.ring[1][c % RING][WP - 1] : l[WP - 1];
      const bool two = lane + 32 < a;
      double w0 = lane < a ? sm.wv[lane] : 0.0, w1 = two ? sm.wv[lane + 32] : 0.0;
      const double l0 = lane < a ? l[lane] : 0.0, l1 = two ? l[lane + 32] : 0.0;
      bar2_arrive(NT + 32);
      if (s1 >= 0) {
        if (s1 < 32) w0 = lane == s1 ? fma(d, l0, w0) : w0;
        else w1 = lane == s1 - 32 ? fma(d, l1, w1) : w1;
      }
      double acc = fma(l0, w0, lane == 0 ? q : 0.0);
      if (a > 32) acc = fma(l1, w1, acc);
      for (int o = steps >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      d = __shfl_sync(0xffffffffu, acc, 0);
      if (lane == 0) {
        sm.dg[c & 1] = d;
        if (outs) out[(int64_t)c * W] = d;
      }
      s1 = s1 < 0 ? (L - 1) % a : (s1 == 0 ? a - 1 : s1 - 1);
      prefetch(c - AHEAD);
    }
    bar(NT + 32);  // the last diagonal entry
  } else {
    const int rt = tid - 32, u = rt / TP, part = rt % TP;
    double V[CP];
    {
      const int sL = L % a;
      auto off = [&](int v) { return v >= sL ? v - sL : v - sL + a; };
      const int k1 = R.k0 + R.L - 1;
      const int64_t p = S.sn_par[k1];
      const int Jp = (int)(S.rows_ptr[p + 1] - S.rows_ptr[p]);
      const double* Fp = ws + S.f_off[p];
      const int32_t* rel = S.rel + S.rows_ptr[k1] + 1;
#pragma unroll
      for (int j = 0; j < CP; ++j) {
        const int v = part + TP * j;
        V[j] = 0.0;
        if (u < a && v < a) {
          const int x = max(off(u), off(v)), y = min(off(u), off(v));
          if (sp.in) V[j] = sp.in[x + (int64_t)y * a];
          else if (sp.top) V[j] = __ldcg(Fp + __ldg(rel + x) + (int64_t)__ldg(rel + y) * Jp);
        }
      }
    }
    bar(NT + 32);
    int s = (L - 1) % a;
    for (int c = L - 1; c >= lo; --c) {
      const double* l = sm.ring[0][c % RING];
      const double* mm = sm.ring[1][c % RING];
      // one accumulator: a warp issues an FP64 instruction every 64 clocks at
      // best, dependent or not
      double a0 = 0.0;
#pragma unroll
      for (int j = 0; j < CP; ++j)
        if (TP * j < a) a0 = fma(V[j], l[part + TP * j], a0);  // slots beyond the window: V = 0
#pragma unroll
      for (int o = 1; o < TP; o <<= 1) a0 += __shfl_xor_sync(0xffffffffu, a0, o);
      if (part == 0 && u < a) sm.wv[u] = a0;
      bar(NT + 32);
      const int s1 = c + 1 < L ? (s + 1 == a ? 0 : s + 1) : -1;  // row c + 1, its diagonal still missing
      double* tv = sm.tv[c & 1];
      const double dnew = sm.dg[(c + 1) & 1];
      if (rt < a) {
        double w = sm.wv[rt];
        if (rt == s1) w = fma(dnew, l[rt], w);
        const double t = MODE == DOWN_HESS ? mm[rt] - w : -w;
        tv[rt] = t;
        int p = rt - s;
        if (p <= 0) p += a;
        if (outs) out[(int64_t)c * W + p] = t;
      }
      bar2_sync(NT + 32);
      // the new row into the registers: column slot s of every row, the
      // threads of row slot s, and the diagonal entry of the row before
      const double mine = u < a ? tv[u] : 0.0;
      const int js = s / TP, ps = s % TP;
      if (part == ps) {
#pragma unroll
        for (int j = 0; j < CP; ++j)
          if (j == js) V[j] = mine;
      }
      if (u == s) {
#pragma unroll
        for (int j = 0; j < CP; ++j) {
          const int v = part + TP * j;
          V[j] = v == s || v >= a ? 0.0 : tv[v];
        }
      } else if (u == s1 && part == s1 % TP) {
#pragma unroll
        for (int j = 0; j < CP; ++j)
          if (j == s1 / TP) V[j] = dnew;
      }
      s = s == 0 ? a - 1 : s - 1;
    }
    bar(NT + 32);
    if (sp.win && u < a) {
      const int sw = lo % a;
      const int p = u >= sw ? u - sw : u - sw + a;
#pragma unroll
      for (int j = 0; j < CP; ++j) {
        const int v = part + TP * j, q = v >= sw ? v - sw : v - sw + a;
        if (v < a && p >= q) sp.win[p + (int64_t)q * a] = p == 0 ? sm.dg[lo & 1] : V[j];
      }
    }
  }
}
constexpr int DNT = 288;
template <int MODE>
__device__ __forceinline__ void down_dispatch(const SymDev& S, const Run& R, const DownSpan& sp, const double* wc,
                                             const double* src, double* out, const double* ws, DownSmem& sm) {
  if (R.a <= 8) down_run<32, 2, 4, MODE>(S, R, sp, wc, src, out, ws, sm);
  else if (R.a <= 16) down_run<64, 4, 4, MODE>(S, R, sp, wc, src, out, ws, sm);
  else if (R.a <= 32) down_run<128, 8, 4, MODE>(S, R, sp, wc, src, out, ws, sm);
  else down_run<256, 16, 4, MODE>(S, R, sp, wc, src, out, ws, sm);
}
// by segments: phase 1: every segment but the first from a zero window, the
// last one from the parent and for good; phase 2: the others from their windows
__device__ __forceinline__ bool down_seg(const SymDev& S, const ChainSeg& g, const Run& R, int phase, double* ws,
                                         DownSpan& sp) {
  const bool last = g.p == g.P - 1;
  if (phase == 1 ? g.p == 0 && g.P > 1 : last) return false;
  sp = DownSpan{g.e - 1, g.s, phase == 2 ? seg_window(R, g.e, ws) : nullptr, last, phase == 2 || last,
                phase == 1 && g.p > 0 ? seg_window(R, g.s, ws) : nullptr};
  return true;
}

// Algorithm 7.2 for one-column fronts (Algorithm 4.1): S_AN = -V L_AN,
// S_NN = D^{-1} - S_AN^T L_AN; V of the child = [S_NN S_AN^T; S_AN V] on the
// child's rows.  kc_grad_post stores V_j of every column and the gradient.
__global__ void __launch_bounds__(DNT) kc_gradient(SymDev S, int task0, const double* Wc, double* Sc,
                                                  const double* ws) {
  __shared__ DownSmem sm;
  const Run R = run_of(S, task0 + blockIdx.x);
  down_dispatch<DOWN_GRAD>(S, R, DownSpan{R.L - 1, 0, nullptr, true, true, nullptr}, Wc + R.base0, nullptr,
                           Sc + R.base0, ws, sm);
}
__global__ void __launch_bounds__(DNT) kc_gradient_seg(SymDev S, int task0, int phase, const double* Wc, double* Sc,
                                                      double* ws) {
  __shared__ DownSmem sm;
  const ChainSeg g = S.cseg[blockIdx.x];
  const Run R = run_of(S, task0 + g.run);
  DownSpan sp;
  if (!down_seg(S, g, R, phase, ws, sp)) return;
  down_dispatch<DOWN_GRAD>(S, R, sp, Wc + R.base0, nullptr, Sc + R.base0, ws, sm);
}
template <bool LIST>
__global__ void __launch_bounds__(MT) kc_grad_post(SymDev S, Columns cols, const double* Sc, double* g, double* Vd,
                                                  const double* ws) {
  int i, step;
  const Run R = run_of_columns<LIST>(S, cols, 1, 0, i, step);
  const Parent P = parent_of(S, R, ws);
  const int a = R.a, lane = threadIdx.x & 31;
  const double* v = Sc + R.base0;
  for (; i < R.L; i += step) {
    double* Vb = Vd + R.v0 + (int64_t)i * R.vstride;
    for (int c = threadIdx.x >> 5; c < a; c += MT / 32) {
      const int col = i + 1 + c;
      for (int r = c + lane; r < a; r += 32) {
        double x;
        if (col < R.L) {
          x = v[(int64_t)col * (a + 1) + (r - c)];
        } else {
          const int pr = __ldg(P.rel + (i + 1 + r - R.L)), pc = __ldg(P.rel + (col - R.L));
          x = __ldcg(P.F + (pr >= pc ? pr + (int64_t)pc * P.J : pc + (int64_t)pr * P.J));
        }
        Vb[r + (int64_t)c * a] = x;
      }
    }
    if (g) {
      const int64_t b = (int64_t)i * (a + 1);
      for (int q = threadIdx.x; q <= a; q += MT) g[R.base0 + b + q] = -v[b + q];
    }
  }
}
// Algorithm 5.1 step 3 for one-column fronts: with w = V' L_A, T_A = M_A - w,
// T_jj = M_jj - 2 L_A^T M_A + L_A^T w; V' of the child = [T_jj T_A^T; T_A V']
// on its rows.  T in place; first
// what of T_jj does not depend on the recursion, in place: M_jj - 2 L_A^T M_A
template <bool LIST>
__global__ void __launch_bounds__(128) kc_down_pre(SymDev S, Columns cols, const double* Wc, double* T, int64_t ldt) {
  int i, step;
  const Run R = run_of_columns<LIST>(S, cols, 4, threadIdx.x >> 5, i, step);
  const int lane = threadIdx.x & 31, W = R.a + 1;
  T += (int64_t)blockIdx.z * ldt + R.base0;
  for (; i < R.L; i += step) {
    double* t = T + (int64_t)i * W;
    const double* l = Wc + R.base0 + (int64_t)i * W;
    double acc = 0.0;
    for (int p = 1 + lane; p < W; p += 32) acc = fma(l[p], t[p], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) t[0] = fma(-2.0, acc, t[0]);
  }
}
__global__ void __launch_bounds__(DNT) kc_hess_down(SymDev S, int task0, const double* Wc, double* T, int64_t ldt,
                                                   const double* ws) {
  __shared__ DownSmem sm;
  const Run R = run_of(S, task0 + blockIdx.x);
  const int64_t y = blockIdx.y;
  double* t = T + y * ldt + R.base0;
  down_dispatch<DOWN_HESS>(S, R, DownSpan{R.L - 1, 0, nullptr, true, true, nullptr}, Wc + R.base0, t, t,
                           ws + y * S.f_total, sm);
}
__global__ void __launch_bounds__(DNT) kc_hess_down_seg(SymDev S, int task0, int phase, const double* Wc, double* T,
                                                       int64_t ldt, double* ws) {
  __shared__ DownSmem sm;
  const ChainSeg g = S.cseg[blockIdx.x];
  const Run R = run_of(S, task0 + g.run);
  const int64_t y = blockIdx.y;
  ws += y * S.f_total;
  DownSpan sp;
  if (!down_seg(S, g, R, phase, ws, sp)) return;
  double* t = T + y * ldt + R.base0;
  down_dispatch<DOWN_HESS>(S, R, sp, Wc + R.base0, t, t, ws, sm);
}

// ---------------------------------------------------------------------------
// Segments.  Along a run the gradient and both Hessian passes are affine in
// the window that passes from front to front: over a segment of columns
//   top-down   V_low  = Psi V_high Psi^T + C,
//   bottom-up  U_high = Psi^T U_low Psi + B,
// with the same a x a matrix Psi (rows: the window at the segment's lower end,
// in terms of the one at its upper end), which depends on L only.  So all
// segments run at once from a zero window (phase 1), the windows at their
// ends follow from one small congruence per segment, and all run again from
// their true windows (phase 2).  Twice the work, but on as many SMs as there
// are segments instead of one: every value is computed by the same recursion
// as in the serial kernels, from windows whose error is that of one more
// congruence.  kc_psi propagates the rows of Psi; its columns are independent
// of each other, so it needs no exchange between threads.
// ---------------------------------------------------------------------------
constexpr int PSX = 16;  // columns of Psi per CTA, four threads each
__global__ void __launch_bounds__(4 * PSX) kc_psi(SymDev S, int task0, const double* Wc, double* Psi) {
  __shared__ double Lb[2][RING][WP];
  const ChainSeg g = S.cseg[blockIdx.x];
  const int tid = threadIdx.x, part = tid & 3, x = blockIdx.y * PSX + (tid >> 2);
  const Run R = run_of(S, task0 + g.run);
  const int a = R.a, W = a + 1;
  if (g.p == 0 || g.p == g.P - 1 || (int)(blockIdx.y * PSX) >= a) return;
  const double* wc = Wc + R.base0;
  double X[AMAX / 4];
  const int se = g.e % a;
#pragma unroll
  for (int j = 0; j < AMAX / 4; ++j) {
    const int v = part + 4 * j, q = v >= se ? v - se : v - se + a;
    X[j] = v < a && q == x ? 1.0 : 0.0;
  }
  auto load = [&](int c0, int b) {  // columns c0, c0 - 1, .. c0 - RING + 1
    for (int k = 0; k < RING; ++k)
      if (c0 - k >= g.s)
        for (int p = tid; p < W; p += 4 * PSX) cp_async8(&Lb[b][k][p], wc + (int64_t)(c0 - k) * W + p);
    cp_async_commit();
  };
  int b = 0, sc = (g.e - 1) % a;
  load(g.e - 1, 0);
  for (int c0 = g.e - 1; c0 >= g.s; c0 -= RING, b ^= 1) {
    __syncthreads();
    load(c0 - RING, b ^ 1);
    cp_async_wait<1>();
    __syncthreads();
    for (int k = 0; k < RING && c0 - k >= g.s; ++k) {
      const double* l = Lb[b][k];
      double y = 0.0;
#pragma unroll
      for (int j = 0; j < AMAX / 4; ++j) {
        const int v = part + 4 * j;
        int p = v - sc;
        if (p <= 0) p += a;
        if (4 * j < a) y = fma(X[j], v < a ? l[p] : 0.0, y);
      }
      y += __shfl_xor_sync(0xffffffffu, y, 1);
      y += __shfl_xor_sync(0xffffffffu, y, 2);
      if (part == (sc & 3)) {
#pragma unroll
        for (int j = 0; j < AMAX / 4; ++j)
          if (j == sc >> 2) X[j] = -y;
      }
      sc = sc == 0 ? a - 1 : sc - 1;
    }
  }
  if (x >= a) return;
  const int ss = g.s % a;
#pragma unroll
  for (int j = 0; j < AMAX / 4; ++j) {
    const int v = part + 4 * j, p = v >= ss ? v - ss : v - ss + a;
    if (v < a) Psi[g.psi + p + (int64_t)x * a] = X[j];
  }
}
// One step of the windows' recursion on every run of three segments or more:
// Z = M V (half 0), then win += Z M^T (half 1, lower), M = Psi (top-down) or
// Psi^T (bottom-up); 16 x 16 outputs per CTA
template <bool UP>
__global__ void __launch_bounds__(256) kc_scan(SymDev S, int task0, int step, int half, const double* Psi,
                                              double* ws) {
  __shared__ double A[16][AMAX + 1], B[AMAX][17];
  const int2 rs = S.crun[blockIdx.y];
  const int p = UP ? 1 + step : rs.y - 2 - step;
  if (p < 1 || p > rs.y - 2) return;
  const ChainSeg g = S.cseg[rs.x + p], src = S.cseg[UP ? rs.x + p - 1 : rs.x + p + 1];
  const Run R = run_of(S, task0 + g.run);
  const int a = R.a, i0 = (blockIdx.x & 3) * 16, j0 = (blockIdx.x >> 2) * 16, tid = threadIdx.x;
  if (i0 >= a || j0 >= a || (half && i0 < j0)) return;
  ws += (int64_t)blockIdx.z * S.f_total;
  const double* M = Psi + g.psi;
  double* win = seg_window(R, g.s, ws);
  double* Z = win + R.fstride;
  const double* V = seg_window(R, src.s, ws);
  auto m = [&](int i, int k) { return UP ? M[k + (int64_t)i * a] : M[i + (int64_t)k * a]; };
  for (int e = tid; e < 16 * AMAX; e += 256) {
    const int i = e & 15, k = e >> 4;
    double x = 0.0, y = 0.0;
    if (k < a) {
      if (i0 + i < a) x = half ? Z[i0 + i + (int64_t)k * a] : m(i0 + i, k);
      if (j0 + i < a) {
        const int j = j0 + i;
        y = half ? m(j, k) : V[max(k, j) + (int64_t)min(k, j) * a];
      }
    }
    A[i][k] = x;
    B[k][i] = y;
  }
  __syncthreads();
  const int i = tid & 15, j = tid >> 4;
  double acc = 0.0;
  for (int k = 0; k < a; ++k) acc = fma(A[i][k], B[k][j], acc);
  if (i0 + i >= a || j0 + j >= a) return;
  if (half == 0) Z[i0 + i + (int64_t)(j0 + j) * a] = acc;
  else if (i0 + i >= j0 + j) win[i0 + i + (int64_t)(j0 + j) * a] += acc;
}

// Algorithm 5.2 steps 1-2 for one-column fronts: V' is the input T on
// A_j x A_j, M_A = T_A + V' L_A, M_jj = T_jj + L_A^T (T_A + M_A),
// K_jj = D M_jj D, K_A = V^{-1} (M_A D).  No column waits for another.
// Writes what step 3 starts from into the front's temporaries: P = K_A + L_A
// K_jj / 2 into the first, Y_jj = K_jj and Y_A = K_A + L_A K_jj into the second.
// Not into the output, which may be the input: other CTAs still read the
// input's columns j+1 .. j+a.
template <bool LIST>
__global__ void __launch_bounds__(MT) kc_ihess_down(SymDev S, Columns cols, const double* Wc, const double* Dd,
                                                   const double* Rd, const double* Tin, int64_t ldt,
                                                   double* ws) {
  __shared__ double B[AMAX][BLD];
  __shared__ double lw[AMAX], tt[AMAX], x[AMAX], yv[AMAX];
  __shared__ double kjj;
  int i, step;
  const Run R = run_of_columns<LIST>(S, cols, 1, 0, i, step);
  const int a = R.a, tid = threadIdx.x, lane = tid & 31;
  const int64_t y = blockIdx.z;
  Tin += y * ldt + R.base0;
  ws += y * S.f_total;
  const Parent P = parent_of(S, R, ws);
  for (; i < R.L; i += step) {
    const int64_t b = (int64_t)i * (a + 1);
    const double dd = Dd[R.d0 + 4 * (int64_t)i];
    stage_window(S, R, i, Tin, P.F, P.J, P.rel, B);
    if (tid < a) {
      lw[tid] = Wc[R.base0 + b + 1 + tid];
      tt[tid] = Tin[b + 1 + tid];
    }
    __syncthreads();
    sym_dot(B, lw, a, yv);
    __syncthreads();
    if (tid < 32) {
      double acc = 0.0;
      for (int r = lane; r < a; r += 32) {
        const double t = tt[r], m = t + yv[r];
        acc = fma(lw[r], t + m, acc);
        x[r] = m * dd;
      }
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) kjj = dd * ((Tin[b] + acc) * dd);
    }
    stage_sym(B, Rd + R.v0 + (int64_t)i * R.vstride, a);
    __syncthreads();
    sym_dot(B, x, a, yv);
    __syncthreads();
    double* Pv = ws + R.f0 + (int64_t)i * R.fstride + (int64_t)(a + 1) * (a + 1);
    double* Yv = Pv + a + 1;
    if (tid < a) {
      const double k = kjj, p = fma(0.5 * lw[tid], k, yv[tid]);
      Pv[1 + tid] = p;
      Yv[1 + tid] = 2.0 * p - yv[tid];
    }
    if (tid == MT - 1) Yv[0] = kjj;
    __syncthreads();
  }
}

// Sums of the columns' rank-one (rank-two) blocks over a run: entry
// (j + r, j) of Z = sum_k x_k y_k^T, the k-th column's vectors covering rows
// k .. k+a.  Nothing depends on the order of the columns, so a warp takes one
// column j of Z, its lanes the rows r, for the columns of the run (stored to
// the output) and for the a columns beyond it (the update block the parent
// adds).
//   product (Algorithm 3.2): x = y = [C; B];
//   inverse Hessian step 3:  -(P L^T + L P^T), rows k+1 .. k+a, added to what
//   kc_ihess_down left in the second temporaries.
// LIST: the grid ends with `beyond` CTAs for the columns beyond each run
template <bool PROD, bool LIST>
__global__ void __launch_bounds__(128) kc_band_sum(SymDev S, Columns cols, int beyond, const double* Gc, double* Out,
                                                  int64_t ldo, double* ws) {
  int j, step;
  Run R;
  const int e = (int)blockIdx.x - (cols.n + 3) / 4;
  if (!LIST || e < 0) {
    R = run_of_columns<LIST>(S, cols, 4, threadIdx.x >> 5, j, step);
  } else {
    R = run_of(S, cols.task0 + e / beyond);
    j = R.L + e % beyond * 4 + (threadIdx.x >> 5);
    step = 1 << 30;
  }
  const int a = R.a, lane = threadIdx.x & 31, W = a + 1;
  const int64_t y = blockIdx.z;
  Out += y * ldo + R.base0;
  ws += y * S.f_total;
  const double* Lw = Gc + R.base0;
  const double* Pw = ws + R.f0 + (int64_t)W * W;
  double* G = ws + R.f0 + (int64_t)(R.L - 1) * R.fstride;
  for (; j < R.L + a; j += step) {
    const int rmax = j < R.L ? a : R.L + a - 1 - j;
    const int kend = PROD ? min(j, R.L - 1) : min(j, R.L) - 1;
    for (int r0 = 0; r0 <= rmax; r0 += 32) {
      const int r = r0 + lane;
      const int klo = max(0, j + r - a);  // the first column that reaches row j + r
      double acc = 0.0;
      for (int k = max(0, j + r0 - a); k <= kend; ++k) {
        if (k >= klo && r <= rmax) {
          const double lj = Lw[(int64_t)k * W + (j - k)], li = Lw[(int64_t)k * W + (j - k) + r];
          if (PROD) {
            acc = fma(li, lj, acc);
          } else {
            const double* pk = Pw + (int64_t)k * R.fstride + (j - k);
            acc = fma(pk[r], lj, acc);
            acc = fma(li, pk[0], acc);
          }
        }
      }
      if (r <= rmax) {
        if (j < R.L) {
          Out[(int64_t)j * W + r] = PROD ? acc : Pw[(int64_t)j * R.fstride + W + r] + acc;
        } else {
          const int q = j - R.L;
          G[(1 + q + r) + (int64_t)(1 + q) * W] = PROD ? acc : -acc;
        }
      }
    }
  }
}

}  // namespace chain
}  // namespace chd

namespace chd_launch {
using namespace chd::chain;
// the columns of the launch's runs, and a grid of m x `per` of them per CTA
// (extra: as many more beyond each run)
static Columns columns(const chd_symbolic* s, int t0, int nt) {
  if (s->run_lmax > 0) return Columns{t0, 0, 0};
  return Columns{t0, s->task_ptr[t0], s->task_ptr[t0 + nt] - s->task_ptr[t0]};
}
static dim3 column_grid(const chd_symbolic* s, const Columns& c, int nt, int per, int m, int extra = 0) {
  auto ctas = [&](int v) { return (v + per - 1) / per; };
  if (c.n > 0) return dim3(ctas(c.n) + nt * ctas(extra), 1, m);
  return dim3(nt, std::min(ctas(s->run_lmax + extra), 32768), m);
}
// Whether m right-hand sides run by segments (chain_by_segments: the rule and
// its evidence)
static bool by_segments(const chd_symbolic* s, int m, const double* psi) {
  return psi && !s->cseg.empty() && chain_by_segments(s, m, 0.8);
}
template <bool UP>
static void scan(const chd_symbolic* s, cudaStream_t st, int t0, int m, const double* psi, double* ws) {
  const int nr = (int)s->crun.size() / 2;
  for (int step = 0; step < s->cseg_steps; ++step)
    for (int half = 0; half < 2; ++half) {
      kc_scan<UP><<<dim3(16, nr, m), 256, 0, st>>>(s->dev, t0, step, half, psi, ws);
      count_launch();
    }
}
// Psi of every inner segment (once per factor)
void chain_psi(const chd_symbolic* s, cudaStream_t st, const double* Wc, double* psi) {
  if (s->cseg.empty() || !psi) return;
  kc_psi<<<dim3((unsigned)s->cseg.size(), AMAX / PSX), 4 * PSX, 0, st>>>(s->dev, s->lvl_ptr[0], Wc, psi);
  count_launch();
}
void chain_factor(const chd_symbolic* s, cudaStream_t st, int t0, int nt, const double* X, double* Lc, double* Wc,
                  double* Dd, double* ws, double* ldet, int64_t* status) {
  kc_factor<<<nt, UPT, 0, st>>>(s->dev, t0, X, Lc, Wc, Dd, ws, status);
  count_launch();
  const Columns c = columns(s, t0, nt);
  const auto post = c.n > 0 ? kc_factor_post<true> : kc_factor_post<false>;
  post<<<column_grid(s, c, nt, 4, 1), 128, 0, st>>>(s->dev, c, Lc, Dd, ldet);
  count_launch();
}
void chain_product(const chd_symbolic* s, cudaStream_t st, int t0, int nt, const double* Lc, double* X, double* ws) {
  const Columns c = columns(s, t0, nt);
  const auto sum = c.n > 0 ? kc_band_sum<true, true> : kc_band_sum<true, false>;
  sum<<<column_grid(s, c, nt, 4, 1, s->run_amax), 128, 0, st>>>(s->dev, c, (s->run_amax + 3) / 4, Lc, X, 0, ws);
  count_launch();
}
void chain_gradient(const chd_symbolic* s, cudaStream_t st, int t0, int nt, const double* Wc, double* Sc, double* g,
                    double* Vd, double* ws, double* psi) {
  if (by_segments(s, 1, psi)) {
    const unsigned ns = (unsigned)s->cseg.size();
    kc_gradient_seg<<<ns, DNT, 0, st>>>(s->dev, t0, 1, Wc, Sc, ws);
    count_launch();
    scan<false>(s, st, t0, 1, psi, ws);
    kc_gradient_seg<<<ns, DNT, 0, st>>>(s->dev, t0, 2, Wc, Sc, ws);
    count_launch();
  } else {
    kc_gradient<<<nt, DNT, 0, st>>>(s->dev, t0, Wc, Sc, ws);
    count_launch();
  }
  const Columns c = columns(s, t0, nt);
  const auto post = c.n > 0 ? kc_grad_post<true> : kc_grad_post<false>;
  post<<<column_grid(s, c, nt, 1, 1), MT, 0, st>>>(s->dev, c, Sc, g, Vd, ws);
  count_launch();
}
void chain_hess_up(const chd_symbolic* s, cudaStream_t st, int t0, int nt, int m, const double* Wc, const double* Vd,
                   const double* Y, int64_t ldy, double* T, int64_t ldt, double* ws, const uint8_t* act,
                   const double* psi) {
  if (!act && by_segments(s, m, psi)) {
    const unsigned ns = (unsigned)s->cseg.size();
    kc_hess_up_seg<<<dim3(ns, m), UPT, 0, st>>>(s->dev, t0, 1, Wc, Y, ldy, T, ldt, ws);
    count_launch();
    scan<true>(s, st, t0, m, psi, ws);
    kc_hess_up_seg<<<dim3(ns, m), UPT, 0, st>>>(s->dev, t0, 2, Wc, Y, ldy, T, ldt, ws);
    count_launch();
  } else {
    kc_hess_up<<<dim3(nt, m), UPT, 0, st>>>(s->dev, t0, Wc, Y, ldy, T, ldt, ws, act);
    count_launch();
  }
  const Columns c = columns(s, t0, nt);
  const auto step2 = c.n > 0 ? kc_hess_m<true> : kc_hess_m<false>;
  step2<<<column_grid(s, c, nt, 1, m), MT, 0, st>>>(s->dev, c, Wc, Vd, T, ldt, act);
  count_launch();
}
void chain_hess_down(const chd_symbolic* s, cudaStream_t st, int t0, int nt, int m, const double* Wc, double* T,
                     int64_t ldt, double* ws, const double* psi) {
  const Columns c = columns(s, t0, nt);
  const auto pre = c.n > 0 ? kc_down_pre<true> : kc_down_pre<false>;
  pre<<<column_grid(s, c, nt, 4, m), 128, 0, st>>>(s->dev, c, Wc, T, ldt);
  count_launch();
  if (by_segments(s, m, psi)) {
    const unsigned ns = (unsigned)s->cseg.size();
    kc_hess_down_seg<<<dim3(ns, m), DNT, 0, st>>>(s->dev, t0, 1, Wc, T, ldt, ws);
    count_launch();
    scan<false>(s, st, t0, m, psi, ws);
    kc_hess_down_seg<<<dim3(ns, m), DNT, 0, st>>>(s->dev, t0, 2, Wc, T, ldt, ws);
    count_launch();
  } else {
    kc_hess_down<<<dim3(nt, m), DNT, 0, st>>>(s->dev, t0, Wc, T, ldt, ws);
    count_launch();
  }
}
void chain_ihess_down(const chd_symbolic* s, cudaStream_t st, int t0, int nt, int m, const double* Wc,
                      const double* Dd, const double* Rd, const double* T, int64_t ldt, double* ws) {
  const Columns c = columns(s, t0, nt);
  const auto down = c.n > 0 ? kc_ihess_down<true> : kc_ihess_down<false>;
  down<<<column_grid(s, c, nt, 1, m), MT, 0, st>>>(s->dev, c, Wc, Dd, Rd, T, ldt, ws);
  count_launch();
}
void chain_ihess_up(const chd_symbolic* s, cudaStream_t st, int t0, int nt, int m, const double* Wc, double* Y,
                    int64_t ldy, double* ws) {
  const Columns c = columns(s, t0, nt);
  const auto sum = c.n > 0 ? kc_band_sum<false, true> : kc_band_sum<false, false>;
  sum<<<column_grid(s, c, nt, 4, m, s->run_amax), 128, 0, st>>>(s->dev, c, (s->run_amax + 3) / 4, Wc, Y, ldy, ws);
  count_launch();
}
}  // namespace chd_launch
