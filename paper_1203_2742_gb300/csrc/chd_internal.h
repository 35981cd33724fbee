// Internal declarations shared by the host symbolic phase, the C ABI and the
// CUDA kernels of the chordal log-det barrier library.
#pragma once

#include <cuda_runtime_api.h>

#include <cstdint>
#include <vector>

#include "chordal_barrier.h"

// One record per position of the task lists (aligned with task_fronts):
// what a warp needs to start a front with one load.  flags:
//   WM_PREV_CHILD      the previous front of the task is a child of this one
//   WM_NEXT_PARENT     the next front of the task is this one's parent
//   WM_ONLY_CHILD_PREV this front's only child is the previous front of the task
constexpr int32_t WM_PREV_CHILD = 1, WM_NEXT_PARENT = 2, WM_ONLY_CHILD_PREV = 4;
struct alignas(16) WMeta {
  int64_t col0;      // first column of N_k
  int64_t base;      // colptr[col0]: offset of the front's values
  int64_t f_off;     // workspace offset (one right-hand side)
  int64_t rows_off;  // rows_ptr[k]
  int64_t d_off;     // offset of the n x n block
  int64_t v_off;     // offset of the a x a block
  int32_t k, n, J, flags;
  int32_t ch_beg, ch_end;  // children of k in ch[ch_beg..ch_end)
  int32_t task, place;     // the task that holds the front, and where in it
};

// Grouped tier (group_tier.cu): the fronts whose gradient, Hessian and
// inverse-Hessian steps run as one launch per step over many fronts.
constexpr int kGroupBlock = 32;       // rows per block of the assembly and of the update tiles
constexpr int kGroupThin = 16;        // thin fronts: up to this many columns
constexpr int kGroupFactor = 32;      // fronts up to this many columns factor in one launch per sub-level
constexpr int kGroupCols = 256;       // widest front of the tier
// sub-levels with a front of more children than this use add_children: 40 children gain
// 7 %, 400 a third, and fronts of few children lose up to 10 % (group_tier.cu)
constexpr int kManyChildren = 64;
// the grouped completion ends the N x N part of a front in one CTA from 33 columns
// on, 0.2 to 0.4 ms up to here; wider ones by the rule at wide_by_sequence
constexpr int kGroupComplete = 64;
constexpr int kGroupSmem = 200 << 10; // dynamic shared memory a kernel of the tier may use
struct alignas(16) GFront {
  int64_t base, f_off, fp_off, d_off, v_off, rel_off;  // values, workspace, parent's workspace, D_NN, V_k, rel of A_k
  int32_t k, n, a, J, Jp;
  int32_t lrb, nb;         // row blocks of 8 << lrb rows of A_k, nb of them (at least one)
  int32_t nbn;             // blocks of N_k
  int32_t ch_beg, ch_end;  // children (extend-add order) in gch
  int32_t pad[2];
};
struct alignas(16) GChild {
  int64_t u_off;    // workspace offset of the child's update block
  int64_t rel_off;  // positions of its A in the parent, in `rel`
  int32_t Jc, k;
  int32_t ptr_off;  // gptr[ptr_off + b]: its first row in block b of the parent
  int32_t pad;
};

// one segment of a chain run (chain_tier.cu): columns s .. e - 1 of run
// `run` (index among level 0's runs), p-th of P from the bottom
struct alignas(16) ChainSeg {
  int32_t run, p, P, s, e, pad;
  int64_t psi;  // offset of its a x a matrix Psi
};
// grouped inverse of V_k: one front
struct alignas(16) GJob {
  int64_t v_off, w_off;  // V_k slot, workspace (a x a)
  int32_t a, k;
};

// grouped completion: one front, blocks of its S-front in the order (A, N)
struct alignas(16) GComp {
  int64_t base, f_off, v_off, d_off, rows_off;
  int32_t k, n, a, J, nA, pad;
};

// Device copy of the symbolic data, passed by value to every kernel.
struct SymDev {
  int64_t n = 0;
  int64_t nsn = 0;             // number of supernodes (fronts)
  const int64_t* colptr = nullptr;   // n+1: CSC of V (analysed order)
  const int32_t* rowind = nullptr;   // nnz: row indices of the CSC (sorted per column)
  const int64_t* sn_ptr = nullptr;   // nsn+1: N_k = [sn_ptr[k], sn_ptr[k+1])
  const int64_t* sn_par = nullptr;   // nsn: clique-tree parent or -1
  const int64_t* rows_ptr = nullptr; // nsn+1: offsets of J_k in `rows`/`rel`
  const int32_t* rel = nullptr;      // position of A_k[r] inside J_par(k) (A part only)
  const int32_t* rows = nullptr;     // J_k (N_k then A_k, increasing), at rows_ptr[k]
  const int64_t* ch_ptr = nullptr;   // nsn+1: children of k in ch[ch_ptr[k]..)
  const int32_t* ch = nullptr;
  const int64_t* ea_ptr = nullptr;   // nsn+1: children whose update blocks k adds (a leaf
  const int32_t* ea = nullptr;       //   group contributes through its first member only)
  const int64_t* f_off = nullptr;    // nsn+1: per-front workspace offsets (doubles)
  const int64_t* d_off = nullptr;    // nsn+1: per-front n_k*n_k block offsets
  const int64_t* v_off = nullptr;    // nsn+1: per-front a_k*a_k block offsets
  const int32_t* task_ptr = nullptr; // ntask+1
  const int32_t* task_fronts = nullptr;
  const WMeta* tmeta = nullptr;      // aligned with task_fronts
  const int32_t* small_fronts = nullptr;  // fronts not in the dense tier
  int64_t small_count = 0;
  const int32_t* cta_fronts = nullptr;    // fronts of the CTA and wide warp tiers (completion)
  int64_t cta_count = 0;
  const int32_t* warp_fronts = nullptr;   // fronts of the warp tier
  int64_t warp_count = 0;
  const int32_t* plain_fronts = nullptr;  // fronts of the warp, wide and CTA tiers (no dense, no group)
  int64_t plain_count = 0;
  // fronts whose update blocks reach front k's: [sub_lo[k], sub_hi[k]] (its
  // subtree, plus the other members when k heads a leaf group)
  const int32_t* sub_lo = nullptr;
  const int32_t* sub_hi = nullptr;
  // pruned Hessian factor (§5.5): per right-hand side y, act[y * nsn + k] != 0
  // iff Y has a nonzero in the columns of that range; null: every front active
  const uint8_t* act = nullptr;
  const int64_t* fc_off = nullptr;        // factored completion: scratch offsets (per front)
  const int32_t* fc_fronts = nullptr;     // factored completion: CTA-handled fronts by level
  // grouped tier: fronts by sub-level, their children, and the work lists
  // (front, low/high 16 bits or block index)
  const GFront* gf = nullptr;
  const GChild* gch = nullptr;
  const int32_t* gptr = nullptr;
  const int2 *gt_up = nullptr, *gt_row = nullptr, *gt_asm = nullptr, *gt_p = nullptr, *gt_gat = nullptr,
             *gt_nn = nullptr, *gt_asmf = nullptr, *gt_wb = nullptr, *gt_fr = nullptr, *gt_out = nullptr;
  const int32_t* gleg = nullptr;
  const ChainSeg* cseg = nullptr;
  const int2* crun = nullptr;  // runs of at least three segments: first segment, number of segments
  const GJob* gj = nullptr;
  const int2 *gv_all = nullptr, *gv_sol = nullptr, *gv_upd = nullptr;
  const int32_t* gv_small = nullptr;
  const GComp* gc = nullptr;
  const int2 *gc_all = nullptr, *gc_sol = nullptr, *gc_upd = nullptr, *gc_back = nullptr, *gc_b = nullptr;
  const int32_t *gc_thin = nullptr, *gc_wide = nullptr, *gc_root = nullptr;
  const int64_t* inst_sn = nullptr;       // instances x supernode ranges
  int64_t ninst = 1;
  int64_t f_total = 0;               // workspace doubles per right-hand side
  int64_t d_total = 0;
  int64_t v_total = 0;
};

struct chd_symbolic {
  int64_t n = 0;
  std::vector<int64_t> perm;       // perm[new] = old
  std::vector<int64_t> colptr;     // n+1
  std::vector<int32_t> rowind;     // nnz(V)
  int64_t nsn = 0;
  std::vector<int64_t> sn_ptr;     // nsn+1
  std::vector<int64_t> sn_par;     // nsn
  std::vector<int64_t> rows_ptr;   // nsn+1
  std::vector<int32_t> rows;       // J_k, N_k first then A_k
  std::vector<int32_t> rel;        // aligned with rows; -1 on the N part
  std::vector<int64_t> ch_ptr;
  std::vector<int32_t> ch;
  std::vector<int64_t> ea_ptr;  // children for the extend-add (see SymDev)
  std::vector<int32_t> ea;
  // leaf groups: supernodes [grp_first[g], grp_first[g] + grp_count[g]) are
  // one-column leaves of one parent with the same A; grp_of[k] = g or -1
  std::vector<int64_t> grp_first, grp_count;
  std::vector<int32_t> grp_of;
  std::vector<int64_t> f_off, d_off, v_off;
  // schedule: tasks are front sequences processed by one CTA; launches
  // group tasks by level (bottom-up order); lvl_ptr indexes tasks.
  std::vector<int32_t> task_ptr, task_fronts, lvl_ptr;
  std::vector<WMeta> tmeta;  // aligned with task_fronts
  // per level: the last lvl_big[l] tasks of the level are single big fronts
  // run by the multi-CTA dense tier
  std::vector<int32_t> lvl_big;
  // per level: the first lvl_r32[l] + lvl_r64[l] tasks are chain-tier runs
  // (|J| <= 32, then |J| <= 64; all zero unless chain_runs)
  std::vector<int32_t> lvl_r32, lvl_r64;
  // lowest level that waits for a chain run, and whether other tasks lie below it
  int32_t run_join = 0, run_overlap = 0;
  // largest a of the runs, and the longest run if a grid of runs x columns of it
  // is full enough (Columns in chain_tier.cu), else 0
  int run_amax = 0, run_lmax = 0;
  // segments of the runs (none when the serial kernels are faster), (first,
  // count) of the runs of at least three, doubles of all Psi, most inner segments
  // of a run; modelled times in us: longest run, longest segment, all runs, one
  // step of the windows
  std::vector<ChainSeg> cseg;
  std::vector<int32_t> crun;
  int64_t cseg_psi = 0;
  int cseg_steps = 0;
  double cseg_serial = 0, cseg_column = 0, cseg_total = 0, cseg_step = 0;
  // per level l, five counts at 5*l: chain runs (|J| <= 32), chain runs
  // (|J| <= 64), warp, wide warp and dense-tier tasks (chd_symbolic_schedule)
  std::vector<int32_t> lvl_counts;
  // per level, after the runs: lvl_warp[l] warp-tier tasks (|J| <= 32),
  // the next lvl_w64[l] wide warp-tier tasks (|J| <= 64)
  std::vector<int32_t> lvl_warp, lvl_w64;
  std::vector<char> is_big;  // per supernode
  std::vector<int32_t> tier;  // per supernode: 0 warp, 3 wide warp, 1 CTA, 2 dense, 4 leaf group
  std::vector<int32_t> small_fronts;
  std::vector<int32_t> cta_fronts;
  std::vector<int32_t> warp_fronts;
  std::vector<int32_t> big_fronts;
  std::vector<int32_t> plain_fronts;
  std::vector<int32_t> sub_lo, sub_hi;
  double flops[5] = {0, 0, 0, 0, 0};
  // independent instances analysed together (chd_analyze_batch): instance i
  // owns columns [inst_n[i], inst_n[i+1]), values [inst_nnz[i], inst_nnz[i+1])
  // and supernodes [inst_sn[i], inst_sn[i+1]) of the analysed numbering
  std::vector<int64_t> inst_n, inst_nnz, inst_sn;
  int64_t max_front = 0;
  int tc_mode = 0;  // chd_opts.tc_products
  // completion with factored update matrices (chd_opts.completion = 1):
  // fronts with a_k > 0 by depth in the clique tree, parents first; the
  // per-front sequence runs one CTA per front (fc_fronts, level l at
  // [fc_lvl[l], fc_lvl[l+1])) or the dense tier (fc_big, fc_big_lvl);
  // fc_off: scratch offset (doubles) of the front's reduction within its
  // level; fc_total: largest level's scratch; fc_flops: Cholesky of every
  // V_k (independent form) and the factored form's arithmetic
  int completion_mode = 0;
  std::vector<int64_t> fc_off;
  std::vector<int32_t> fc_fronts, fc_lvl, fc_big, fc_big_lvl;
  int64_t fc_total = 0;
  double fc_flops[2] = {0, 0};
  // grouped tier: sub-levels glvl[l] .. glvl[l+1]) of level l (the i-th fronts
  // of the level's CTA tasks, and with the first the thin dense fronts);
  // gidx: index in gf or -1.  Work lists as (front, code) pairs with the
  // sub-levels' ranges gs_*; gs_rn: largest row block (doubles) of a
  // sub-level, gs_np: most factor panels, gs_thin: whether it has fronts of
  // at most kGroupFactor columns; gleg: CTA-tier fronts outside the tier.
  std::vector<GFront> gf;
  std::vector<GChild> gch;
  std::vector<int32_t> gptr, gidx, glvl;
  std::vector<int32_t> gt_up, gt_row, gt_asm, gt_p, gt_gat, gt_nn, gt_asmf, gt_wb, gt_fr, gt_out, gleg;
  std::vector<int32_t> gs_up, gs_row, gs_asm, gs_p, gs_gat, gs_asmf, gs_wb, gs_out, gs_rn, gs_np, gs_thin, gs_many, gs_leg;
  int g_rnmax = 0, g_nmax = 0, g_amax = 0;
  // grouped inverse: fronts by decreasing a, their lower tiles, and per panel
  // of 32 columns the row blocks to solve and the tiles to update
  std::vector<GJob> gj;
  std::vector<char> in_gj;  // per supernode
  std::vector<int32_t> gv_all, gv_sol, gv_upd, gv_sol_ptr, gv_upd_ptr;
  std::vector<int32_t> gv_small;  // supernodes of at most 32 ancestors
  // grouped completion: fronts by decreasing a and the lists of its steps;
  // gc_thin: indices of fronts of at most 32 columns, gc_wide: supernodes of
  // the others, gc_root: supernodes of more than 32 columns and no ancestors, one
  // CTA each, gc_rest: CTA-tier supernodes outside the grouped form, which take the
  // dense tier's sequences
  std::vector<GComp> gc;
  std::vector<char> in_gc;
  std::vector<int32_t> gc_all, gc_sol, gc_upd, gc_sol_ptr, gc_upd_ptr, gc_back, gc_b, gc_thin, gc_wide, gc_root, gc_rest;
  int gc_amax = 0;
  // device mirror
  SymDev dev;
  void* dev_buf = nullptr;
  int dev_id = -1;
};

// Execution resources of the dense tier: side streams on which independent
// big fronts run concurrently (forked from and joined back to the caller's
// stream with events), and one scratch slice per stream (slice 0: the
// caller's stream) for split-K partial products, ending with the counter of
// the Cholesky panel kernel.  The first kWideSlices slices are large; the
// rest hold the counter and small partial products only.
constexpr int kSideStreams = 32;
// The last of the side streams take second halves of dense fronts (Posts in
// kernels.cu), with the scratch sizes of the caller's stream.  Two: four gave
// the same times (er5000 factor 5.95 against 5.98 ms), and four with the other
// side streams' scratch lost 2 of 41 ms on the Hessian of 64 right-hand sides
// of a 150 x 150 grid, whose products then ran two right-hand sides at a time.
constexpr int kPostStreams = 2;
constexpr int kAuxStreams = 3;  // chain runs, warp tier, wide warp tier beside the caller's stream
constexpr int kWideSlices = 9;
struct Exec {
  int nside = 0;
  cudaStream_t side[kSideStreams] = {};
  cudaEvent_t fork = nullptr;
  cudaEvent_t join[kSideStreams] = {};
  double* slice[kSideStreams + 1] = {};
  int64_t slice_cap[kSideStreams + 1] = {};
  // scratch of the tensor-core products (digit planes), per stream slot
  void* tc[kSideStreams + 1] = {};
  size_t tc_cap[kSideStreams + 1] = {};
  int64_t* status = nullptr;  // the factor's status (tensor-core timeouts)
  int tc_mode = 0;
  double* psi = nullptr;      // chain segments' matrices, when the pattern has segments
  // streams for the other launches of a level, with their fork and join events
  int naux = 0;
  cudaStream_t aux[kAuxStreams] = {};
  cudaEvent_t aux_fork[kAuxStreams] = {}, aux_join[kAuxStreams] = {};
};

// Whether m right-hand sides of the chain runs are faster by segments than `gain`
// times the serial kernels, with the times of the analysis (us): the serial
// kernels take an SM per run and right-hand side, at least as long as the longest
// run; by segments every column is done twice, all segments sharing the SMs, and
// every inner segment adds two launches of small products over the runs that have
// one (kMaxScanRuns of them at most: a grid dimension indexes them).
constexpr size_t kMaxScanRuns = 65535;
inline bool chain_by_segments(const chd_symbolic* s, int m, double gain) {
  const double share = m * s->cseg_total / 152.0, runs = (double)s->crun.size() / 2;
  const double serial = share > s->cseg_serial ? share : s->cseg_serial;
  const double seg = 2.0 * (share > s->cseg_column ? share : s->cseg_column) +
                     s->cseg_steps * s->cseg_step * (m * runs > 40.0 ? m * runs / 40.0 : 1.0);
  return seg < gain * serial;
}

// Formation of V_k^{-1} by the size a of V_k: up to kInvVGroup rows the
// grouped kernels over all fronts at once (kv_* in group_tier.cu; 12000 fronts
// of 61 rows: 9.4 ms with one CTA per front, 5.0 ms grouped), beyond that a launch
// sequence per front whose trailing products run on the tensor cores.  The upper
// factor of V_k (Hessian factor) has no grouped form: one CTA (k_inv_v) below
// kInvVMulti rows, else a sequence per front.
constexpr int kInvVMulti = 96;
constexpr int kInvVGroup = 512;

// What one dense-tier front sequence runs with: its stream, the split-K
// scratch slice (may be null), the tensor-core scratch (may be null), the
// factor's status and the tensor-core mode of the analysis.
struct Slot {
  cudaStream_t st = nullptr;
  double* xs = nullptr;
  int64_t xcap = 0;
  void* tc = nullptr;
  size_t tc_cap = 0;
  int64_t* status = nullptr;
  int tc_mode = 0;
};

// A captured launch sequence of one kind of call (see capi.cpp): the
// arguments it was captured with, and the launch count of one replay.
struct GraphKey {
  const void* p[4] = {nullptr, nullptr, nullptr, nullptr};
  int64_t v[4] = {0, 0, 0, 0};
  bool operator==(const GraphKey& o) const {
    for (int i = 0; i < 4; ++i)
      if (p[i] != o.p[i] || v[i] != o.v[i]) return false;
    return true;
  }
};
struct GraphSlot {
  GraphKey key;
  bool seen = false;
  bool capture_failed = false;
  cudaGraphExec_t exec = nullptr;
  int64_t launches = 0;
};
enum GraphKind {
  G_FACTOR = 0,
  G_GRADIENT,
  G_HESSIAN,
  G_INV_HESSIAN,
  G_INV_V,
  G_COMPLETE,
  G_PRODUCT,
  G_HFACTOR,
  G_HFACTOR_ADJ,
  G_HFACTOR_SPARSE,
  G_Q,
  G_KINDS
};

// A factor object: device-resident factor blocks, cached projected inverse
// and the per-right-hand-side front workspace (all owned by the object).
struct chd_factor {
  chd_symbolic* sym = nullptr;
  cudaStream_t stream = nullptr;
  void* block = nullptr;  // one allocation holding everything below but ws
  double* Lc = nullptr;
  double* Wc = nullptr;
  double* Sc = nullptr;
  double* Dd = nullptr;
  double* Vd = nullptr;
  double* Rd = nullptr;      // per front, once have_R: V_k^{-1} (lower), or chol(V_k) for dense-tier fronts
  double* Qd = nullptr;      // per front, once have_Q: Cholesky factor of P V_k P (P the order reversal),
                             // i.e. the upper factor Q of V_k = Q Q^T held reversed (Hessian factor, §5.4)
  double* ldet = nullptr;
  double* scalar = nullptr;  // [0] log det
  int64_t* status = nullptr; // [0] code, [1] supernode, [2] column
  double* ws = nullptr;      // per-right-hand-side front workspace
  double* fcs = nullptr;     // factored completion: scratch of the reductions (own allocation)
  Exec ex;                   // dense-tier streams and split-K scratch
  double* inst_sum = nullptr;  // per-instance log det sums (batched symbolic objects)
  int64_t ws_rhs = 0;        // capacity in right-hand sides
  void* act_buf = nullptr;   // pruned Hessian factor: int32 counts, then uint8 flags, per (RHS, front)
  int64_t act_rhs = 0;       // capacity of act_buf in right-hand sides
  size_t ws_limit = 0;       // caller's cap on the workspace (0: library default)
  bool have_S = false;
  bool have_psi = false;     // ex.psi belongs to the current factor
  bool have_R = false;
  bool have_Q = false;
  // CUDA graphs of the launch sequences, replayed on the private stream gs
  bool graphs_on = true;
  int64_t graph_limit = 8192;  // longest launch sequence that is captured
  cudaStream_t gs = nullptr;
  cudaEvent_t g_in = nullptr, g_out = nullptr;
  GraphSlot graphs[G_KINDS];
};

// Host helpers implemented in symbolic.cpp
chd_status chd_symbolic_build(int64_t n, const int64_t* colptr, const int32_t* rowind,
                              const chd_opts& opts, chd_symbolic* s);
chd_status chd_symbolic_upload(chd_symbolic* s);
chd_status chd_order_pattern(int64_t n, const int64_t* colptr, const int32_t* rowind, const chd_opts& opts,
                             std::vector<int64_t>& perm);

inline int64_t front_n(const chd_symbolic* s, int64_t k) { return s->sn_ptr[k + 1] - s->sn_ptr[k]; }
inline int64_t front_J(const chd_symbolic* s, int64_t k) { return s->rows_ptr[k + 1] - s->rows_ptr[k]; }
