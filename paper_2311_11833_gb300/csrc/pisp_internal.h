// Internal declarations shared by the CUDA translation units of libpisp.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "../../include/pisp.h"

namespace pisp {

// Launchers set kernel attributes (shared-memory limits) and read the SM
// count once per device: these are per-device properties, so the flags are
// indexed by the current device.
constexpr int kMaxDevices = 64;
inline int current_device() {
  int d = 0;
  if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= kMaxDevices) return 0;
  return d;
}

// Limit of a bounded wait on the device, stated in polls 64 ns apart (0: the
// default).  The polls of a long wait grow apart, so the limit is kept as the time
// asleep between them; with the polls themselves the default is about 0.4 s.
constexpr int64_t kWaitPolls = 1 << 22;
inline int64_t wait_limit_ns(int64_t polls) {
  return 64 * (polls <= 0 ? kWaitPolls : polls < INT64_MAX / 64 ? polls : INT64_MAX / 64);
}

constexpr int kCtrStride = 8;  // ints between completion counters: a 32-byte sector each

// A child as its parent's assembly needs it; mask (parents of at most 32 rows):
// the parent's rows that its update rows land on.
struct alignas(16) ChildDesc {
  int64_t fo;  // front_off
  int32_t ns, F;
  uint32_t mask;
  int32_t pad[3];
};

// Device view of the symbolic structure (all arrays live on the device).
struct SymDev {
  const int32_t* c0;         // [S] first permuted column of each supernode
  const int32_t* ns;         // [S] pivots
  const int32_t* ms;         // [S] update rows
  const int32_t* inst;       // [S] instance of each supernode
  const int64_t* front_off;  // [S+1] prefix of F^2
  const int64_t* vec_off;    // [S+1] prefix of F
  const int64_t* row_off;    // [S] offset into rows/emap
  const int32_t* child_off;  // [S+1]
  const int32_t* child;      // children, ascending
  const ChildDesc* cdesc;    // [S] their records, in the same order
  const int64_t* amap_off;   // [S+1]
  const int32_t* amap_src;   // A value index
  const int32_t* amap_dst;   // position i + j*F in the front
  const int64_t* amap_coff;  // [sum F + 1] first entry of column j of front s at vec_off[s] + j
  const int32_t* rows;       // update rows (permuted global index)
  const int32_t* emap;       // position of each update row in the parent front
  const int32_t* parent;     // [S] parent supernode or -1
  const int64_t* inv_off;    // [sum F + 1] contributions to position vec_off[s] + j
  const int32_t* inv_child;  //   contributing child
  const int32_t* inv_a;      //   its update-row index
  const int32_t* inv_cF;     //   the child's front size
  const int32_t* inv_col;    //   position in the child's front
  const int32_t* perm;       // [N] perm[new] = old
  const int32_t* iperm;      // [N] iperm[old] = new
  const int32_t* row_inst;   // [N] instance of each original row
  const int64_t* row_ptr;    // [N+1] CSR of A (original order)
  const int32_t* col;        // [nnz]
  const int64_t* at_ptr;     // [N+1] CSC of A: entries of column j at at_ptr[j]..at_ptr[j+1]
  const int32_t* at_src;     //   their CSR entry indices
  const int64_t* inv_pos;    // inverse extend-add map as positions: vec_off[child] + inv_col
  const int32_t* pcol;       // [nnz] permuted column of every CSR entry
  const int32_t* at_prow;    // [nnz] permuted row of every CSC entry
  int64_t N;
  int32_t S;
};

// Shifts and combination weights, passed by value to kernels.
struct Shifts {
  double t[PISP_K_MAX];
  double w[PISP_K_MAX];
  int32_t K;
};

// One level of the assembly forest, split by front size.
struct LevelPlan {
  // small fronts (factored in shared memory), grouped by size class
  struct Group {
    int64_t off;      // offset into the device list of small fronts
    int32_t count;    // fronts in the group
    int32_t maxF;     // largest front in the group
    int32_t cluster;  // 0: one CTA per (front, k); C > 0: clusters of C CTAs
  };
  Group groups[9];  // up to 8, 16, 32, 64 rows; clusters of 1, 2, 4, 8; the rest
  int32_t n_groups = 0;
  // big fronts (blocked factorisation in global memory)
  int64_t big_off = 0;
  int32_t big_count = 0;
  int32_t big_maxF = 0;
  int32_t big_maxns = 0;
  // tile-DAG schedule of the big fronts (see launch_factor_big_dag)
  int64_t dag_task_off = 0;   // offset into the device task list
  int32_t dag_tasks = 0;
  int64_t dag_flag_off = 0;   // offset into the device flag area (per level)
  int32_t dag_flags = 0;
  int32_t dag_owner = 0;      // 1: the tasks are owner tiles
  int32_t own_ch = 0;         //    rows per owner tile (a multiple of 32)
  // algorithmic bytes per perturbation (a + b * R) of each kernel family,
  // used for the achieved-bandwidth figures of the profiling interface
  double bytes_fsmall = 0, bytes_fbig = 0;
  double bytes_fwd_a = 0, bytes_fwd_b = 0, bytes_bwd_a = 0, bytes_bwd_b = 0;
};

// Host copies needed to size the launches of the big-front path.
struct BigFrontHost {
  int32_t F, ns;
};

// One task of the tile-DAG factorisation of a level's big fronts.  Column
// blocks are 32 wide; kind 0 assembles block j, kind 1 factors the panel of
// pivots [32p, 32p+32), kind 2 applies panel p to block j (triangular solve
// of its U rows, then the trailing update of the rows below).  flags points
// at the (front, k) pair's counters: J "updates applied" per column block,
// then P "panel done" flags.
//
// The owner schedule (kind 3) uses the same record: one task per (front b,
// perturbation k, 32-column block j, row chunk q in p), flags pointing at the
// pair's P x Q "rows released" and P x J "U rows released" flags.
enum DagKind { kDagAsm = 0, kDagPanel = 1, kDagUpdate = 2, kDagOwner = 3 };
struct DagTask {
  int32_t kind, b, k, p, j, flags;
};

// Tasks of the one-launch factorisation (factor policy 4), all levels:
//   kFacSeg8/16/32: s = offset of a group in the list of fronts of at most
//              32 rows, q = first task, j = tasks in the group; task i is (front
//              list[s + i / K], k = i % K), 256 / SEG tasks per record;
//   kFacCta  : front s, perturbation k, factored in shared memory;
//   kFacOwner: owner tile (column block j, row chunk q) of front s,
//              perturbation k; flags = offset of the (front, k) pair's
//              release flags.
enum FactorKind { kFacSeg8 = 0, kFacSeg16 = 1, kFacSeg32 = 2, kFacCta = 3, kFacOwner = 4 };
struct FactorTask {
  int32_t kind, s, k, q, j, flags;
};

// Builds the task list of one level (b indexes the level's big-front list).
void build_dag_tasks(const BigFrontHost* big, int32_t nbig, int32_t K, std::vector<DagTask>& out,
                     int32_t& nflags);
// Owner tiles (32-column block j, chunk q of CH rows) of one level, sorted by
// (j, q) so that a tile only waits on tiles with smaller tickets; the record
// carries q in its p field.
void build_owner_tasks(const BigFrontHost* big, int32_t nbig, int32_t K, int32_t CH,
                       std::vector<DagTask>& out, int32_t& nflags);

// ---- factor (factor.cu) ----
// Each launcher returns the number of kernels launched (>= 0) or -1 on a
// launch error.  Small fronts of one level (shared-memory path):
int launch_factor_small(int precision, const SymDev& sd, const LevelPlan& lp,
                        const int32_t* d_small, const double* vals, const double* D,
                        const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol,
                        cudaStream_t st);
// One size-class group of a level (the groups of a level are independent):
int launch_factor_small_group(int precision, const SymDev& sd, const LevelPlan& lp, int g,
                              const int32_t* d_small, const double* vals, const double* D,
                              const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol,
                              cudaStream_t st);
// Big fronts of one level (blocked path):
int launch_factor_big(int precision, const SymDev& sd, const LevelPlan& lp, const int32_t* d_big,
                      const BigFrontHost* big_host, const double* vals, const double* D,
                      const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol,
                      cudaStream_t st);
// Big fronts of one level as one persistent launch over the level's task
// list (tile DAG, or owner tiles when lp.dag_owner); ticket (1 int)
// and flags (lp.dag_flags ints) must be zero; err is set if a bounded
// dependency wait gave up.  tc != 0: FP32 owner-tile updates on the tensor
// cores (3xTF32, tcgen05).
int launch_factor_big_dag(int precision, const SymDev& sd, const LevelPlan& lp, const int32_t* d_big,
                          const DagTask* tasks, int* ticket, int* flags, int* err,
                          const double* vals, const double* D, const Shifts& sh, void* fronts,
                          int32_t* status, int32_t* badcol, int tc, cudaStream_t st);
// The whole factorisation in one persistent launch (factor policy 4): ticket
// (1 int), fdone (S*K counters, kCtrStride apart) and flags must be zero; need[s]
// = the tasks of the children of s (per k).
int launch_factor_persistent(int precision, const SymDev& sd, const FactorTask* tasks, int ntasks, int* ticket,
                             int* fdone, const int* need, int* flags, int* err, const int32_t* wlist,
                             const double* vals, const double* D, const Shifts& sh, void* fronts,
                             int32_t* status, int32_t* badcol, int CH, size_t smem, int64_t polls, int tc,
                             int ctas, cudaStream_t st);
// widest front the one-launch factorisation keeps in shared memory (wider:
// owner tiles), and its dynamic shared memory per CTA
int persistent_cta_front_limit(int precision);
size_t factor_persistent_smem(int precision, int CH, bool has_owner, int maxCtaF);
size_t tc_staging_bytes();  // more of it for the tensor-core form
// largest front the tile-DAG path takes (its panel must fit in shared memory)
int max_dag_front(int precision);
// rows per owner tile for a level whose widest front is maxF (tc != 0: leave
// room for the tensor-core staging)
int owner_chunk_rows(int precision, int maxF, int tc);
// largest front (in elements of the given precision) the shared-memory path takes
int small_front_limit(int precision);
// CTAs per cluster for a front of size F factored in distributed shared
// memory: 0 for F <= 64 (single-CTA kernel), -1 if the front does not fit
// (blocked path in global memory)
int front_cluster_size(int F, int precision);
// largest front the blocked path can take (its panel must fit in shared memory)
int max_big_front(int precision);
// widest front a solve takes
int max_solve_front(int precision);

// ---- solve (solve_persistent.h; solve.cu) ----
// Work unit of the solves: 16 bytes, read at once.  x = kind | d << 4.
//   kUnitSeg8/16/32 (forward, and backward with one right-hand side, or with many
//     pivots to few right-hand sides): 256 / SEG consecutive segment tasks of one group (a task = one front, a group of d
//     consecutive shifts, one chunk of 8 right-hand sides or the only one): a =
//     the group's first front record, b = first task, c = tasks in the group;
//   kUnitCol (backward, several right-hand sides): 8 consecutive warp tasks of
//     one group (a task = one front, one group of 32 columns (k, r)), a, b, c as
//     above;
//   kUnitCta: one front (record a) with at most 32 pivots, for the shift b and
//     RHS chunk c, or for the column group b;
//   kUnitWide: a front (record a) with more than 32 pivots, b = shift | d << 4 |
//     q << 8 with q the 256 rows taken, RHS chunk c of d right-hand sides (as many
//     in all units of a direction).
enum UnitKind { kUnitSeg8 = 0, kUnitSeg16 = 1, kUnitSeg32 = 2, kUnitCol = 3, kUnitCta = 4, kUnitWide = 5 };
struct SolveUnit {
  int32_t x, a, b, c;
};

// What a solve task needs to know of its front, in unit-list order: one
// 64-byte read in place of a chain of lookups.  needF = its children's tasks,
// needB = its parent's, as the completion counters count them.
enum FrontWhole { kSelfWhole = 1, kParentWhole = 2 };
struct alignas(16) FrontDesc {
  int32_t c0, ns, F, inst;
  int64_t fo, vo;  // prefix sums of F^2 and F
  int64_t ro;      // first update row in `rows`
  int32_t parent, s;
  int32_t needF, needB;
  int32_t flag;   // more than 32 pivots: first of its counters in `wide`
  int32_t whole;  // FrontWhole: counted at group 0 only
};

constexpr int kSolveChunk = 8;  // right-hand sides of a segment task, where there are several

// xd_mode: what a backward solve does with its FP64 output
enum XdMode { kXdStore = 0, kXdAdd = 1 };

// Arguments of one solve launch (solve_persistent.h says what the arrays hold).
template <typename T>
struct SolveArgs {
  const FrontDesc* desc;
  const int64_t *inv_off, *inv_pos;
  const int32_t *rows, *perm;
  const SolveUnit* units;
  int32_t first, nunits;  // the launch's units are first .. first + nunits - 1
  const int* ucount;      // length of a compacted list, or nullptr: nunits
  const uint8_t* act;     // per-instance flags of the adaptive sweeps, or nullptr: all
  int* ticket;            // zero
  int* done;              // [S][NG] finished tasks, zero; nullptr (one launch per stage): nothing to wait for
  int* wide;              // solved blocks per (front with more than 32 pivots, shift, chunk), zero
  int* err;               // set if a wait gave up
  int64_t wait_ns;        // most time asleep in one wait
  const T* fronts;
  const double* b;        // broadcast right-hand side, or nullptr: rk
  const T* rk;
  T* V;
  T* xt;
  double* xd;             // FP64 output, or nullptr
  int32_t xd_mode, R, K, RV, RX, vec, vecd;
  int32_t NG;     // groups of the completion counters: K shifts, or ceil(K RV / 32) column groups
  int32_t stage;  // per-warp shared memory of the column tasks (set by the launch)
};

// row strides of the vectors for R right-hand sides: in the factor precision
// (16-byte accesses) and in FP64
inline int32_t rhs_stride(int precision, int32_t R) {
  const int32_t n = precision == PISP_FP32 ? 4 : 2;
  return R <= 2 && R < n ? R : (R + n - 1) / n * n;
}
inline int32_t rhs_stride64(int32_t R) { return R == 1 ? 1 : (R + 1) / 2 * 2; }

// One launch of the forward (L, or U^T with trans) or backward (U, L^T) solve;
// ctas = resident CTAs per SM it is compiled for with several right-hand sides
// (2, 3, 4; <= 0, or transposed: 2); wide = the most right-hand sides of a task of a
// front with more than 32 pivots, 0 if there is none; segs: the list has backward
// segments of several right-hand sides.  Returns the kernels launched or -1.
template <typename T, bool FWD>
int launch_solve_dir(bool trans, const SolveArgs<T>& a, int32_t nunits, int32_t wide, bool segs, int32_t ctas,
                     cudaStream_t st);
constexpr int kWideUnitRows = 256;  // rows of a task of a front with more than 32 pivots
int launch_combine(const SymDev& sd, const double* X, const Shifts& sh, int32_t R, double* x,
                   cudaStream_t st);
// The instances still iterating in the adaptive sweeps (device arrays
// written by the stopping test): act[g] flags, their number *nact, their ids
// ai[0..nact) in increasing order, and arow[q] = the rows of ai[0..q)
// (arow[nact] = all their rows).  Active row a belongs to instance ai[q] for
// the largest q with arow[q] <= a, at original row inst_off[ai[q]] + a - arow[q].
struct ActiveSet {
  const uint8_t* act;
  const int32_t* nact;
  const int32_t* ai;
  const int64_t* arow;
  const int64_t* inst_off;  // [G+1] first original row of each instance
};
// Rows a residual launch covers: every row; every row with Rk = 0 on the rows
// of instances that have stopped (whose correction is then exactly 0, for a
// solve that is not gated); only the rows of the active set.
enum ResidualMode { kResAll = 0, kResZeroStopped = 1, kResActive = 2 };
int launch_residual_per_k(int precision, const SymDev& sd, const double* vals, const double* D,
                          const Shifts& sh, const double* b, const double* X, int32_t R,
                          void* Rk, const ActiveSet& as, int mode, cudaStream_t st);
// Per instance g of the active set: X += Y on its rows, then per RHS r the
// largest |Y| and |X| over its rows and all k, atomically maxed into
// dmax/xmax [G][R] (zero on entry) as bit patterns.
int launch_refine_stats(int precision, const SymDev& sd, const ActiveSet& as, double* X, const void* Y, int32_t K,
                        int32_t R, unsigned long long* dmax, unsigned long long* xmax, cudaStream_t st);
// One CTA: the stopping test after sweep s = *sweep + 1 (s >= S: every
// instance stops), *sweep = s, nsw[g] = the sweeps instance g took, dmax /
// xmax zeroed again, then the active set: pre[g] = the active instances
// before g (G+1 ints), *nact, ai [G], arow [G+1].  has_cond: sets the
// conditional `cond` of a device-side sweep loop to continue while an
// instance is active and s < S.
int launch_refine_decide(int32_t G, int32_t R, double tol, int32_t S, int32_t* sweep,
                         cudaGraphConditionalHandle cond, int has_cond, uint8_t* act, unsigned long long* dmax,
                         unsigned long long* xmax, double* prevd, int32_t* nsw, int32_t* pre, int32_t* nact,
                         int32_t* ai, int64_t* arow, const int64_t* inst_off, cudaStream_t st);
// Every instance active, no sweep done: act, pre, *nact, ai, arow, *sweep.
int launch_refine_init(int32_t G, uint8_t* act, int32_t* pre, int32_t* nact, int32_t* ai, int64_t* arow,
                       const int64_t* inst_off, int32_t* sweep, cudaStream_t st);
// In-order compaction of the forward and backward unit lists to the units
// whose instance range [lo, hi] (rf, rb: int32 pairs) holds an active
// instance, into cf / cb with lengths in ucount[0..1]; cnt holds
// compact_scratch(nf, nb) ints of scratch.  Returns the kernels launched.
int compact_scratch(int32_t nf, int32_t nb);
int launch_compact_units(const SolveUnit* uf, const int32_t* rf, int32_t nf, SolveUnit* cf, const SolveUnit* ub,
                         const int32_t* rb, int32_t nb, SolveUnit* cb, const int32_t* pre, int32_t* cnt,
                         int32_t* ucount, cudaStream_t st);
// FP64 residuals of the transposed perturbed systems (adjoint sweeps)
int launch_residual_T_per_k(int precision, const SymDev& sd, const double* vals, const double* D,
                            const Shifts& sh, const double* g, const double* Lam, int32_t R,
                            void* Rk, cudaStream_t st);
int launch_residual(const SymDev& sd, const double* vals, const double* b, const double* x,
                    int32_t R, double* r, cudaStream_t st);
int launch_axpy(int64_t n, const double* y, double* x, cudaStream_t st);
int launch_grad_values(const SymDev& sd, const double* Lam, const double* X, const Shifts& sh,
                       int32_t R, double* grad, cudaStream_t st);
int launch_fill_nan_failed(const SymDev& sd, const int32_t* status, int32_t K, int32_t R,
                           double* x, cudaStream_t st);

}  // namespace pisp
