// C ABI of libpisp: handle, symbolic upload, level plans and the host-side
// orchestration of the level-scheduled factor / solve launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <climits>
#include <cmath>
#include <cstring>
#include <memory>
#include <new>
#include <stdexcept>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/pisp.h"
#include "pisp_internal.h"
#include "symbolic.h"

namespace {

struct Buf {
  void* p = nullptr;
  size_t bytes = 0;
  ~Buf() { release(); }
  void release() {
    if (p) cudaFree(p);
    p = nullptr;
    bytes = 0;
  }
  // grow-only device buffer; returns false on allocation failure
  bool ensure(size_t want) {
    want = std::max<size_t>(want, 256);
    if (want <= bytes) return true;
    release();
    if (cudaMalloc(&p, want) != cudaSuccess) {
      cudaGetLastError();
      p = nullptr;
      return false;
    }
    bytes = want;
    return true;
  }
  template <typename T>
  T* as() const { return reinterpret_cast<T*>(p); }
};

thread_local std::string g_last_error;  // for calls without a valid handle, per host thread

}  // namespace

struct pisp_handle {
  int device = 0;
  cudaStream_t stream = nullptr;
  std::string err;
  bool analyzed = false, factored = false, solved = false;
  pisp::Symbolic sym;
  double analyze_ms = 0.0;
  // device symbolic
  Buf c0, ns, ms, inst, front_off, vec_off, row_off, child_off, child, cdesc, amap_off, amap_src,
      amap_dst, amap_coff, rows, emap, perm, iperm, row_inst, row_ptr, col, parent, inv_off, inv_child, inv_a, inv_pos,
      inv_cF, inv_col, at_ptr, at_src, pcol, at_prow;
  // persistent solve schedule (depends on K and R)
  int32_t schedule = 0;
  int32_t factor_policy = 0;
  int32_t units_K = 0, units_R = 0;
  int32_t n_units_f = 0, n_units_b = 0;
  int32_t units_wide[2] = {};                 // right-hand sides of a task of a front with more than 32 pivots, per direction
  bool units_segs = false;                    // the backward list has segments of several right-hand sides
  size_t ctr_tickets = 0, ctr_half = 0;       // tickets, and all counters, of one direction
  std::vector<int32_t> lvl_units_f, lvl_units_b;  // first unit of each stage (one launch per stage)
  // front records in unit-list order; counters, forward then backward: the
  // tickets, the finished tasks per (front, column group), the solved blocks of
  // the fronts with more than 32 pivots
  Buf units_f, units_b, desc, ctr, serr;
  // adaptive FP64 residual sweeps (pisp_set_refinement): stopping tolerance
  // (0 = every sweep for every instance), the instance range [lo, hi] of
  // each persistent solve unit, the compacted unit lists and their lengths,
  // per-instance flags / sweep counts / correction sizes, instance offsets
  double sweep_tol = 0.0;
  int32_t last_sweeps = 0;
  bool last_adaptive = false, any_solve = false;
  bool last_loop = false;       // the last solve's sweeps ran as a device-side loop
  int32_t loop_kernels = 0;     // kernels per iteration of that loop
  cudaStream_t body_stream = nullptr;  // captures the loop's body
  std::vector<double> inst_w;  // solve work of each instance (front entries)
  // supernodes by level, and by instance, the widest fronts of each first
  std::vector<int32_t> by_level, by_inst;
  Buf rng_f, rng_b, units_fc, units_bc, ucount, r_act, r_pre, r_dmax, r_xmax, r_prevd, r_nsw, d_inst_off;
  Buf r_nact, r_ai, r_arow, r_ccnt, r_sweep;
  // bounded waits of the persistent solves: polls before giving up (0 = the
  // default), and the test hook that makes one dependency unreachable
  int64_t wait_polls = 0;
  int32_t wait_unreachable = 0;
  // persistent solve tiling (pisp_options.solve_kfuse / solve_warp_maxF)
  int32_t kfuse = 1, warp_maxF = 32, solve_ctas = 0;
  int32_t factor_smem_maxF = 0;  // one-launch factorisation: widest shared-memory front (0 = limit)
  int32_t factor_tc = 0;         // FP32 owner-tile updates on the tensor cores
  int32_t factor_ctas = 0;       // one-launch factorisation: resident CTAs per SM (2 or 3; 0 = 2)
  pisp::SymDev sd{};
  // level plans (depend on the factor precision)
  int plan_precision = 0;
  std::vector<pisp::LevelPlan> plans;
  std::vector<int32_t> h_small, h_big;
  std::vector<pisp::BigFrontHost> h_bigF;
  std::vector<pisp::DagTask> h_dag;
  int32_t dag_max_flags = 0;
  Buf d_small, d_big, d_dag, dag_ticket, dag_flags;
  // one-launch factorisation (factor policy 4): all-level task list, the
  // list of fronts of at most 32 rows, completion targets, counters and owner release flags
  int32_t n_ftasks = 0, fac_CH = 32, fac_nflags = 0;
  size_t fac_smem = 0;
  bool fac_single = false;  // the plan is one launch (one_launch), at fac_ctas CTAs per SM
  int32_t fac_ctas = 0;
  double fac_bytes = 0;
  Buf d_ftasks, d_fwl, d_fneed, fdone, fflags, fticket;
  // numeric state
  int32_t K = 0, precision = 0, K_hint = 1, plan_K = 0;
  double t[PISP_K_MAX] = {}, beta[PISP_K_MAX] = {}, w_last[PISP_K_MAX] = {};
  Buf fronts, vals, D, status, badcol;
  // solve state
  int32_t R = 0;
  Buf V, X, Y, Rk, Lam, X2, rtmp, dtmp;
  // host-buffer entry point staging; b is copied on its own stream, after
  // the values and D and during the factorisation
  Buf in_vals, in_D, in_b, out_x;
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t copy_ev[2] = {};
  int launches = 0;
  // library-owned CUDA graph of one factor + solve step (pisp_graph_capture)
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t graph_exec = nullptr;
  cudaStream_t cap_stream = nullptr;
  cudaEvent_t cap_ev = nullptr;
  bool graph_valid = false;
  bool capturing = false;  // inside pisp_graph_capture's own factor + solve calls
  void drop_graph() {
    if (graph_exec) cudaGraphExecDestroy(graph_exec);
    if (graph) cudaGraphDestroy(graph);
    graph_exec = nullptr;
    graph = nullptr;
    graph_valid = false;
  }
  // profiling: CUDA events bracketing each kernel family per level
  // sweep = -1: a whole device-side sweep loop (launches per iteration, and
  // the bytes of one sweep over every instance split into rows and solve
  // work, scaled at collection per iteration by the share it covered)
  struct Bracket {
    int fam, e0, e1, launches;
    double bytes;
    int sweep;
    double bytes_rows, bytes_work;
  };
  bool prof_on = false;
  std::vector<cudaEvent_t> prof_ev;
  int prof_next = 0;
  std::vector<Bracket> prof_br;
  double prof_ms[PISP_PROF_FAMILIES] = {}, prof_bytes[PISP_PROF_FAMILIES] = {};
  int64_t prof_launches[PISP_PROF_FAMILIES] = {};
  // side streams for the independent size classes of a level, forked from
  // and joined back into `stream` with events (parallel branches when the
  // caller captures the work into a CUDA graph)
  static constexpr int kSide = 3;
  cudaStream_t side[kSide] = {}, big_side = nullptr;  // big_side: the level's wide fronts
  cudaEvent_t fork_ev = nullptr, join_ev[kSide] = {}, big_join = nullptr;
  ~pisp_handle() {
    drop_graph();
    if (cap_stream) cudaStreamDestroy(cap_stream);
    if (copy_stream) cudaStreamDestroy(copy_stream);
    for (cudaEvent_t e : copy_ev)
      if (e) cudaEventDestroy(e);
    if (body_stream) cudaStreamDestroy(body_stream);
    if (cap_ev) cudaEventDestroy(cap_ev);
    for (cudaEvent_t e : prof_ev) cudaEventDestroy(e);
    for (int i = 0; i < kSide; ++i) {
      if (side[i]) cudaStreamDestroy(side[i]);
      if (join_ev[i]) cudaEventDestroy(join_ev[i]);
    }
    if (big_side) cudaStreamDestroy(big_side);
    if (big_join) cudaEventDestroy(big_join);
    if (fork_ev) cudaEventDestroy(fork_ev);
  }
};

namespace {

size_t esize(int precision) { return precision == PISP_FP32 ? 4 : 8; }

// NVTX range over one ABI call, so that profilers can scope a capture to a
// phase (factor, solve, ...); without an attached tool it costs a pointer test.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

int fail(pisp_handle* h, int code, const std::string& msg) {
  if (h) h->err = msg; else g_last_error = msg;
  return code;
}

#define CK(call)                                                                       \
  do {                                                                                 \
    cudaError_t e_ = (call);                                                           \
    if (e_ != cudaSuccess)                                                             \
      return fail(h, PISP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// The handle's device is made current for one ABI call and the caller's
// current device is restored when the call returns, so the library never
// leaves a different device current behind (streams and buffers stay bound to
// the handle's device).
struct DeviceScope {
  int prev = -1;
  DeviceScope() = default;
  DeviceScope(const DeviceScope&) = delete;
  DeviceScope& operator=(const DeviceScope&) = delete;
  ~DeviceScope() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

int set_device(pisp_handle* h, DeviceScope& scope) {
  if (h->device < 0)
    return fail(h, PISP_ERR_INVALID_ARG, "host-only handle (device -1): numeric calls need a device");
  int cur = -1;
  CK(cudaGetDevice(&cur));
  if (cur != h->device) {
    CK(cudaSetDevice(h->device));
    if (scope.prev < 0) scope.prev = cur;
  }
  return PISP_OK;
}

// Copies v to b, which keeps its allocation when it is large enough: on the
// handle's stream, so that work in flight there reads the old contents to its end
// and what is queued next reads the new ones (a copy on the legacy stream is
// ordered with neither when the handle's stream is a non-blocking one).  v may be
// freed afterwards.  While the stream is being captured the copy is not to become
// part of the graph.
template <typename T>
int upload(pisp_handle* h, Buf& b, const T* v, size_t n) {
  if (!b.ensure(n * sizeof(T))) return fail(h, PISP_ERR_OOM, "device allocation failed");
  if (n == 0) return PISP_OK;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  CK(cudaStreamIsCapturing(h->stream, &cs));
  if (cs != cudaStreamCaptureStatusNone) {
    CK(cudaMemcpy(b.p, v, n * sizeof(T), cudaMemcpyHostToDevice));
    return PISP_OK;
  }
  CK(cudaMemcpyAsync(b.p, v, n * sizeof(T), cudaMemcpyHostToDevice, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return PISP_OK;
}
template <typename T>
int upload(pisp_handle* h, Buf& b, const std::vector<T>& v) {
  return upload(h, b, v.data(), v.size());
}

// The schedules are built inside the first factorisation and the first solve of a
// pattern (and when K, the precision or R change), so they cost a user with one
// pattern a call what they cost: linear passes over the supernodes, no sorts.
// list stably sorted by key in [0, n); start[v] = the first entry of key v, start[n]
// their number.
template <typename Key>
std::vector<int32_t> sorted_by(const std::vector<int32_t>& list, size_t n, std::vector<int32_t>& start, Key key) {
  std::vector<int32_t> at(n + 1, 0), out(list.size());
  for (int32_t s : list) ++at[key(s) + 1];
  for (size_t v = 0; v < n; ++v) at[v + 1] += at[v];
  start = at;
  for (int32_t s : list) out[at[key(s)]++] = s;
  return out;
}

// Runs a step that allocates host memory: no C++ exception may cross the C boundary.
template <typename Step>
int no_throw(pisp_handle* h, Step step) {
  try {
    return step();
  } catch (const std::bad_alloc&) {
    return fail(h, PISP_ERR_OOM, "out of host memory");
  } catch (const std::exception& e) {
    return fail(h, PISP_ERR_INVALID_ARG, e.what());
  }
}

#define TRY(x)            \
  do {                    \
    int rc_ = (x);        \
    if (rc_) return rc_;  \
  } while (0)

// Level by level, the path of a front of size F > 64: 0 = one CTA with the front in
// shared memory, C >= 1 = a cluster of C CTAs (distributed shared memory), -1 = the
// global-memory path.  Policy 1: clusters wherever the front fits in at most 8 CTAs'
// shared memory; the others: one CTA while the front fits.
int factor_path(const pisp_handle* h, int F, int precision) {
  if (h->factor_policy == 1) return pisp::front_cluster_size(F, precision);
  return F <= pisp::small_front_limit(precision) ? 0 : -1;
}

// Routing of policy 0, by (front, shift) pairs: beyond kManyTasks a factorisation
// has work for every SM.
constexpr int64_t kManyTasks = 8192;

// CTAs of the one-launch factorisation that an SM holds (at most 3) beside the
// shared memory of the owner tiles, which grows with the widest front in FP32.
int tile_ctas(const pisp_handle* h, int precision) {
  const int F = h->sym.max_front;
  if (F <= pisp::persistent_cta_front_limit(precision)) return 3;
  const size_t smem = pisp::factor_persistent_smem(precision, pisp::owner_chunk_rows(precision, F, h->factor_tc), true, 0) +
                      (precision == PISP_FP32 && h->factor_tc ? pisp::tc_staging_bytes() : 0);
  return (int)std::min<size_t>(3, 228 * 1024 / (smem + 1536));  // an SM's, and what a CTA takes beside
}

// Whether the factorisation is one persistent launch: under policy 4, and under
// policy 0 by what was measured (us level by level / in one launch, K 4).  In FP32 it
// saves the launches and the waits between levels and size classes: 1354 buses
// 344 / 245, 777 buses 230 / 191, 5 grids 280 / 192, 64 grids 1784 / 897; with a
// root of 1596 rows the owner tiles are all that counts, and those alone on an SM
// with 255 registers a thread are ahead (10000 buses 1671 / 1786).  The owner tiles'
// shared memory bounds the CTAs an SM holds for all the other fronts too, so a batch
// with one wide front goes level by level from some number of pairs on.  With room
// for three CTAs one launch was ahead or even wherever it was measured (150 grids of
// 200 buses and one of 3000, 55 k pairs: 600 / 521; 600 and one, 206 k: 935 / 880).
// For two, the other grids decide (one of 5000 buses, with 150 of 200 buses, 58 k:
// 855 / 784; with 100 of 1000, 170 k: 1907 / 1746; with 600 of 200, 210 k: 1134 /
// 1323; with 1500, 513 k: 1694 / 2513).  For one, few pairs do (one of 6000 buses:
// 10 k 919 / 765; with 150 of 200 buses, 59 k: 1008 / 1066; with 600, 211 k: 1244 /
// 2043; with 100 of 1000, 171 k: 1941 / 2510; the one-launch figures past the lines
// are with fronts of up to 160 rows by CTAs).
// In FP64 tiles are small.  One grid's fronts are bound by the FP64 pipe whichever
// way they are launched (300 buses 154 / 156, 1354 buses 565 / 570; 118 buses 99 /
// 122: the one-launch form takes segments for fronts of at most 32 rows); many grids'
// fronts fill the SMs (48 grids 3939 / 2470, with the bodies of that time).
// Fronts that wait for no others (dense systems) need no more than a launch a size
// class, and no counters, while a CTA holds each: FP32, K 4, 16 systems of 40 rows
// 36 / 39, of 97 81 / 90, of 160 139 / 156, of 200 (owner tiles) 191 / 144, of 9 to 137
// 110 / 122; 100 systems, K 10, of 40 rows 73 / 118; FP64, of 128 rows 2065 / 2490.
bool one_launch(const pisp_handle* h, int precision, int32_t K) {
  if (h->factor_policy != 0) return h->factor_policy == 4;
  const int64_t tasks = (int64_t)h->sym.sn.size() * K;
  if (h->sym.n_levels == 1 && h->sym.max_front <= 160) return false;
  if (precision != PISP_FP32) return tasks >= kManyTasks;
  const int room = tile_ctas(h, precision);
  return h->sym.max_front <= 1024 && tasks < (room >= 3 ? INT64_MAX : room == 2 ? 24 * kManyTasks : 4 * kManyTasks);
}

// Task list of the one-launch factorisation (one_launch): per level,
// bottom-up, the owner tiles of the fronts wider than the shared-memory
// limit (in (block, chunk) order, every tile after the ones it waits for),
// then one task per (front, k) for the shared-memory fronts, then the segment
// tasks of the fronts of at most 32 rows by size class, 256 / SEG a record.
int build_persistent_factor(pisp_handle* h, int precision, int32_t K) {
  const pisp::Symbolic& S = h->sym;
  int smem_maxF = h->factor_smem_maxF;
  h->fac_ctas = h->factor_ctas;
  if (h->factor_policy == 0) {
    // many fronts: three CTAs an SM with the fronts that three can hold (64 grids
    // 871 us, 994 with two; 48 grids in FP64 1914, 2173 with two), but compiled for
    // two, with more registers, where the tiles leave no room for three (one of 6000
    // buses, K 8: 1051 us, 1182 compiled for three; 150 grids of 200 buses and one of
    // 5000, K 4: 784, 851); few: two (2000 buses 341 us, 364 with three)
    const bool many = (int64_t)S.sn.size() * K >= kManyTasks;
    smem_maxF = many ? (precision == PISP_FP32 ? 128 : 64) : 0;
    h->fac_ctas = many && tile_ctas(h, precision) >= 3 ? 3 : 2;
  }
  const int Fc = smem_maxF > 0 ? std::min(smem_maxF, pisp::persistent_cta_front_limit(precision))
                               : pisp::persistent_cta_front_limit(precision);
  int maxBig = 0, maxCta = 0;
  for (const auto& sn : S.sn) {
    if (sn.F() > Fc) maxBig = std::max(maxBig, sn.F());
    else if (sn.F() > 32) maxCta = std::max(maxCta, sn.F());
  }
  const int CH = maxBig > 0 ? pisp::owner_chunk_rows(precision, maxBig, h->factor_tc) : 32;
  std::vector<pisp::FactorTask> ft;
  std::vector<int32_t> wl, ntask(S.sn.size(), 1);  // tasks per (front, k)
  int64_t nflags = 0;
  for (int l = 0; l < S.n_levels; ++l) {
    // the level's fronts from the widest down: owner tiles, CTAs, segments
    const auto at = h->by_level.begin() + S.level_off[l], end = h->by_level.begin() + S.level_off[l + 1];
    auto past = [&](auto from, int F) { return std::find_if(from, end, [&](int32_t q) { return S.sn[q].F() <= F; }); };
    const auto cta = past(at, Fc), seg32 = past(cta, 32), seg16 = past(seg32, 16), seg8 = past(seg16, 8);
    const std::vector<int32_t> big(at, cta);
    if (!big.empty()) {
      std::vector<pisp::BigFrontHost> bh;
      for (int32_t sn : big) bh.push_back({S.sn[sn].F(), S.sn[sn].ns()});
      std::vector<pisp::DagTask> tk;
      int32_t nfl = 0;
      pisp::build_owner_tasks(bh.data(), (int32_t)bh.size(), K, CH, tk, nfl);
      for (const auto& t : tk)
        ft.push_back({pisp::kFacOwner, big[t.b], t.k, t.p, t.j, (int32_t)(nflags + t.flags)});
      for (size_t b = 0; b < big.size(); ++b)
        ntask[big[b]] = ((bh[b].F + 31) / 32) * ((bh[b].F + CH - 1) / CH);
      nflags += nfl;
      if (nflags >= INT32_MAX) return fail(h, PISP_ERR_UNSUPPORTED, "too many factor flags");
    }
    for (auto q = cta; q != seg32; ++q)
      for (int k = 0; k < K; ++k) ft.push_back({pisp::kFacCta, *q, k, 0, 0, 0});
    for (int w = 2; w >= 0; --w) {
      const auto from = w == 2 ? seg32 : (w == 1 ? seg16 : seg8), to = w == 2 ? seg16 : (w == 1 ? seg8 : end);
      const int64_t off = (int64_t)wl.size(), tasks = (to - from) * K;
      if (off + (to - from) >= INT32_MAX || tasks >= INT32_MAX)
        return fail(h, PISP_ERR_UNSUPPORTED, "too many factor tasks");
      wl.insert(wl.end(), from, to);
      for (int64_t b = 0; b < tasks; b += 256 / (8 << w))
        ft.push_back({pisp::kFacSeg8 + w, (int32_t)off, 0, (int32_t)b, (int32_t)tasks, 0});
    }
  }
  std::vector<int32_t> need(S.sn.size(), 0);
  for (size_t q = 0; q < S.sn.size(); ++q)
    if (S.sn[q].parent >= 0) need[S.sn[q].parent] += ntask[q];
  if ((int64_t)ft.size() >= INT32_MAX) return fail(h, PISP_ERR_UNSUPPORTED, "too many factor tasks");
  TRY(upload(h, h->d_ftasks, ft));
  TRY(upload(h, h->d_fwl, wl));
  TRY(upload(h, h->d_fneed, need));
  if (!h->fdone.ensure(S.sn.size() * (size_t)K * pisp::kCtrStride * sizeof(int)) || !h->fflags.ensure((size_t)nflags * sizeof(int)) ||
      !h->fticket.ensure(sizeof(int)))
    return fail(h, PISP_ERR_OOM, "device allocation failed (factor schedule)");
  h->n_ftasks = (int32_t)ft.size();
  h->fac_CH = CH;
  h->fac_nflags = (int32_t)nflags;
  h->fac_smem = pisp::factor_persistent_smem(precision, CH, maxBig > 0, maxCta);
  return PISP_OK;
}

// The factorisation's schedule: one launch (build_persistent_factor), or level by
// level, its fronts grouped by size: fronts factored in shared memory into classes,
// wider ones into the global-memory paths.  Either way the algorithmic bytes per
// level and perturbation: what each kernel family must read and write at least
// (values, indices, factor entries, vectors).
int build_plans(pisp_handle* h, int precision) {
  const pisp::Symbolic& S = h->sym;
  h->plan_precision = 0;  // until all of it is in place
  h->units_K = h->units_R = 0;
  h->plans.assign(S.n_levels, pisp::LevelPlan());
  auto path = [&](int F) { return F > 64 ? factor_path(h, F, precision) : 0; };
  const double p = (double)esize(precision);
  for (const pisp::Supernode& sn : S.sn) {
    pisp::LevelPlan& lp = h->plans[sn.level];
    const size_t s = &sn - S.sn.data();
    const double F = sn.F(), ns = sn.ns(), ms = sn.ms;
    const double amap = (double)(S.amap_off[s + 1] - S.amap_off[s]);
    const double fac = amap * 16 + ns * 12 + F * F * p;
    if (path(sn.F()) < 0) lp.bytes_fbig += fac + 2 * F * F * p;
    else lp.bytes_fsmall += fac;
    lp.bytes_fwd_a += ns * 4 + (ns * F - ns * (ns + 1) / 2) * p;
    lp.bytes_fwd_b += ns * 8 + F * p;
    lp.bytes_bwd_a += ms * 4 + (ns * (ns + 1) / 2 + ns * ms) * p;
    lp.bytes_bwd_b += ms * 8 + ns * p + ns * 8;
    if (sn.parent < 0) continue;
    // as a child of its parent
    const pisp::Supernode& up = S.sn[sn.parent];
    pisp::LevelPlan& lq = h->plans[up.level];
    (path(up.F()) < 0 ? lq.bytes_fbig : lq.bytes_fsmall) += ms * ms * p + ms * 4;
    lq.bytes_fwd_a += ms * 4;
    lq.bytes_fwd_b += ms * p;
  }
  h->fac_single = one_launch(h, precision, h->K_hint);
  if (h->fac_single) {
    TRY(build_persistent_factor(h, precision, h->K_hint));
    h->fac_bytes = 0;
    for (const auto& lp : h->plans) h->fac_bytes += lp.bytes_fsmall + lp.bytes_fbig;
    h->plan_precision = precision;
    return PISP_OK;
  }
  h->h_small.clear();
  h->h_big.clear();
  h->h_bigF.clear();
  h->h_dag.clear();
  h->dag_max_flags = 0;
  for (int l = 0; l < S.n_levels; ++l) {
    pisp::LevelPlan& lp = h->plans[l];
    lp.big_off = (int64_t)h->h_big.size();
    // from the narrowest front up, in the order of their numbers among equals
    int last = 0;
    for (int64_t hi = S.level_off[l + 1]; hi > S.level_off[l];) {
      int64_t lo = hi - 1;
      const int F = S.sn[h->by_level[lo]].F();
      while (lo > S.level_off[l] && S.sn[h->by_level[lo - 1]].F() == F) --lo;
      const int C = path(F);
      if (C < 0) {
        for (int64_t q = lo; q < hi; ++q) {
          const int32_t s = h->by_level[q];
          h->h_big.push_back(s);
          h->h_bigF.push_back({F, S.sn[s].ns()});
          lp.big_maxns = std::max(lp.big_maxns, S.sn[s].ns());
        }
        lp.big_count += (int32_t)(hi - lo);
        lp.big_maxF = F;
      } else {
        // on-chip fronts: segment classes up to 32 (one class of CTAs in FP64), a
        // class of CTAs up to 64, then clusters of 1..8 CTAs or single CTAs
        const int cls = F > 64 ? 100 + C : F > 32 ? 64 : precision != PISP_FP32 ? 32 : F > 16 ? 32 : F > 8 ? 16 : 8;
        if (cls != last) lp.groups[lp.n_groups++] = {(int64_t)h->h_small.size(), 0, 0, C};
        last = cls;
        pisp::LevelPlan::Group& G = lp.groups[lp.n_groups - 1];
        h->h_small.insert(h->h_small.end(), h->by_level.begin() + lo, h->by_level.begin() + hi);
        G.count += (int32_t)(hi - lo);
        G.maxF = F;
      }
      hi = lo;
    }
    // big fronts as one persistent launch per level: owner tiles (policy 0,
    // any front size) or the tile DAG (policy 2, while a panel fits in shared
    // memory); else (and under policies 1 and 3) one panel launch and one
    // update launch per 32 pivots
    const bool owner = h->factor_policy == 0;
    const bool dag = h->factor_policy == 2 && lp.big_maxF <= pisp::max_dag_front(precision);
    if (lp.big_count > 0 && (owner || dag)) {
      std::vector<pisp::DagTask> tk;
      int32_t nfl = 0;
      if (owner) {
        lp.own_ch = pisp::owner_chunk_rows(precision, lp.big_maxF, h->factor_tc);
        pisp::build_owner_tasks(h->h_bigF.data() + lp.big_off, lp.big_count, h->K_hint, lp.own_ch, tk, nfl);
      }
      else
        pisp::build_dag_tasks(h->h_bigF.data() + lp.big_off, lp.big_count, h->K_hint, tk, nfl);
      lp.dag_owner = owner ? 1 : 0;
      lp.dag_task_off = (int64_t)h->h_dag.size();
      lp.dag_tasks = (int32_t)tk.size();
      lp.dag_flags = nfl;
      h->h_dag.insert(h->h_dag.end(), tk.begin(), tk.end());
      h->dag_max_flags = std::max(h->dag_max_flags, nfl);
    }
  }
  TRY(upload(h, h->d_small, h->h_small));
  TRY(upload(h, h->d_big, h->h_big));
  TRY(upload(h, h->d_dag, h->h_dag));
  if (!h->dag_ticket.ensure(sizeof(int)) || !h->dag_flags.ensure((size_t)h->dag_max_flags * sizeof(int)))
    return fail(h, PISP_ERR_OOM, "device allocation failed (factor schedule)");
  h->plan_precision = precision;
  return PISP_OK;
}

// groups of the completion counters (SolveArgs::NG)
int counter_groups(const pisp_handle* h, int32_t K, int32_t R, bool fwd) {
  return fwd || R == 1 ? K : (K * pisp::rhs_stride(h->precision, R) + 31) / 32;
}

// Work units of the solves.  Fronts with more than 32 pivots are CTA tasks per
// (256 rows, shift, RHS chunk); other fronts wider than h->warp_maxF (at least
// 32) CTA tasks per (shift, RHS chunk of 8); the rest segment tasks of 8, 16 or
// 32 lanes by their size, one per group of h->kfuse consecutive shifts and RHS
// chunk of 8.  Backward solves of several right-hand sides take column groups
// instead: one CTA task, or one warp's task (8 a unit), per front and group; fronts
// with many pivots to few right-hand sides (few_columns) segments of 32 lanes.
// The forward list goes by the fronts' height above the leaves, the backward
// list by their depth below the root: each as soon as what it waits for can be
// done, so that the CTAs in flight hold ready units (by falling height, a
// root's leaf children would come last, and fronts next to the leaves wait in
// line behind chains of tall ones: 150 us against 106 us for the backward solve
// of the 2000-bus grid).  Within a stage the CTA tasks come first, those with
// the longest way to go before the others, then the warps' tasks from the widest
// down, by instance, so that the adaptive sweeps' compaction drops whole units.
// The fronts' records are listed in the order the units name them.
struct UnitList {
  std::vector<pisp::SolveUnit> units;
  std::vector<int32_t> rng;    // [lo, hi] instance range per unit
  std::vector<int32_t> order;  // front of each record
  std::vector<int32_t> start;  // first unit of each stage, and the number of units
};

// Right-hand sides of a task of a front with more than 32 pivots, by the most such
// tasks that a stage would have with one each.  FP32: four, whose chains of steps
// overlap in the warp that solves a block, or eight, a warp each, where such tasks fill
// the SMs (two CTAs each) and the kernel has the registers: 100 dense systems of 97
// rows, K 10, R 8, forward + backward, 50 + 48 us, 74 + 70 with four; 4 of 97, K 6, R 4,
// 15 + 15.  FP64, whose pipe is what the columns of a task wait for: one while those
// fill the SMs (4 systems of 97 rows, K 6, R 4: 22 + 25 us, 33 + 40 with two in one
// warp), then two and four, a warp each (40 grids to 1500 buses, K 4, R 8: 208 + 208, 197
// + 213 with one, 228 + 245 with four; 128 to 3000: 1014 + 784, 1025 + 831, 941 + 710),
// and eight where even those fill them many times (100 of 64 rows, K 10, R 32: 343 + 485
// us, 400 + 531 with four; 712 + 973 with two in one warp).
int wide_rhs(const pisp_handle* h, int64_t tasks, int32_t R) {
  if (R == 1) return 1;
  constexpr int64_t kCtas = 2 * 152;
  if (h->precision == PISP_FP32) return R > 4 && h->solve_ctas <= 2 && tasks * ((R + 7) / 8) >= kCtas ? 8 : 4;
  const int64_t n = tasks * R;
  return n <= kCtas ? 1 : (n <= 4 * kCtas ? 2 : (n <= 32 * kCtas ? 4 : 8));
}

// Whether the backward solve of R > 1 right-hand sides takes a front of at most 32
// rows by segments and not by columns: a warp's 32 columns share n^2 / 2 steps on
// it, a segment's 8 right-hand sides n steps each, so that few columns, or many
// pivots, leave the columns behind (dense systems, K 4, FP64, columns / segments: 32 rows,
// R 2 55 / 18 us, R 8 56 / 45, R 32 56 / 46, and with 1000 pairs 58 / 158; 16 rows, R 4 22
// / 18; FP32, 32 rows, R 2 28 / 14, R 8 29 / 18; 24 rows, R 8 20 / 20).  Compiled for
// more than two CTAs an SM the kernel has no registers for both.
bool few_columns(const pisp_handle* h, const pisp::Supernode& n, int32_t R) {
  return h->solve_ctas <= 2 && n.F() <= 32 && n.ns() > std::max(8, 3 * R);
}

// Whether a front counts its tasks of a backward solve of R > 1 right-hand sides
// together, because they are cut by shift.
bool whole_front(const pisp_handle* h, const pisp::Supernode& n, int32_t R) {
  return n.ns() > 32 || few_columns(h, n, R);
}

// tasks[s]: tasks of front s per completion counter
int build_unit_list(pisp_handle* h, int32_t K, int32_t R, const std::vector<int32_t>& stage, int32_t stages,
                    const std::vector<int32_t>& left, bool fwd, std::vector<int32_t>& tasks, int32_t& wide,
                    UnitList& out) {
  const pisp::Symbolic& S = h->sym;
  const int NG = counter_groups(h, K, R, fwd);
  const bool cols = !fwd && R > 1;
  const int kf = std::max(1, std::min(h->kfuse, (int)K));
  const int rchunks = R == 1 ? 1 : (R + pisp::kSolveChunk - 1) / pisp::kSolveChunk;
  // by stage, within it by instance and from the widest front down
  std::vector<int32_t> at;
  const std::vector<int32_t> lst = sorted_by(h->by_inst, stages, at, [&](int32_t q) { return stage[q]; });
  out.order.reserve(S.sn.size());
  auto cta_unit = [&](int32_t sn, const pisp::SolveUnit& u) {
    out.units.push_back(u);
    out.rng.push_back(S.sn[sn].instance);
    out.rng.push_back(S.sn[sn].instance);
  };
  auto wide_rows = [&](int32_t sn) {  // tasks of 256 rows
    return ((fwd ? S.sn[sn].F() : S.sn[sn].ns()) + pisp::kWideUnitRows - 1) / pisp::kWideUnitRows;
  };
  int64_t most = 0;
  for (int32_t st = 0; st < stages; ++st) {
    int64_t n = 0;
    for (int32_t e = at[st]; e < at[st + 1]; ++e)
      if (S.sn[lst[e]].ns() > 32) n += (int64_t)wide_rows(lst[e]) * K;
    most = std::max(most, n);
  }
  const int rc = wide_rhs(h, most, R);
  std::vector<int32_t> cta, seg[4];  // segments of 8, 16, 32 lanes; warps
  for (int32_t st = 0; st < stages; ++st) {
    out.start.push_back((int32_t)out.units.size());
    cta.clear();
    for (auto& g : seg) g.clear();
    for (int32_t e = at[st]; e < at[st + 1]; ++e) {
      const int32_t sn = lst[e];
      const int F = S.sn[sn].F(), ns = S.sn[sn].ns();
      if (ns > 32 || F > std::max(32, h->warp_maxF)) cta.push_back(sn);
      else seg[cols ? (few_columns(h, S.sn[sn], R) ? 2 : 3) : (F > 16 ? 2 : (F > 8 ? 1 : 0))].push_back(sn);
      tasks[sn] = !cols ? rchunks : whole_front(h, S.sn[sn], R) ? K * rchunks : 1;
    }
    std::sort(cta.begin(), cta.end(), [&](int32_t a, int32_t b) {
      if (left[a] != left[b]) return left[a] > left[b];
      const int fa = S.sn[a].F(), fb = S.sn[b].F();
      return fa != fb ? fa > fb : a < b;
    });
    for (int32_t sn : cta) {
      const int32_t slot = (int32_t)out.order.size();
      out.order.push_back(sn);
      if (S.sn[sn].ns() <= 32) {
        for (int g = 0; g < NG; ++g)
          for (int c = 0; c < tasks[sn]; ++c) cta_unit(sn, {pisp::kUnitCta, slot, g, c});
        continue;
      }
      const int ch = (R + rc - 1) / rc, nq = wide_rows(sn);
      wide = rc;
      tasks[sn] = cols ? nq * K * ch : nq * ch;
      // the rows solved first, first: a task waits only for tasks before it
      for (int q = 0; q < nq; ++q)
        for (int k = 0; k < K; ++k)
          for (int c = 0; c < ch; ++c)
            cta_unit(sn, {pisp::kUnitWide, slot, k | rc << 4 | (fwd ? q : nq - 1 - q) << 8, c});
    }
    for (int w = 3; w >= 0; --w) {
      std::vector<int32_t>& g = seg[w];
      if (g.empty()) continue;
      const int kind = w == 3 ? pisp::kUnitCol : (w == 2 ? pisp::kUnitSeg32 : (w == 1 ? pisp::kUnitSeg16 : pisp::kUnitSeg8));
      const int per_unit = w == 3 ? 8 : 256 / (8 << w);
      const int64_t per_front = w == 3 ? NG : (int64_t)((K + kf - 1) / kf) * rchunks;
      const int32_t off = (int32_t)out.order.size();
      const int64_t n = (int64_t)g.size() * per_front;
      if (n >= INT32_MAX) return fail(h, PISP_ERR_UNSUPPORTED, "too many solve tasks");
      out.order.insert(out.order.end(), g.begin(), g.end());
      for (int64_t b = 0; b < n; b += per_unit) {
        out.units.push_back({kind | (w == 3 ? 0 : kf << 4), off, (int32_t)b, (int32_t)n});
        out.rng.push_back(S.sn[g[b / per_front]].instance);
        out.rng.push_back(S.sn[g[(std::min(n, b + per_unit) - 1) / per_front]].instance);
      }
    }
  }
  if (out.units.size() >= (size_t)INT32_MAX) return fail(h, PISP_ERR_UNSUPPORTED, "too many solve tasks");
  out.start.push_back((int32_t)out.units.size());
  return PISP_OK;
}

int build_units(pisp_handle* h, int32_t K, int32_t R) {
  h->units_K = h->units_R = 0;  // until all of it is in place
  const pisp::Symbolic& S = h->sym;
  const size_t nS = S.sn.size();
  // parents have larger numbers than their children
  std::vector<int32_t> height(nS), depth(nS, 0);
  for (size_t q = 0; q < nS; ++q) height[q] = S.sn[q].level;
  int32_t deepest = -1;
  for (size_t q = nS; q-- > 0;) {
    if (S.sn[q].parent >= 0) depth[q] = depth[S.sn[q].parent] + 1;
    deepest = std::max(deepest, depth[q]);
  }
  UnitList f, b;
  std::vector<int32_t> nf(nS, 1), nb(nS, 1);
  int32_t wide[2] = {};
  TRY(build_unit_list(h, K, R, height, S.n_levels, depth, true, nf, wide[0], f));
  TRY(build_unit_list(h, K, R, depth, deepest + 1, height, false, nb, wide[1], b));
  // completion targets: forward, every task of a front's children; backward,
  // every task of its parent, as the counters count them
  const int NG = std::max(counter_groups(h, K, R, true), counter_groups(h, K, R, false));
  auto whole = [&](int32_t q) { return R > 1 && whole_front(h, S.sn[q], R); };  // backward
  std::vector<int32_t> need(nS, 0);
  for (size_t q = 0; q < nS; ++q)
    if (S.sn[q].parent >= 0) need[S.sn[q].parent] += nf[q];
  if (h->wait_unreachable) {
    // test hook: one front's completion target can never be reached, so the
    // waits on it (its parent's in the forward pass, its children's in the
    // backward pass) run out of polls
    for (size_t q = 0; q < nS; ++q)
      if (S.sn[q].parent >= 0) {
        need[S.sn[q].parent] += 1;
        nb[q] += 1;
        break;
      }
  }
  // counters of the fronts with more than 32 pivots (at most one per right-hand side)
  std::vector<int32_t> flag(nS, 0);
  int64_t nflags = 0;
  for (size_t q = 0; q < nS; ++q)
    if (S.sn[q].ns() > 32) {
      flag[q] = (int32_t)nflags;
      nflags += (int64_t)K * R;
      if (nflags >= INT32_MAX) return fail(h, PISP_ERR_UNSUPPORTED, "too many solve tasks");
    }
  // the records, forward order, then backward order; read in the fronts' own order
  std::unique_ptr<pisp::FrontDesc[]> desc(new pisp::FrontDesc[2 * nS]);
  std::vector<int32_t> at_f(nS), at_b(nS);
  for (size_t q = 0; q < nS; ++q) {
    at_f[f.order[q]] = (int32_t)q;
    at_b[b.order[q]] = (int32_t)q;
  }
  for (size_t q = 0; q < nS; ++q) {
    const int32_t sn = (int32_t)q;
    const pisp::Supernode& n = S.sn[q];
    desc[at_f[q]] = desc[nS + at_b[q]] = {
        n.c0, n.ns(), n.F(), n.instance, S.front_off[q], S.vec_off[q], n.row_off, n.parent, sn, need[q],
        n.parent >= 0 ? nb[n.parent] : 0, flag[q],
        (whole(sn) ? pisp::kSelfWhole : 0) | (n.parent >= 0 && whole(n.parent) ? pisp::kParentWhole : 0)};
  }
  TRY(upload(h, h->units_f, f.units));
  TRY(upload(h, h->units_b, b.units));
  TRY(upload(h, h->rng_f, f.rng));
  TRY(upload(h, h->rng_b, b.rng));
  TRY(upload(h, h->desc, desc.get(), 2 * nS));
  if (!h->units_fc.ensure(f.units.size() * sizeof(pisp::SolveUnit)) ||
      !h->units_bc.ensure(b.units.size() * sizeof(pisp::SolveUnit)) || !h->ucount.ensure(2 * sizeof(int32_t)) ||
      !h->serr.ensure(sizeof(int)) || !h->ctr.ensure(2 * (f.start.size() + b.start.size() + 8 + (nS * (size_t)NG + (size_t)nflags) * pisp::kCtrStride) * sizeof(int)))
    return fail(h, PISP_ERR_OOM, "device allocation failed (solve schedule)");
  h->n_units_f = (int32_t)f.units.size();
  h->n_units_b = (int32_t)b.units.size();
  h->lvl_units_f = f.start;
  h->lvl_units_b = b.start;
  h->units_wide[0] = wide[0];
  h->units_wide[1] = wide[1];
  h->units_segs = false;
  for (const pisp::Supernode& n : S.sn) h->units_segs = h->units_segs || (R > 1 && few_columns(h, n, R));
  h->ctr_tickets = (f.start.size() + b.start.size()) / 8 * 8 + 8;  // more than one per stage
  h->ctr_half = h->ctr_tickets + (nS * (size_t)NG + (size_t)nflags) * pisp::kCtrStride;
  h->units_K = K;
  h->units_R = R;
  return PISP_OK;
}

int set_weights(pisp_handle* h, const double* w, double* out) {
  if (w) {
    for (int k = 0; k < h->K; ++k) {
      if (!std::isfinite(w[k])) return fail(h, PISP_ERR_INVALID_ARG, "non-finite weight");
      out[k] = w[k];
    }
  } else {
    for (int k = 0; k < h->K; ++k) out[k] = h->beta[k];
  }
  return PISP_OK;
}

pisp::Shifts make_shifts(const pisp_handle* h, const double* w) {
  pisp::Shifts sh{};
  sh.K = h->K;
  for (int k = 0; k < h->K; ++k) {
    sh.t[k] = h->t[k];
    sh.w[k] = w[k];
  }
  return sh;
}

const char* kFamilyNames[PISP_PROF_FAMILIES] = {"factor_small", "factor_big", "forward",
                                                "backward",     "residual",   "combine",
                                                "factor_persistent", "sweep_loop"};

// Event record that also works inside a stream capture: there it must become
// an event-record node of the graph (external record) to be timed on replay.
void record_event(pisp_handle* h, cudaEvent_t e, cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(st, &cs);
  cudaEventRecordWithFlags(e, st,
                           cs == cudaStreamCaptureStatusActive ? cudaEventRecordExternal
                                                               : cudaEventRecordDefault);
}

// Records a start event of a profiling bracket; returns its index or -1.
int prof_begin(pisp_handle* h, cudaStream_t st = nullptr) {
  if (!h->prof_on) return -1;
  if (h->prof_next + 2 > (int)h->prof_ev.size()) {
    for (int q = 0; q < 64; ++q) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) return -1;
      h->prof_ev.push_back(e);
    }
  }
  const int i = h->prof_next;
  h->prof_next += 2;
  record_event(h, h->prof_ev[i], st ? st : h->stream);
  return i;
}

// Closes the bracket on the stream it was opened on (default: the handle's).
void prof_end(pisp_handle* h, int i, int fam, double bytes, int launches, cudaStream_t st = nullptr) {
  if (i < 0 || launches <= 0) return;
  record_event(h, h->prof_ev[i + 1], st ? st : h->stream);
  h->prof_br.push_back({fam, i, i + 1, launches, bytes, 0, 0.0, 0.0});
}

int count(pisp_handle* h, int n) {
  if (n < 0) {
    cudaError_t e = cudaGetLastError();
    return fail(h, PISP_ERR_CUDA, std::string("kernel launch failed: ") + cudaGetErrorString(e));
  }
  h->launches += n;
  return PISP_OK;
}

// Right-hand sides and outputs of one forward + backward solve: b (FP64,
// broadcast, original order) or rk (factor precision, per shift, permuted
// order); xt the solution in the factor precision, xd (may be null) in FP64,
// stored or added (solve_persistent.h).
struct SolveIO {
  const double* b;
  const void* rk;
  void* xt;
  double* xd;
  int xd_mode;
};

template <typename T>
int solve_pass_t(pisp_handle* h, bool trans, const SolveIO& io, int32_t R, const uint8_t* act) {
  const int L = h->sym.n_levels;
  double bf = 0, bb = 0;
  for (int l = 0; l < L; ++l) {
    bf += h->K * (h->plans[l].bytes_fwd_a + h->plans[l].bytes_fwd_b * R);
    bb += h->K * (h->plans[l].bytes_bwd_a + h->plans[l].bytes_bwd_b * R);
  }
  if (io.xd && io.xd_mode == pisp::kXdAdd) bb += 16.0 * h->sym.N * h->K * R;
  const bool cmp = act != nullptr;  // gated: the compacted lists (whole lists before the first test)
  const bool persistent = h->schedule == 0;
  int* ctr = h->ctr.as<int>();
  const size_t nd = h->ctr_half;
  pisp::SolveArgs<T> a{};
  a.inv_off = h->sd.inv_off;
  a.inv_pos = h->sd.inv_pos;
  a.rows = h->sd.rows;
  a.perm = h->sd.perm;
  a.act = act;
  a.err = h->serr.as<int>();
  a.wait_ns = pisp::wait_limit_ns(h->wait_polls);
  a.fronts = h->fronts.as<T>();
  a.b = io.b;
  a.rk = (const T*)io.rk;
  a.V = h->V.as<T>();
  a.xt = (T*)io.xt;
  a.xd = io.xd;
  a.xd_mode = io.xd_mode;
  a.R = R;
  a.K = h->K;
  a.RV = pisp::rhs_stride(h->precision, R);
  a.RX = pisp::rhs_stride64(R);
  a.vec = a.RV % (16 / (int)sizeof(T)) == 0;
  a.vecd = a.RX % 2 == 0;
  CK(cudaMemsetAsync(ctr, 0, 2 * nd * sizeof(int), h->stream));
  for (int dir = 0; dir < 2; ++dir) {  // forward, backward
    a.desc = h->desc.as<pisp::FrontDesc>() + (dir == 0 ? 0 : h->sym.sn.size());
    const int pb = prof_begin(h);
    int n = 0;
    auto go = [&](int count) {
      return dir == 0 ? pisp::launch_solve_dir<T, true>(trans, a, count, h->units_wide[dir], false, h->solve_ctas, h->stream)
                      : pisp::launch_solve_dir<T, false>(trans, a, count, h->units_wide[dir], h->units_segs, h->solve_ctas,
                                                         h->stream);
    };
    const int total = dir == 0 ? h->n_units_f : h->n_units_b;
    a.NG = counter_groups(h, h->K, R, dir == 0);
    a.ticket = ctr + (dir == 0 ? 0 : nd);
    a.wide = a.ticket + h->ctr_tickets + h->sym.sn.size() * (size_t)a.NG * pisp::kCtrStride;
    if (persistent) {
      a.units = (dir == 0 ? (cmp ? h->units_fc : h->units_f) : (cmp ? h->units_bc : h->units_b)).as<pisp::SolveUnit>();
      a.ucount = cmp ? h->ucount.as<int>() + dir : nullptr;
      a.nunits = total;
      a.done = a.ticket + h->ctr_tickets;
      n = go(total);
    } else {
      a.units = (dir == 0 ? h->units_f : h->units_b).as<pisp::SolveUnit>();
      const auto& lv = dir == 0 ? h->lvl_units_f : h->lvl_units_b;
      for (size_t l = 0; l + 1 < lv.size() && n >= 0; ++l) {
        a.first = lv[l];
        a.nunits = lv[l + 1] - lv[l];
        const int m = go(a.nunits);
        n = m < 0 ? -1 : n + m;
        ++a.ticket;
      }
    }
    TRY(count(h, n));
    prof_end(h, pb, dir == 0 ? PISP_PROF_FORWARD : PISP_PROF_BACKWARD, dir == 0 ? bf : bb, n);
  }
  return PISP_OK;
}

// forward + backward over all levels with L U, or with trans with U^T L^T.
// Adaptive sweeps (persistent schedule): act skips the fronts of instances
// that have stopped and the compacted unit lists are walked.
int solve_pass(pisp_handle* h, bool trans, const SolveIO& io, int32_t R, const uint8_t* act = nullptr) {
  if (h->units_K != h->K || h->units_R != R) TRY(no_throw(h, [&] { return build_units(h, h->K, R); }));
  return h->precision == PISP_FP32 ? solve_pass_t<float>(h, trans, io, R, act)
                                   : solve_pass_t<double>(h, trans, io, R, act);
}

// The uncorrected solve of b into X (FP64): with FP64 factors X is itself the
// working solution, with FP32 factors that is Y.
SolveIO first_solve(pisp_handle* h, const double* b, double* X) {
  if (h->precision == PISP_FP64) return {b, nullptr, X, nullptr, pisp::kXdStore};
  return {b, nullptr, h->Y.p, X, pisp::kXdStore};
}

// Sweeps per instance of the last solve, and for s = 1 .. max_sweeps the
// fraction of the solve work (front entries, fs[s]) and of the rows (fr[s])
// that sweep s covered (index 0 unused).  Synchronises the stream.
int sweep_fractions(pisp_handle* h, int max_sweeps, std::vector<int32_t>& nsw, std::vector<double>& fs,
                    std::vector<double>& fr) {
  const int32_t G = h->sym.G;
  nsw.assign(G, h->last_sweeps);
  if (h->last_adaptive) {
    CK(cudaMemcpyAsync(nsw.data(), h->r_nsw.p, (size_t)G * sizeof(int32_t), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
  }
  fs.assign(max_sweeps + 1, 0.0);
  fr.assign(max_sweeps + 1, 0.0);
  double ws = 0.0, wr = 0.0;
  for (int g = 0; g < G; ++g) {
    const double rows = (double)(h->sym.inst_off[g + 1] - h->sym.inst_off[g]);
    ws += h->inst_w[g];
    wr += rows;
    for (int s = 1; s <= std::min(max_sweeps, nsw[g]); ++s) {
      fs[s] += h->inst_w[g];
      fr[s] += rows;
    }
  }
  for (int s = 1; s <= max_sweeps; ++s) {
    fs[s] = ws > 0 ? fs[s] / ws : 0.0;
    fr[s] = wr > 0 ? fr[s] / wr : 0.0;
  }
  return PISP_OK;
}

// Algorithmic bytes of one forward + backward pass (all instances), as the
// brackets count them.
double solve_bytes(const pisp_handle* h, int32_t R) {
  double b = 0.0;
  for (int l = 0; l < h->sym.n_levels; ++l)
    b += h->K * (h->plans[l].bytes_fwd_a + h->plans[l].bytes_fwd_b * R + h->plans[l].bytes_bwd_a +
                 h->plans[l].bytes_bwd_b * R);
  return b;
}

// One adaptive sweep for the instances still iterating, the body of the
// device-side sweep loop: the FP64 residuals of their rows, the gated solves
// of their corrections (compacted unit lists of the persistent schedule; the
// per-level schedule solves every row, with zero residuals outside the active
// set), the corrections added to their solutions with the correction and
// solution sizes, the stopping test (which drives the loop's conditional
// `cond`) and the active set and unit lists of the next sweep.  No profiling
// brackets: a conditional body holds no events.
int sweep_body(pisp_handle* h, const double* rhs, double* X_out, int32_t R, int32_t S, const pisp::Shifts& sh,
               cudaGraphConditionalHandle cond) {
  const bool persistent = h->schedule == 0;
  const int32_t G = h->sym.G;
  uint8_t* act = h->r_act.as<uint8_t>();
  const pisp::ActiveSet as{act, h->r_nact.as<int32_t>(), h->r_ai.as<int32_t>(), h->r_arow.as<int64_t>(),
                           h->d_inst_off.as<int64_t>()};
  TRY(count(h, pisp::launch_residual_per_k(h->precision, h->sd, h->vals.as<double>(), h->D.as<double>(), sh, rhs,
                                           X_out, R, h->Rk.p, as,
                                           persistent ? pisp::kResActive : pisp::kResZeroStopped, h->stream)));
  // the corrections go to Y only: the stats launch below adds them to X
  const bool prof_was = h->prof_on;
  h->prof_on = false;
  const int rc = solve_pass(h, false, {nullptr, h->Rk.p, h->Y.p, nullptr, pisp::kXdStore}, R,
                            persistent ? act : nullptr);
  h->prof_on = prof_was;
  TRY(rc);
  TRY(count(h, pisp::launch_refine_stats(h->precision, h->sd, as, X_out, h->Y.p, h->K, R,
                                         h->r_dmax.as<unsigned long long>(), h->r_xmax.as<unsigned long long>(),
                                         h->stream)));
  TRY(count(h, pisp::launch_refine_decide(G, R, h->sweep_tol, S, h->r_sweep.as<int32_t>(), cond, 1, act,
                                          h->r_dmax.as<unsigned long long>(), h->r_xmax.as<unsigned long long>(),
                                          h->r_prevd.as<double>(), h->r_nsw.as<int32_t>(), h->r_pre.as<int32_t>(),
                                          h->r_nact.as<int32_t>(), h->r_ai.as<int32_t>(), h->r_arow.as<int64_t>(),
                                          h->d_inst_off.as<int64_t>(), h->stream)));
  if (persistent)
    TRY(count(h, pisp::launch_compact_units(
                     h->units_f.as<pisp::SolveUnit>(), h->rng_f.as<int32_t>(), h->n_units_f,
                     h->units_fc.as<pisp::SolveUnit>(), h->units_b.as<pisp::SolveUnit>(), h->rng_b.as<int32_t>(),
                     h->n_units_b, h->units_bc.as<pisp::SolveUnit>(), h->r_pre.as<int32_t>(),
                     h->r_ccnt.as<int32_t>(), h->ucount.as<int32_t>(), h->stream)));
  return PISP_OK;
}

// The adaptive sweeps as a device-side loop: a WHILE conditional node added
// to graph g after deps (its body one sweep_body, captured on a side stream
// into the node's body graph) that runs while the stopping test leaves an
// instance active, at most S times.
int add_sweep_loop(pisp_handle* h, cudaGraph_t g, const cudaGraphNode_t* deps, size_t ndeps,
                   cudaGraphNode_t* node_out, const double* rhs, double* X_out, int32_t R, int32_t S,
                   const pisp::Shifts& sh) {
  cudaGraphConditionalHandle cond = 0;
  CK(cudaGraphConditionalHandleCreate(&cond, g, 1, cudaGraphCondAssignDefault));
  cudaGraphNodeParams np{};
  np.type = cudaGraphNodeTypeConditional;
  np.conditional.handle = cond;
  np.conditional.type = cudaGraphCondTypeWhile;
  np.conditional.size = 1;
  std::vector<cudaGraphNode_t> dv(deps, deps + ndeps);
  CK(cudaGraphAddNode(node_out, g, dv.data(), nullptr, dv.size(), &np));
  cudaGraph_t body = np.conditional.phGraph_out[0];
  if (!h->body_stream) CK(cudaStreamCreateWithFlags(&h->body_stream, cudaStreamNonBlocking));
  CK(cudaStreamBeginCaptureToGraph(h->body_stream, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
  const cudaStream_t outer = h->stream;
  h->stream = h->body_stream;
  const int launches0 = h->launches;
  const int rc = sweep_body(h, rhs, X_out, R, S, sh, cond);
  h->loop_kernels = h->launches - launches0;
  h->stream = outer;
  cudaGraph_t body_out = nullptr;
  const cudaError_t e = cudaStreamEndCapture(h->body_stream, &body_out);
  TRY(rc);
  if (e != cudaSuccess) return fail(h, PISP_ERR_CUDA, std::string("sweep loop capture: ") + cudaGetErrorString(e));
  return PISP_OK;
}

// The sweep loop on h->stream: inside a stream capture in progress, as a node
// of the graph being captured; otherwise as a graph of its own, built,
// launched once and destroyed.  Its construction overlaps the work already queued;
// the call then returns when the loop is done, since destroying an executable graph
// waits for it (64 grids: 2521 us in pisp_solve of a step of 2597).
int run_sweep_loop(pisp_handle* h, const double* rhs, double* X_out, int32_t R, int32_t S, const pisp::Shifts& sh) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaGraph_t g = nullptr;
  const cudaGraphNode_t* deps = nullptr;
  size_t ndeps = 0;
  CK(cudaStreamGetCaptureInfo(h->stream, &cs, nullptr, &g, &deps, nullptr, &ndeps));
  cudaGraphNode_t node = nullptr;
  if (cs == cudaStreamCaptureStatusActive) {
    if (!g) return fail(h, PISP_ERR_CUDA, "stream capture without a graph");
    TRY(add_sweep_loop(h, g, deps, ndeps, &node, rhs, X_out, R, S, sh));
    CK(cudaStreamUpdateCaptureDependencies(h->stream, &node, nullptr, 1, cudaStreamSetCaptureDependencies));
    return PISP_OK;
  }
  CK(cudaGraphCreate(&g, 0));
  int rc = add_sweep_loop(h, g, nullptr, 0, &node, rhs, X_out, R, S, sh);
  cudaGraphExec_t ge = nullptr;
  if (rc == PISP_OK && cudaGraphInstantiate(&ge, g, 0) != cudaSuccess)
    rc = fail(h, PISP_ERR_CUDA, std::string("sweep loop instantiate: ") + cudaGetErrorString(cudaGetLastError()));
  cudaGraphDestroy(g);
  TRY(rc);
  const cudaError_t e = cudaGraphLaunch(ge, h->stream);
  cudaGraphExecDestroy(ge);
  if (e != cudaSuccess) return fail(h, PISP_ERR_CUDA, std::string("sweep loop launch: ") + cudaGetErrorString(e));
  return PISP_OK;
}

// Per-perturbation solves of `rhs` (broadcast, original order) into X_out,
// followed by at most `sweeps` FP64 residual corrections of every x_k: all of
// them for every instance, or (pisp_set_refinement) per instance until its
// stopping test holds, as a device-side loop.
int solve_core(pisp_handle* h, const double* rhs, double* X_out, int32_t R, int32_t sweeps,
               const pisp::Shifts& sh) {
  TRY(solve_pass(h, false, first_solve(h, rhs, X_out), R));
  const double N = (double)h->sym.N, KR = (double)h->K * R;
  const bool adapt = h->sweep_tol > 0.0 && sweeps > 0;
  const int32_t G = h->sym.G;
  h->last_sweeps = sweeps;
  h->last_adaptive = adapt;
  h->last_loop = false;
  h->any_solve = true;
  if (!adapt) {
    const pisp::ActiveSet none{};
    for (int it = 0; it < sweeps; ++it) {
      const int pb = prof_begin(h);
      const int n = pisp::launch_residual_per_k(h->precision, h->sd, h->vals.as<double>(), h->D.as<double>(), sh, rhs,
                                                X_out, R, h->Rk.p, none, pisp::kResAll, h->stream);
      TRY(count(h, n));
      prof_end(h, pb, PISP_PROF_RESIDUAL, h->sym.nnzA * 12.0 + N * 20.0 + N * R * 8.0 + 2.0 * N * KR * 8.0, n);
      TRY(solve_pass(h, false, {nullptr, h->Rk.p, h->Y.p, X_out, pisp::kXdAdd}, R));
    }
    return PISP_OK;
  }
  const size_t gr = (size_t)G * R * sizeof(unsigned long long);
  if (!h->r_act.ensure((size_t)G) || !h->r_pre.ensure((size_t)(G + 1) * sizeof(int32_t)) ||
      !h->r_nsw.ensure((size_t)G * sizeof(int32_t)) || !h->r_dmax.ensure(gr) || !h->r_xmax.ensure(gr) ||
      !h->r_prevd.ensure((size_t)G * R * sizeof(double)) || !h->r_nact.ensure(sizeof(int32_t)) ||
      !h->r_ai.ensure((size_t)G * sizeof(int32_t)) || !h->r_arow.ensure((size_t)(G + 1) * sizeof(int64_t)) ||
      !h->r_sweep.ensure(sizeof(int32_t)) ||
      !h->r_ccnt.ensure((size_t)pisp::compact_scratch(h->n_units_f, h->n_units_b) * sizeof(int32_t)))
    return fail(h, PISP_ERR_OOM, "device allocation failed (adaptive sweeps)");
  // every instance active; the compacted unit lists are the whole lists
  CK(cudaMemsetAsync(h->r_dmax.p, 0, gr, h->stream));
  CK(cudaMemsetAsync(h->r_xmax.p, 0, gr, h->stream));
  TRY(count(h, pisp::launch_refine_init(G, h->r_act.as<uint8_t>(), h->r_pre.as<int32_t>(), h->r_nact.as<int32_t>(),
                                        h->r_ai.as<int32_t>(), h->r_arow.as<int64_t>(),
                                        h->d_inst_off.as<int64_t>(), h->r_sweep.as<int32_t>(), h->stream)));
  if (h->schedule == 0)
    TRY(count(h, pisp::launch_compact_units(
                     h->units_f.as<pisp::SolveUnit>(), h->rng_f.as<int32_t>(), h->n_units_f,
                     h->units_fc.as<pisp::SolveUnit>(), h->units_b.as<pisp::SolveUnit>(), h->rng_b.as<int32_t>(),
                     h->n_units_b, h->units_bc.as<pisp::SolveUnit>(), h->r_pre.as<int32_t>(),
                     h->r_ccnt.as<int32_t>(), h->ucount.as<int32_t>(), h->stream)));
  const int pb = prof_begin(h);
  TRY(run_sweep_loop(h, rhs, X_out, R, sweeps, sh));
  h->last_loop = true;
  if (pb >= 0) {  // the loop as one bracket; bytes and launches are scaled at collection
    record_event(h, h->prof_ev[pb + 1], h->stream);
    h->prof_br.push_back({PISP_PROF_SWEEP_LOOP, pb, pb + 1, h->loop_kernels, 0.0, -1,
                          h->sym.nnzA * 12.0 + N * 20.0 + N * R * 8.0 + 5.0 * N * KR * 8.0, solve_bytes(h, R)});
  }
  return PISP_OK;
}

int ensure_solve_buffers(pisp_handle* h, int32_t R) {
  const size_t kv = (size_t)h->K * pisp::rhs_stride(h->precision, R) * esize(h->precision);
  const size_t nk = (size_t)h->sym.N * h->K * pisp::rhs_stride64(R) * sizeof(double);
  if (!h->V.ensure(kv * h->sym.vec_off.back()) || !h->X.ensure(nk) || !h->Y.ensure(kv * h->sym.N) ||
      !h->Rk.ensure(kv * h->sym.N))
    return fail(h, PISP_ERR_OOM, "device allocation failed (solve workspace)");
  return PISP_OK;
}

}  // namespace

extern "C" {

const char* pisp_last_error(const pisp_handle* h) {
  return h ? h->err.c_str() : g_last_error.c_str();
}

int pisp_create(pisp_handle** out, int device, void* stream) {
  if (!out) return fail(nullptr, PISP_ERR_INVALID_ARG, "null output pointer");
  *out = nullptr;
  if (device != -1) {
    int ndev = 0;
    cudaError_t e = cudaGetDeviceCount(&ndev);
    if (e != cudaSuccess || device < 0 || device >= ndev)
      return fail(nullptr, PISP_ERR_CUDA, "no such CUDA device");
  }
  pisp_handle* h = new pisp_handle();
  h->device = device;
  h->stream = reinterpret_cast<cudaStream_t>(stream);
  *out = h;
  return PISP_OK;
}

int pisp_destroy(pisp_handle* h) {
  if (!h) return PISP_OK;
  if (h->device < 0) {
    delete h;
    return PISP_OK;
  }
  int cur = -1;
  cudaGetDevice(&cur);
  if (cur != h->device) cudaSetDevice(h->device);
  delete h;
  if (cur >= 0) cudaSetDevice(cur);
  return PISP_OK;
}

int pisp_set_stream(pisp_handle* h, void* stream) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  h->stream = reinterpret_cast<cudaStream_t>(stream);
  return PISP_OK;
}

}  // extern "C"

namespace {

int analyze_impl(pisp_handle* h, int32_t G, const int32_t* n, const int64_t* row_ptr,
                 const int32_t* col_idx, const pisp_options* opt) {
  NvtxRange nvtx_("pisp_analyze");
  h->drop_graph();
  DeviceScope dev_scope_;
  if (G < 1 || !n || !row_ptr) return fail(h, PISP_ERR_INVALID_ARG, "bad instance description");
  int64_t N = 0;
  for (int g = 0; g < G; ++g) N += n[g] < 0 ? 0 : n[g];
  if (row_ptr[N] > 0 && !col_idx) return fail(h, PISP_ERR_INVALID_ARG, "null col_idx");
  if (h->device >= 0) {
    TRY(set_device(h, dev_scope_));
    if (!h->fork_ev) {  // side streams of the factorisation (created outside any capture)
      CK(cudaEventCreateWithFlags(&h->fork_ev, cudaEventDisableTiming));
      for (int i = 0; i < pisp_handle::kSide; ++i) {
        CK(cudaStreamCreateWithFlags(&h->side[i], cudaStreamNonBlocking));
        CK(cudaEventCreateWithFlags(&h->join_ev[i], cudaEventDisableTiming));
      }
      CK(cudaStreamCreateWithFlags(&h->big_side, cudaStreamNonBlocking));
      CK(cudaEventCreateWithFlags(&h->big_join, cudaEventDisableTiming));
    }
  }
  pisp::SymbolicOptions so;
  h->schedule = opt ? opt->solve_schedule : 0;
  h->factor_policy = opt ? opt->factor_policy : 0;
  h->kfuse = opt && opt->solve_kfuse > 0 ? opt->solve_kfuse : 1;
  h->warp_maxF = opt && opt->solve_warp_maxF > 0 ? opt->solve_warp_maxF : 32;
  h->solve_ctas = opt && opt->solve_ctas_per_sm > 0 ? std::min(4, std::max(2, opt->solve_ctas_per_sm)) : 0;
  h->factor_smem_maxF = opt && opt->factor_smem_maxF > 0 ? opt->factor_smem_maxF : 0;
  h->factor_tc = opt && opt->factor_tc ? 1 : 0;
  h->factor_ctas = opt && opt->factor_ctas_per_sm > 0 ? opt->factor_ctas_per_sm : 0;
  h->units_K = h->units_R = 0;
  if (opt) {
    so.ordering = opt->ordering;
    if (opt->relax_small >= 0) so.relax_small = opt->relax_small;
    if (opt->relax_zeros >= 0) so.relax_zeros = opt->relax_zeros;
    if (opt->analyze_threads < 0) return fail(h, PISP_ERR_INVALID_ARG, "analyze_threads must be >= 0");
    so.threads = opt->analyze_threads;
  }
  h->analyzed = h->factored = h->solved = false;
  h->any_solve = h->last_adaptive = false;
  h->plan_precision = 0;
  const auto t0 = std::chrono::steady_clock::now();
  std::string msg = pisp::analyze(G, n, row_ptr, col_idx, so, h->sym);
  h->analyze_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  if (!msg.empty()) return fail(h, PISP_ERR_INVALID_ARG, msg);
  msg = pisp::validate(h->sym);
  if (!msg.empty()) return fail(h, PISP_ERR_BOUNDS, msg);
  const pisp::Symbolic& S = h->sym;
  if (S.max_front > 46340) return fail(h, PISP_ERR_UNSUPPORTED, "front larger than 46340");
  if (h->device < 0) {  // host-only handle: symbolic structure for inspection only
    h->analyzed = true;
    return PISP_OK;
  }
  // upload the structure
  const int nS = (int)S.sn.size();
  std::vector<int32_t> c0(nS), ns(nS), ms(nS), inst(nS), child_off(nS + 1), par(nS);
  std::vector<int64_t> row_off(nS);
  for (int s = 0; s < nS; ++s) {
    c0[s] = S.sn[s].c0;
    ns[s] = S.sn[s].ns();
    ms[s] = S.sn[s].ms;
    inst[s] = S.sn[s].instance;
    par[s] = S.sn[s].parent;
    row_off[s] = S.sn[s].row_off;
  }
  for (int s = 0; s <= nS; ++s) child_off[s] = (int32_t)S.child_off[s];
  std::vector<int32_t> row_inst(S.N);
  for (int g = 0; g < G; ++g)
    for (int64_t i = S.inst_off[g]; i < S.inst_off[g + 1]; ++i) row_inst[i] = g;
  std::vector<int64_t> rp(row_ptr, row_ptr + S.N + 1);
  std::vector<int32_t> cl(col_idx ? col_idx : nullptr, col_idx ? col_idx + S.nnzA : nullptr);
  TRY(upload(h, h->c0, c0));
  TRY(upload(h, h->ns, ns));
  TRY(upload(h, h->ms, ms));
  TRY(upload(h, h->inst, inst));
  TRY(upload(h, h->front_off, S.front_off));
  TRY(upload(h, h->vec_off, S.vec_off));
  TRY(upload(h, h->row_off, row_off));
  TRY(upload(h, h->child_off, child_off));
  TRY(upload(h, h->child, S.child));
  {
    std::vector<pisp::ChildDesc> cd(S.child.size());
    for (int s = 0; s < nS; ++s)
      for (int64_t q = S.child_off[s]; q < S.child_off[s + 1]; ++q) {
        const pisp::Supernode& c = S.sn[S.child[q]];
        cd[q] = {S.front_off[S.child[q]], c.ns(), c.F(), 0, {}};
        if (S.sn[s].F() <= 32)
          for (int32_t a = 0; a < c.ms; ++a) cd[q].mask |= 1u << S.emap[c.row_off + a];
      }
    TRY(upload(h, h->cdesc, cd));
  }
  TRY(upload(h, h->amap_off, S.amap_off));
  TRY(upload(h, h->amap_src, S.amap_src));
  TRY(upload(h, h->amap_dst, S.amap_dst));
  TRY(upload(h, h->amap_coff, S.amap_coff));
  TRY(upload(h, h->rows, S.rows));
  TRY(upload(h, h->emap, S.emap));
  TRY(upload(h, h->perm, S.perm));
  TRY(upload(h, h->iperm, S.iperm));
  TRY(upload(h, h->row_inst, row_inst));
  TRY(upload(h, h->d_inst_off, S.inst_off));
  h->inst_w.assign(G, 0.0);
  for (int s = 0; s < nS; ++s) h->inst_w[S.sn[s].instance] += (double)S.sn[s].F() * S.sn[s].F();
  {
    std::vector<int32_t> order(nS), start;
    for (int s = 0; s < nS; ++s) order[s] = s;
    order = sorted_by(order, (size_t)S.max_front + 1, start, [&](int32_t s) { return S.max_front - S.sn[s].F(); });
    h->by_level = sorted_by(order, S.n_levels, start, [&](int32_t s) { return S.sn[s].level; });
    h->by_inst = sorted_by(order, G, start, [&](int32_t s) { return S.sn[s].instance; });
  }
  TRY(upload(h, h->row_ptr, rp));
  TRY(upload(h, h->col, cl));
  TRY(upload(h, h->parent, par));
  TRY(upload(h, h->inv_off, S.inv_off));
  TRY(upload(h, h->inv_child, S.inv_child));
  TRY(upload(h, h->inv_a, S.inv_a));
  {
    std::vector<int64_t> pos(S.inv_col.size());
    for (size_t q = 0; q < pos.size(); ++q) pos[q] = S.vec_off[S.inv_child[q]] + S.inv_col[q];
    TRY(upload(h, h->inv_pos, pos));
    std::vector<int32_t> pc(cl.size());
    for (size_t e = 0; e < pc.size(); ++e) pc[e] = S.iperm[cl[e]];
    TRY(upload(h, h->pcol, pc));
  }
  TRY(upload(h, h->inv_cF, S.inv_cF));
  TRY(upload(h, h->inv_col, S.inv_col));
  {
    // columns of A (CSC by counting sort): permuted row and CSR entry of every entry
    // of column j, for the transposed residuals of the adjoint sweeps
    std::vector<int64_t> atp(S.N + 1, 0);
    for (int64_t e = 0; e < S.nnzA; ++e) ++atp[cl[e] + 1];
    for (int64_t j = 0; j < S.N; ++j) atp[j + 1] += atp[j];
    std::vector<int32_t> atr(S.nnzA), ats(S.nnzA);
    std::vector<int64_t> fill(atp.begin(), atp.end() - 1);
    for (int64_t i = 0; i < S.N; ++i)
      for (int64_t e = rp[i]; e < rp[i + 1]; ++e) {
        const int64_t q = fill[cl[e]]++;
        atr[q] = S.iperm[i];
        ats[q] = (int32_t)e;
      }
    TRY(upload(h, h->at_ptr, atp));
    TRY(upload(h, h->at_src, ats));
    TRY(upload(h, h->at_prow, atr));
  }
  pisp::SymDev& sd = h->sd;
  sd.c0 = h->c0.as<int32_t>();
  sd.ns = h->ns.as<int32_t>();
  sd.ms = h->ms.as<int32_t>();
  sd.inst = h->inst.as<int32_t>();
  sd.front_off = h->front_off.as<int64_t>();
  sd.vec_off = h->vec_off.as<int64_t>();
  sd.row_off = h->row_off.as<int64_t>();
  sd.child_off = h->child_off.as<int32_t>();
  sd.child = h->child.as<int32_t>();
  sd.cdesc = h->cdesc.as<pisp::ChildDesc>();
  sd.amap_off = h->amap_off.as<int64_t>();
  sd.amap_src = h->amap_src.as<int32_t>();
  sd.amap_dst = h->amap_dst.as<int32_t>();
  sd.amap_coff = h->amap_coff.as<int64_t>();
  sd.rows = h->rows.as<int32_t>();
  sd.emap = h->emap.as<int32_t>();
  sd.perm = h->perm.as<int32_t>();
  sd.iperm = h->iperm.as<int32_t>();
  sd.row_inst = h->row_inst.as<int32_t>();
  sd.row_ptr = h->row_ptr.as<int64_t>();
  sd.col = h->col.as<int32_t>();
  sd.parent = h->parent.as<int32_t>();
  sd.inv_off = h->inv_off.as<int64_t>();
  sd.inv_child = h->inv_child.as<int32_t>();
  sd.inv_a = h->inv_a.as<int32_t>();
  sd.inv_pos = h->inv_pos.as<int64_t>();
  sd.pcol = h->pcol.as<int32_t>();
  sd.at_prow = h->at_prow.as<int32_t>();
  sd.inv_cF = h->inv_cF.as<int32_t>();
  sd.inv_col = h->inv_col.as<int32_t>();
  sd.at_ptr = h->at_ptr.as<int64_t>();
  sd.at_src = h->at_src.as<int32_t>();
  sd.N = S.N;
  sd.S = nS;
  h->analyzed = true;
  return PISP_OK;
}

}  // namespace

extern "C" {

int pisp_analyze(pisp_handle* h, int32_t G, const int32_t* n, const int64_t* row_ptr,
                 const int32_t* col_idx, const pisp_options* opt) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  return no_throw(h, [&] { return analyze_impl(h, G, n, row_ptr, col_idx, opt); });
}

int pisp_match_rows(int32_t n, const int64_t* row_ptr, const int32_t* col_idx, int32_t* row_perm) {
  if (n < 0 || (n > 0 && (!row_ptr || !row_perm))) return fail(nullptr, PISP_ERR_INVALID_ARG, "bad arguments");
  if (n == 0) return PISP_OK;
  if (row_ptr[0] != 0) return fail(nullptr, PISP_ERR_INVALID_ARG, "row_ptr[0] must be 0");
  for (int32_t i = 0; i < n; ++i)
    if (row_ptr[i + 1] < row_ptr[i]) return fail(nullptr, PISP_ERR_INVALID_ARG, "row_ptr must be nondecreasing");
  if (row_ptr[n] > 0 && !col_idx) return fail(nullptr, PISP_ERR_INVALID_ARG, "null col_idx");
  for (int64_t e = 0; e < row_ptr[n]; ++e)
    if (col_idx[e] < 0 || col_idx[e] >= n) return fail(nullptr, PISP_ERR_INVALID_ARG, "column index out of range");
  std::vector<int32_t> row_of_col;
  const std::string err = pisp::match_rows(n, row_ptr, col_idx, row_of_col);
  if (!err.empty()) return fail(nullptr, PISP_ERR_INVALID_ARG, err);
  std::copy(row_of_col.begin(), row_of_col.end(), row_perm);
  return PISP_OK;
}

int pisp_weights(const double* t, int32_t K, double* beta) {
  if (!t || !beta || K < 1 || K > PISP_K_MAX)
    return fail(nullptr, PISP_ERR_INVALID_ARG, "pisp_weights: bad arguments");
  for (int k = 0; k < K; ++k) {
    if (!std::isfinite(t[k])) return fail(nullptr, PISP_ERR_INVALID_ARG, "non-finite shift");
    for (int l = 0; l < k; ++l)
      if (t[l] == t[k]) return fail(nullptr, PISP_ERR_INVALID_ARG, "shifts must be distinct");
  }
  // Lagrange basis polynomial of node t_k evaluated at 0: the unique weights
  // with sum_k beta_k t_k^j = [j == 0] for j < K.
  for (int k = 0; k < K; ++k) {
    long double p = 1.0L;
    for (int l = 0; l < K; ++l)
      if (l != k) p *= (long double)t[l] / ((long double)t[l] - (long double)t[k]);
    beta[k] = (double)p;
  }
  return PISP_OK;
}

int pisp_factor_perturbed(pisp_handle* h, const double* values, const double* D,
                          const double* t, int32_t K, int32_t precision) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (!h->capturing) h->graph_valid = false;
  NvtxRange nvtx_("pisp_factor_perturbed");
  if (!h->analyzed) return fail(h, PISP_ERR_NOT_ANALYZED, "pisp_analyze has not succeeded");
  if (K < 1 || K > PISP_K_MAX || !t) return fail(h, PISP_ERR_INVALID_ARG, "K must be in 1..16");
  if (precision != PISP_FP32 && precision != PISP_FP64)
    return fail(h, PISP_ERR_INVALID_ARG, "precision must be PISP_FP32 or PISP_FP64");
  const pisp::Symbolic& S = h->sym;
  if ((S.nnzA > 0 && !values) || (S.N > 0 && !D)) return fail(h, PISP_ERR_INVALID_ARG, "null values or D");
  // the owner tiles (policy 0) take fronts of any size; the per-panel path,
  // which the other policies fall back to, needs a panel in shared memory
  if (S.max_front > pisp::max_solve_front(precision) ||
      (h->factor_policy != 0 && h->factor_policy != 4 && S.max_front > pisp::max_big_front(precision)))
    return fail(h, PISP_ERR_UNSUPPORTED, "front too large for this precision");
  double beta[PISP_K_MAX];
  if (pisp_weights(t, K, beta) != PISP_OK) return fail(h, PISP_ERR_INVALID_ARG, g_last_error);
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  h->factored = h->solved = false;
  h->K_hint = K;
  if (h->plan_precision != precision || h->plan_K != K) TRY(no_throw(h, [&] { return build_plans(h, precision); }));
  h->plan_K = K;
  h->K = K;
  h->precision = precision;
  for (int k = 0; k < K; ++k) {
    h->t[k] = t[k];
    h->beta[k] = beta[k];
  }
  if (!h->fronts.ensure((size_t)K * S.front_elems * esize(precision)) ||
      !h->vals.ensure(S.nnzA * sizeof(double)) || !h->D.ensure(S.N * sizeof(double)) ||
      !h->status.ensure((size_t)S.G * K * sizeof(int32_t)) ||
      !h->badcol.ensure((size_t)S.G * K * sizeof(int32_t)))
    return fail(h, PISP_ERR_OOM, "device allocation failed (factor workspace)");
  if (S.nnzA) CK(cudaMemcpyAsync(h->vals.p, values, S.nnzA * sizeof(double), cudaMemcpyDeviceToDevice, h->stream));
  if (S.N) CK(cudaMemcpyAsync(h->D.p, D, S.N * sizeof(double), cudaMemcpyDeviceToDevice, h->stream));
  CK(cudaMemsetAsync(h->status.p, 0, (size_t)S.G * K * sizeof(int32_t), h->stream));
  CK(cudaMemsetAsync(h->badcol.p, 0x7f, (size_t)S.G * K * sizeof(int32_t), h->stream));
  if (!h->serr.ensure(sizeof(int))) return fail(h, PISP_ERR_OOM, "device allocation failed");
  CK(cudaMemsetAsync(h->serr.p, 0, sizeof(int), h->stream));
  h->launches = 0;
  const pisp::Shifts sh = make_shifts(h, h->beta);
  if (h->fac_single) {
    // every level, every shift and every instance in one persistent launch
    CK(cudaMemsetAsync(h->fticket.p, 0, sizeof(int), h->stream));
    CK(cudaMemsetAsync(h->fdone.p, 0, S.sn.size() * (size_t)K * pisp::kCtrStride * sizeof(int), h->stream));
    if (h->fac_nflags) CK(cudaMemsetAsync(h->fflags.p, 0, (size_t)h->fac_nflags * sizeof(int), h->stream));
    const int pb = prof_begin(h);
    const int n = pisp::launch_factor_persistent(
        precision, h->sd, h->d_ftasks.as<pisp::FactorTask>(), h->n_ftasks, h->fticket.as<int>(), h->fdone.as<int>(),
        h->d_fneed.as<int>(), h->fflags.as<int>(), h->serr.as<int>(), h->d_fwl.as<int32_t>(), h->vals.as<double>(),
        h->D.as<double>(), sh, h->fronts.p, h->status.as<int32_t>(), h->badcol.as<int32_t>(), h->fac_CH,
        h->fac_smem, h->factor_policy == 4 ? h->wait_polls : 0, h->factor_tc, h->fac_ctas, h->stream);
    TRY(count(h, n));
    prof_end(h, pb, PISP_PROF_FACTOR, K * h->fac_bytes, n);
    h->factored = true;
    return PISP_OK;
  }
  for (int l = 0; l < S.n_levels; ++l) {
    // The fronts of a level are independent: its wide fronts (owner kernel)
    // and each size class of its narrow ones go to their own streams, forked
    // from the work queued so far and joined before the next level (parallel
    // branches when the caller captures the work into a CUDA graph).
    const pisp::LevelPlan& lp = h->plans[l];
    const bool mixed = lp.big_count > 0 && lp.n_groups > 0;
    const int used = lp.n_groups > 1 ? std::min(lp.n_groups - 1, pisp_handle::kSide) : 0;
    if (used > 0 || mixed) CK(cudaEventRecord(h->fork_ev, h->stream));
    for (int i = 0; i < used; ++i) CK(cudaStreamWaitEvent(h->side[i], h->fork_ev, 0));
    const cudaStream_t bst = mixed ? h->big_side : h->stream;
    if (mixed) CK(cudaStreamWaitEvent(bst, h->fork_ev, 0));
    if (lp.big_count > 0) {
      const int pb = prof_begin(h, bst);
      int n = 0;
      if (lp.dag_tasks > 0) {
        CK(cudaMemsetAsync(h->dag_ticket.p, 0, sizeof(int), bst));
        CK(cudaMemsetAsync(h->dag_flags.p, 0, (size_t)lp.dag_flags * sizeof(int), bst));
        n = pisp::launch_factor_big_dag(precision, h->sd, lp, h->d_big.as<int32_t>(),
                                        h->d_dag.as<pisp::DagTask>(), h->dag_ticket.as<int>(),
                                        h->dag_flags.as<int>(), h->serr.as<int>(), h->vals.as<double>(),
                                        h->D.as<double>(), sh, h->fronts.p, h->status.as<int32_t>(),
                                        h->badcol.as<int32_t>(), h->factor_tc, bst);
      } else {
        n = pisp::launch_factor_big(precision, h->sd, lp, h->d_big.as<int32_t>(), h->h_bigF.data(),
                                    h->vals.as<double>(), h->D.as<double>(), sh, h->fronts.p,
                                    h->status.as<int32_t>(), h->badcol.as<int32_t>(), bst);
      }
      TRY(count(h, n));
      prof_end(h, pb, PISP_PROF_FACTOR_BIG, K * lp.bytes_fbig, n, bst);
    }
    if (lp.n_groups > 0) {
      const int pb = prof_begin(h);
      int n = 0;
      for (int g = 0; g < lp.n_groups && n >= 0; ++g) {
        const cudaStream_t st = g == 0 ? h->stream : h->side[(g - 1) % pisp_handle::kSide];
        const int m = pisp::launch_factor_small_group(precision, h->sd, lp, g, h->d_small.as<int32_t>(),
                                                      h->vals.as<double>(), h->D.as<double>(), sh,
                                                      h->fronts.p, h->status.as<int32_t>(),
                                                      h->badcol.as<int32_t>(), st);
        n = m < 0 ? -1 : n + m;
      }
      for (int i = 0; i < used; ++i) {
        CK(cudaEventRecord(h->join_ev[i], h->side[i]));
        CK(cudaStreamWaitEvent(h->stream, h->join_ev[i], 0));
      }
      TRY(count(h, n));
      prof_end(h, pb, PISP_PROF_FACTOR_SMALL, K * lp.bytes_fsmall, n);
    }
    if (mixed) {
      CK(cudaEventRecord(h->big_join, bst));
      CK(cudaStreamWaitEvent(h->stream, h->big_join, 0));
    }
  }
  h->factored = true;
  return PISP_OK;
}

int pisp_solve(pisp_handle* h, const double* b, int32_t R, const double* w, double* x,
               int32_t sweeps) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (!h->capturing) h->graph_valid = false;
  NvtxRange nvtx_("pisp_solve");
  if (!h->factored) return fail(h, PISP_ERR_NOT_FACTORED, "no factorisation");
  if (R < 1 || sweeps < 0) return fail(h, PISP_ERR_INVALID_ARG, "R must be >= 1, sweeps >= 0");
  if (h->sym.N > 0 && (!b || !x)) return fail(h, PISP_ERR_INVALID_ARG, "null b or x");
  if (b == x && b) return fail(h, PISP_ERR_INVALID_ARG, "x may not alias b");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  TRY(set_weights(h, w, h->w_last));
  // from here on the kept solutions go, and with more right-hand sides than fit
  // the workspace too: until this solve is queued nothing may be made of them
  h->solved = false;
  TRY(ensure_solve_buffers(h, R));
  const pisp::Shifts sh = make_shifts(h, h->w_last);
  TRY(solve_core(h, b, h->X.as<double>(), R, sweeps, sh));
  const int pb = prof_begin(h);
  const int n = pisp::launch_combine(h->sd, h->X.as<double>(), sh, R, x, h->stream);
  TRY(count(h, n));
  prof_end(h, pb, PISP_PROF_COMBINE, (double)h->sym.N * R * 8.0 * (h->K + 1) + h->sym.N * 4.0, n);
  TRY(count(h, pisp::launch_fill_nan_failed(h->sd, h->status.as<int32_t>(), h->K, R, x, h->stream)));
  h->R = R;
  h->solved = true;
  return PISP_OK;
}

int pisp_combine(pisp_handle* h, const double* w, double* x) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  NvtxRange nvtx_("pisp_combine");
  if (!h->solved) return fail(h, PISP_ERR_NOT_FACTORED, "pisp_solve has not run");
  if (h->sym.N > 0 && !x) return fail(h, PISP_ERR_INVALID_ARG, "null x");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  double ww[PISP_K_MAX];
  TRY(set_weights(h, w, ww));
  const pisp::Shifts sh = make_shifts(h, ww);
  TRY(count(h, pisp::launch_combine(h->sd, h->X.as<double>(), sh, h->R, x, h->stream)));
  TRY(count(h, pisp::launch_fill_nan_failed(h->sd, h->status.as<int32_t>(), h->K, h->R, x, h->stream)));
  return PISP_OK;
}

int pisp_refine(pisp_handle* h, const double* b, double* x, int32_t R, int32_t iters,
                int32_t sweeps) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (!h->capturing) h->graph_valid = false;
  NvtxRange nvtx_("pisp_refine");
  if (!h->factored) return fail(h, PISP_ERR_NOT_FACTORED, "no factorisation");
  if (R < 1 || iters < 0 || sweeps < 0) return fail(h, PISP_ERR_INVALID_ARG, "bad R/iters/sweeps");
  if (h->sym.N > 0 && (!b || !x)) return fail(h, PISP_ERR_INVALID_ARG, "null b or x");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  // more right-hand sides than the last solve may reallocate the store of the
  // kept per-perturbation solutions: they are then gone, and pisp_combine /
  // pisp_adjoint refuse until the next pisp_solve
  if (h->solved && R > h->R) h->solved = false;
  TRY(ensure_solve_buffers(h, R));
  const size_t nkr = (size_t)h->sym.N * h->K * pisp::rhs_stride64(R) * sizeof(double);
  const size_t nr = (size_t)h->sym.N * R * sizeof(double);
  if (!h->X2.ensure(nkr) || !h->rtmp.ensure(nr) || !h->dtmp.ensure(nr))
    return fail(h, PISP_ERR_OOM, "device allocation failed (refine workspace)");
  const pisp::Shifts sh = make_shifts(h, h->beta);
  for (int it = 0; it < iters; ++it) {
    TRY(count(h, pisp::launch_residual(h->sd, h->vals.as<double>(), b, x, R, h->rtmp.as<double>(), h->stream)));
    TRY(solve_core(h, h->rtmp.as<double>(), h->X2.as<double>(), R, sweeps, sh));
    TRY(count(h, pisp::launch_combine(h->sd, h->X2.as<double>(), sh, R, h->dtmp.as<double>(), h->stream)));
    TRY(count(h, pisp::launch_axpy((int64_t)h->sym.N * R, h->dtmp.as<double>(), x, h->stream)));
  }
  TRY(count(h, pisp::launch_fill_nan_failed(h->sd, h->status.as<int32_t>(), h->K, R, x, h->stream)));
  return PISP_OK;
}

int pisp_adjoint(pisp_handle* h, const double* g, const double* w, double* grad_b,
                 double* grad_values, int32_t sweeps) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  NvtxRange nvtx_("pisp_adjoint");
  if (!h->solved) return fail(h, PISP_ERR_NOT_FACTORED, "pisp_solve has not run");
  if (h->sym.N > 0 && !g) return fail(h, PISP_ERR_INVALID_ARG, "null g");
  if (sweeps < 0) return fail(h, PISP_ERR_INVALID_ARG, "sweeps must be >= 0");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  double ww[PISP_K_MAX];
  TRY(set_weights(h, w, ww));
  const int32_t R = h->R;
  if (!h->Lam.ensure((size_t)h->sym.N * h->K * pisp::rhs_stride64(R) * sizeof(double)))
    return fail(h, PISP_ERR_OOM, "device allocation failed (adjoint workspace)");
  const pisp::Shifts sh = make_shifts(h, ww);
  TRY(solve_pass(h, true, first_solve(h, g, h->Lam.as<double>()), R));
  // FP64 residual sweeps of every lambda_k on the transposed systems, as the
  // forward sweeps do for x_k: with FP32 factors the adjoint then reaches the
  // FP64 definition too (Rk and Y are the solve's workspace, sized for R)
  for (int it = 0; it < sweeps; ++it) {
    TRY(count(h, pisp::launch_residual_T_per_k(h->precision, h->sd, h->vals.as<double>(), h->D.as<double>(), sh, g,
                                               h->Lam.as<double>(), R, h->Rk.p, h->stream)));
    TRY(solve_pass(h, true, {nullptr, h->Rk.p, h->Y.p, h->Lam.as<double>(), pisp::kXdAdd}, R));
  }
  if (grad_b) TRY(count(h, pisp::launch_combine(h->sd, h->Lam.as<double>(), sh, R, grad_b, h->stream)));
  if (grad_values)
    TRY(count(h, pisp::launch_grad_values(h->sd, h->Lam.as<double>(), h->X.as<double>(), sh, R,
                                          grad_values, h->stream)));
  return PISP_OK;
}

int pisp_graph_capture(pisp_handle* h, const double* values, const double* D, const double* t,
                       int32_t K, int32_t precision, const double* b, int32_t R, const double* w,
                       double* x, int32_t sweeps, const double* g, double* grad_b, double* grad_values,
                       int32_t adjoint_sweeps) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  NvtxRange nvtx_("pisp_graph_capture");
  if (!h->analyzed) return fail(h, PISP_ERR_NOT_ANALYZED, "pisp_analyze has not succeeded");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  h->drop_graph();
  // one eager step: checks the arguments, allocates every workspace the step
  // needs (nothing may be allocated during the capture) and leaves its results
  auto step = [&]() -> int {
    TRY(pisp_factor_perturbed(h, values, D, t, K, precision));
    TRY(pisp_solve(h, b, R, w, x, sweeps));
    if (g) TRY(pisp_adjoint(h, g, w, grad_b, grad_values, adjoint_sweeps));
    return PISP_OK;
  };
  TRY(step());
  if (h->prof_on) {  // only the brackets recorded into the graph are replayed
    h->prof_next = 0;
    h->prof_br.clear();
  }
  if (!h->cap_stream) {
    CK(cudaStreamCreateWithFlags(&h->cap_stream, cudaStreamNonBlocking));
    CK(cudaEventCreateWithFlags(&h->cap_ev, cudaEventDisableTiming));
  }
  // capture on a private stream ordered after the work queued so far
  CK(cudaEventRecord(h->cap_ev, h->stream));
  CK(cudaStreamWaitEvent(h->cap_stream, h->cap_ev, 0));
  const cudaStream_t user = h->stream;
  h->stream = h->cap_stream;
  h->capturing = true;
  cudaError_t e = cudaStreamBeginCapture(h->cap_stream, cudaStreamCaptureModeThreadLocal);
  int rc = e == cudaSuccess ? step() : PISP_ERR_CUDA;
  cudaGraph_t gr = nullptr;
  const cudaError_t e2 = e == cudaSuccess ? cudaStreamEndCapture(h->cap_stream, &gr) : e;
  h->capturing = false;
  h->stream = user;
  if (rc) {
    if (gr) cudaGraphDestroy(gr);
    return rc;
  }
  if (e2 != cudaSuccess || !gr)
    return fail(h, PISP_ERR_CUDA, std::string("stream capture failed: ") + cudaGetErrorString(e2));
  h->graph = gr;
  CK(cudaGraphInstantiate(&h->graph_exec, h->graph, 0));
  h->graph_valid = true;
  return PISP_OK;
}

int pisp_graph_launch(pisp_handle* h) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (!h->graph_valid || !h->graph_exec)
    return fail(h, PISP_ERR_INVALID_ARG, "no valid captured step (pisp_graph_capture)");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  CK(cudaGraphLaunch(h->graph_exec, h->stream));
  return PISP_OK;
}

int pisp_set_wait_limit(pisp_handle* h, int64_t polls, int32_t unreachable) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (polls < 0) return fail(h, PISP_ERR_INVALID_ARG, "polls must be >= 0");
  h->wait_polls = polls;
  h->wait_unreachable = unreachable ? 1 : 0;
  h->units_K = h->units_R = 0;  // the next persistent solve rebuilds its targets
  h->graph_valid = false;
  return PISP_OK;
}

int pisp_set_refinement(pisp_handle* h, double tol) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (!(tol >= 0.0) || !std::isfinite(tol)) return fail(h, PISP_ERR_INVALID_ARG, "tol must be finite and >= 0");
  h->sweep_tol = tol;
  return PISP_OK;
}

int pisp_refinement_stats(pisp_handle* h, int32_t* sweeps_per_instance, double* work, double* rows,
                          int32_t max_sweeps) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (max_sweeps < 0) return fail(h, PISP_ERR_INVALID_ARG, "max_sweeps must be >= 0");
  if (!h->any_solve) return fail(h, PISP_ERR_NOT_FACTORED, "no solve");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  std::vector<int32_t> nsw;
  std::vector<double> fs, fr;
  TRY(sweep_fractions(h, std::max(max_sweeps, 1), nsw, fs, fr));
  if (sweeps_per_instance) std::copy(nsw.begin(), nsw.end(), sweeps_per_instance);
  for (int q = 0; q < max_sweeps; ++q) {
    if (work) work[q] = fs[q + 1];
    if (rows) rows[q] = fr[q + 1];
  }
  return PISP_OK;
}

int pisp_get_status(pisp_handle* h, int32_t* per_instance_k, int32_t* first_bad_col) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (!h->factored) return fail(h, PISP_ERR_NOT_FACTORED, "no factorisation");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  const size_t n = (size_t)h->sym.G * h->K;
  std::vector<int32_t> st(n), bc(n);
  CK(cudaMemcpyAsync(st.data(), h->status.p, n * sizeof(int32_t), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaMemcpyAsync(bc.data(), h->badcol.p, n * sizeof(int32_t), cudaMemcpyDeviceToHost, h->stream));
  int serr = 0;
  CK(cudaMemcpyAsync(&serr, h->serr.p, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  if (serr) {
    h->err = "a bounded dependency wait of the persistent solve gave up";
    return PISP_ERR_TIMEOUT;
  }
  int worst = PISP_OK;
  for (size_t q = 0; q < n; ++q) {
    int code = PISP_OK;
    if (st[q] & 1) code = PISP_ERR_ZERO_PIVOT;
    else if (st[q] & 2) code = PISP_ERR_NONFINITE;
    if (per_instance_k) per_instance_k[q] = code;
    if (first_bad_col) first_bad_col[q] = code ? bc[q] : -1;
    if (code == PISP_ERR_ZERO_PIVOT || (code && worst == PISP_OK)) worst = code;
  }
  return worst;
}

int pisp_get_stats(const pisp_handle* h, pisp_stats* o) {
  if (!h || !o) return PISP_ERR_INVALID_ARG;
  if (!h->analyzed) return PISP_ERR_NOT_ANALYZED;
  const pisp::Symbolic& S = h->sym;
  std::memset(o, 0, sizeof(*o));
  o->N = S.N;
  o->nnzA = S.nnzA;
  o->nnzL = S.nnzL;
  o->nnzF_stored = S.nnzF_stored;
  o->front_elems = S.front_elems;
  o->G = S.G;
  o->n_supernodes = (int32_t)S.sn.size();
  o->n_levels = S.n_levels;
  o->max_front = S.max_front;
  o->etree_height = S.etree_height;
  o->K = h->K;
  o->precision = h->precision;
  o->gpu_launches = h->launches;
  if (h->last_loop && h->loop_kernels > 0 && h->r_sweep.p) {
    // a device-side sweep loop counted its body once: add its further iterations
    pisp_handle* hh = const_cast<pisp_handle*>(h);
    DeviceScope dev_scope_;
    if (set_device(hh, dev_scope_) == PISP_OK) {
      int32_t iters = 0;
      if (cudaMemcpyAsync(&iters, h->r_sweep.p, sizeof(int32_t), cudaMemcpyDeviceToHost, h->stream) == cudaSuccess &&
          cudaStreamSynchronize(h->stream) == cudaSuccess && iters > 1)
        o->gpu_launches += h->loop_kernels * (iters - 1);
    }
  }
  o->flops_factor = S.flops_factor;
  o->flops_solve = S.flops_solve;
  o->analyze_ms = h->analyze_ms;
  return PISP_OK;
}

int pisp_get_perm(const pisp_handle* h, int32_t* perm) {
  if (!h || !perm) return PISP_ERR_INVALID_ARG;
  if (!h->analyzed) return PISP_ERR_NOT_ANALYZED;
  std::copy(h->sym.perm.begin(), h->sym.perm.end(), perm);
  return PISP_OK;
}

int pisp_get_supernodes(const pisp_handle* h, int32_t* c0, int32_t* c1, int32_t* ms,
                        int32_t* rows) {
  if (!h) return PISP_ERR_INVALID_ARG;
  if (!h->analyzed) return PISP_ERR_NOT_ANALYZED;
  const auto& S = h->sym;
  for (size_t s = 0; s < S.sn.size(); ++s) {
    if (c0) c0[s] = S.sn[s].c0;
    if (c1) c1[s] = S.sn[s].c1;
    if (ms) ms[s] = S.sn[s].ms;
  }
  if (rows) std::copy(S.rows.begin(), S.rows.end(), rows);
  return PISP_OK;
}

int pisp_get_front(pisp_handle* h, int32_t s, int32_t k, double* out, int32_t* F_out) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (!h->factored) return fail(h, PISP_ERR_NOT_FACTORED, "no factorisation");
  if (s < 0 || s >= (int32_t)h->sym.sn.size() || k < 0 || k >= h->K)
    return fail(h, PISP_ERR_INVALID_ARG, "supernode or k out of range");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  const int64_t F = h->sym.sn[s].F();
  if (F_out) *F_out = (int32_t)F;
  if (!out) return PISP_OK;
  const size_t es = esize(h->precision);
  const size_t off = ((size_t)h->K * h->sym.front_off[s] + (size_t)k * F * F) * es;
  std::vector<unsigned char> buf(F * F * es);
  CK(cudaMemcpyAsync(buf.data(), (const char*)h->fronts.p + off, buf.size(), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  for (int64_t q = 0; q < F * F; ++q)
    out[q] = es == 4 ? (double)reinterpret_cast<const float*>(buf.data())[q]
                     : reinterpret_cast<const double*>(buf.data())[q];
  return PISP_OK;
}

int pisp_get_pivot_range(pisp_handle* h, double* min_abs, double* max_abs) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (!h->factored) return fail(h, PISP_ERR_NOT_FACTORED, "no factorisation");
  if (!min_abs || !max_abs) return fail(h, PISP_ERR_INVALID_ARG, "null output");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  const pisp::Symbolic& S = h->sym;
  const int K = h->K;
  const size_t es = esize(h->precision);
  const size_t GK = (size_t)S.G * K;
  std::vector<double> lo(GK, HUGE_VAL), hi(GK, 0.0);
  std::vector<char> bad(GK, 0);
  // pivots of perturbation k, permuted column c, at buf[k * N + c]
  std::vector<unsigned char> buf((size_t)S.N * K * es);
  for (size_t s = 0; s < S.sn.size(); ++s) {
    const pisp::Supernode& sn = S.sn[s];
    const int64_t F = sn.F(), ns = sn.ns();
    for (int k = 0; k < K; ++k) {
      // u_jj of the front's pivot block sits at j + j*F of the column-major
      // F x F front of (s, k): every (F + 1)-th element, ns of them
      const char* src = (const char*)h->fronts.p + ((size_t)K * S.front_off[s] + (size_t)k * F * F) * es;
      CK(cudaMemcpy2DAsync(buf.data() + ((size_t)k * S.N + sn.c0) * es, es, src, (size_t)(F + 1) * es, es,
                           (size_t)ns, cudaMemcpyDeviceToHost, h->stream));
    }
  }
  CK(cudaStreamSynchronize(h->stream));
  for (size_t s = 0; s < S.sn.size(); ++s) {
    const pisp::Supernode& sn = S.sn[s];
    for (int k = 0; k < K; ++k) {
      const size_t q = (size_t)sn.instance * K + k;
      for (int32_t c = sn.c0; c < sn.c1; ++c) {
        const size_t e = (size_t)k * S.N + c;
        const double u = std::fabs(es == 4 ? (double)reinterpret_cast<const float*>(buf.data())[e]
                                           : reinterpret_cast<const double*>(buf.data())[e]);
        if (!std::isfinite(u)) bad[q] = 1;
        lo[q] = std::min(lo[q], u);
        hi[q] = std::max(hi[q], u);
      }
    }
  }
  for (size_t q = 0; q < GK; ++q) {
    const bool empty = lo[q] == HUGE_VAL;  // an instance with no unknowns
    min_abs[q] = bad[q] || empty ? NAN : lo[q];
    max_abs[q] = bad[q] || empty ? NAN : hi[q];
  }
  return PISP_OK;
}

int pisp_solve_host(pisp_handle* h, const double* values_host, const double* D_host,
                    const double* t, int32_t K, int32_t precision, const double* b_host,
                    int32_t R, double* x_host, int32_t sweeps) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  NvtxRange nvtx_("pisp_solve_host");
  h->graph_valid = false;
  if (!h->analyzed) return fail(h, PISP_ERR_NOT_ANALYZED, "pisp_analyze has not succeeded");
  if (R < 1) return fail(h, PISP_ERR_INVALID_ARG, "R must be >= 1");
  const pisp::Symbolic& S = h->sym;
  if ((S.nnzA && !values_host) || (S.N && (!D_host || !b_host || !x_host)))
    return fail(h, PISP_ERR_INVALID_ARG, "null host buffer");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  const size_t nv = S.nnzA * sizeof(double), nd = S.N * sizeof(double);
  const size_t nb = (size_t)S.N * R * sizeof(double);
  if (!h->in_vals.ensure(nv) || !h->in_D.ensure(nd) || !h->in_b.ensure(nb) || !h->out_x.ensure(nb))
    return fail(h, PISP_ERR_OOM, "device allocation failed (host staging)");
  if (!h->copy_stream) {
    CK(cudaStreamCreateWithFlags(&h->copy_stream, cudaStreamNonBlocking));
    for (cudaEvent_t& e : h->copy_ev) CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  }
  if (nv) CK(cudaMemcpyAsync(h->in_vals.p, values_host, nv, cudaMemcpyHostToDevice, h->stream));
  if (nd) CK(cudaMemcpyAsync(h->in_D.p, D_host, nd, cudaMemcpyHostToDevice, h->stream));
  // b after the values and D (the factorisation needs those first), copied
  // while the factorisation runs; the solve waits for it
  CK(cudaEventRecord(h->copy_ev[0], h->stream));
  CK(cudaStreamWaitEvent(h->copy_stream, h->copy_ev[0], 0));
  if (nb) CK(cudaMemcpyAsync(h->in_b.p, b_host, nb, cudaMemcpyHostToDevice, h->copy_stream));
  CK(cudaEventRecord(h->copy_ev[1], h->copy_stream));
  TRY(pisp_factor_perturbed(h, h->in_vals.as<double>(), h->in_D.as<double>(), t, K, precision));
  CK(cudaStreamWaitEvent(h->stream, h->copy_ev[1], 0));
  TRY(pisp_solve(h, h->in_b.as<double>(), R, nullptr, h->out_x.as<double>(), sweeps));
  if (nb) CK(cudaMemcpyAsync(x_host, h->out_x.p, nb, cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return PISP_OK;
}

int pisp_profile(pisp_handle* h, int32_t on) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  if (on) {
    DeviceScope dev_scope_;
    TRY(set_device(h, dev_scope_));
    while (h->prof_ev.size() < 2048) {  // events exist before any stream capture
      cudaEvent_t e;
      CK(cudaEventCreate(&e));
      h->prof_ev.push_back(e);
    }
    h->prof_on = true;
    h->prof_next = 0;
    h->prof_br.clear();
  } else {
    h->prof_on = false;
  }
  return PISP_OK;
}

int pisp_profile_collect(pisp_handle* h) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  DeviceScope dev_scope_;
  TRY(set_device(h, dev_scope_));
  CK(cudaStreamSynchronize(h->stream));
  bool loop = false;
  for (const auto& b : h->prof_br) loop = loop || b.sweep == -1;
  std::vector<int32_t> nsw;
  std::vector<double> fs, fr;
  if (loop && h->last_adaptive) TRY(sweep_fractions(h, std::max(h->last_sweeps, 1), nsw, fs, fr));
  for (const auto& b : h->prof_br) {
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, h->prof_ev[b.e0], h->prof_ev[b.e1]));
    h->prof_ms[b.fam] += ms;
    if (b.sweep == -1) {  // a device-side loop: one iteration per sweep any instance took
      int iters = 0;
      double by = 0.0;
      for (int s = 1; s < (int)fs.size(); ++s)
        if (fr[s] > 0.0) {
          ++iters;
          by += fr[s] * b.bytes_rows + fs[s] * b.bytes_work;
        }
      h->prof_bytes[b.fam] += by;
      h->prof_launches[b.fam] += (int64_t)b.launches * iters;
      continue;
    }
    h->prof_bytes[b.fam] += b.bytes;
    h->prof_launches[b.fam] += b.launches;
  }
  return PISP_OK;
}

int pisp_profile_read(pisp_handle* h, int32_t family, double* ms, double* bytes,
                      int64_t* launches) {
  if (!h || family < 0 || family >= PISP_PROF_FAMILIES)
    return fail(h, PISP_ERR_INVALID_ARG, "bad profiling family");
  if (ms) *ms = h->prof_ms[family];
  if (bytes) *bytes = h->prof_bytes[family];
  if (launches) *launches = h->prof_launches[family];
  return PISP_OK;
}

int pisp_profile_reset(pisp_handle* h) {
  if (!h) return fail(h, PISP_ERR_INVALID_ARG, "null handle");
  for (int f = 0; f < PISP_PROF_FAMILIES; ++f) {
    h->prof_ms[f] = h->prof_bytes[f] = 0.0;
    h->prof_launches[f] = 0;
  }
  return PISP_OK;
}

const char* pisp_profile_name(int32_t family) {
  return (family >= 0 && family < PISP_PROF_FAMILIES) ? kFamilyNames[family] : "";
}

}  // extern "C"
