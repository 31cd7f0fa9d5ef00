// The triangular solves of every front, shift and right-hand side as one
// kernel per direction: L y = v (forward) and U x = y (backward), or for the
// adjoint U^T y = v and L^T x = y with the same factors.  Included by one
// translation unit per (factor precision, direction).
//
// Layouts (T = factor precision):
//   V   [sum F][K][RV]  T, front vectors: row vec_off[s] + i of front s holds
//                       the forward solution of its pivot rows and the
//                       contribution of its update rows to the parent
//   xt  [N][K][RV]      T, solution in permuted row order (read back by the
//                       descendants' backward solves)
//   xd  [N][K][RX]      FP64, solution or running sum, permuted row order
//   rk  [N][K][RV]      T, per-shift right-hand sides, permuted row order
//   b   [N][R]          FP64, broadcast right-hand side, original row order
// RV and RX round R up so that rows are read and written with 16-byte accesses;
// the padding holds anything and reaches no result.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "pisp_internal.h"

namespace pisp {
namespace {

constexpr int kSolveThreads = 256;
constexpr int kSolveWarps = kSolveThreads / 32;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kBS = 33;                              // padded row of a staged 32 x 32 block
// Shared memory a launch may ask for.  The most is asked for by column tasks of
// FP64 factors with two right-hand sides, whose 32 columns are 16 shifts (K = 16:
// 158720 bytes, one CTA an SM); checked at compile time with the layouts below.
constexpr int kSolveSmemMax = 160 * 1024;

__device__ __forceinline__ int ld_relaxed(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// One thread waits until *f >= need, asleep between polls for at most wait_ns in
// all; then gives up and records it.  Returns the count seen.  Whatever thread group continues is
// ordered after the acquiring load by the caller's barrier; the data themselves
// are read past L1.  The polls in between are relaxed (an acquiring one drops
// the SM's L1 lines each time, under the CTAs at work beside it) and end with an
// acquiring load, not a fence: that also waits for the thread's own stores,
// 0.6 us more a level of the tree.  They grow apart, by an eighth of the time
// waited up to 1 us, and every counter has a sector of its own (kCtrStride):
// hundreds of pollers on a few lines fill the L2 slices that hold them, ahead of
// the results and the counts they wait for.
__device__ __forceinline__ int wait_count(const int* f, int need, int* err, int64_t wait_ns) {
  int v = ld_acquire(f);
  if (v >= need) return v;
  unsigned ns = 32;
  for (int64_t left = wait_ns; left > 0;) {
    __nanosleep(ns);
    if (ld_relaxed(f) >= need) break;
    left -= ns;
    ns += ns < 1024 ? ns >> 3 : 0;
  }
  v = ld_acquire(f);
  if (v < need) atomicExch(err, 1);
  return v;
}

// Counts one finished task; the release covers the writes of the group whose
// barrier precedes it.
__device__ __forceinline__ void publish(int* f) {
  asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(f) : "memory");
}

// Completion counters.  Tasks cover a group of columns (one shift, or in the
// backward solve of several right-hand sides 32 (k, r) columns), and a front
// counts per group, so that the groups run through the tree independently.
// Forward, a front waits for the tasks of its children, counted at itself;
// backward, for those of its parent, counted at the parent.  Backward with
// several right-hand sides a front solved by segments or with more than 32 pivots is
// cut by shift, and counts all its tasks together (at group 0).
template <typename T>
__device__ __forceinline__ void wait_children(const SolveArgs<T>& a, const FrontDesc& d, int g) {
  if (a.done && d.needF > 0) wait_count(a.done + ((int64_t)d.s * a.NG + g) * kCtrStride, d.needF, a.err, a.wait_ns);
}
template <typename T>
__device__ __forceinline__ void publish_up(const SolveArgs<T>& a, const FrontDesc& d, int g) {
  if (!a.done || d.parent < 0) return;
  int* c = a.done + (int64_t)d.parent * a.NG * kCtrStride;
  publish(c + g * kCtrStride);
}
template <typename T>
__device__ __forceinline__ void wait_parent(const SolveArgs<T>& a, const FrontDesc& d, int g) {
  if (!a.done || d.parent < 0) return;
  const int* c = a.done + (int64_t)d.parent * a.NG * kCtrStride;
  if (d.whole & kParentWhole) wait_count(c, d.needB, a.err, a.wait_ns);
  else if (d.whole & kSelfWhole)
    for (int q = 0; q < a.NG; ++q) wait_count(c + q * kCtrStride, d.needB, a.err, a.wait_ns);
  else wait_count(c + g * kCtrStride, d.needB, a.err, a.wait_ns);
}
template <typename T>
__device__ __forceinline__ void publish_self(const SolveArgs<T>& a, const FrontDesc& d, int g) {
  if (a.done) publish(a.done + ((int64_t)d.s * a.NG + (d.whole & kSelfWhole ? 0 : g)) * kCtrStride);
}

template <typename T> struct Vec16;
template <> struct Vec16<float> { using V = float4; static constexpr int N = 4; };
template <> struct Vec16<double> { using V = double2; static constexpr int N = 2; };

// x[r] = p[r] for r < n, zero beyond; p lies in rows of stride RV (see above),
// so a whole 16-byte vector that holds one wanted value may be read.  Reads
// past L1: other CTAs of the same launch write these values.
template <typename T, int NR>
__device__ __forceinline__ void ld_row(const T* p, int n, bool vec, T (&x)[NR]) {
  using V = typename Vec16<T>::V;
  constexpr int N = Vec16<T>::N;
  if constexpr (NR % N == 0) {
    if (vec) {
#pragma unroll
      for (int q = 0; q < NR / N; ++q) {
        union { V v; T t[N]; } u;
        if (q * N < n) {
          u.v = __ldcg(reinterpret_cast<const V*>(p) + q);
        } else {
#pragma unroll
          for (int e = 0; e < N; ++e) u.t[e] = T(0);
        }
#pragma unroll
        for (int e = 0; e < N; ++e) x[q * N + e] = u.t[e];
      }
      return;
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) x[r] = r < n ? __ldcg(p + r) : T(0);
}

template <typename T, int NR>
__device__ __forceinline__ void st_row(T* p, int n, bool vec, const T (&x)[NR]) {
  using V = typename Vec16<T>::V;
  constexpr int N = Vec16<T>::N;
  if constexpr (NR % N == 0) {
    if (vec) {
#pragma unroll
      for (int q = 0; q < NR / N; ++q)
        if (q * N < n) {
          union { V v; T t[N]; } u;
#pragma unroll
          for (int e = 0; e < N; ++e) u.t[e] = x[q * N + e];
          reinterpret_cast<V*>(p)[q] = u.v;
        }
      return;
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r)
    if (r < n) p[r] = x[r];
}

// FP64 output: *p = x, or *p += x
template <typename T>
__device__ __forceinline__ void st_xd(double* p, int mode, T x) {
  *p = mode == kXdAdd ? *p + (double)x : (double)x;
}

// FP64 output row: p[r] = x[r] (mode kXdStore) or p[r] += x[r] (kXdAdd)
template <typename T, int NR>
__device__ __forceinline__ void st_xd_row(double* p, int n, bool vec, int mode, const T (&x)[NR]) {
  if constexpr (NR % 2 == 0) {
    if (vec) {
      double2* q = reinterpret_cast<double2*>(p);
#pragma unroll
      for (int i = 0; i < NR / 2; ++i)
        if (2 * i < n) {
          double2 v = make_double2((double)x[2 * i], (double)x[2 * i + 1]);
          if (mode == kXdAdd) {
            const double2 o = q[i];
            v.x += o.x;
            v.y += o.y;
          }
          q[i] = v;
        }
      return;
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r)
    if (r < n) p[r] = mode == kXdAdd ? p[r] + (double)x[r] : (double)x[r];
}

// broadcast right-hand side row (FP64, caller's memory)
template <typename T, int NR>
__device__ __forceinline__ void ld_b(const double* p, int n, T (&x)[NR]) {
  if constexpr (NR % 2 == 0) {
    if (n == NR && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
      const double2* q = reinterpret_cast<const double2*>(p);
#pragma unroll
      for (int i = 0; i < NR / 2; ++i) {
        const double2 v = __ldg(q + i);
        x[2 * i] = (T)v.x;
        x[2 * i + 1] = (T)v.y;
      }
      return;
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) x[r] = r < n ? (T)__ldg(p + r) : T(0);
}

// *p if ok, else 0.  Volatile: the load is issued where it stands.  Left to
// the compiler, loads meant to run under a dependency wait or a diagonal solve
// sink to their first use behind it, one memory latency per step of the chain
// (a 22-row front's backward solve took 10 us that way).
__device__ __forceinline__ float ld_early(const float* p, bool ok) {
  float v;
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n mov.f32 %0, 0f00000000;\n @q ld.global.nc.f32 %0, [%1];\n}"
               : "=f"(v) : "l"(p), "r"((int)ok));
  return v;
}
__device__ __forceinline__ double ld_early(const double* p, bool ok) {
  double v;
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n mov.f64 %0, 0d0000000000000000;\n @q ld.global.nc.f64 %0, [%1];\n}"
               : "=d"(v) : "l"(p), "r"((int)ok));
  return v;
}
__device__ __forceinline__ int32_t ld_early(const int32_t* p, bool ok) {
  int32_t v;
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n mov.b32 %0, 0;\n @q ld.global.nc.b32 %0, [%1];\n}"
               : "=r"(v) : "l"(p), "r"((int)ok));
  return v;
}
__device__ __forceinline__ int64_t ld_early(const int64_t* p, bool ok) {
  int64_t v;
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n mov.b64 %0, 0;\n @q ld.global.nc.b64 %0, [%1];\n}"
               : "=l"(v) : "l"(p), "r"((int)ok));
  return v;
}
__device__ __forceinline__ float ld_early(const float* p) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
__device__ __forceinline__ double ld_early(const double* p) {
  double v;
  asm volatile("ld.global.nc.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}
// Nothing that reads memory moves across: the reads of an unrolled loop stay
// near their use.  (Hoisted to its top they cost more registers than there are,
// and the spills come back from L2: the waits' fences empty L1.)
__device__ __forceinline__ void keep_order() { asm volatile("" ::: "memory"); }
// x is computed by here
__device__ __forceinline__ void settle(float& x) { asm volatile("" : "+f"(x)); }
__device__ __forceinline__ void settle(double& x) { asm volatile("" : "+d"(x)); }

// coefficient (i, j) of the triangular matrix being solved with, 0 unless ok
template <typename T, bool TRANS>
__device__ __forceinline__ T coef(const T* f, int F, int i, int j, bool ok = true) {
  return ld_early(TRANS ? f + j + (int64_t)i * F : f + i + (int64_t)j * F, ok);
}

__device__ __forceinline__ FrontDesc ld_desc(const FrontDesc* d) {
  FrontDesc r;
  const int4* s = reinterpret_cast<const int4*>(d);
  int4* o = reinterpret_cast<int4*>(&r);
#pragma unroll
  for (int q = 0; q < 4; ++q) o[q] = __ldg(s + q);
  return r;
}

// Where the value of one front position comes from before the solve: its
// right-hand side entry (pivot positions) and the children's contributions,
// added in child order.  None of this depends on the children's results, so
// it is loaded before the dependency wait.
struct Gather {
  int64_t e0 = 0, e1 = 0, p0 = 0, p1 = 0;
  int64_t row = -1;  // right-hand side row, or -1
};

template <typename T>
__device__ __forceinline__ Gather gather_begin(const SolveArgs<T>& a, const FrontDesc& d, int j, bool on) {
  Gather g;
  if (!on) return g;
  g.e0 = ld_early(a.inv_off + d.vo + j, true);
  g.e1 = ld_early(a.inv_off + d.vo + j + 1, true);
  if (j < d.ns) g.row = a.b ? (int64_t)ld_early(a.perm + d.c0 + j, true) : (int64_t)(d.c0 + j);
  g.p0 = ld_early(a.inv_pos + g.e0, g.e0 < g.e1);
  g.p1 = ld_early(a.inv_pos + g.e0 + 1, g.e0 + 1 < g.e1);
  return g;
}

// right-hand side entries r0 .. r0 + n of the position's row, for shift k
template <typename T, int NR>
__device__ __forceinline__ void gather_rhs(const SolveArgs<T>& a, const Gather& g, int k, int r0, int n, bool vec,
                                           T (&v)[NR]) {
#pragma unroll
  for (int r = 0; r < NR; ++r) v[r] = T(0);
  if (g.row < 0) return;
  if (a.b) {
    ld_b<T, NR>(a.b + g.row * a.R + r0, n, v);
  } else {
    ld_row<T, NR>(a.rk + (g.row * a.K + k) * a.RV + r0, n, vec, v);
  }
}

// NB contributions in flight at a time (a root's position has dozens, each a
// memory latency away), added in child order whatever NB is.
template <typename T, int NR, int NB>
__device__ __forceinline__ void gather_children(const SolveArgs<T>& a, const Gather& g, int k, int r0, int n,
                                                bool vec, T (&v)[NR]) {
  if (g.e0 >= g.e1) return;
  const T* Vk = a.V + (int64_t)k * a.RV + r0;
  const int64_t st = (int64_t)a.K * a.RV;
  int64_t q[NB];
#pragma unroll
  for (int t = 0; t < NB; ++t)
    q[t] = t == 0 ? g.p0 : t == 1 ? g.p1 : ld_early(a.inv_pos + g.e0 + t, g.e0 + t < g.e1);
  for (int64_t e = g.e0;;) {
    const int m = (int)min((int64_t)NB, g.e1 - e);
    T x[NB][NR];
#pragma unroll
    for (int t = 0; t < NB; ++t) ld_row<T, NR>(Vk + q[t] * st, t < m ? n : 0, vec, x[t]);
    e += NB;
#pragma unroll
    for (int t = 0; t < NB; ++t) q[t] = ld_early(a.inv_pos + e + t, e + t < g.e1);
#pragma unroll
    for (int t = 0; t < NB; ++t)
      if (t < m) {
#pragma unroll
        for (int r = 0; r < NR; ++r) v[r] += x[t][r];
      }
    if (e >= g.e1) return;
  }
}

// ---------------------------------------------------------------------------
// Segment tasks (forward solves, and backward solves of one right-hand side):
// SEG lanes (8, 16 or 32) solve one (front, chunk of NR = 1 or 8 right-hand
// sides) for one or more shifts; lane i owns front position i with its NR values
// in registers and its coefficients, loaded before the dependency wait, and the
// triangular solve is a chain of shuffles.  For SEG < 32 the whole front fits;
// for SEG = 32 the positions beyond the first 32 are handled in further blocks
// of 32 (at most 32 pivots).  Loops run to
// warp-uniform bounds (coefficients beyond a front are zero), so segments with
// different fronts never diverge around a shuffle; all lanes call together.
// ---------------------------------------------------------------------------
struct SegTask {
  bool active = false;
  int r0 = 0, nr = 0, k0 = 0, k1 = 0;
};

template <typename T>
__device__ __forceinline__ SegTask seg_task(const SolveArgs<T>& a, const SolveUnit& U, unsigned q, int nrw,
                                            FrontDesc& d) {
  SegTask t;
  const int kf = U.x >> 4;
  const unsigned nch = (unsigned)((a.R + nrw - 1) / nrw), nkg = (unsigned)((a.K + kf - 1) / kf);
  d.ns = d.F = 0;
  if (q < (unsigned)U.c) {
    const unsigned slot = q / (nch * nkg), rem = q - slot * nch * nkg;
    const unsigned kg = rem / nch;
    d = ld_desc(a.desc + U.a + slot);
    t.active = !a.act || a.act[d.inst];
    t.k0 = (int)kg * kf;
    t.k1 = min(a.K, t.k0 + kf);
    t.r0 = (int)(rem - kg * nch) * nrw;
    t.nr = min(nrw, a.R - t.r0);
    if (!t.active) d.ns = d.F = 0;
  }
  return t;
}

template <typename T, int SEG, bool TRANS, int NR>
__device__ __forceinline__ void seg_forward(const SolveArgs<T>& a, const SegTask& t, const FrontDesc& d, int sl,
                                            T* yb) {
  const int ns = d.ns, F = d.F;
  const int nr = t.active ? t.nr : 0;
  const bool vec = a.vec;
  const int nsw = __reduce_max_sync(kFull, ns);
  const int nb = SEG < 32 ? 1 : (F + 31) / 32;             // uniform for SEG = 32
  const int nkw = __reduce_max_sync(kFull, t.k1 - t.k0);  // shifts per task (uniform)
  const int nrw = __reduce_max_sync(kFull, nr);
  const Gather g = gather_begin<T>(a, d, sl, sl < F);
  for (int kk = 0; kk < nkw; ++kk) {
    const int k = min(t.k0 + kk, max(t.k1 - 1, 0));
    const bool kon = t.k0 + kk < t.k1 && t.active;
    const T* f = a.fronts + a.K * d.fo + (int64_t)k * F * F;
    T C[8], v[NR];
    auto load8 = [&](int cb) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int c = cb + q;
        C[q] = coef<T, TRANS>(f, F, sl, c, kon && c < ns && sl > c && sl < F);
      }
    };
    load8(0);
    T rd = T(1);
    if (TRANS && kon && sl < ns) rd = T(1) / __ldg(f + (int64_t)sl * (F + 1));
    const int n = (kon && sl < F) ? nr : 0;
    if (n) {
      gather_rhs<T, NR>(a, g, k, t.r0, n, vec, v);
    } else {
#pragma unroll
      for (int r = 0; r < NR; ++r) v[r] = T(0);
    }
    if (TRANS) settle(rd);
#pragma unroll
    for (int r = 0; r < NR; ++r) settle(v[r]);
    if (kon && sl == 0) wait_children(a, d, k);
    __syncwarp();
    if (n) gather_children<T, NR, (NR == 1 ? 4 : 2)>(a, g, k, t.r0, n, vec, v);
    for (int cb = 0; cb < nsw; cb += 8) {  // eight pivots at a time: most fronts have no more
      if (cb > 0) load8(cb);
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int c = cb + q;
        if (c >= nsw) break;
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (r < nrw) {
            if (TRANS && sl == c) v[r] *= rd;
            v[r] -= C[q] * __shfl_sync(kFull, v[r], c, SEG);
          }
      }
    }
    T* Vs = a.V + (d.vo * a.K + k) * a.RV + t.r0;
    const int64_t st = (int64_t)a.K * a.RV;
    if (n) st_row<T, NR>(Vs + sl * st, n, vec, v);
    if (SEG == 32 && nb > 1) {
#pragma unroll
      for (int r = 0; r < NR; ++r) yb[sl * NR + r] = v[r];
      __syncwarp();
      for (int bk = 1; bk < nb; ++bk) {
        const int i = bk * 32 + sl;
        const int ni = (kon && i < F) ? nr : 0;
        if (ni) {
          const Gather gi = gather_begin<T>(a, d, i, true);
          T w[NR];
#pragma unroll
          for (int r = 0; r < NR; ++r) w[r] = T(0);
          gather_children<T, NR, (NR == 1 ? 4 : 2)>(a, gi, k, t.r0, ni, vec, w);
#pragma unroll 4
          for (int c = 0; c < ns; ++c) {
            const T l = __ldg(TRANS ? f + c + (int64_t)i * F : f + i + (int64_t)c * F);
#pragma unroll
            for (int r = 0; r < NR; ++r) w[r] -= l * yb[c * NR + r];
          }
          st_row<T, NR>(Vs + i * st, ni, vec, w);
        }
      }
    }
    __syncwarp();  // also: yb is reused by the next shift
    if (kon && sl == 0) publish_up(a, d, k);
  }
}

template <typename T, int SEG, bool TRANS>
__device__ __forceinline__ void seg_backward(const SolveArgs<T>& a, const SegTask& t, const FrontDesc& d, int sl) {
  const int ns = d.ns, F = d.F;
  const int Fw = min(SEG, __reduce_max_sync(kFull, F));
  const int nb = SEG < 32 ? 1 : (F + 31) / 32;
  const int nkw = __reduce_max_sync(kFull, t.k1 - t.k0);
  const int64_t K = a.K;
  // permuted row of this lane's position: a pivot row, or an ancestor's row
  const int64_t row = sl < ns ? d.c0 + sl : ld_early(a.rows + d.ro + sl - ns, sl < F);
  for (int kk = 0; kk < nkw; ++kk) {
    const int k = min(t.k0 + kk, max(t.k1 - 1, 0));
    const bool kon = t.k0 + kk < t.k1 && t.active;
    const T* f = a.fronts + K * d.fo + (int64_t)k * F * F;
    T C[SEG];
#pragma unroll
    for (int j = 0; j < SEG; ++j) C[j] = coef<T, TRANS>(f, F, sl, j, kon && sl < ns && j > sl && j < F);
    T rd = T(1), v = T(0);
    if (!TRANS && kon && sl < ns) rd = T(1) / __ldg(f + (int64_t)sl * (F + 1));
    if (kon && sl < ns) v = __ldcg(a.V + (d.vo + sl) * K + k);
    if (!TRANS) settle(rd);
    if (kon && sl == 0) wait_parent(a, d, k);
    __syncwarp();
    if (kon && sl >= ns && sl < F) v = __ldcg(a.xt + row * K + k);
    if (SEG == 32 && nb > 1) {
      // positions beyond the first 32: ancestors' solutions, 32 at a time
      for (int j0 = 32; j0 < F; j0 += 32) {
        const int j = j0 + sl;
        const T x = kon && j < F ? __ldcg(a.xt + __ldg(a.rows + d.ro + j - ns) * K + k) : T(0);
        const int m = min(32, F - j0);
#pragma unroll 8
        for (int jj = 0; jj < m; ++jj) {
          const T u = (kon && sl < ns) ? __ldg(TRANS ? f + j0 + jj + (int64_t)sl * F : f + sl + (int64_t)(j0 + jj) * F) : T(0);
          v -= u * __shfl_sync(kFull, x, jj);
        }
      }
    }
#pragma unroll
    for (int j = SEG - 1; j >= 0; --j) {
      if (j >= Fw) continue;
      if (!TRANS && sl == j) v *= rd;  // rd = 1 beyond the pivots
      v -= C[j] * __shfl_sync(kFull, v, j, SEG);
    }
    if (kon && sl < ns) {
      a.xt[row * K + k] = v;
      if (a.xd) st_xd<T>(a.xd + row * K + k, a.xd_mode, v);
    }
    __syncwarp();
    if (kon && sl == 0) publish_self(a, d, k);
  }
}

// The same for several right-hand sides and a front of at most 32 rows a warp, eight
// columns of coefficients at a time.
template <typename T, bool TRANS, int NR>
__device__ __forceinline__ void seg_backward_rhs(const SolveArgs<T>& a, const SegTask& t, const FrontDesc& d, int sl) {
  const int ns = d.ns, F = d.F;
  const int nr = t.nr;
  const bool vec = a.vec;
  const int top = (F - 1) & ~7;
  const int64_t row = sl < ns ? d.c0 + sl : ld_early(a.rows + d.ro + sl - ns, sl < F);
  if (!t.active) return;
  for (int k = t.k0; k < t.k1; ++k) {
    const T* f = a.fronts + a.K * d.fo + (int64_t)k * F * F;
    T C[8], v[NR];
    auto load8 = [&](int jb) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int j = jb + q;
        C[q] = coef<T, TRANS>(f, F, sl, j, sl < ns && j > sl && j < F);
      }
    };
    load8(top);
    T rd = T(1);
    if (!TRANS && sl < ns) rd = T(1) / __ldg(f + (int64_t)sl * (F + 1));
    const int n = sl < F ? nr : 0;
    ld_row<T, NR>(a.V + ((d.vo + sl) * a.K + k) * a.RV + t.r0, sl < ns ? n : 0, vec, v);
    if (!TRANS) settle(rd);
    if (sl == 0) wait_parent(a, d, 0);
    __syncwarp();
    T* x = a.xt + (row * a.K + k) * a.RV + t.r0;
    if (n && sl >= ns) ld_row<T, NR>(x, n, vec, v);
    for (int jb = top; jb >= 0; jb -= 8) {
      if (jb != top) load8(jb);
#pragma unroll
      for (int q = 7; q >= 0; --q) {
        const int j = jb + q;
        if (j >= F) continue;
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (r < nr) {
            if (!TRANS && sl == j) v[r] *= rd;  // rd = 1 beyond the pivots
            v[r] -= C[q] * __shfl_sync(kFull, v[r], j);
          }
      }
    }
    if (n && sl < ns) {
      st_row<T, NR>(x, n, vec, v);
      if (a.xd) st_xd_row<T, NR>(a.xd + (row * a.K + k) * a.RX + t.r0, n, a.vecd, a.xd_mode, v);
    }
    __syncwarp();
    if (sl == 0) publish_self(a, d, 0);
  }
}

// One warp, lane = row of a staged 32 x 32 triangle B (zero outside it, rd =
// reciprocal diagonal, 1 where unit): v becomes the solution.
template <typename T, bool LOWER, bool UNIT>
__device__ __forceinline__ T block_solve(const T* B, const T* rd, T v, int nb, int lane) {
#pragma unroll 4
  for (int q = 0; q < nb; ++q) {
    const int c = LOWER ? q : nb - 1 - q;
    T y = __shfl_sync(kFull, v, c);
    if (!UNIT) y *= rd[c];
    v -= B[lane * kBS + c] * y;
  }
  return UNIT ? v : v * rd[lane];
}

// the diagonal block (ns <= 32 pivots) into B and its reciprocal pivots into
// rd, by the whole CTA
template <typename T, bool LOWER, bool UNIT, bool TRANS>
__device__ __forceinline__ void stage_block(T* B, T* rd, const T* f, int F, int ns, int tid) {
  T x[4], dg = T(1);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int q = tid + kSolveThreads * t;
    // lanes run along the contiguous index
    const int i = TRANS ? q >> 5 : q & 31, c = TRANS ? q & 31 : q >> 5;
    x[t] = coef<T, TRANS>(f, F, i, c, i < ns && c < ns && (LOWER ? i > c : i < c));
  }
  if (!UNIT && tid < 32) dg = ld_early(f + (int64_t)tid * (F + 1), tid < ns);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const int q = tid + kSolveThreads * t;
    const int i = TRANS ? q >> 5 : q & 31, c = TRANS ? q & 31 : q >> 5;
    B[i * kBS + c] = x[t];
  }
  if (!UNIT && tid < 32) rd[tid] = tid < ns ? T(1) / dg : T(1);
}

// Shared memory of a front of the two kinds below, in elements: the diagonal
// block, its reciprocal pivots, then the pivots' values (forward) or the warps'
// partial sums (backward)
constexpr int kThinRd = 32 * kBS, kThinV = kThinRd + 32;
constexpr int thin_smem(bool fwd, int nr) { return kThinV + (fwd ? 32 * nr : kSolveWarps * 32); }

// Wider fronts with at most 32 pivots, one (front, shift, chunk) a CTA: every
// thread keeps its row's values and coefficients in registers; only the pivot
// rows meet in shared memory.
template <typename T, bool TRANS, int NR>
__device__ __forceinline__ void thin_forward(const SolveArgs<T>& a, const FrontDesc& d, int k, int r0, int nr, T* sm) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int ns = d.ns, F = d.F;
  const bool vec = a.vec && (r0 % Vec16<T>::N == 0);
  T* B = sm;                    // 32 x kBS
  T* rdv = B + kThinRd;         // 32
  T* y = B + kThinV;            // 32 x NR
  const T* f = a.fronts + a.K * d.fo + (int64_t)k * F * F;
  stage_block<T, true, !TRANS, TRANS>(B, rdv, f, F, ns, tid);
  Gather g = gather_begin<T>(a, d, tid, tid < F);
  T C[8], v[NR];
  auto load8 = [&](int i, int cb) {
#pragma unroll
    for (int q = 0; q < 8; ++q) C[q] = coef<T, TRANS>(f, F, i, cb + q, cb + q < ns && i >= ns && i < F);
  };
  load8(tid, 0);
  gather_rhs<T, NR>(a, g, k, r0, nr, vec, v);
#pragma unroll
  for (int r = 0; r < NR; ++r) settle(v[r]);
  if (tid == 0) wait_children(a, d, k);
  __syncthreads();
  if (tid < F) gather_children<T, NR, (NR == 1 ? 8 : 2)>(a, g, k, r0, nr, vec, v);
  if (tid < 32) {
#pragma unroll
    for (int r = 0; r < NR; ++r) y[tid * NR + r] = tid < ns ? v[r] : T(0);
  }
  __syncthreads();
  for (int r = wid; r < nr; r += kSolveWarps)
    y[lane * NR + r] = block_solve<T, true, !TRANS>(B, rdv, y[lane * NR + r], ns, lane);
  __syncthreads();
  T* Vs = a.V + (d.vo * a.K + k) * a.RV + r0;
  const int64_t st = (int64_t)a.K * a.RV;
  for (int i = tid; i < F; i += kSolveThreads) {
    if (i < ns) {
#pragma unroll
      for (int r = 0; r < NR; ++r) v[r] = y[i * NR + r];
    } else {
      if (i >= kSolveThreads) {
        g = gather_begin<T>(a, d, i, true);
        load8(i, 0);
#pragma unroll
        for (int r = 0; r < NR; ++r) v[r] = T(0);
        gather_children<T, NR, (NR == 1 ? 8 : 2)>(a, g, k, r0, nr, vec, v);
      }
      for (int cb = 0; cb < ns; cb += 8) {
        if (cb > 0) load8(i, cb);
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (cb + q >= ns) break;
#pragma unroll
          for (int r = 0; r < NR; ++r) v[r] -= C[q] * y[(cb + q) * NR + r];
        }
      }
    }
    st_row<T, NR>(Vs + i * st, nr, vec, v);
  }
  __syncthreads();
  if (tid == 0) publish_up(a, d, k);
}

// z -= U12 x_R over the update rows, then the diagonal block.  Thread (p, jj)
// sums over every JG-th update row j for pivot p; the partial sums meet by
// shuffles within a warp and in shared memory across warps, in a fixed order.
// Lanes run along the contiguous index of the coefficients: the pivots, or
// with TRANS the update rows.
template <typename T, bool TRANS>
__device__ __forceinline__ void thin_backward1(const SolveArgs<T>& a, const FrontDesc& d, int k, T* sm) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int ns = d.ns, F = d.F, ms = F - ns;
  const int64_t K = a.K;
  T* B = sm;                    // 32 x kBS
  T* rdv = B + kThinRd;         // 32
  T* part = B + kThinV;         // 8 warps x 32
  const T* f = a.fronts + K * d.fo + (int64_t)k * F * F;
  stage_block<T, false, TRANS, TRANS>(B, rdv, f, F, ns, tid);
  const int lp = ns <= 1 ? 0 : 32 - __clz(ns - 1);  // log2 of the pivots rounded up
  const int JG = kSolveThreads >> lp;               // 8 .. 256
  const int p = TRANS ? tid / JG : tid & ((1 << lp) - 1);
  const int jj = TRANS ? tid & (JG - 1) : tid >> lp;
  const T z = wid == 0 && lane < ns ? __ldcg(a.V + (d.vo + lane) * K + k) : T(0);
  // the first coefficient and row index do not depend on the parent
  const bool on = p < ns;
  T acc = T(0);
  T u = coef<T, TRANS>(f, F, p, ns + jj, on && jj < ms);
  int64_t row = ld_early(a.rows + d.ro + jj, jj < ms);
  if (tid == 0) wait_parent(a, d, k);
  __syncthreads();
  for (int j = jj; j < ms; j += JG) {
    const T x = __ldcg(a.xt + row * K + k), uc = u;
    const int jn = j + JG;
    u = coef<T, TRANS>(f, F, p, ns + jn, on && jn < ms);
    row = ld_early(a.rows + d.ro + jn, jn < ms);
    acc += uc * x;
  }
  // lanes of one pivot: lane = p + (jj << lp), or with TRANS jj in the low bits
  const int o0 = TRANS ? 1 : 1 << lp, o1 = TRANS ? min(32, JG) : 32;
  for (int o = o0; o < o1; o <<= 1) acc += __shfl_xor_sync(kFull, acc, o);
  if (TRANS) {
    // a warp holds 32 / JG pivots (JG < 32) or a JG / 32-th part of one
    if ((lane & (min(32, JG) - 1)) == 0) part[(JG >= 32 ? wid & (JG / 32 - 1) : 0) * 32 + p] = acc;
  } else if (lane < (1 << lp)) {
    part[wid * 32 + lane] = acc;
  }
  __syncthreads();
  if (wid == 0) {
    const int np = TRANS ? max(1, JG / 32) : kSolveWarps;
    T v = T(0);
    if (lane < ns) {
      T s = part[lane];
      for (int w = 1; w < np; ++w) s += part[w * 32 + lane];
      v = z - s;
    }
    v = block_solve<T, false, TRANS>(B, rdv, v, ns, lane);
    if (lane < ns) {
      const int64_t o = (int64_t)(d.c0 + lane) * K + k;
      a.xt[o] = v;
      if (a.xd) st_xd<T>(a.xd + o, a.xd_mode, v);
    }
    __syncwarp();
    if (lane == 0) publish_self(a, d, k);
  }
}

// ---------------------------------------------------------------------------
// Backward solves of several right-hand sides, fronts with at most 32 pivots (but for
// those with many pivots to few right-hand sides, kUnitSeg32): a
// warp takes one front for 32 of its K x RV columns (k, r), one a lane.
// Structure is read once for the 32 columns, V and xt a whole row segment at a
// time, and no lane idles on a front's shape; the columns of the front are
// worked through in blocks of 8, 8 pivots a lane in registers, against 8 x 8
// blocks of coefficients that the warp stages in shared memory (cp.async, a
// block ahead), one set per shift among its columns, read as 16-byte broadcasts.
// (With lane = front row, as in the forward solve, 3 of 4 lanes idle on the few
// pivot rows, and the 256-grid batch (K = 4, R = 8) took 560 us a solve against
// 445.  The same form of the forward solve was slower, 680 us against 430: it
// walks a front's rows block by block, a memory latency each, where the lanes
// of a segment task gather all of them at once.)
// ---------------------------------------------------------------------------
template <typename T> struct Stage { static constexpr int LD = sizeof(T) == 4 ? 68 : 66; };  // per shift

// per-warp stage: two buffers of nk sets, the reciprocal pivots of a block (nk x 9)
template <typename T>
__host__ __device__ constexpr int col_stage(int nk) { return 2 * nk * Stage<T>::LD + (nk * 9 + 3) / 4 * 4; }

template <typename T>
struct Cols {
  int col, k, kl, klo, nk, r;
  bool on;
  __device__ __forceinline__ Cols(const SolveArgs<T>& a, int g, int lane) {
    const int n = a.K * a.RV;
    const int c0 = g * 32, c1 = min(c0 + 31, n - 1);
    col = min(c0 + lane, c1);
    on = c0 + lane <= c1;
    k = col / a.RV;
    r = col - k * a.RV;
    klo = c0 / a.RV;
    nk = c1 / a.RV - klo + 1;
    kl = k - klo;
  }
};

__device__ __forceinline__ void cp_async(float* d, const float* s, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(d)), "l"(s),
               "r"(ok ? 4 : 0));
}
__device__ __forceinline__ void cp_async(double* d, const double* s, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(d)), "l"(s),
               "r"(ok ? 8 : 0));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// coefficients (i0 + ii, j0 + jj) of the nk shifts from klo on into S[kk][ii][jj],
// zero outside rows [0, iend) x columns [0, jend) and, on the diagonal block,
// below the diagonal
template <typename T, bool TRANS>
__device__ __forceinline__ void stage8(T* S, const T* f0, int F, int nk, int i0, int iend, int j0, int jend, int lane) {
  const int lo = lane & 7, hi = lane >> 3;
  // lanes run along the contiguous index of the front's columns
  for (int q = 0; q < 2 * nk; ++q) {
    const int kk = q >> 1, h = (q & 1) * 4 + hi;
    const int ii = TRANS ? h : lo, jj = TRANS ? lo : h;
    const int i = i0 + ii, j = j0 + jj;
    const bool ok = i < iend && j < jend && i < j;
    const T* p = f0 + (int64_t)kk * F * F;
    cp_async(S + kk * Stage<T>::LD + ii * 8 + jj, ok ? (TRANS ? p + j + (int64_t)i * F : p + i + (int64_t)j * F) : p, ok);
  }
  cp_commit();
}

// reciprocal pivots p0 .. p0 + 7 of the nk shifts, 1 past the pivots
template <typename T>
__device__ __forceinline__ void stage_pivots(T* rd, const T* f0, int F, int nk, int p0, int ns, int lane) {
  for (int e = lane; e < 8 * nk; e += 32) {
    const int kk = e >> 3, p = p0 + (e & 7);
    const T u = ld_early(f0 + (int64_t)kk * F * F + (int64_t)p * (F + 1), p < ns);
    rd[kk * 9 + (e & 7)] = p < ns ? T(1) / u : T(1);
  }
}

// acc[i] -= sum_j S[i][j] x[j], from the last column down
template <typename T>
__device__ __forceinline__ void apply8(T (&acc)[8], const T* S, const T (&x)[8]) {
  using V = typename Vec16<T>::V;
  constexpr int N = Vec16<T>::N;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    if (i % 4 == 0) keep_order();
#pragma unroll
    for (int j = 8 - N; j >= 0; j -= N) {
      union { V v; T t[N]; } u;
      u.v = *reinterpret_cast<const V*>(S + i * 8 + j);
#pragma unroll
      for (int e = N - 1; e >= 0; --e) acc[i] -= u.t[e] * x[j + e];
    }
  }
}

// one block of 8 columns j0 .. of the solution: pivots' values (already
// solved) or ancestors', rows one a lane for 32 positions from `base` on
template <typename T>
__device__ __forceinline__ void ld_x8(const SolveArgs<T>& a, const Cols<T>& c, int64_t rowl, int j0, int F, T (&x)[8]) {
  const int64_t st = (int64_t)a.K * a.RV;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int64_t row = __shfl_sync(kFull, rowl, (j0 + j) & 31);
    x[j] = j0 + j < F ? __ldcg(a.xt + row * st + c.col) : T(0);
  }
}

// nw warps share the front (nw = 8: the CTA's, with `red` for their partial
// sums): the blocks of update columns are dealt out, warp 0 solves the pivots.
template <typename T, bool TRANS>
__device__ __forceinline__ void col_backward(const SolveArgs<T>& a, const FrontDesc& d, int g, int w, int nw, T* S,
                                             T* red) {
  const int lane = threadIdx.x & 31;
  const Cols<T> c(a, g, lane);
  const int ns = d.ns, F = d.F;
  const int nb = (F + 7) >> 3, nsb = (ns + 7) >> 3;
  const int64_t st = (int64_t)a.K * a.RV;
  const T* f0 = a.fronts + a.K * d.fo + (int64_t)c.klo * F * F;
  T* S1 = S + c.nk * Stage<T>::LD;
  T* rd = S1 + c.nk * Stage<T>::LD;
  const int so = c.kl * Stage<T>::LD;
  const T* Vs = a.V + d.vo * st + c.col;
  auto row_of = [&](int j) -> int64_t {  // permuted row of position j
    return j < ns ? d.c0 + j : ld_early(a.rows + d.ro + j - ns, j < F);
  };
  int buf = 0, rbase = -1;
  int64_t rowl = 0;
  bool waited = false;
  for (int pb = nsb - 1; pb >= 0; --pb) {
    const int p0 = pb * 8;
    T z[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) z[i] = T(0);
    if (nw == 1) {
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (p0 + i < ns) z[i] = __ldcg(Vs + (p0 + i) * st);
    }
    int jb = nb - 1 - w;  // this warp's blocks of columns, from the last down
    if (jb >= nsb) stage8<T, TRANS>(S, f0, F, c.nk, p0, ns, jb * 8, F, lane);
    buf = 0;
    if (!TRANS && w == 0) stage_pivots(rd, f0, F, c.nk, p0, ns, lane);
    if (jb >= nsb && (jb * 8 & ~31) != rbase) {
      rbase = jb * 8 & ~31;
      rowl = row_of(rbase + lane);
    }
    if (!waited) {
      if (w == 0 && lane == 0) wait_parent(a, d, g);
      if (nw > 1) __syncthreads();
      else __syncwarp();
      waited = true;
    }
    T x[8];
    if (jb >= nsb) ld_x8(a, c, rowl, jb * 8, F, x);
    while (jb >= nsb) {
      const int jn = jb - nw;
      T* Sn = buf ? S : S1;
      const T* Sc = (buf ? S1 : S) + so;
      T xn[8];
      if (jn >= nsb) {
        stage8<T, TRANS>(Sn, f0, F, c.nk, p0, ns, jn * 8, F, lane);
        if ((jn * 8 & ~31) != rbase) {
          rbase = jn * 8 & ~31;
          rowl = row_of(rbase + lane);
        }
        ld_x8(a, c, rowl, jn * 8, F, xn);
      } else {
        cp_commit();
      }
      cp_wait<1>();
      __syncwarp();
      apply8(z, Sc, x);
      __syncwarp();
      buf ^= 1;
      jb = jn;
#pragma unroll
      for (int j = 0; j < 8; ++j) x[j] = xn[j];
    }
    if (nw > 1) {
      // the warps' partial sums, added in their order, then the forward solution
      if (w > 0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) red[((w - 1) * 8 + i) * 32 + lane] = z[i];
      }
      __syncthreads();
      if (w == 0) {
        for (int q = 0; q < nw - 1; ++q) {
#pragma unroll
          for (int i = 0; i < 8; ++i) z[i] += red[(q * 8 + i) * 32 + lane];
        }
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (p0 + i < ns) z[i] += __ldcg(Vs + (p0 + i) * st);
      }
      __syncthreads();  // red is used again by the next pivot block
    }
    if (w == 0) {
      // the columns next to the pivots: later pivot blocks, then the diagonal
      // block, whose positions past the pivots hold ancestors' values
      for (int jb2 = nsb - 1; jb2 > pb; --jb2) {
        stage8<T, TRANS>(S, f0, F, c.nk, p0, ns, jb2 * 8, F, lane);
        T y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int jp = jb2 * 8 + j;
          const int64_t row = jp < ns ? d.c0 + jp : (jp < F ? __ldg(a.rows + d.ro + jp - ns) : -1);
          y[j] = row >= 0 ? __ldcg(a.xt + row * st + c.col) : T(0);
        }
        cp_wait<0>();
        __syncwarp();
        apply8(z, S + so, y);
        __syncwarp();
      }
      stage8<T, TRANS>(S, f0, F, c.nk, p0, ns, p0, F, lane);
      if (p0 + 8 > ns) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (p0 + i >= ns && p0 + i < F) z[i] = __ldcg(a.xt + __ldg(a.rows + d.ro + p0 + i - ns) * st + c.col);
      }
      cp_wait<0>();
      __syncwarp();
      const T* Sc = S + so;
#pragma unroll
      for (int j = 7; j >= 0; --j) {
        if (!TRANS) z[j] *= rd[c.kl * 9 + j];  // 1 past the pivots
#pragma unroll
        for (int i = 0; i < j; ++i) z[i] -= Sc[i * 8 + j] * z[j];
      }
      __syncwarp();
      if (c.on) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (p0 + i < ns) {
            const int64_t row = d.c0 + p0 + i;
            a.xt[row * st + c.col] = z[i];
            if (a.xd && c.r < a.R) st_xd<T>(a.xd + (row * a.K + c.k) * a.RX + c.r, a.xd_mode, z[i]);
          }
      }
    }
  }
  cp_wait<0>();
  __syncwarp();
}

// ---------------------------------------------------------------------------
// Fronts with more than 32 pivots: a CTA takes 256 rows of one (front, shift,
// chunk of RC right-hand sides), a row and its RC values per thread, so that
// 32 pivots are one warp's rows.  Per block of 32 pivots the owning warp solves
// the diagonal block in registers (its triangle staged in shared memory at the
// start), hands the 32 x RC solution to
// the CTA through shared memory, and every warp with rows still to do takes it
// in: 32 coefficients in registers, loaded a block ahead, against values read
// as broadcasts.  One barrier a block; the warp that owns the next block starts
// on it at once.  A front with more than 256 rows is that many CTA tasks: each
// reads the blocks solved by the others from global memory, as many at a time as
// their counter says are there, and waits only for tasks with smaller tickets.
// The bound is the chain of blocks: apply 32 coefficients, solve 32 pivots.
// (One CTA walking all the rows of a front, values in shared memory and blocks
// solved one right-hand side a warp, took 6.7 us a block on a 1600-row root,
// 3.2 us on a 320-row one.)
// Many such tasks share the SMs' pipes, and a block that one warp solves leaves its
// SM's idle: there the owning warp hands its block to as many warps as there are
// right-hand sides and takes the solution back, two barriers a block (kSpread;
// 100 dense systems of 97 rows, K 10, R 8, FP32: 50 us forward, 70 without).
// ---------------------------------------------------------------------------
constexpr int kWideRows = kSolveThreads;
constexpr int kTri = 32 * kBS + 32;  // a staged triangle and its reciprocal pivots
// right-hand sides of a task compiled for the spread form (at most), and for the other
template <typename T> constexpr int kWideSpread = 8;
template <typename T> constexpr int kWideAlone = sizeof(T) == 8 ? 1 : 4;
template <typename T, int RC> constexpr bool kSpread = RC == kWideSpread<T>;

template <typename T> struct WideTile { static constexpr int C = sizeof(T) == 8 ? 8 : 16, LD = C + 1; };

// L[c] = coefficient (i, col0 + c), c < nb, of this thread's row i (rows past
// lim repeat the last one).  The columns of a row are F apart in memory unless
// TRANS, where they are contiguous: the warp then loads rows, lanes along the
// columns, and turns them in its shared-memory area, 16 columns at a time.
template <typename T, bool TRANS>
__device__ __forceinline__ void load_panel(T (&L)[32], const T* f, int F, int i, int lim, int col0, int nb, T* tile,
                                           int lane) {
  if (!TRANS) {
    const T* p = f + min(i, lim - 1) + (int64_t)col0 * F;
    if (nb == 32) {
#pragma unroll
      for (int c = 0; c < 32; ++c, p += F) L[c] = ld_early(p);
    } else {
#pragma unroll
      for (int c = 0; c < 32; ++c, p += F) L[c] = ld_early(p, c < nb);
    }
  } else {
    constexpr int C = WideTile<T>::C, LD = WideTile<T>::LD;
    const int i0 = i - lane, lr = lane / C, lc = lane % C;
#pragma unroll
    for (int h = 0; h < 32 / C; ++h) {
      T x[C];
#pragma unroll
      for (int q = 0; q < C; ++q) {
        const int row = min(i0 + q * (32 / C) + lr, lim - 1), c = h * C + lc;
        x[q] = ld_early(f + col0 + c + (int64_t)row * F, c < nb);
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < C; ++q) tile[(q * (32 / C) + lr) * LD + lc] = x[q];
      __syncwarp();
#pragma unroll
      for (int c = 0; c < C; ++c) L[h * C + c] = tile[lane * LD + c];
    }
  }
}

// w -= sum_c L[c] y(c, :), y 32 rows of RC values in shared memory (zero where
// the coefficients are)
template <typename T, int RC>
__device__ __forceinline__ void apply_panel(const T (&L)[32], T (&w)[RC], const T* y, int nr) {
  if constexpr (sizeof(T) == 8 && RC > 1) {  // the FP64 pipe's time is the columns': only those there are
#pragma unroll
    for (int r = 0; r < RC; ++r)
      if (r < nr) {
#pragma unroll
        for (int c = 0; c < 32; ++c) {
          if (c % 8 == 0) keep_order();
          w[r] -= L[c] * y[c * RC + r];
        }
      }
  } else {
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      if (c % (16 / RC) == 0) keep_order();
#pragma unroll
      for (int r = 0; r < RC; ++r) w[r] -= L[c] * y[c * RC + r];
    }
  }
}

// The CTA: block `own` (its warp's number) of nb <= 32 pivots, handed over in y [32][RC] by
// the warp that owns it, solved one right-hand side a warp.  All threads call.
template <typename T, bool LOWER, bool UNIT, int RC>
__device__ __forceinline__ void spread_solve(const T* B, int own, T* y, int nr, int nb, int wid, int lane) {
  __syncthreads();
  if (wid < nr) {
    const T* Bo = B + own * kTri;
    y[lane * RC + wid] = block_solve<T, LOWER, UNIT>(Bo, Bo + 32 * kBS, y[lane * RC + wid], nb, lane);
  }
  __syncthreads();
}

// This warp's diagonal block (nb pivots from p0) into B, zero outside the
// triangle, and unless UNIT the reciprocal pivots behind it (1 past the pivots).
template <typename T, bool LOWER, bool UNIT, bool TRANS>
__device__ __forceinline__ void stage_triangle(T* B, const T* f, int F, int p0, int nb, int lane) {
  T rd = T(1);
  if (!UNIT) rd = ld_early(f + (int64_t)(p0 + lane) * (F + 1), lane < nb);
#pragma unroll 1
  for (int h = 0; h < 32; h += 8) {
    T x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = TRANS ? h + q : lane, c = TRANS ? lane : h + q;
      x[q] = coef<T, TRANS>(f, F, p0 + i, p0 + c, i < nb && c < nb && (LOWER ? i > c : i < c));
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) B[(TRANS ? h + q : lane) * kBS + (TRANS ? lane : h + q)] = x[q];
  }
  if (!UNIT) B[32 * kBS + lane] = lane < nb ? T(1) / rd : T(1);
  __syncwarp();
}

// One warp, lane = row: v becomes the solution with the staged triangle.
// FP32: four pivots per step, every lane forming the four solved values itself
// (in the order their own lanes would), which quarters the chain of shuffles.
// FP64 goes one at a time: its multiply-adds, at 2 a clock and SM, cost more
// than the shuffles.  Rows already solved meet zero coefficients and keep
// their values (FP64 leaves out the steps past the nb pivots of a short block).
template <typename T, bool LOWER, bool UNIT, int RC>
__device__ __forceinline__ void triangle_solve(const T* B, T (&v)[RC], int nb, int lane) {
  const T* bl = B + lane * kBS;
  const T* rd = B + 32 * kBS;
  if constexpr (sizeof(T) == 8) {
#pragma unroll 4
    for (int q = 0; q < nb; ++q) {
      const int c = LOWER ? q : nb - 1 - q;
      const T b = bl[c], rc = UNIT ? T(1) : rd[c];
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        T y = __shfl_sync(kFull, v[r], c);
        if (!UNIT) y *= rc;
        v[r] -= b * y;
      }
    }
  } else {
#pragma unroll 2
    for (int q = 0; q < 32; q += 4) {
      // positions of the four pivots in the order they are solved
      const int c0 = LOWER ? q : 31 - q, c1 = LOWER ? q + 1 : 30 - q, c2 = LOWER ? q + 2 : 29 - q,
                c3 = LOWER ? q + 3 : 28 - q;
      const T t10 = B[c1 * kBS + c0], t20 = B[c2 * kBS + c0], t21 = B[c2 * kBS + c1];
      const T t30 = B[c3 * kBS + c0], t31 = B[c3 * kBS + c1], t32 = B[c3 * kBS + c2];
      const T b0 = bl[c0], b1 = bl[c1], b2 = bl[c2], b3 = bl[c3];
#pragma unroll
      for (int r = 0; r < RC; ++r) {
        T y0 = __shfl_sync(kFull, v[r], c0), y1 = __shfl_sync(kFull, v[r], c1);
        T y2 = __shfl_sync(kFull, v[r], c2), y3 = __shfl_sync(kFull, v[r], c3);
        if (!UNIT) y0 *= rd[c0];
        y1 -= t10 * y0;
        if (!UNIT) y1 *= rd[c1];
        y2 -= t20 * y0;
        y2 -= t21 * y1;
        if (!UNIT) y2 *= rd[c2];
        y3 -= t30 * y0;
        y3 -= t31 * y1;
        y3 -= t32 * y2;
        if (!UNIT) y3 *= rd[c3];
        v[r] -= b0 * y0;
        v[r] -= b1 * y1;
        v[r] -= b2 * y2;
        v[r] -= b3 * y3;
      }
    }
  }
  if (!UNIT) {
#pragma unroll
    for (int r = 0; r < RC; ++r) v[r] *= rd[lane];
  }
}

// whether right-hand sides r0 .. r0 + nr fill pairs of a row but for its padding: a
// chunk of four or eight does, one of one or two (FP64) may not
template <typename T>
__device__ __forceinline__ bool whole_pairs(const SolveArgs<T>& a, int r0, int nr) {
  return sizeof(T) == 4 || (r0 % 2 == 0 && (nr % 2 == 0 || r0 + nr == a.R));
}

template <typename T, bool TRANS, int RC>
__device__ __forceinline__ void wide_forward(const SolveArgs<T>& a, const FrontDesc& d, int k, int q, int ch, int rc,
                                             int r0, int nr, T* sm) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int ns = d.ns, F = d.F;
  const bool vec = a.vec && whole_pairs<T>(a, r0, nr);
  T* ys = sm;                                    // kWideRows x RC: solved blocks
  T* B = ys + kWideRows * RC + wid * kTri;       // this warp's triangle
  T* tile = ys + kWideRows * RC + kSolveWarps * kTri + wid * 32 * WideTile<T>::LD;  // TRANS
  __shared__ int s_seen;
  const T* f = a.fronts + a.K * d.fo + (int64_t)k * F * F;
  const int64_t st = (int64_t)a.K * a.RV;
  T* Vs = a.V + (d.vo * a.K + k) * a.RV + r0;
  const int nblk = (ns + 31) >> 5, b0 = q * kSolveWarps;  // blocks; the first of this CTA's rows
  const int i = q * kWideRows + tid;
  const int mine = b0 + wid;                              // block of this warp's rows
  const int last = min(mine, nblk - 1);                   // last block this warp takes part in
  const bool rows = i - lane < F;                         // this warp has rows
  const bool shared = F > kWideRows;                      // other CTAs take this front's other rows
  int* flag = a.wide + (int64_t)(d.flag + (k * ((a.R + rc - 1) / rc) + ch)) * kCtrStride;
  if (mine < nblk) stage_triangle<T, true, !TRANS, TRANS>(B, f, F, mine * 32, min(32, ns - mine * 32), lane);
  Gather g = gather_begin<T>(a, d, i, i < F);
  if (tid == 0) wait_children(a, d, k);
  __syncthreads();
  constexpr int GR = RC < 4 ? RC : 4;
  T w[RC];
#pragma unroll
  for (int rg = 0; rg < RC; rg += GR) {
    T x[GR];
#pragma unroll
    for (int r = 0; r < GR; ++r) x[r] = T(0);
    const int n = i < F ? min(GR, nr - rg) : 0;
    if (n > 0) {
      gather_rhs<T, GR>(a, g, k, r0 + rg, n, vec, x);
      gather_children<T, GR, (GR == 1 ? 8 : sizeof(T) == 4 ? 4 : 2)>(a, g, k, r0 + rg, n, vec, x);
    }
#pragma unroll
    for (int r = 0; r < GR; ++r) w[rg + r] = x[r];
  }
  T L[32];
  if (rows && (mine > 0 || b0 >= nblk)) load_panel<T, TRANS>(L, f, F, i, F, 0, min(32, ns), tile, lane);
  // blocks solved by other CTAs
  const int next = min(b0, nblk);
  for (int p = 0; p < next;) {
    if (tid == 0) s_seen = wait_count(flag, p + 1, a.err, a.wait_ns);
    __syncthreads();  // also: the blocks before are taken in
    const int m = min(next, min(max(s_seen, p + 1), p + kSolveWarps)) - p;
    if (tid < m * 32) {
      const int c = p * 32 + tid;  // below ns: only the last block is short, and it is in no CTA's way
      T y[RC];
#pragma unroll
      for (int r = 0; r < RC; ++r) y[r] = T(0);
      if (c < ns) ld_row<T, RC>(Vs + c * st, nr, vec, y);
#pragma unroll
      for (int r = 0; r < RC; ++r) ys[tid * RC + r] = y[r];
    }
    __syncthreads();
    for (int e = 0; e < m; ++e, ++p) {
      if (!rows) continue;
      apply_panel<T, RC>(L, w, ys + e * 32 * RC, nr);
      if (p + 1 <= last && p + 1 != mine)
        load_panel<T, TRANS>(L, f, F, i, F, (p + 1) * 32, min(32, ns - (p + 1) * 32), tile, lane);
    }
  }
  if (next > 0) __syncthreads();
  // this CTA's own blocks
  for (int p = b0; p < min(b0 + kSolveWarps, nblk); ++p) {
    T* y = ys + (p & 1) * 32 * RC;
    const int nb = min(32, ns - p * 32);
    if constexpr (kSpread<T, RC>) {
      if (mine == p) {
#pragma unroll
        for (int r = 0; r < RC; ++r) y[lane * RC + r] = lane < nb ? w[r] : T(0);
      }
      spread_solve<T, true, !TRANS, RC>(ys + kWideRows * RC, p - b0, y, nr, nb, wid, lane);
    }
    if (mine == p) {
      // rows past the pivots in this warp (a short last block) have zeros in
      // the triangle: their coefficients follow below
      if constexpr (kSpread<T, RC>) {
#pragma unroll
        for (int r = 0; r < RC; ++r) w[r] = lane < nb ? y[lane * RC + r] : w[r];
      } else {
        triangle_solve<T, true, !TRANS, RC>(B, w, nb, lane);
#pragma unroll
        for (int r = 0; r < RC; ++r) y[lane * RC + r] = lane < nb ? w[r] : T(0);
      }
      if (i < ns) st_row<T, RC>(Vs + i * st, nr, vec, w);
      if (nb < 32) load_panel<T, TRANS>(L, f, F, i, F, p * 32, nb, tile, lane);
    }
    if constexpr (kSpread<T, RC>) __syncwarp();
    else __syncthreads();
    if (shared && mine == p && lane == 0) publish(flag);  // behind the barrier: off the chain of blocks
    if (rows && (mine > p || (mine == p && p * 32 + 32 > ns))) {
      if (mine > p) {
        apply_panel<T, RC>(L, w, y, nr);
      } else {
        T u[RC];
#pragma unroll
        for (int r = 0; r < RC; ++r) u[r] = w[r];
        apply_panel<T, RC>(L, u, y, nr);
#pragma unroll
        for (int r = 0; r < RC; ++r) w[r] = i >= ns ? u[r] : w[r];
      }
      if (p + 1 <= last && p + 1 != mine)
        load_panel<T, TRANS>(L, f, F, i, F, (p + 1) * 32, min(32, ns - (p + 1) * 32), tile, lane);
    }
  }
  if (i >= ns && i < F) st_row<T, RC>(Vs + i * st, nr, vec, w);
  __syncthreads();
  if (tid == 0) publish_up(a, d, k);
}

// The rows are the pivots, solved from the last block up; the update rows'
// values, known, come first as further blocks of columns.
template <typename T, bool TRANS, int RC>
__device__ __forceinline__ void wide_backward(const SolveArgs<T>& a, const FrontDesc& d, int k, int q, int ch, int rc,
                                              int r0, int nr, T* sm) {
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int ns = d.ns, F = d.F, ms = F - ns;
  const bool vec = a.vec && whole_pairs<T>(a, r0, nr);
  T* ys = sm;
  T* B = ys + kWideRows * RC + wid * kTri;
  T* tile = ys + kWideRows * RC + kSolveWarps * kTri + wid * 32 * WideTile<T>::LD;
  __shared__ int s_seen;
  const T* f = a.fronts + a.K * d.fo + (int64_t)k * F * F;
  const int64_t st = (int64_t)a.K * a.RV;
  T* xk = a.xt + (int64_t)k * a.RV + r0;
  const int nblk = (ns + 31) >> 5, b0 = q * kSolveWarps;
  const int hi = min(b0 + kSolveWarps, nblk) - 1;  // last block of this CTA's rows
  const int i = q * kWideRows + tid;
  const int mine = b0 + wid;
  const bool rows = i - lane < ns;
  const bool shared = ns > kWideRows;
  int* flag = a.wide + (int64_t)(d.flag + (k * ((a.R + rc - 1) / rc) + ch)) * kCtrStride;
  if (rows) stage_triangle<T, false, TRANS, TRANS>(B, f, F, mine * 32, min(32, ns - mine * 32), lane);
  T w[RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) w[r] = T(0);
  if (i < ns) ld_row<T, RC>(a.V + ((d.vo + i) * a.K + k) * a.RV + r0, nr, vec, w);
  T L[32];
  if (ms > 0) {
    if (rows) load_panel<T, TRANS>(L, f, F, i, ns, ns, min(32, ms), tile, lane);
    if (tid == 0) wait_parent(a, d, k);
    __syncthreads();
    for (int j0 = 0; j0 < ms; j0 += kWideRows) {
      const int m = min(kWideRows, ms - j0);
      T y[RC];
#pragma unroll
      for (int r = 0; r < RC; ++r) y[r] = T(0);
      if (tid < m) ld_row<T, RC>(xk + __ldg(a.rows + d.ro + j0 + tid) * st, nr, vec, y);
#pragma unroll
      for (int r = 0; r < RC; ++r) ys[tid * RC + r] = y[r];
      __syncthreads();
      for (int e = 0; e < m; e += 32) {
        if (!rows) continue;
        apply_panel<T, RC>(L, w, ys + e * RC, nr);
        const int jn = j0 + e + 32;
        if (jn < ms) load_panel<T, TRANS>(L, f, F, i, ns, ns + jn, min(32, ms - jn), tile, lane);
      }
      __syncthreads();
    }
  }
  // blocks solved by other CTAs, then this CTA's own (a warp's rows need the
  // blocks above its own)
  const int top = nblk - 1;
  if (rows && mine < top) load_panel<T, TRANS>(L, f, F, i, ns, top * 32, ns - top * 32, tile, lane);
  for (int p = top; p > hi;) {
    if (tid == 0) s_seen = wait_count(flag, nblk - p, a.err, a.wait_ns);
    __syncthreads();
    const int m = min(p - hi, min(max(s_seen, nblk - p) - (top - p), kSolveWarps));
    const int lo = p - m + 1;
    if (tid < m * 32) {
      const int c = lo * 32 + tid;
      T y[RC];
#pragma unroll
      for (int r = 0; r < RC; ++r) y[r] = T(0);
      if (c < ns) ld_row<T, RC>(xk + (d.c0 + c) * st, nr, vec, y);
#pragma unroll
      for (int r = 0; r < RC; ++r) ys[tid * RC + r] = y[r];
    }
    __syncthreads();
    for (; p >= lo; --p) {
      if (!rows) continue;
      apply_panel<T, RC>(L, w, ys + (p - lo) * 32 * RC, nr);
      if (p - 1 > mine) load_panel<T, TRANS>(L, f, F, i, ns, (p - 1) * 32, 32, tile, lane);
    }
  }
  if (top > hi) __syncthreads();
  for (int p = hi; p >= b0; --p) {
    T* y = ys + (p & 1) * 32 * RC;
    if constexpr (kSpread<T, RC>) {
      if (mine == p) {
#pragma unroll
        for (int r = 0; r < RC; ++r) y[lane * RC + r] = w[r];
      }
      spread_solve<T, false, TRANS, RC>(ys + kWideRows * RC, p - b0, y, nr, min(32, ns - p * 32), wid, lane);
    }
    if (mine == p) {
      if constexpr (kSpread<T, RC>) {
#pragma unroll
        for (int r = 0; r < RC; ++r) w[r] = y[lane * RC + r];
      } else {
        triangle_solve<T, false, TRANS, RC>(B, w, min(32, ns - p * 32), lane);
#pragma unroll
        for (int r = 0; r < RC; ++r) y[lane * RC + r] = i < ns ? w[r] : T(0);
      }
      if (i < ns) st_row<T, RC>(xk + (d.c0 + i) * st, nr, vec, w);
    }
    if constexpr (kSpread<T, RC>) __syncwarp();
    else __syncthreads();
    if (shared && mine == p && lane == 0) publish(flag);
    if (mine < p) {
      apply_panel<T, RC>(L, w, y, nr);
      if (p - 1 > mine) load_panel<T, TRANS>(L, f, F, i, ns, (p - 1) * 32, 32, tile, lane);
    }
  }
  if (i < ns && a.xd)
    st_xd_row<T, RC>(a.xd + ((int64_t)(d.c0 + i) * a.K + k) * a.RX + r0, nr, a.vecd && whole_pairs<T>(a, r0, nr),
                     a.xd_mode, w);
  __syncthreads();
  if (tid == 0) publish_self(a, d, k);
}

// ---------------------------------------------------------------------------
// One launch per direction.  CTAs take work units in ticket order (forward by
// height above the leaves, backward by depth below the root): a unit is one CTA
// task, or 256 / SEG segment tasks, or 8 warps' tasks of 32 columns.  A task
// waits for its children or its parent (completion counters above), that is for
// units with smaller tickets, which running CTAs already hold, so the schedule
// cannot deadlock whatever the number of resident CTAs, and every wait is
// bounded.  (Taking the next ticket while a unit runs hides its latency but
// parks a unit behind one that waits.)  In the adaptive sweeps the list is the
// in-order subsequence of units holding a front of an instance still iterating.
// Without completion counters (one launch per stage) nothing waits but the
// tasks of one front with more than 32 pivots for each other.
// ---------------------------------------------------------------------------
template <typename T, bool FWD, bool TRANS, int RC>
__device__ __forceinline__ void wide_task(const SolveArgs<T>& a, int slot, int b, int ch, T* sm) {
  const FrontDesc d = ld_desc(a.desc + slot);
  if (a.act && !a.act[d.inst]) return;
  const int rc = sizeof(T) == 8 && RC > 1 ? b >> 4 & 15 : RC;
  const int r0 = ch * rc, nr = min(rc, a.R - r0);
  const int k = b & 15, q = b >> 8;  // shift; rows [256 q, 256 q + 256)
  if (FWD) wide_forward<T, TRANS, RC>(a, d, k, q, ch, rc, r0, nr, sm);
  else wide_backward<T, TRANS, RC>(a, d, k, q, ch, rc, r0, nr, sm);
}
// The same with registers of its own: with several right-hand sides the other
// tasks of the kernel spill less beside it.
template <typename T, bool FWD, bool TRANS, int RC>
__device__ __noinline__ void wide_call(const SolveArgs<T>& a, int slot, int b, int ch, T* sm) {
  wide_task<T, FWD, TRANS, RC>(a, slot, b, ch, sm);
}

// WIDE: right-hand sides that the tasks of fronts with more than 32 pivots are compiled
// for; one call of one form, since a second would have each keep registers for the other.
// SEGS: backward segments of several right-hand sides, a kernel of their own for the same
// reason (2000 buses, six solves of 16 right-hand sides: 310 us, 317 with them compiled in)
template <typename T, bool FWD, bool TRANS, int MINB, bool ONE, int WIDE, bool SEGS>
__global__ void __launch_bounds__(kSolveThreads, MINB) k_solve(const __grid_constant__ SolveArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_unit[2];
  T* sm = reinterpret_cast<T*>(smraw);
  const int tid = threadIdx.x, wid = tid >> 5;
  const int nunits = a.ucount ? *a.ucount : a.nunits;
  const int4* units = reinterpret_cast<const int4*>(a.units) + a.first;
  for (int par = 0;; par ^= 1) {
    if (tid == 0) s_unit[par] = atomicAdd(a.ticket, 1);
    __syncthreads();  // also: the unit before is done with shared memory
    const int u = s_unit[par];
    if (u >= nunits) return;
    const int4 uq = __ldg(units + u);
    const SolveUnit U{uq.x, uq.y, uq.z, uq.w};
    const int kind = U.x & 15;
    if (kind == kUnitWide) {
      if constexpr (ONE) wide_task<T, FWD, TRANS, 1>(a, U.a, U.b, U.c, sm);
      else wide_call<T, FWD, TRANS, WIDE>(a, U.a, U.b, U.c, sm);
    } else if constexpr (FWD || ONE) {
      constexpr int NR = ONE ? 1 : 8;
      FrontDesc d;
      if (kind == kUnitCta) {
        d = ld_desc(a.desc + U.a);
        // a front of an instance whose sweeps have stopped is skipped: no front
        // of another instance depends on it (CTA-uniform test)
        if (!a.act || a.act[d.inst]) {
          if constexpr (FWD) thin_forward<T, TRANS, NR>(a, d, U.b, U.c * NR, min(NR, a.R - U.c * NR), sm);
          else thin_backward1<T, TRANS>(a, d, U.b, sm);
        }
      } else if (kind == kUnitSeg8) {
        const SegTask t = seg_task<T>(a, U, (unsigned)U.b + tid / 8, NR, d);
        if constexpr (FWD) seg_forward<T, 8, TRANS, NR>(a, t, d, tid % 8, nullptr);
        else seg_backward<T, 8, TRANS>(a, t, d, tid % 8);
      } else if (kind == kUnitSeg16) {
        const SegTask t = seg_task<T>(a, U, (unsigned)U.b + tid / 16, NR, d);
        if constexpr (FWD) seg_forward<T, 16, TRANS, NR>(a, t, d, tid % 16, nullptr);
        else seg_backward<T, 16, TRANS>(a, t, d, tid % 16);
      } else {
        const SegTask t = seg_task<T>(a, U, (unsigned)U.b + tid / 32, NR, d);
        if constexpr (FWD) seg_forward<T, 32, TRANS, NR>(a, t, d, tid % 32, sm + wid * 32 * NR);
        else seg_backward<T, 32, TRANS>(a, t, d, tid % 32);
      }
    } else if (SEGS && kind == kUnitSeg32) {
      FrontDesc d;
      const SegTask t = seg_task<T>(a, U, (unsigned)U.b + wid, 8, d);
      seg_backward_rhs<T, TRANS, 8>(a, t, d, tid & 31);
    } else {
      // a CTA task, its 8 warps sharing the front, or per warp task q of the
      // group: front q / NG, columns [32 g, 32 g + 32), g = q % NG
      const bool cta = kind == kUnitCta;
      unsigned slot = U.a, g = U.b;
      bool on = true;
      if (!cta) {
        const unsigned q = (unsigned)U.b + wid;
        on = q < (unsigned)U.c;
        const unsigned f = q / (unsigned)a.NG;
        g = q - f * a.NG;
        slot = U.a + (on ? f : 0);
      }
      const FrontDesc d = ld_desc(a.desc + slot);
      if (on && (!a.act || a.act[d.inst])) {  // uniform over the CTA for a CTA task
        col_backward<T, TRANS>(a, d, (int)g, cta ? wid : 0, cta ? kSolveWarps : 1, sm + (int64_t)wid * a.stage,
                               sm + (int64_t)kSolveWarps * a.stage);
        if (cta ? tid == 0 : (tid & 31) == 0) publish_self(a, d, (int)g);
      }
    }
  }
}

template <typename T, bool FWD, bool TRANS, int MINB, bool ONE, int WIDE, bool SEGS = false>
int launch_one(const SolveArgs<T>& a, int nunits, size_t smem, cudaStream_t st) {
  static std::atomic<int> nsm_dev[kMaxDevices];
  const int dev = current_device();
  int nsm = nsm_dev[dev].load(std::memory_order_acquire);
  if (!nsm) {
    cudaFuncSetAttribute(k_solve<T, FWD, TRANS, MINB, ONE, WIDE, SEGS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSolveSmemMax);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    nsm = std::max(nsm, 1);
    nsm_dev[dev].store(nsm, std::memory_order_release);
  }
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_solve<T, FWD, TRANS, MINB, ONE, WIDE, SEGS>, kSolveThreads, smem);
  const int grid = std::max(1, std::min(nunits, std::max(1, occ) * nsm));
  k_solve<T, FWD, TRANS, MINB, ONE, WIDE, SEGS><<<grid, kSolveThreads, smem, st>>>(a);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace

// elements of a launch's column tasks (8 warps' stages and partial sums), and of
// its tasks of fronts with more than 32 pivots, `wide` right-hand sides each
template <typename T>
constexpr size_t col_smem(int nk) { return (size_t)kSolveWarps * col_stage<T>(nk) + (size_t)(kSolveWarps - 1) * 8 * 32; }
template <typename T>
constexpr size_t wide_smem(int wide, bool trans) {
  return (size_t)kWideRows * wide + (size_t)kSolveWarps * kTri + (trans ? (size_t)kSolveWarps * 32 * WideTile<T>::LD : 0);
}

template <typename T, bool FWD>
int launch_solve_dir(bool trans, const SolveArgs<T>& a0, int32_t nunits, int32_t wide, bool segs, int32_t ctas,
                     cudaStream_t st) {
  if (nunits <= 0) return 0;
  SolveArgs<T> a = a0;
  size_t e;
  if (FWD || a.R == 1) {
    const int nr = a.R == 1 ? 1 : 8;
    e = std::max(thin_smem(FWD, nr), kSolveWarps * 32 * nr);
  } else {
    // most shifts among 32 columns
    const int nk = std::min(a.K, (31 + a.RV - 1) / a.RV + 1);
    a.stage = col_stage<T>(nk);
    e = col_smem<T>(nk);
  }
  const bool spread = wide > kWideAlone<T>;
  if (wide > 0) e = std::max(e, wide_smem<T>(a.R == 1 ? 1 : spread ? kWideSpread<T> : kWideAlone<T>, trans));
  const size_t smem = e * sizeof(T);
  static_assert(col_smem<T>(PISP_K_MAX) * sizeof(T) <= kSolveSmemMax && wide_smem<T>(kWideSpread<T>, true) * sizeof(T) <= kSolveSmemMax &&
                    std::max(thin_smem(FWD, 8), kSolveWarps * 32 * 8) * sizeof(T) <= kSolveSmemMax,
                "every launch of a solve fits");
  if (a.R == 1)
    return trans ? launch_one<T, FWD, true, 2, true, 1>(a, nunits, smem, st)
                 : launch_one<T, FWD, false, 2, true, 1>(a, nunits, smem, st);
  constexpr int A = kWideAlone<T>, W = kWideSpread<T>;
  if constexpr (!FWD) {
    if (segs && spread)
      return trans ? launch_one<T, FWD, true, 2, false, W, true>(a, nunits, smem, st)
                   : launch_one<T, FWD, false, 2, false, W, true>(a, nunits, smem, st);
    if (segs)
      return trans ? launch_one<T, FWD, true, 2, false, A, true>(a, nunits, smem, st)
                   : launch_one<T, FWD, false, 2, false, A, true>(a, nunits, smem, st);
  }
  if (spread)  // the registers of two CTAs an SM
    return trans ? launch_one<T, FWD, true, 2, false, W>(a, nunits, smem, st)
                 : launch_one<T, FWD, false, 2, false, W>(a, nunits, smem, st);
  if (trans) return launch_one<T, FWD, true, 2, false, A>(a, nunits, smem, st);
  if (ctas >= 4) return launch_one<T, FWD, false, 4, false, A>(a, nunits, smem, st);
  if (ctas == 3) return launch_one<T, FWD, false, 3, false, A>(a, nunits, smem, st);
  return launch_one<T, FWD, false, 2, false, A>(a, nunits, smem, st);
}

}  // namespace pisp
