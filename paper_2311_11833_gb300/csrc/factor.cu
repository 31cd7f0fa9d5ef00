// Pivot-free multifrontal LU of all K perturbed matrices (Alg. 1, Eq. xap / xam).
//
// Each supernode s owns a dense front of size F = ns + ms per perturbation k:
//   1. assembly: P (A + t_k D) P^T entries that belong to s, plus the
//      Schur complements (update blocks) of its children (extend-add);
//   2. ns steps of right-looking elimination WITHOUT pivoting: the pivot
//      order is the static one fixed by the symbolic phase (Sec. II-C).
// Fronts at the same level of the assembly forest are independent; one
// launch covers all of them, all K perturbations (grid.y / grid.z) and all
// instances of a batch.  Small fronts are factored in shared memory, one CTA
// per (front, k); large fronts use a blocked right-looking scheme in global
// memory (panel factorisation, row-block triangular solve, tiled update).
//
// Storage: front s of perturbation k occupies F*F contiguous elements
// (column-major) at K*front_off[s] + k*F*F.  After factorisation it holds
// L11\U11, L21, U12 and the Schur complement F22 that the parent reads.
#include <atomic>
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <type_traits>
#include <vector>

#include "pisp_internal.h"

namespace pisp {
namespace {

constexpr int kSmemCap = 225 * 1024;  // dynamic shared memory budget per CTA
constexpr int kStatusZero = 1;        // status bits: exact zero pivot
constexpr int kStatusNonfinite = 2;   //              Inf / NaN pivot

template <typename T>
__device__ __forceinline__ void check_pivot(T piv, const SymDev& sd, int s, int k, int K,
                                            int col, int32_t* status, int32_t* badcol) {
  const double p = (double)piv;
  int code = 0;
  if (!isfinite(p)) code = kStatusNonfinite;
  else if (p == 0.0) code = kStatusZero;
  if (code) {
    const int g = sd.inst[s];
    atomicOr(&status[g * K + k], code);
    atomicMin(&badcol[g * K + k], col);
  }
}

// Pivot-free LU of a panel in shared memory: rows p0..F-1 of nb <= 32
// columns, P[i + c*ld] = front(i, p0 + c).  Warps take rows; lane j of a warp
// updates column j, so a row costs one instruction group.  The warp that
// finishes row p0+c+1 during step c also copies it to the other half of a
// double-buffered pivot row, so each pivot costs one block barrier.  An odd
// ld keeps the lanes' column accesses on distinct banks.
template <typename T>
__device__ __forceinline__ void panel_factor_rows(T* P, int ld, int F, int p0, int nb,
                                                  T (*prow)[32], const SymDev& sd, int s, int k,
                                                  int K, int colbase, int32_t* status,
                                                  int32_t* badcol) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (wid == 0 && lane < nb) prow[0][lane] = P[p0 + lane * ld];
  for (int c = 0; c < nb; ++c) {
    __syncthreads();
    const T* pr = prow[c & 1];
    const int pc = p0 + c;
    const T piv = pr[c];
    if (threadIdx.x == 0) check_pivot(piv, sd, s, k, K, colbase + c, status, badcol);
    const T rp = T(1) / piv;
    const T pj = (lane > c && lane < nb) ? pr[lane] : T(0);
    for (int i = pc + 1 + wid; i < F; i += nw) {
      const T l = P[i + c * ld] * rp;
      __syncwarp();
      if (lane == c) P[i + c * ld] = l;
      else if (lane > c && lane < nb) P[i + lane * ld] -= l * pj;
      if (i == pc + 1 && c + 1 < nb) {
        __syncwarp();
        if (lane < nb) prow[(c + 1) & 1][lane] = P[i + lane * ld];
      }
    }
  }
  __syncthreads();
}

// Pivot-free elimination of a panel in shared memory: rows 0..Mr-1, nb <= 32
// columns, P[i + c*ld] (ld odd).  Per pivot: scale the column by one
// reciprocal, then lane j of each warp updates column j of the warp's rows;
// the loops carry no integer division.
template <typename T>
__device__ __forceinline__ void panel_eliminate(T* P, int ld, int Mr, int nb, const SymDev& sd,
                                                int s, int k, int K, int colbase, int32_t* status,
                                                int32_t* badcol) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  for (int c = 0; c < nb; ++c) {
    const T piv = P[c + c * ld];
    if (tid == 0) check_pivot(piv, sd, s, k, K, colbase + c, status, badcol);
    const T rp = T(1) / piv;
    for (int i = c + 1 + tid; i < Mr; i += nt) P[i + c * ld] *= rp;
    __syncthreads();
    if (lane > c && lane < nb) {
      const T u = P[c + lane * ld];
      T* col = P + lane * ld;
      const T* lc = P + c * ld;
      for (int i = c + 1 + wid; i < Mr; i += nw) col[i] -= lc[i] * u;
    }
    __syncthreads();
  }
}

// Children's update columns added into the destination columns [d0, d0 + w)
// and rows [R0, R1) of front s, stored at dst[(row - R0) + (col - d0) * ld].  Each
// destination column belongs to one warp (col - d0 = warp, warp + warps, ...),
// which walks the column's inverse extend-add list in child order: every element
// receives its contributions in child order, with no barrier between children,
// and a group of 8 x 32 child rows is loaded before any of them is added.  Owner
// tiles keep this form: their columns are tall, and the flat form below is no
// faster there (10000 buses 2401 us of tiles against 2424).
template <typename T>
__device__ __forceinline__ void extend_add_columns(const SymDev& sd, int s, int k, int K,
                                                   const T* __restrict__ fronts, T* dst, int ld,
                                                   int d0, int w, int R0, int R1, int wid, int nw) {
  const int lane = threadIdx.x & 31;
  const int64_t vo = sd.vec_off[s];
  for (int dc = wid; dc < w; dc += nw) {
    const int64_t e0 = sd.inv_off[vo + d0 + dc], e1 = sd.inv_off[vo + d0 + dc + 1];
    T* dcol = dst + (int64_t)dc * ld;
    for (int64_t eb = e0; eb < e1; eb += 32) {
      const int ne = (int)min((int64_t)32, e1 - eb);
      int ca = 0, cF = 1, ccol = 0;
      int64_t cfo = 0, cro = 0;
      if (lane < ne) {
        const int ch = sd.inv_child[eb + lane];
        ca = sd.inv_a[eb + lane];
        cF = sd.inv_cF[eb + lane];
        ccol = sd.inv_col[eb + lane];
        cfo = sd.front_off[ch];
        cro = sd.row_off[ch];
      }
      for (int e = 0; e < ne; ++e) {
        const int eF = __shfl_sync(0xffffffffu, cF, e);
        const int ecol = __shfl_sync(0xffffffffu, ccol, e);
        const int cns = ecol - __shfl_sync(0xffffffffu, ca, e);
        const int cms = eF - cns;
        const int32_t* em = sd.emap + __shfl_sync(0xffffffffu, cro, e);
        const T* scol = fronts + (int64_t)K * __shfl_sync(0xffffffffu, cfo, e) + (int64_t)k * eF * eF +
                        (int64_t)ecol * eF + cns;
        for (int a0 = 0; a0 < cms; a0 += 256) {
          int r[8];
          T v[8];
#pragma unroll
          for (int t = 0; t < 8; ++t) {
            const int a = a0 + lane + 32 * t;
            r[t] = a < cms ? em[a] : -1;
            v[t] = a < cms ? scol[a] : T(0);
          }
#pragma unroll
          for (int t = 0; t < 8; ++t)
            if (r[t] >= R0 && r[t] < R1) dcol[r[t] - R0] += v[t];
        }
        __syncwarp();
      }
    }
  }
}

// The CTA: entries [e0, e1) of the assembly map, EB at a time per thread, so that
// the two dependent reads of an entry are paid once for EB of them (a 486-row
// dense front's tiles spent 33 us each on them one by one).
template <typename T, typename Put>
__device__ __forceinline__ void add_entries(const SymDev& sd, const double* __restrict__ vals, int64_t e0, int64_t e1,
                                            Put put) {
  constexpr int EB = 8;
  const int nt = blockDim.x;
  for (int64_t e = e0 + threadIdx.x; e < e1; e += (int64_t)EB * nt) {
    int d[EB], at[EB];
    double v[EB];
#pragma unroll
    for (int q = 0; q < EB; ++q) {
      const bool in = e + q * nt < e1;
      d[q] = in ? sd.amap_dst[e + q * nt] : -1;
      at[q] = in ? sd.amap_src[e + q * nt] : 0;
    }
#pragma unroll
    for (int q = 0; q < EB; ++q) v[q] = d[q] >= 0 ? vals[at[q]] : 0.0;
#pragma unroll
    for (int q = 0; q < EB; ++q)
      if (d[q] >= 0) put(d[q], (T)v[q]);
  }
}

// One warp: the children's update blocks added into the destination columns
// [d0, d1) of front s, rows [R0, R1), stored at dst[row + col * ld] (dst is
// where row 0 of column 0 would be).  The columns'
// entries of the inverse extend-add map are consecutive; 32 are resolved at a
// time, one a lane, and four child columns are in flight at a time (two rows a
// lane), so that a memory latency covers four contributions and not one.  The
// additions to an element follow a fixed order.
template <typename T>
__device__ __forceinline__ void extend_add_flat(const SymDev& sd, int s, int k, int K, const T* __restrict__ fronts,
                                                T* dst, int ld, int d0, int d1, int R0, int R1) {
  constexpr int NE = 4;
  const int lane = threadIdx.x & 31;
  const int64_t vo = sd.vec_off[s];
  const int64_t e1 = sd.inv_off[vo + d1];
  for (int64_t eb = sd.inv_off[vo + d0]; eb < e1; eb += 32) {
    const int ne = (int)min((int64_t)32, e1 - eb);
    int64_t src = 0, ro = 0;
    int cms = 0, dc = 0;
    if (lane < ne) {
      const int ch = sd.inv_child[eb + lane], ca = sd.inv_a[eb + lane];
      const int cF = sd.inv_cF[eb + lane], col = sd.inv_col[eb + lane];
      ro = sd.row_off[ch];
      cms = cF - (col - ca);
      src = (int64_t)K * sd.front_off[ch] + (int64_t)k * cF * cF + (int64_t)col * cF + (col - ca);
      dc = sd.emap[ro + ca] * ld;
    }
    for (int g = 0; g < ne; g += NE) {
      const T* p[NE];
      const int32_t* em[NE];
      int m[NE], d[NE], most = 0;
#pragma unroll
      for (int q = 0; q < NE; ++q) {
        p[q] = fronts + __shfl_sync(0xffffffffu, src, g + q);
        em[q] = sd.emap + __shfl_sync(0xffffffffu, ro, g + q);
        m[q] = __shfl_sync(0xffffffffu, cms, g + q);
        d[q] = __shfl_sync(0xffffffffu, dc, g + q);
        most = max(most, m[q]);
      }
      for (int a = lane; a < most + lane; a += 64) {  // warp-uniform trips
        int r0[NE], r1[NE];
        T v0[NE], v1[NE];
#pragma unroll
        for (int q = 0; q < NE; ++q) {
          r0[q] = a < m[q] ? em[q][a] : -1;
          v0[q] = a < m[q] ? __ldcg(p[q] + a) : T(0);
          r1[q] = a + 32 < m[q] ? em[q][a + 32] : -1;
          v1[q] = a + 32 < m[q] ? __ldcg(p[q] + a + 32) : T(0);
        }
#pragma unroll
        for (int q = 0; q < NE; ++q) {
          if (r0[q] >= R0 && r0[q] < R1) dst[r0[q] + d[q]] += v0[q];
          if (r1[q] >= R0 && r1[q] < R1) dst[r1[q] + d[q]] += v1[q];
          __syncwarp();  // the next contribution may land on another lane's element
        }
      }
    }
  }
}

// leading dimension of a front in shared memory: odd, so that rows and columns
// both fall on distinct banks
__host__ __device__ __forceinline__ int front_ld(int F) { return F | 1; }

// Pivot-free LU of ns pivots of the F x F front f (leading dimension ld) in
// shared memory, by the whole CTA, in panels of NB pivots: one warp factors the
// panel's diagonal block in registers (lane = row), then threads take the rows
// below it and the columns beside it, one each, and 4 x 4 register tiles update
// the rest: three barriers a panel.  (One pivot at a time, two barriers and a
// pass over the whole front in shared memory each, a 213-row front took 500 us.)
template <typename T>
__device__ __forceinline__ void front_lu(T* f, int ld, int F, int ns, T* rinv, const SymDev& sd, int s, int k, int K,
                                         int32_t* status, int32_t* badcol) {
  constexpr int NB = 16;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int c0 = sd.c0[s];
  for (int p0 = 0; p0 < ns; p0 += NB) {
    const int nb = min(NB, ns - p0);
    T* fd = f + p0 + p0 * ld;  // the diagonal block
    if (tid < 32) {
      T d[NB];
#pragma unroll
      for (int c = 0; c < NB; ++c) d[c] = lane < nb && c < nb ? fd[lane + c * ld] : T(0);
#pragma unroll 1
      for (int c = 0; c < nb; ++c) {  // d[0] is column c: the row moves down a place each step
        const T piv = __shfl_sync(0xffffffffu, d[0], c);
        if (lane == 0) check_pivot(piv, sd, s, k, K, c0 + p0 + c, status, badcol);
        const T rp = T(1) / piv;
        if (lane == 0) rinv[c] = rp;
        const T l = lane > c ? d[0] * rp : T(0);
        if (lane < nb) fd[lane + c * ld] = lane > c ? l : d[0];
#pragma unroll
        for (int j = 1; j < NB; ++j) d[j - 1] = d[j] - l * __shfl_sync(0xffffffffu, d[j], c);
      }
    }
    __syncthreads();
    const int t0 = p0 + nb, m = F - t0;
    for (int q = tid; q < 2 * m; q += nt) {
      // a row below, L(i, :) = A(i, :) U^-1, or a column beside, U(:, j) = L^-1 A(:, j)
      const bool low = q < m;
      T* v = low ? f + t0 + q + p0 * ld : f + p0 + (t0 + q - m) * ld;
      const int vs = low ? ld : 1, ds = low ? ld : 1;  // strides of the vector, and of the block's row or column
      T x[NB];
#pragma unroll
      for (int c = 0; c < NB; ++c) x[c] = c < nb ? v[c * vs] : T(0);
#pragma unroll 1
      for (int c = 0; c < nb; ++c) {
        const T y = low ? x[0] * rinv[c] : x[0];
        v[c * vs] = y;
        const T* e = fd + c * (ld + 1);  // the pivot; then along its row (U) or column (L)
#pragma unroll
        for (int j = 1; j < NB; ++j) x[j - 1] = x[j] - (c + j < nb ? e[j * ds] * y : T(0));
      }
    }
    __syncthreads();
    // 64 x 64 tiles, 16 x 16 threads, one tile per 256 threads
    const int tx = tid & 15, ty = (tid >> 4) & 15, tpd = (m + 63) >> 6;
    for (int t = tid >> 8; t < tpd * tpd; t += nt >> 8) {
      const int ib = t0 + (t % tpd) * 64 + tx, jb = t0 + (t / tpd) * 64 + ty;
      T acc[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
      const T* lp = f + p0 * ld;
      const T* up = f + p0;
#pragma unroll 2
      for (int c = 0; c < nb; ++c) {
        T l[4], u[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) l[a] = ib + 16 * a < F ? lp[ib + 16 * a + c * ld] : T(0);
#pragma unroll
        for (int b = 0; b < 4; ++b) u[b] = jb + 16 * b < F ? up[c + (jb + 16 * b) * ld] : T(0);
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a][b] += l[a] * u[b];
      }
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a)
          if (ib + 16 * a < F && jb + 16 * b < F) f[ib + 16 * a + (jb + 16 * b) * ld] -= acc[a][b];
    }
    __syncthreads();
  }
}

// The same one pivot at a time: the column scaled by all threads, then the trailing
// columns dealt out to the warps, two barriers a pivot.  The form of FP64, whose pipe
// (2 FMA a clock per SM) gains nothing from panels: a 40-row front 40 us, a 160-row
// one 509.
template <typename T>
__device__ __forceinline__ void front_lu_columns(T* f, int ld, int F, int ns, const SymDev& sd, int s, int k, int K,
                                                 int32_t* status, int32_t* badcol) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const int c0 = sd.c0[s];
  for (int p = 0; p < ns; ++p) {
    T* lc = f + p * ld;
    const T piv = lc[p];
    if (tid == 0) check_pivot(piv, sd, s, k, K, c0 + p, status, badcol);
    const T rp = T(1) / piv;
    for (int i = p + 1 + tid; i < F; i += nt) lc[i] *= rp;
    __syncthreads();
    for (int j = p + 1 + wid; j < F; j += nw) {
      T* col = f + j * ld;
      const T u = col[p];
      for (int i = p + 1 + lane; i < F; i += 32) col[i] -= lc[i] * u;
    }
    __syncthreads();
  }
}

// The same with the trailing elements dealt out to the threads one by one, where
// three CTAs share an SM's FP64 pipe and every idle lane of an instruction costs as
// much as a busy one: one barrier a pivot: warp 0 takes the next pivot's column
// first, inverts the pivot and scales the column while the other warps update the
// rest (48 grids 1983 us, 2015 by columns).  A CTA by itself is slower this way (a
// 40-row front 46 us against 40, a 160-row one 540 against 509).
template <typename T>
__device__ __forceinline__ void front_lu_flat(T* f, int ld, int F, int ns, const SymDev& sd, int s, int k, int K,
                                              int32_t* status, int32_t* badcol) {
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const int c0 = sd.c0[s];
  for (int p = -1; p < ns; ++p) {
    // column p is scaled; eliminate it from columns p+1 .. F-1, and prepare column p+1
    const T* lc = f + p * ld;
    if (tid < 32) {
      if (p + 1 < ns) {
        T* col = f + (p + 1) * ld;
        const T u = p >= 0 ? col[p] : T(0);
        T piv = col[p + 1];
        if (p >= 0) piv -= lc[p + 1] * u;
        if (lane == 0) check_pivot(piv, sd, s, k, K, c0 + p + 1, status, badcol);
        const T rp = T(1) / piv;
        __syncwarp();
        for (int i = p + 1 + lane; i < F; i += 32) {
          T x = col[i];
          if (p >= 0) x -= lc[i] * u;
          col[i] = i == p + 1 ? x : x * rp;
        }
      }
    }
    if (p >= 0 && p + 1 < F) {
      const int m = F - p - 1, j0 = p + 1 < ns ? p + 2 : p + 1;  // rows p+1.., columns j0..
      const int total = m * (F - j0);
      // warp 0 comes last, after its column
      const int first = nt > 32 ? (tid + nt - 32) % nt : tid;
      const int qs = nt / m, rs = nt - qs * m;
      int c = first / m, r = first - c * m;
      const T* lp = lc + p + 1;
      const T* up = f + p + j0 * ld;
      T* xp = f + p + 1 + j0 * ld;
      for (int e = first; e < total; e += 4 * nt) {
        int at[4];
        T x[4], l[4], u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const bool in = e + q * nt < total;
          at[q] = in ? r + c * ld : -1;
          if (in) {
            l[q] = lp[r];
            u[q] = up[c * ld];
            x[q] = xp[at[q]];
          }
          r += rs;
          c += qs;
          if (r >= m) {
            r -= m;
            ++c;
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (at[q] >= 0) xp[at[q]] = x[q] - l[q] * u[q];
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Fronts in shared memory, one CTA (256 threads, or a multiple) per (front, k):
// assembly (original entries, t_k D, the children's Schur complements), pivot-
// free LU, write to the front storage.  f: F x front_ld(F) values.
// ---------------------------------------------------------------------------
template <typename T, bool FLAT>
__device__ __forceinline__ void front_cta(const SymDev& sd, int s, int k, const double* __restrict__ vals,
                                          const double* __restrict__ D, const Shifts& sh,
                                          T* __restrict__ fronts, int32_t* status, int32_t* badcol, T* f, T* rinv) {
  const int K = sh.K;
  const int ns = sd.ns[s], ms = sd.ms[s], F = ns + ms, ld = front_ld(F);
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  for (int q = tid; q < F * ld; q += nt) f[q] = T(0);
  __syncthreads();
  // entries of A owned by this front (duplicates add up)
  const int64_t a0 = sd.amap_off[s], a1 = sd.amap_off[s + 1];
  add_entries<T>(sd, vals, a0, a1, [&](int d, T v) { atomicAdd(&f[d + d / F * (ld - F)], v); });
  // the perturbation t_k D on the pivot diagonal
  const double tk = sh.t[k];
  const int c0 = sd.c0[s];
  for (int c = tid; c < ns; c += nt) atomicAdd(&f[c * (ld + 1)], (T)(tk * D[sd.perm[c0 + c]]));
  __syncthreads();
  // extend-add, every warp its share of the columns
  extend_add_flat<T>(sd, s, k, K, fronts, f, ld, (int)((int64_t)F * wid / nw), (int)((int64_t)F * (wid + 1) / nw), 0, F);
  __syncthreads();
  if constexpr (sizeof(T) == 8 && FLAT) front_lu_flat<T>(f, ld, F, ns, sd, s, k, K, status, badcol);
  else if constexpr (sizeof(T) == 8) front_lu_columns<T>(f, ld, F, ns, sd, s, k, K, status, badcol);
  else front_lu<T>(f, ld, F, ns, rinv, sd, s, k, K, status, badcol);
  T* out = fronts + (int64_t)K * sd.front_off[s] + (int64_t)k * F * F;
  for (int j = wid; j < F; j += nw)
    for (int i = lane; i < F; i += 32) out[i + (int64_t)j * F] = f[i + j * ld];
}

template <typename T>
__global__ void __launch_bounds__(512) k_front_small(SymDev sd, const int32_t* __restrict__ list,
                                                     const double* __restrict__ vals, const double* __restrict__ D,
                                                     Shifts sh, T* __restrict__ fronts, int32_t* status,
                                                     int32_t* badcol) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ T rinv[16];
  front_cta<T, false>(sd, list[blockIdx.x], blockIdx.y, vals, D, sh, fronts, status, badcol,
               reinterpret_cast<T*>(smraw), rinv);
}

// ---------------------------------------------------------------------------
// Fronts of at most 32 rows: SEG lanes (8, 16 or 32) per (front, k), lane =
// row, the front in the segment's SEG x SEG shared-memory area f.  A child's
// update block is added a column at a time, four in flight: the child's rows
// land on the rows of a 32-bit mask, so lane i reads child row popcount(mask
// below i), and the columns are the mask's bits in turn.  The elimination takes
// four columns at a time too, all reads before the writes.  Loops are short and
// rolled, and run to warp-uniform bounds; all lanes of a warp call together.
// (The same in registers, unrolled to static indices, is 1500 instructions that
// a level runs once per SM: fetching them doubled the factorisation of the 118-
// bus grid.)
// ---------------------------------------------------------------------------
template <typename T, int SEG>
__device__ __forceinline__ void front_seg(const SymDev& sd, int s, int k, bool on, int sl,
                                          const double* __restrict__ vals, const double* __restrict__ D,
                                          const Shifts& sh, T* __restrict__ fronts, int32_t* status,
                                          int32_t* badcol, T* f) {
  const int K = sh.K;
  int ns = 0, F = 0, c0 = 0, cb = 0, ce = 0;
  int64_t a0 = 0, a1 = 0, fo = 0;
  if (on) {
    ns = sd.ns[s];
    F = ns + sd.ms[s];
    c0 = sd.c0[s];
    a0 = sd.amap_off[s];
    a1 = sd.amap_off[s + 1];
    cb = sd.child_off[s];
    ce = sd.child_off[s + 1];
    fo = sd.front_off[s];
  }
  const int Fw = __reduce_max_sync(0xffffffffu, F), nsw = __reduce_max_sync(0xffffffffu, ns);
  for (int j = 0; j < Fw; ++j) f[sl + j * SEG] = T(0);
  __syncwarp();
  for (int64_t q = a0 + sl; q < a1; q += SEG) {
    const int d = sd.amap_dst[q];
    atomicAdd(&f[d + d / F * (SEG - F)], (T)vals[sd.amap_src[q]]);
  }
  if (sl < ns) atomicAdd(&f[sl * (SEG + 1)], (T)(sh.t[k] * D[sd.perm[c0 + sl]]));
  __syncwarp();
  // children, SEG records at a time, one a lane
  const int most = __reduce_max_sync(0xffffffffu, ce - cb);
  for (int b = 0; b < most; b += SEG) {
    int64_t cfo = 0;
    int cns = 0, cF = 0;
    unsigned cm = 0;
    if (cb + b + sl < ce) {
      const ChildDesc cd = sd.cdesc[cb + b + sl];
      cfo = cd.fo;
      cns = cd.ns;
      cF = cd.F;
      cm = cd.mask;
    }
    const int nc = min(SEG, most - b);
    for (int c = 0; c < nc; ++c) {
      unsigned mask = __shfl_sync(0xffffffffu, cm, c, SEG);
      const int eF = __shfl_sync(0xffffffffu, cF, c, SEG), ens = __shfl_sync(0xffffffffu, cns, c, SEG);
      const int64_t efo = __shfl_sync(0xffffffffu, cfo, c, SEG);
      const bool mine = (mask >> sl) & 1u;
      const T* p = fronts + (int64_t)K * efo + (int64_t)k * eF * eF + ens + __popc(mask & ((1u << sl) - 1u)) +
                   (int64_t)ens * eF;
      const int cols = __reduce_max_sync(0xffffffffu, __popc(mask));
      for (int e = 0; e < cols; e += 4) {
        int j[4];
        T v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          j[q] = mine && mask ? __ffs(mask) - 1 : -1;
          mask &= mask - 1;
          v[q] = j[q] >= 0 ? __ldcg(p) : T(0);
          p += eF;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (j[q] >= 0) f[sl + j[q] * SEG] += v[q];
      }
    }
  }
  __syncwarp();
  for (int p = 0; p < nsw; ++p) {
    const bool act = p < ns;
    const T piv = act ? f[p * (SEG + 1)] : T(1);
    if (act && sl == 0) check_pivot(piv, sd, s, k, K, c0 + p, status, badcol);
    const T rp = T(1) / piv;
    const bool below = act && sl > p && sl < F;
    const T l = below ? f[sl + p * SEG] * rp : T(0);
    if (below) f[sl + p * SEG] = l;
    for (int j = p + 1; j < Fw; j += 4) {
      T u[4], x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const bool in = below && j + q < F;
        u[q] = in ? f[p + (j + q) * SEG] : T(0);
        x[q] = in ? f[sl + (j + q) * SEG] : T(0);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (below && j + q < F) f[sl + (j + q) * SEG] = x[q] - l * u[q];
    }
    __syncwarp();
  }
  T* out = fronts + (int64_t)K * fo + (int64_t)k * F * F + sl;
  for (int j = 0; j < Fw; ++j)
    if (j < F && sl < F) out[j * F] = f[sl + j * SEG];
}

template <int SEG>
__global__ void __launch_bounds__(256) k_front_seg(SymDev sd, const int32_t* __restrict__ list, int ntasks,
                                                   const double* __restrict__ vals, const double* __restrict__ D,
                                                   Shifts sh, float* __restrict__ fronts, int32_t* status,
                                                   int32_t* badcol) {
  __shared__ float area[256 * SEG];
  const int q = (int)((blockIdx.x * 256 + threadIdx.x) / SEG);
  const bool on = q < ntasks;
  const int s = on ? list[q / sh.K] : 0, k = on ? q % sh.K : 0;
  front_seg<float, SEG>(sd, s, k, on, threadIdx.x % SEG, vals, D, sh, fronts, status, badcol,
                        area + threadIdx.x / SEG * SEG * SEG);
}

// ---------------------------------------------------------------------------
// Big fronts, step 1: assembly, one CTA per (column tile, front, k).  Each
// CTA owns TW columns, so children are added in a fixed order: the result is
// deterministic.
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t lower_bound_col(const int32_t* dst, int64_t lo, int64_t hi,
                                                   int F, int j) {
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (dst[mid] / F < j) lo = mid + 1; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ int lower_bound_i(const int32_t* a, int n, int x) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

template <typename T>
__global__ void __launch_bounds__(256) k_assemble_big(SymDev sd, const int32_t* __restrict__ list,
                                                      const double* __restrict__ vals,
                                                      const double* __restrict__ D, Shifts sh,
                                                      T* __restrict__ fronts, int TW) {
  const int s = list[blockIdx.y];
  const int k = blockIdx.z;
  const int K = sh.K;
  const int ns = sd.ns[s], ms = sd.ms[s], F = ns + ms;
  const int j0 = blockIdx.x * TW;
  if (j0 >= F) return;
  const int j1 = min(F, j0 + TW);
  const int tid = threadIdx.x, nt = blockDim.x;
  T* f = fronts + (int64_t)K * sd.front_off[s] + (int64_t)k * F * F;
  const int64_t nz = (int64_t)F * (j1 - j0);
  for (int64_t q = tid; q < nz; q += nt) f[(int64_t)j0 * F + q] = T(0);
  __syncthreads();
  const int64_t a0 = sd.amap_off[s], a1 = sd.amap_off[s + 1];
  const int64_t lo = lower_bound_col(sd.amap_dst, a0, a1, F, j0);
  const int64_t hi = lower_bound_col(sd.amap_dst, lo, a1, F, j1);
  for (int64_t q = lo + tid; q < hi; q += nt) atomicAdd(&f[sd.amap_dst[q]], (T)vals[sd.amap_src[q]]);
  const double tk = sh.t[k];
  const int c0 = sd.c0[s];
  for (int c = j0 + tid; c < min(j1, ns); c += nt)
    atomicAdd(&f[(int64_t)c * (F + 1)], (T)(tk * D[sd.perm[c0 + c]]));
  __syncthreads();
  for (int ci = sd.child_off[s]; ci < sd.child_off[s + 1]; ++ci) {
    const int c = sd.child[ci];
    const int cns = sd.ns[c], cms = sd.ms[c], cF = cns + cms;
    const int32_t* em = sd.emap + sd.row_off[c];
    const int b0 = lower_bound_i(em, cms, j0);
    const int b1 = lower_bound_i(em, cms, j1);
    if (b1 > b0) {
      const T* cf = fronts + (int64_t)K * sd.front_off[c] + (int64_t)k * cF * cF;
      const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
      for (int b = b0 + wid; b < b1; b += nw) {
        T* dcol = f + (int64_t)em[b] * F;
        const T* scol = cf + (int64_t)(cns + b) * cF + cns;
        for (int a = lane; a < cms; a += 32) dcol[em[a]] += scol[a];
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Big fronts, step 2: factor the panel of columns [p0, p0+NB) (rows p0..F-1)
// in shared memory, then solve the row block U[p0:p0+NB, p0+NB:F] with the
// panel's unit lower triangle.  One CTA per (front, k).
// ---------------------------------------------------------------------------
template <typename T, int NB>
__global__ void __launch_bounds__(512) k_panel_big(SymDev sd, const int32_t* __restrict__ list,
                                                   int K, T* __restrict__ fronts, int p0,
                                                   int32_t* status, int32_t* badcol) {
  extern __shared__ __align__(16) unsigned char smraw[];
  T* P = reinterpret_cast<T*>(smraw);
  const int s = list[blockIdx.x];
  const int k = blockIdx.y;
  const int ns = sd.ns[s], F = ns + sd.ms[s];
  if (p0 >= ns) return;
  const int nbe = min(NB, ns - p0);
  const int Mr = F - p0;
  const int ld = Mr | 1;
  const int tid = threadIdx.x, nt = blockDim.x;
  T* f = fronts + (int64_t)K * sd.front_off[s] + (int64_t)k * F * F;
  const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  for (int c = wid; c < nbe; c += nw)
    for (int i = lane; i < Mr; i += 32) P[i + c * ld] = f[(p0 + i) + (int64_t)(p0 + c) * F];
  __syncthreads();
  panel_eliminate<T>(P, ld, Mr, nbe, sd, s, k, K, sd.c0[s] + p0, status, badcol);
  for (int c = wid; c < nbe; c += nw)
    for (int i = lane; i < Mr; i += 32) f[(p0 + i) + (int64_t)(p0 + c) * F] = P[i + c * ld];
  // row block of U: columns j >= p0 + nbe
  for (int j = p0 + nbe + tid; j < F; j += nt) {
    T* col = f + (int64_t)j * F + p0;
    T u[NB];
#pragma unroll
    for (int q = 0; q < NB; ++q) u[q] = (q < nbe) ? col[q] : T(0);
#pragma unroll
    for (int q = 1; q < NB; ++q) {
      T a = u[q];
#pragma unroll
      for (int r = 0; r < NB - 1; ++r)
        if (r < q) a -= P[q + r * ld] * u[r];
      u[q] = a;
    }
#pragma unroll
    for (int q = 0; q < NB; ++q)
      if (q < nbe) col[q] = u[q];
  }
}

// ---------------------------------------------------------------------------
// Big fronts, step 3: trailing update C -= L_panel * U_panel on 64x64 tiles.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_update_big(SymDev sd, const int32_t* __restrict__ list,
                                                    int K, T* __restrict__ fronts, int p0,
                                                    int nb) {
  const int s = list[blockIdx.y];
  const int k = blockIdx.z;
  const int ns = sd.ns[s], F = ns + sd.ms[s];
  if (p0 >= ns) return;
  const int nbe = min(nb, ns - p0);
  const int t0 = p0 + nbe;
  const int m = F - t0;
  if (m <= 0) return;
  const int tpd = (m + 63) / 64;
  if ((int)blockIdx.x >= tpd * tpd) return;
  const int i0 = t0 + (blockIdx.x % tpd) * 64;
  const int j0 = t0 + (blockIdx.x / tpd) * 64;
  T* f = fronts + (int64_t)K * sd.front_off[s] + (int64_t)k * F * F;
  __shared__ T As[32][64];
  __shared__ T Bs[32][65];
  const int tid = threadIdx.x;
  for (int e = tid; e < 64 * 32; e += 256) {
    const int r = e % 64, q = e / 64;
    As[q][r] = (q < nbe && i0 + r < F) ? f[(i0 + r) + (int64_t)(p0 + q) * F] : T(0);
  }
  for (int e = tid; e < 64 * 32; e += 256) {
    const int q = e % 32, c = e / 32;
    Bs[q][c] = (q < nbe && j0 + c < F) ? f[(p0 + q) + (int64_t)(j0 + c) * F] : T(0);
  }
  __syncthreads();
  const int tx = tid % 16, ty = tid / 16;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
  for (int q = 0; q < nbe; ++q) {
    T a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = As[q][tx + 16 * i];
#pragma unroll
    for (int j = 0; j < 4; ++j) b[j] = Bs[q][ty + 16 * j];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] += a[i] * b[j];
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = i0 + tx + 16 * i, c = j0 + ty + 16 * j;
      if (r < F && c < F) f[r + (int64_t)c * F] -= acc[i][j];
    }
}

// ---------------------------------------------------------------------------
// Mid-size fronts: one thread-block cluster of C CTAs per (front, k).  The
// front's columns are dealt out to the CTAs in widths cw (a multiple of 32)
// and live in their shared memory for the whole factorisation.  For each
// panel of 32 pivots the owning CTA factors it locally, one cluster barrier
// publishes it, and every CTA copies the panel over distributed shared
// memory, solves its part of the U row block and applies a register-tiled
// update to its columns.  Only the owner's panel columns are ever read
// remotely and they are not written after being factored, so one barrier per
// panel suffices; a final barrier keeps every CTA resident until the last
// remote read is done.
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ int cluster_cw(int F, int C) {
  return (((F + C - 1) / C) + 31) / 32 * 32;
}

template <typename T>
__host__ __device__ __forceinline__ size_t cluster_smem(int F, int C) {
  const size_t cw = (size_t)cluster_cw(F, C);
  return ((size_t)F * cw + (C > 1 ? (size_t)F * 32 : 0) + 32 * 33) * sizeof(T);
}

template <typename T>
__global__ void __launch_bounds__(256) k_front_cluster(SymDev sd, const int32_t* __restrict__ list,
                                                       int C, const double* __restrict__ vals,
                                                       const double* __restrict__ D, Shifts sh,
                                                       T* __restrict__ fronts, int32_t* status,
                                                       int32_t* badcol) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char smraw[];
  const int rank = (int)cl.block_rank();
  const int s = list[blockIdx.x / C];
  const int k = blockIdx.y;
  const int K = sh.K;
  const int ns = sd.ns[s], ms = sd.ms[s], F = ns + ms;
  const int cw = cluster_cw(F, C);
  const int j0 = min(F, rank * cw), j1 = min(F, j0 + cw);
  const int nc = j1 - j0;
  T* M = reinterpret_cast<T*>(smraw);                  // my columns, F x cw, ld F
  T* Lp = M + (size_t)F * cw;                           // copy of a remote panel
  T* L11 = Lp + (C > 1 ? (size_t)F * 32 : 0);           // 32 x 33 unit-lower block
  __shared__ T prow[2][32];
  const int tid = threadIdx.x, nt = blockDim.x;
  const int c0 = sd.c0[s];
  // 1. assembly of my columns
  for (int q = tid; q < F * nc; q += nt) M[q] = T(0);
  __syncthreads();
  if (nc > 0) {
    const int64_t a0 = sd.amap_off[s], a1 = sd.amap_off[s + 1];
    const int64_t lo = lower_bound_col(sd.amap_dst, a0, a1, F, j0);
    const int64_t hi = lower_bound_col(sd.amap_dst, lo, a1, F, j1);
    for (int64_t q = lo + tid; q < hi; q += nt)
      atomicAdd(&M[sd.amap_dst[q] - j0 * F], (T)vals[sd.amap_src[q]]);
    const double tk = sh.t[k];
    for (int c = j0 + tid; c < min(j1, ns); c += nt)
      atomicAdd(&M[c + (c - j0) * F], (T)(tk * D[sd.perm[c0 + c]]));
  }
  __syncthreads();
  for (int ci = sd.child_off[s]; ci < sd.child_off[s + 1]; ++ci) {
    const int c = sd.child[ci];
    const int cns = sd.ns[c], cms = sd.ms[c], cF = cns + cms;
    const int32_t* em = sd.emap + sd.row_off[c];
    const int b0 = lower_bound_i(em, cms, j0);
    const int b1 = lower_bound_i(em, cms, j1);
    if (b1 > b0) {
      const T* cf = fronts + (int64_t)K * sd.front_off[c] + (int64_t)k * cF * cF;
      const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
      for (int b = b0 + wid; b < b1; b += nw) {
        T* dcol = M + (size_t)(em[b] - j0) * F;
        const T* scol = cf + (int64_t)(cns + b) * cF + cns;
        for (int a = lane; a < cms; a += 32) dcol[em[a]] += scol[a];
      }
    }
    __syncthreads();
  }
  // 2. blocked right-looking elimination, 32 pivots per panel
  const int tx = tid & 15, ty = tid >> 4;
  for (int p0 = 0; p0 < ns; p0 += 32) {
    const int nb = min(32, ns - p0);
    const int owner = p0 / cw;
    if (rank == owner) panel_factor_rows<T>(M + (size_t)(p0 - j0) * F, F, F, p0, nb, prow, sd, s, k,
                                            K, c0 + p0, status, badcol);
    cl.sync();
    const int jlo = max(j0, p0 + nb);
    if (jlo < j1) {
      const T* Ls;                                       // Ls[i + c*F] = front(i, p0 + c)
      if (rank == owner) {
        Ls = M + (size_t)(p0 - j0) * F;
      } else {
        const T* R = cl.map_shared_rank(M, owner) + (size_t)(p0 - owner * cw) * F;
        const int hr = F - p0;
        for (int e = tid; e < hr * nb; e += nt) {
          const int i = p0 + e % hr, c = e / hr;
          Lp[i + c * F] = R[i + c * F];
        }
        Ls = Lp;
      }
      __syncthreads();
      for (int e = tid; e < 32 * 32; e += nt) {
        const int r = e >> 5, c = e & 31;
        L11[r * 33 + c] = (r < nb && c < r) ? Ls[(p0 + r) + c * F] : T(0);
      }
      __syncthreads();
      // (a) U row block of my columns: unit-lower triangular solve, one column per thread
      for (int j = jlo + tid; j < j1; j += nt) {
        T* col = M + (size_t)(j - j0) * F + p0;
        T u[32];
#pragma unroll
        for (int r = 0; r < 32; ++r) u[r] = (r < nb) ? col[r] : T(0);
#pragma unroll
        for (int r = 1; r < 32; ++r) {
          T a = u[r];
#pragma unroll
          for (int c = 0; c < 31; ++c)
            if (c < r) a -= L11[r * 33 + c] * u[c];
          u[r] = a;
        }
#pragma unroll
        for (int r = 0; r < 32; ++r)
          if (r < nb) col[r] = u[r];
      }
      __syncthreads();
      // (b) trailing update of my columns, 64 x 64 tiles, 4 x 4 per thread
      const int r0 = p0 + nb;
      for (int rb = r0; rb < F; rb += 64) {
        for (int cb = jlo; cb < j1; cb += 64) {
          T acc[4][4];
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
          for (int c = 0; c < nb; ++c) {
            T av[4], bv[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
              const int i = rb + tx + 16 * a;
              av[a] = (i < F) ? Ls[i + c * F] : T(0);
            }
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const int j = cb + ty + 16 * b;
              bv[b] = (j < j1) ? M[(p0 + c) + (size_t)(j - j0) * F] : T(0);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
              for (int b = 0; b < 4; ++b) acc[a][b] += av[a] * bv[b];
          }
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const int i = rb + tx + 16 * a, j = cb + ty + 16 * b;
              if (i < F && j < j1) M[i + (size_t)(j - j0) * F] -= acc[a][b];
            }
        }
      }
      __syncthreads();
    }
  }
  cl.sync();
  T* out = fronts + (int64_t)K * sd.front_off[s] + (int64_t)k * F * F + (int64_t)j0 * F;
  for (int e = tid; e < F * nc; e += nt) out[e] = M[e];
}

// ---------------------------------------------------------------------------
// Big fronts as a tile DAG, one persistent launch per level.  Column blocks
// are 32 wide.  Tasks: ASM(j) assembles block j; PANEL(p) factors the panel
// of pivots [32p, 32p+32) in shared memory; UPDATE(p, j) applies panel p to
// block j (unit-lower solve of its 32 U rows, then the trailing update of all
// rows below).  PANEL(p+1) waits only for UPDATE(p, p+1), so the next panel
// starts while the rest of step p is still updating (look-ahead).  CTAs take
// tasks in ticket order and wait only for tasks with smaller tickets; every
// wait is bounded and sets *err when it gives up.
// ---------------------------------------------------------------------------
constexpr int64_t kDagWaitPolls = kWaitPolls;

__device__ __forceinline__ int dag_ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void dag_st_release(int* p, int v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ void dag_wait(const int* f, int need, int* err) {
  if (dag_ld_acquire(f) >= need) return;
  for (int64_t i = 0; i < kDagWaitPolls; ++i) {
    __nanosleep(64);
    if (dag_ld_acquire(f) >= need) return;
  }
  atomicExch(err, 1);
}

template <typename T>
__global__ void __launch_bounds__(256) k_big_dag(SymDev sd, const int32_t* __restrict__ big,
                                                 const DagTask* __restrict__ tasks, int ntasks,
                                                 int* ticket, int* flags, int* err,
                                                 const double* __restrict__ vals,
                                                 const double* __restrict__ D, Shifts sh,
                                                 T* __restrict__ fronts, int32_t* status,
                                                 int32_t* badcol) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_t;
  const int K = sh.K;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5;
  for (;;) {
    if (tid == 0) s_t = atomicAdd(ticket, 1);
    __syncthreads();
    const int u = s_t;
    __syncthreads();
    if (u >= ntasks) return;
    const DagTask t = tasks[u];
    const int s = big[t.b];
    const int k = t.k;
    const int ns = sd.ns[s], F = ns + sd.ms[s];
    const int J = (F + 31) / 32;
    int* stepdone = flags + t.flags;
    int* paneldone = stepdone + J;
    T* f = fronts + (int64_t)K * sd.front_off[s] + (int64_t)k * F * F;
    int publish_at = -1, publish_val = 0;
    if (t.kind == kDagAsm) {
      const int j0 = 32 * t.j, j1 = min(F, j0 + 32);
      const int64_t nz = (int64_t)F * (j1 - j0);
      for (int64_t q = tid; q < nz; q += nt) f[(int64_t)j0 * F + q] = T(0);
      __syncthreads();
      const int64_t a0 = sd.amap_off[s], a1 = sd.amap_off[s + 1];
      const int64_t lo = lower_bound_col(sd.amap_dst, a0, a1, F, j0);
      const int64_t hi = lower_bound_col(sd.amap_dst, lo, a1, F, j1);
      for (int64_t q = lo + tid; q < hi; q += nt) atomicAdd(&f[sd.amap_dst[q]], (T)vals[sd.amap_src[q]]);
      const double tk = sh.t[k];
      const int c0 = sd.c0[s];
      for (int c = j0 + tid; c < min(j1, ns); c += nt)
        atomicAdd(&f[(int64_t)c * (F + 1)], (T)(tk * D[sd.perm[c0 + c]]));
      __syncthreads();
      for (int ci = sd.child_off[s]; ci < sd.child_off[s + 1]; ++ci) {
        const int c = sd.child[ci];
        const int cns = sd.ns[c], cms = sd.ms[c], cF = cns + cms;
        const int32_t* em = sd.emap + sd.row_off[c];
        const int b0 = lower_bound_i(em, cms, j0);
        const int b1 = lower_bound_i(em, cms, j1);
        if (b1 > b0) {
          const T* cf = fronts + (int64_t)K * sd.front_off[c] + (int64_t)k * cF * cF;
          for (int b = b0 + wid; b < b1; b += (nt >> 5)) {
            T* dcol = f + (int64_t)em[b] * F;
            const T* scol = cf + (int64_t)(cns + b) * cF + cns;
            for (int a = lane; a < cms; a += 32) dcol[em[a]] += scol[a];
          }
        }
        __syncthreads();
      }
      publish_at = t.j;
      publish_val = 1;
    } else if (t.kind == kDagPanel) {
      if (tid == 0) dag_wait(&stepdone[t.p], t.p + 1, err);
      __syncthreads();
      T* P = reinterpret_cast<T*>(smraw);
      const int r0 = 32 * t.p;
      const int nb = min(32, ns - r0);
      const int Mr = F - r0;
      const int ld = Mr | 1;
      for (int c = wid; c < nb; c += (nt >> 5))
        for (int i = lane; i < Mr; i += 32) P[i + c * ld] = __ldcg(f + (r0 + i) + (int64_t)(r0 + c) * F);
      __syncthreads();
      panel_eliminate<T>(P, ld, Mr, nb, sd, s, k, K, sd.c0[s] + r0, status, badcol);
      for (int c = wid; c < nb; c += (nt >> 5))
        for (int i = lane; i < Mr; i += 32) f[(r0 + i) + (int64_t)(r0 + c) * F] = P[i + c * ld];
      publish_at = J + t.p;
      publish_val = 1;
    } else {
      const int p = t.p, j = t.j;
      const int r0 = 32 * p;
      const int nb = min(32, ns - r0);
      const int jc0 = max(32 * j, r0 + nb), jc1 = min(32 * j + 32, F);
      const int w = jc1 - jc0;
      if (tid == 0) {
        dag_wait(&paneldone[p], 1, err);
        dag_wait(&stepdone[j], p + 1, err);
      }
      __syncthreads();
      T* Ls = reinterpret_cast<T*>(smraw);       // 32 x 33: unit-lower L11 of panel p
      T* Us = Ls + 32 * 33;                       // 32 x 33: U rows of this block
      for (int e = tid; e < 32 * 32; e += nt) {
        const int r = e & 31, c = e >> 5;
        Ls[r * 33 + c] = (r < nb && c < r) ? __ldcg(f + (r0 + r) + (int64_t)(r0 + c) * F) : T(0);
        Us[r * 33 + c] = (r < nb && c < w) ? __ldcg(f + (r0 + r) + (int64_t)(jc0 + c) * F) : T(0);
      }
      __syncthreads();
      if (wid == 0) {
        T uu[32];
#pragma unroll
        for (int r = 0; r < 32; ++r) uu[r] = Us[r * 33 + lane];
#pragma unroll
        for (int r = 1; r < 32; ++r) {
          T a = uu[r];
#pragma unroll
          for (int c = 0; c < 31; ++c)
            if (c < r) a -= Ls[r * 33 + c] * uu[c];
          uu[r] = a;
        }
#pragma unroll
        for (int r = 0; r < 32; ++r) {
          Us[r * 33 + lane] = uu[r];
          if (r < nb && lane < w) f[(r0 + r) + (int64_t)(jc0 + lane) * F] = uu[r];
        }
      }
      __syncthreads();
      for (int i = r0 + nb + tid; i < F; i += nt) {
        T l[32], cv[32];
#pragma unroll
        for (int c = 0; c < 32; ++c) l[c] = (c < nb) ? __ldcg(f + i + (int64_t)(r0 + c) * F) : T(0);
#pragma unroll
        for (int col = 0; col < 32; ++col) cv[col] = (col < w) ? __ldcg(f + i + (int64_t)(jc0 + col) * F) : T(0);
#pragma unroll
        for (int col = 0; col < 32; ++col) {
          T a = T(0);
#pragma unroll
          for (int c = 0; c < 32; ++c) a += l[c] * Us[c * 33 + col];
          cv[col] -= a;
        }
#pragma unroll
        for (int col = 0; col < 32; ++col)
          if (col < w) f[i + (int64_t)(jc0 + col) * F] = cv[col];
      }
      publish_at = j;
      publish_val = p + 2;
    }
    __threadfence();
    __syncthreads();
    if (tid == 0 && publish_at >= 0) dag_st_release(&stepdone[publish_at], publish_val);
  }
}

template <typename T>
int big_dag_impl(const SymDev& sd, const LevelPlan& lp, const int32_t* d_big, const DagTask* tasks,
                 int* ticket, int* flags, int* err, const double* vals, const double* D,
                 const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol, cudaStream_t st) {
  if (lp.dag_tasks == 0) return 0;
  static std::atomic<int> nsm_dev[kMaxDevices];
  const int dev = current_device();
  int nsm = nsm_dev[dev].load(std::memory_order_acquire);
  if (!nsm) {
    cudaFuncSetAttribute(k_big_dag<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    nsm_dev[dev].store(nsm, std::memory_order_release);
  }
  const size_t smem = std::max((size_t)(lp.big_maxF + 1) * 32, (size_t)2 * 32 * 33) * sizeof(T);
  int occ = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_big_dag<T>, 256, smem);
  const int grid = std::max(1, std::min(lp.dag_tasks, std::max(1, occ) * std::max(nsm, 1)));
  k_big_dag<T><<<grid, 256, smem, st>>>(sd, d_big + lp.big_off, tasks + lp.dag_task_off, lp.dag_tasks,
                                        ticket, flags, err, vals, D, sh, (T*)fronts, status, badcol);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

// ---------------------------------------------------------------------------
// Big fronts, owner tiles: one persistent launch per level.  A task is a
// tile: the 32-column block j of one (front, k) restricted to a chunk of CH
// rows (CH a multiple of 32; a whole column when CH >= F).  The CTA that takes
// it keeps the tile in shared memory from assembly to its final value:
//   1. assembly of the tile: the original entries (per-column ranges of the
//      assembly map), t_k D on the diagonal, and the children's update
//      columns through the inverse extend-add map.  Each destination column
//      belongs to one warp, which adds its contributions in child order, so
//      the sums are deterministic with no barrier between children;
//   2. every earlier panel p, in pivot order (left-looking form of the
//      static-pivot elimination of Sec. II-C): the tile holding panel p's
//      pivot rows waits for L11(p), solves the block's U rows and releases
//      them for the chunks below; every tile below the pivot rows waits for
//      those U rows and for its own chunk's rows of L21(p), then subtracts
//      L21(p) U(p, j) from its rows;
//   3. if the block holds pivots: the tile holding the diagonal block factors
//      it in shared memory, eliminates its rows below
//      it and releases them; the tiles of the chunks below wait for that,
//      then eliminate their rows with the released U rows and reciprocal
//      pivots.  Tiles are written to the front storage before their release
//      flags (st.release.gpu) are set.
// The same per-element sequence of multiply-adds as panel_eliminate is used
// for the panel, so the pivot block and L21 match the per-panel path.
// Tasks are taken in ticket order from a list sorted by (block, chunk):
// every wait is on a tile earlier in that order, already held by a running
// CTA, so the schedule cannot deadlock whatever the residency, and every wait
// is bounded.
// ---------------------------------------------------------------------------
constexpr int kOwnThreads = 256;
constexpr unsigned kOwnFull = 0xffffffffu;

// U rows r0..r0+nb-1 of the block, solved with the unit lower L11 in Ls
// (row-major, ld 33): warp g takes columns [4g, 4g+4), lane r holds row r and
// receives row q's final values by shuffle.  The loop body is small so one
// warp's instruction stream stays cached.  Us gets the U rows row-major (32
// per row, zero beyond w and nb) for the update.  Needs 8 warps.
template <typename T>
__device__ __forceinline__ void own_trsm(T* Bk, int ld, int r0, int nb, int w, const T* Ls, T* Us) {
  const int lane = threadIdx.x & 31, cb = (threadIdx.x >> 5) * 4;
  T x[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = (lane < nb && cb + i < w) ? Bk[r0 + lane + (cb + i) * ld] : T(0);
  for (int q = 0; q + 1 < nb; ++q) {
    T u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = __shfl_sync(kOwnFull, x[i], q);
    if (lane > q) {
      const T l = Ls[lane * 33 + q];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] -= l * u[i];
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const bool in = lane < nb && cb + i < w;
    if (in) Bk[r0 + lane + (cb + i) * ld] = x[i];
    Us[lane * 32 + cb + i] = in ? x[i] : T(0);
  }
}

// rows [i0, i1) of an FP64 tile: x(i, :) -= L(i, r0..r0+nb-1) U, L from the front
// storage, U from Us; lane = row, four columns a warp.
// A warp has a quarter of the SM's FP64 pipe at most, so all eight take part (two
// warps of 16 columns took 18 us a panel).
__device__ __forceinline__ void own_update_few64(double* Bt, int ld, int R0, const double* f, int F, int r0, int nb,
                                                 const double* Us, int i0, int i1, int w) {
  const int cb = 4 * (threadIdx.x >> 5);
  if (cb >= w) return;
  for (int i = i0 + (threadIdx.x & 31); i < i1; i += 32) {
    double l[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) l[c] = c < nb ? __ldcg(f + i + (int64_t)(r0 + c) * F) : 0.0;
    double* row = Bt + (i - R0) + cb * ld;
    double x[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) x[c] = row[c * ld];
#pragma unroll
    for (int c = 0; c < 32; ++c)
      if (c < nb) {
#pragma unroll
        for (int g = 0; g < 4; ++g) x[g] -= l[c] * Us[c * 32 + cb + g];
      }
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (cb + c < w) row[c * ld] = x[c];
  }
}

// own_eliminate_rows in FP64: the whole CTA takes one pivot column at a time, the
// elements dealt out one by one (a row a thread, 32 rows were one warp's work, a
// quarter of the pipe: 19 us)
__device__ __forceinline__ void own_eliminate_flat(double* Bt, int ld, int R0, int i0, int i1, int np, int w,
                                                   const double* Us, const double* rinv) {
  const int m = i1 - i0;
  if (m <= 0) return;
  double* t = Bt + (i0 - R0);
  for (int c = -1; c < np; ++c) {
    // column c is scaled; its update of the others, and column c + 1 scaled
    const int j0 = c + 1 < np ? c + 1 : w, n = c >= 0 ? w - c - 1 : 1;
    const int total = c >= 0 ? m * n : m;
    for (int e = threadIdx.x; e < total; e += blockDim.x) {
      const int g = e / m, r = e - g * m, j = c + 1 + g;
      double x = t[r + j * ld];
      if (c >= 0) x -= t[r + c * ld] * Us[c * 32 + j];
      if (j == j0) x *= rinv[j];
      t[r + j * ld] = x;
    }
    __syncthreads();
  }
}

// own_trsm in FP64: the warp's four columns stay in the tile and a step's
// elements, rows below q of the four, are dealt out to the lanes one by one: an
// FP64 instruction takes its 16 clocks whether its lanes are needed or not.
__device__ __forceinline__ void own_trsm_flat(double* Bk, int ld, int nb, int w, const double* Ls, double* Us) {
  const int lane = threadIdx.x & 31, cb = (threadIdx.x >> 5) * 4, wc = min(4, w - cb);
  for (int q = 0; q + 1 < nb; ++q) {
    const int m = nb - 1 - q;
    for (int e = lane; e < m * wc; e += 32) {
      const int c = e / m, r = q + 1 + e - c * m;
      double* col = Bk + (cb + c) * ld;
      col[r] -= Ls[r * 33 + q] * col[q];
    }
    __syncwarp();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
    Us[lane * 32 + cb + i] = lane < nb && cb + i < w ? Bk[lane + (cb + i) * ld] : 0.0;
}

// pivot-free LU of the np x w diagonal block D (rows = the block's pivots) in
// shared memory: lane = column, warp g = rows g, g + 8, g + 16, g + 24, and
// two pivots per barrier.  Columns keep their unscaled values during the
// elimination and are scaled once at the end; every thread forms the
// multipliers, the second pivot and the second pivot's row and column entries
// after the first elimination itself, as the same expressions in the same
// order as the one-pivot-at-a-time elimination (so every thread holds the
// values the owners of those entries store).  Writes the reciprocal pivots to
// rinv and the U rows, row-major, to Us.
template <typename T>
__device__ __forceinline__ void own_factor_diag(T* D, int ld, int np, int w, T* Us, T* rinv,
                                                const SymDev& sd, int s, int k, int K, int colbase,
                                                int32_t* status, int32_t* badcol) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int c = 0;
  for (; c + 1 < np; c += 2) {
    const T p0 = D[c + c * ld], b = D[(c + 1) + c * ld], e = D[c + (c + 1) * ld];
    const T p1raw = D[(c + 1) + (c + 1) * ld];
    const T rp0 = T(1) / p0;
    const T l1 = b * rp0;
    const T p1 = p1raw - l1 * e;
    const T rp1 = T(1) / p1;
    if (threadIdx.x == 0) {
      check_pivot(p0, sd, s, k, K, colbase + c, status, badcol);
      check_pivot(p1, sd, s, k, K, colbase + c + 1, status, badcol);
      rinv[c] = rp0;
      rinv[c + 1] = rp1;
    }
    // row c + 1 and column c + 1 are read unmodified by every thread in this
    // step, so their new values are stored only after the barrier (nothing
    // reads them again before the step after next)
    T held[4];
    int hmask = 0;
    if (lane > c && lane < w) {
      const T u0 = D[c + lane * ld];
      const T u1 = D[(c + 1) + lane * ld] - l1 * u0;
      T a0[4], a1[4], d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = wid + 8 * i;
        a0[i] = r < np ? D[r + c * ld] : T(0);
        a1[i] = r < np ? D[r + (c + 1) * ld] : T(0);
        d[i] = r < np ? D[r + lane * ld] : T(0);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = wid + 8 * i;
        held[i] = T(0);
        if (r > c && r < np) {
          const T m0 = a0[i] * rp0;
          T v = d[i] - m0 * u0;
          if (r > c + 1 && lane > c + 1) {
            const T m1 = (a1[i] - m0 * e) * rp1;
            v = v - m1 * u1;
            D[r + lane * ld] = v;
          } else {
            held[i] = v;
            hmask |= 1 << i;
          }
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (hmask & (1 << i)) D[(wid + 8 * i) + lane * ld] = held[i];
  }
  __syncthreads();
  if (c < np) {  // odd count: the last pivot updates nothing below it
    if (threadIdx.x == 0) {
      const T piv = D[c + c * ld];
      check_pivot(piv, sd, s, k, K, colbase + c, status, badcol);
      rinv[c] = T(1) / piv;
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = wid + 8 * i;
    T v = T(0);
    if (r < np && lane < w) {
      v = D[r + lane * ld];
      if (lane < r) D[r + lane * ld] = v * rinv[lane];
    }
    Us[r * 32 + lane] = (r < np && lane < w && lane >= r) ? v : T(0);
  }
}

// The same in FP64: one pivot at a time with one barrier each, the trailing
// elements dealt out to warps 1 to 7 one by one.  Warp 0 takes the next pivot's
// column: its update, the one reciprocal, the scaled column.  (Every warp
// dividing twice a barrier kept the FP64 pipe, 16 clocks an instruction, busy for
// most of a block's 75 us.)  The operations on an element are the same.
__device__ __forceinline__ void own_factor_diag_flat(double* D, int ld, int np, int w, double* Us, double* rinv,
                                                     const SymDev& sd, int s, int k, int K, int colbase,
                                                     int32_t* status, int32_t* badcol) {
  const int tid = threadIdx.x, lane = tid & 31;
  for (int p = -1; p < np; ++p) {
    const double* lc = D + p * ld;
    if (tid < 32) {
      if (p + 1 < np) {
        double* col = D + (p + 1) * ld;
        const double u = p >= 0 ? col[p] : 0.0;
        double piv = col[p + 1];
        if (p >= 0) piv -= lc[p + 1] * u;
        if (lane == 0) check_pivot(piv, sd, s, k, K, colbase + p + 1, status, badcol);
        const double rp = 1.0 / piv;
        if (lane == 0) rinv[p + 1] = rp;
        __syncwarp();
        const int i = p + 1 + lane;
        if (i < np) {
          double x = col[i];
          if (p >= 0) x -= lc[i] * u;
          col[i] = i == p + 1 ? x : x * rp;
        }
      }
    } else if (p >= 0) {
      const int m = np - p - 1, j0 = p + 1 < np ? p + 2 : p + 1, total = m * (w - j0);
      for (int e = tid - 32; e < total; e += blockDim.x - 32) {
        const int c = e / m, r = e - c * m;
        double* x = D + (p + 1 + r) + (j0 + c) * ld;
        *x -= lc[p + 1 + r] * D[p + (j0 + c) * ld];
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < 32 * 32; e += blockDim.x) {
    const int r = e >> 5, c = e & 31;
    Us[e] = (r < np && c < w && c >= r) ? D[r + c * ld] : 0.0;
  }
}

// rows [i0, i1) of the tile (stored from row R0), all below the factored
// diagonal block: one thread per row scales by the reciprocal pivots and
// eliminates in pivot order (the remaining columns of a block that straddles
// the end of the pivots are updated too).
template <typename T>
__device__ __forceinline__ void own_eliminate_rows(T* Bt, int ld, int R0, int i0, int i1, int np, int w,
                                                   const T* Us, const T* rinv) {
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    T* row = Bt + (i - R0);
    T x[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) x[c] = (c < w) ? row[c * ld] : T(0);
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      if (c < np) {
        const T l = x[c] * rinv[c];
        x[c] = l;
#pragma unroll
        for (int cc = c + 1; cc < 32; ++cc) x[cc] -= l * Us[c * 32 + cc];
      }
    }
#pragma unroll
    for (int c = 0; c < 32; ++c)
      if (c < w) row[c * ld] = x[c];
  }
}

// ---------------------------------------------------------------------------
// Tensor-core form of an owner tile's trailing update (FP32 factors only):
//     x(i, c) -= sum_{cc < nb} L(i, r0 + cc) U(cc, c)
// for the tile's rows, 128 rows at a time, on the 5th-generation tensor cores
// (tcgen05.mma, kind::tf32, M = 128, N = 32, K = 8 per instruction, FP32
// accumulator in tensor memory).  TF32 keeps 10 mantissa bits, so every FP32
// operand is split as hi + lo (hi = TF32 rounding of x, lo = TF32 rounding of
// x - hi) and the product is formed as hi*hi + hi*lo + lo*hi ("3xTF32"): the
// dropped lo*lo term and the rounding of lo are below FP32 rounding of the
// sum, so the update keeps FP32 accuracy.  Operands are staged in shared
// memory in the no-swizzle K-major core-matrix layout: 8 rows x 16 bytes per
// core matrix, K-adjacent core matrices 128 bytes apart, 8-row groups 1024
// bytes apart.
// ---------------------------------------------------------------------------
struct TcCtx {
  int on;          // 1: owner-tile updates on the tensor cores
  float* sA;       // [2][128 * 32] hi / lo of 128 rows of L
  float* sB;       // [2][32 * 32]  hi / lo of the 32 U rows (as N x K)
  uint32_t tmem;   // 32 tensor-memory columns: the 128 x 32 FP32 accumulator
  uint32_t mbar;   // shared-memory address of the MMA-completion barrier
  uint32_t phase;  // parity of the next completion of that barrier
};
constexpr int kTcSmemFloats = 2 * 128 * 32 + 2 * 32 * 32;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ float tf32_round(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// offset of element (row r, k) of a rows x 32 K-major operand
__device__ __forceinline__ int tc_kmaj(int r, int k) {
  return (r >> 3) * 256 + (k >> 2) * 32 + (r & 7) * 4 + (k & 3);
}

// shared-memory matrix descriptor: start address, leading-dimension (K) and
// stride-dimension (8-row group) byte offsets, fixed field 0b001, no swizzle
__device__ __forceinline__ uint64_t tc_sdesc(uint32_t addr) {
  uint64_t d = (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)(128 >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Allocates the CTA's 32 tensor-memory columns (warp 0) and initialises the
// completion barrier; every thread of the CTA calls it.
__device__ __forceinline__ void tc_setup(TcCtx& tc, uint32_t* s_taddr, uint64_t* s_mbar) {
  if (!tc.on) return;
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(smem_addr(s_taddr)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(s_mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  tc.tmem = *s_taddr;
  tc.mbar = smem_addr(s_mbar);
  tc.phase = 0;
}

// Frees the tensor memory; every thread of the CTA calls it before exiting.
__device__ __forceinline__ void tc_teardown(const TcCtx& tc) {
  if (!tc.on) return;
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tc.tmem));
}

// rows [i0, i1) of the tile (stored from row R0): x(i, c) -= L(i, r0..r0+nb-1) U
// for c < w, L from the front storage, U from Us (32 x 32 row-major, zero
// beyond nb rows and w columns).  Needs kOwnThreads (8 warps) threads.
__device__ __noinline__ void tc_update_rows(float* Bt, int ld, int R0, const float* f, int F, int r0, int nb,
                                               const float* Us, int i0, int i1, int w, TcCtx& tc, int* err) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5;
  float* sAh = tc.sA;
  float* sAl = tc.sA + 128 * 32;
  float* sBh = tc.sB;
  float* sBl = tc.sB + 32 * 32;
  for (int q = tid; q < 32 * 32; q += nt) {  // B(k, n) = U(k, n), staged as N x K
    const int n = q & 31, k = q >> 5;
    const float u = Us[k * 32 + n], hi = tf32_round(u);
    sBh[tc_kmaj(n, k)] = hi;
    sBl[tc_kmaj(n, k)] = tf32_round(u - hi);
  }
  const int ksteps = (nb + 7) >> 3;
  // instruction descriptor: FP32 accumulator, TF32 A and B, both K-major,
  // N = 32, M = 128
  const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((32u >> 3) << 17) | ((128u >> 4) << 24);
  for (int m0 = i0; m0 < i1; m0 += 128) {
    for (int q = tid; q < 128 * 32; q += nt) {  // A(r, k) = L(m0 + r, r0 + k), zero outside
      const int r = q & 127, k = q >> 7, i = m0 + r;
      const float a = (i < i1 && k < nb) ? __ldcg(f + i + (int64_t)(r0 + k) * F) : 0.f;
      const float hi = tf32_round(a);
      sAh[tc_kmaj(r, k)] = hi;
      sAl[tc_kmaj(r, k)] = tf32_round(a - hi);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (tid == 0) {
      uint32_t acc = 0;
      for (int ks = 0; ks < ksteps; ++ks) {
        for (int term = 0; term < 3; ++term) {  // hi*hi, hi*lo, lo*hi
          const uint64_t da = tc_sdesc(smem_addr(term == 2 ? sAl : sAh) + ks * 256);
          const uint64_t db = tc_sdesc(smem_addr(term == 1 ? sBl : sBh) + ks * 256);
          asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                       " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}" ::"r"(tc.tmem),
                       "l"(da), "l"(db), "r"(idesc), "r"(acc));
          acc = 1;
        }
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc.mbar));
    }
    {  // bounded wait for the MMAs of this block
      uint32_t done = 0;
      for (int it = 0; it < (1 << 24) && !done; ++it)
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done)
                     : "r"(tc.mbar), "r"(tc.phase));
      if (!done && tid == 0) atomicExch(err, 1);
      tc.phase ^= 1;
    }
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // warp w reads tensor-memory lanes 32 (w % 4) .. + 31 (rows), columns
    // 16 (w / 4) .. + 15
    uint32_t v[16];
    const uint32_t ta = tc.tmem + ((uint32_t)(32 * (wid & 3)) << 16) + 16 * (wid >> 2);
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]),
                   "=r"(v[15])
                 : "r"(ta));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    const int row = m0 + 32 * (wid & 3) + lane;
    if (row < i1) {
      float* x = Bt + (row - R0);
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        const int col = 16 * (wid >> 2) + c;
        if (col < w) x[col * ld] -= __uint_as_float(v[c]);
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();  // sA / the accumulator are reused by the next block
  }
}

// ---------------------------------------------------------------------------
// FP32 owner tiles on the FP32 pipe.  A tile's rows are worked through in chunks
// of kOwnChunk, and a panel's flag counts what is final of it: 1 = the pivot
// rows, 2 + c = also the rows of chunks 0 .. c, kOwnDone = all.  A tile follows
// the panel before it chunk by chunk, so a panel costs the chain of panels one
// chunk and the pivot block, not two passes over the column (10000 buses, 1596
// rows, K 8: 2.40 ms of owner tiles, 2.95 before).  U rows are read four values a time,
// which both of a thread's rows use: read one by one, shared memory took four
// times as long as the multiply-adds.
// ---------------------------------------------------------------------------
constexpr int kOwnChunk = 256;
constexpr int kOwnDone = 1 << 20;

// waits as dag_wait; returns the value seen
__device__ __forceinline__ int own_wait(const int* f, int need, int* err) {
  int v = dag_ld_acquire(f);
  for (int64_t i = 0; v < need && i < kDagWaitPolls; ++i) {
    __nanosleep(64);
    v = dag_ld_acquire(f);
  }
  if (v < need) {
    atomicExch(err, 1);
    v = need;
  }
  return v;
}

// rows [i0, i1) of the tile: x(i, :) -= L(i, r0..r0+nb-1) U.  A thread takes NR
// rows, 128 apart, and 16 columns; L comes from the front storage CB columns
// ahead of their use.
template <int NR, int CB>
__device__ __forceinline__ void own_update_rows_of(float* Bt, int ld, int R0, const float* f, int F, int r0, int nb,
                                                 const float* Us, int i0, int i1, int w) {
  const int cb = 16 * (threadIdx.x >> 7), pr = threadIdx.x & 127;
  if (cb >= w) return;
  const float* lp = f + (int64_t)r0 * F;
  float l[2][NR][CB];
  auto fetch = [&](float (&d)[NR][CB], int i, int c0) {
#pragma unroll
    for (int h = 0; h < NR; ++h)
#pragma unroll
      for (int c = 0; c < CB; ++c)
        d[h][c] = i + 128 * h < i1 && c0 + c < nb ? __ldcg(lp + i + 128 * h + (int64_t)(c0 + c) * F) : 0.f;
  };
  fetch(l[0], i0 + pr, 0);
  for (int i = i0 + pr; i < i1; i += 128 * NR) {
    float* row = Bt + (i - R0) + cb * ld;
    float x[NR][16];
#pragma unroll
    for (int c = 0; c < 16; ++c) {
#pragma unroll
      for (int h = 0; h < NR; ++h) x[h][c] = i + 128 * h < i1 ? row[c * ld + 128 * h] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < 32 / CB; ++q) {
      if (q + 1 < 32 / CB) fetch(l[(q + 1) & 1], i, CB * q + CB);
      else fetch(l[0], i + 128 * NR, 0);
      if (CB * q < nb) {
#pragma unroll
        for (int c = 0; c < CB; ++c) {
          const float4* u = reinterpret_cast<const float4*>(Us + (CB * q + c) * 32 + cb);
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            const float4 v = u[g];
#pragma unroll
            for (int h = 0; h < NR; ++h) {
              x[h][4 * g] -= l[q & 1][h][c] * v.x;
              x[h][4 * g + 1] -= l[q & 1][h][c] * v.y;
              x[h][4 * g + 2] -= l[q & 1][h][c] * v.z;
              x[h][4 * g + 3] -= l[q & 1][h][c] * v.w;
            }
          }
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 16; ++c) {
#pragma unroll
      for (int h = 0; h < NR; ++h)
        if (i + 128 * h < i1) row[c * ld + 128 * h] = x[h][c];
    }
  }
}

// by the registers of the kernel: 255 for the tiles alone, 128 or 80 in the one-launch form
template <int REGS>
__device__ __forceinline__ void own_update_pairs(float* Bt, int ld, int R0, const float* f, int F, int r0, int nb,
                                                 const float* Us, int i0, int i1, int w) {
  own_update_rows_of<(REGS >= 128 ? 2 : 1), (REGS >= 255 ? 16 : 8)>(Bt, ld, R0, f, F, r0, nb, Us, i0, i1, w);
}

// the same for at most 32 rows: lane = row, four columns a warp (8 warps)
__device__ __forceinline__ void own_update_few(float* Bt, int ld, int R0, const float* f, int F, int r0, int nb,
                                               const float* Us, int i0, int i1, int w) {
  const int i = i0 + (threadIdx.x & 31), cb = 4 * (threadIdx.x >> 5);
  if (i >= i1 || cb >= w) return;
  float l[32];
#pragma unroll
  for (int c = 0; c < 32; ++c) l[c] = c < nb ? __ldcg(f + i + (int64_t)(r0 + c) * F) : 0.f;
  float* row = Bt + (i - R0) + cb * ld;
  float x[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) x[c] = row[c * ld];
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    const float4 v = *reinterpret_cast<const float4*>(Us + c * 32 + cb);
    x[0] -= l[c] * v.x;
    x[1] -= l[c] * v.y;
    x[2] -= l[c] * v.z;
    x[3] -= l[c] * v.w;
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) row[c * ld] = x[c];
}

// own_eliminate_rows with the U rows read four at a time
__device__ __forceinline__ void own_eliminate_quads(float* Bt, int ld, int R0, int i0, int i1, int np,
                                                    const float* Us, const float* rinv) {
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    float* row = Bt + (i - R0);
    float x[32];
#pragma unroll
    for (int c = 0; c < 32; ++c) x[c] = row[c * ld];
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      if (c < np) {
        const float l = x[c] * rinv[c];
        x[c] = l;
#pragma unroll
        for (int g = (c + 1) / 4; g < 8; ++g) {
          const float4 v = *reinterpret_cast<const float4*>(Us + c * 32 + 4 * g);
          const float u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (4 * g + e > c) x[4 * g + e] -= l * u[e];
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 32; ++c) row[c * ld] = x[c];
  }
}

// The panels' updates and the own pivots of a tile that holds its pivot rows'
// chunk and is worked through in chunks (Us, Ls: 32 x 32 and 32 x 33 floats,
// 16-byte aligned).  Returns with every row of the tile from the first pivot
// down written and released; the U rows above remain to be written.
template <int REGS>
__device__ __forceinline__ void own_follow(const SymDev& sd, int s, int k, int K, int j, int q, int CH, int ns, int F,
                                           int P, int J, int Q, int* Lf, int* Uf, int* err, float* f,
                                           int32_t* status, int32_t* badcol, float* Us, float* Ls, float* Bt,
                                           float* rinv) {
  __shared__ int s_have;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const int ld = CH + 1, j0 = j << 5, w = min(32, F - j0), R0 = q * CH, R1 = min(F, R0 + CH);
  const int pe = min(j, P), qj = j0 / CH;
  const bool piv = j < P && q == qj;  // the tile holds its block's diagonal
  const int np = min(32, ns - j0);
  const int last = (R1 - 1 - R0) / kOwnChunk;
  auto release = [&](int v) {
    __syncthreads();
    if (tid == 0) dag_st_release(Lf + j * Q + q, v);
  };
  auto store = [&](int i0, int i1) {
    for (int c = wid; c < w; c += nw) {
      float* dst = f + (int64_t)(j0 + c) * F;
      const float* src = Bt + c * ld - R0;
      for (int i = i0 + lane; i < i1; i += 32) dst[i] = src[i];
    }
  };
  auto have = [&](int p, int need) {  // the stage of panel p, at least `need`
    if (tid == 0) s_have = own_wait(Lf + p * Q + q, need, err);
    __syncthreads();
    const int v = s_have;
    __syncthreads();
    return v;
  };
  int seen = 0;  // stage of panel j - 1
  for (int p = 0; p < pe; ++p) {
    const int r0 = p << 5, nb = min(32, ns - r0), qp = r0 / CH;
    if (q < qp) break;
    int v = 0;
    if (q == qp) {
      v = have(p, 1);
      for (int e = tid; e < 32 * 32; e += nt) {
        const int r = e & 31, c = e >> 5;
        Ls[r * 33 + c] = (r < nb && c < r) ? __ldcg(f + (r0 + r) + (int64_t)(r0 + c) * F) : 0.f;
      }
      __syncthreads();
      own_trsm<float>(Bt + (r0 - R0), ld, 0, nb, w, Ls, Us);
      __syncthreads();
      if (qp + 1 < Q) {  // tiles below read these U rows
        for (int c = wid; c < w; c += nw)
          for (int r = lane; r < nb; r += 32) f[(r0 + r) + (int64_t)(j0 + c) * F] = Bt[(r0 - R0 + r) + c * ld];
        __syncthreads();
        if (tid == 0) dag_st_release(Uf + p * J + j, 1);
      }
    } else {
      if (tid == 0) dag_wait(Uf + p * J + j, 1, err);
      v = have(p, 2);
      for (int e = tid; e < 32 * 32; e += nt) {
        const int r = e >> 5, c = e & 31;
        Us[e] = (r < nb && c < w) ? __ldcg(f + (r0 + r) + (int64_t)(j0 + c) * F) : 0.f;
      }
      __syncthreads();
    }
    const int i0 = q == qp ? r0 + nb : R0;  // the rows below the panel's pivots
    if (piv && p + 1 == pe) {  // goes on below, with the block's own pivots
      seen = v;
      break;
    }
    for (int c = (i0 - R0) / kOwnChunk; c <= last;) {
      if (v < 2 + c) v = have(p, 2 + c);
      const int ce = min(v - 1, last + 1);  // chunks below ce are there
      own_update_pairs<REGS>(Bt, ld, R0, f, F, r0, nb, Us, max(i0, R0 + c * kOwnChunk), min(R1, R0 + ce * kOwnChunk), w);
      c = ce;
    }
    __syncthreads();
  }
  if (!piv) return;
  // panel j - 1 (32 pivots, its rows below end at j0) and the own pivots: the pivot rows, then chunk by chunk
  const int p = j - 1, r0 = j0 - 32;
  if (j > 0) {
    const int c = (j0 + np - 1 - R0) / kOwnChunk;
    if (seen < 2 + c) seen = have(p, 2 + c);
    own_update_few(Bt, ld, R0, f, F, r0, 32, Us, j0, j0 + np, w);
    __syncthreads();
  }
  own_factor_diag<float>(Bt + (j0 - R0), ld, np, w, Ls, rinv, sd, s, k, K, sd.c0[s] + j0, status, badcol);
  __syncthreads();
  store(j0, j0 + np);
  release(1);
  for (int c = (j0 + np - R0) / kOwnChunk; c <= last; ++c) {
    const int a = max(j0 + np, R0 + c * kOwnChunk), b = min(R1, R0 + (c + 1) * kOwnChunk);
    if (j > 0) {
      if (seen < 2 + c) seen = have(p, 2 + c);
      own_update_pairs<REGS>(Bt, ld, R0, f, F, r0, 32, Us, a, b, w);
      __syncthreads();
    }
    own_eliminate_quads(Bt, ld, R0, a, b, np, Ls, rinv);
    __syncthreads();
    store(a, b);
    if (c < last) release(2 + c);
  }
  release(kOwnDone);
}

// One owner tile: the 32-column block j of front s, perturbation k,
// restricted to the row chunk q of CH rows (see above).  `flags` points at
// the (front, k) pair's release flags.  Needs kOwnThreads threads and the
// shared memory layout of the owner kernels (Us, Ls, Bt, rinv).
template <typename T, bool TC, int REGS>
__device__ __forceinline__ void owner_tile(const SymDev& sd, int s, int k, int j, int q, int* flags, int CH,
                                           int* err, const double* __restrict__ vals,
                                           const double* __restrict__ D, const Shifts& sh,
                                           T* __restrict__ fronts, int32_t* status, int32_t* badcol,
                                           T* Us, T* Ls, T* Bt, T* rinv, TcCtx& tc) {
  const int K = sh.K;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
  const int ld = CH + 1;
  const int ns = sd.ns[s], F = ns + sd.ms[s];
  const int P = (ns + 31) >> 5, J = (F + 31) >> 5, Q = (F + CH - 1) / CH;
  const int j0 = j << 5, w = min(32, F - j0);
  const int R0 = q * CH, R1 = min(F, R0 + CH);
  int* Lf = flags;            // [P][Q]: rows of chunk q of panel block p final
  int* Uf = Lf + P * Q;       // [P][J]: U rows of panel p in block j final
  T* f = fronts + (int64_t)K * sd.front_off[s] + (int64_t)k * F * F;
  const int64_t vo = sd.vec_off[s];

  // 1. assembly of the tile: rows [R0, R1) of columns [j0, j0 + w)
  for (int e = tid; e < ld * w; e += nt) Bt[e] = T(0);
  __syncthreads();
  {
    const int64_t a0 = sd.amap_coff[vo + j0], a1 = sd.amap_coff[vo + j0 + w];
    add_entries<T>(sd, vals, a0, a1, [&](int d, T v) {
      const int c = d / F, i = d - c * F;
      if (i >= R0 && i < R1) atomicAdd(&Bt[(i - R0) + (c - j0) * ld], v);
    });
    const double tk = sh.t[k];
    const int c0 = sd.c0[s];
    for (int c = max(j0, R0) + tid; c < min(min(j0 + w, ns), R1); c += nt)
      atomicAdd(&Bt[(c - R0) + (c - j0) * ld], (T)(tk * D[sd.perm[c0 + c]]));
  }
  __syncthreads();
  extend_add_columns<T>(sd, s, k, K, fronts, Bt, ld, j0, w, R0, R1, wid, nw);
  __syncthreads();

  // 2. the updates of every earlier panel, in pivot order; panels whose
  //    pivot rows lie below the tile do not touch it
  constexpr bool kFollow = std::is_same<T, float>::value && !TC;
  if constexpr (kFollow)
    own_follow<REGS>(sd, s, k, K, j, q, CH, ns, F, P, J, Q, Lf, Uf, err, f, status, badcol, Us, Ls, Bt, rinv);
  const int pe = kFollow ? 0 : min(j, P);
  for (int p = 0; p < pe; ++p) {
    const int r0 = p << 5, nb = min(32, ns - r0), qp = r0 / CH;
    if (q < qp) break;
    if (q == qp) {
      // the tile holds panel p's pivot rows: solve this block's U rows
      if (tid == 0) dag_wait(Lf + p * Q + qp, kOwnDone, err);
      __syncthreads();
      for (int e = tid; e < 32 * 32; e += nt) {
        const int r = e & 31, c = e >> 5;
        Ls[r * 33 + c] = (r < nb && c < r) ? __ldcg(f + (r0 + r) + (int64_t)(r0 + c) * F) : T(0);
      }
      __syncthreads();
      if constexpr (sizeof(T) == 8) own_trsm_flat(Bt + (r0 - R0), ld, nb, w, Ls, Us);
      else own_trsm<T>(Bt + (r0 - R0), ld, 0, nb, w, Ls, Us);
      __syncthreads();
      if (qp + 1 < Q) {  // chunks below read these U rows
        for (int c = wid; c < w; c += nw)
          for (int r = lane; r < nb; r += 32) f[(r0 + r) + (int64_t)(j0 + c) * F] = Bt[(r0 - R0 + r) + c * ld];
        __threadfence();
        __syncthreads();
        if (tid == 0) dag_st_release(Uf + p * J + j, 1);
      }
      if constexpr (TC && std::is_same<T, float>::value)
        tc_update_rows(Bt, ld, R0, f, F, r0, nb, Us, r0 + nb, R1, w, tc, err);
      else if constexpr (sizeof(T) == 8)
        own_update_few64(Bt, ld, R0, f, F, r0, nb, Us, r0 + nb, R1, w);
      __syncthreads();
    } else {
      // a chunk below panel p: its U rows of this block come from the
      // chunk holding the pivot rows, its L rows from this chunk's tile of
      // panel p
      if (tid == 0) {
        dag_wait(Uf + p * J + j, 1, err);
        dag_wait(Lf + p * Q + q, kOwnDone, err);
      }
      __syncthreads();
      for (int e = tid; e < 32 * 32; e += nt) {
        const int r = e >> 5, c = e & 31;
        Us[e] = (r < nb && c < w) ? __ldcg(f + (r0 + r) + (int64_t)(j0 + c) * F) : T(0);
      }
      __syncthreads();
      if constexpr (TC && std::is_same<T, float>::value)
        tc_update_rows(Bt, ld, R0, f, F, r0, nb, Us, R0, R1, w, tc, err);
      else if constexpr (sizeof(T) == 8)
        own_update_few64(Bt, ld, R0, f, F, r0, nb, Us, R0, R1, w);
      __syncthreads();
    }
  }

  // 3. the block's own pivots
  const int qj = j0 / CH;
  if (j < P) {
    const int np = min(32, ns - j0);
    if (q == qj && !kFollow) {
      if constexpr (sizeof(T) == 8)
        own_factor_diag_flat(Bt + (j0 - R0), ld, np, w, Us, rinv, sd, s, k, K, sd.c0[s] + j0, status, badcol);
      else
        own_factor_diag<T>(Bt + (j0 - R0), ld, np, w, Us, rinv, sd, s, k, K, sd.c0[s] + j0, status, badcol);
      __syncthreads();
      if constexpr (sizeof(T) == 8) own_eliminate_flat(Bt, ld, R0, j0 + np, R1, np, w, Us, rinv);
      else own_eliminate_rows<T>(Bt, ld, R0, j0 + np, R1, np, w, Us, rinv);
      __syncthreads();
    } else if (q > qj) {
      // rows below the diagonal block's chunk: its factored rows come from
      // the front storage once that tile has released them
      if (tid == 0) dag_wait(Lf + j * Q + qj, 1, err);
      __syncthreads();
      for (int e = tid; e < 32 * 32; e += nt) {
        const int r = e >> 5, c = e & 31;
        Us[e] = (r < np && c < w && c >= r) ? __ldcg(f + (j0 + r) + (int64_t)(j0 + c) * F) : T(0);
      }
      if (tid < np) rinv[tid] = T(1) / __ldcg(f + (int64_t)(j0 + tid) * (F + 1));
      __syncthreads();
      if constexpr (sizeof(T) == 8) own_eliminate_flat(Bt, ld, R0, R0, R1, np, w, Us, rinv);
      else own_eliminate_rows<T>(Bt, ld, R0, R0, R1, np, w, Us, rinv);
      __syncthreads();
    }
  }

  // 4. write the tile; tiles holding L rows of this block release them
  //    (rows from the first pivot down first, then the U rows above)
  const bool rel = j < P && q >= qj;
  const int rs = (rel && q == qj) ? j0 : R0;
  if (!(kFollow && rel && q == qj)) {
  for (int c = wid; c < w; c += nw) {
    T* dst = f + (int64_t)(j0 + c) * F;
    const T* src = Bt + c * ld;
    for (int i = rs + lane; i < R1; i += 32) dst[i] = src[i - R0];
  }
  if (rel) {
    __threadfence();
    __syncthreads();
    if (tid == 0) dag_st_release(Lf + j * Q + q, kOwnDone);
  }
  }
  for (int c = wid; c < w; c += nw) {
    T* dst = f + (int64_t)(j0 + c) * F;
    const T* src = Bt + c * ld;
    for (int i = R0 + lane; i < rs; i += 32) dst[i] = src[i - R0];
  }
}

template <typename T, bool TC>
__global__ void __launch_bounds__(kOwnThreads) k_front_owner(SymDev sd, const int32_t* __restrict__ big,
                                                             const DagTask* __restrict__ tasks, int ntasks,
                                                             int* ticket, int* flags, int* err,
                                                             const double* __restrict__ vals,
                                                             const double* __restrict__ D, Shifts sh,
                                                             T* __restrict__ fronts, int32_t* status,
                                                             int32_t* badcol, int CH) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_t;
  __shared__ T rinv[32];
  __shared__ uint32_t s_taddr;
  __shared__ __align__(8) uint64_t s_mbar;
  T* Us = reinterpret_cast<T*>(smraw);  // 32 x 32 row-major: U rows of the current panel
  T* Ls = Us + 32 * 32;                 // 32 x 33 row-major: unit-lower L11 of the current panel
  T* Bt = Ls + 32 * 33;                 // (CH + 1) x 32 column-major: the owned tile
  float* tcs = reinterpret_cast<float*>(Bt + (size_t)(CH + 1) * 32);  // tensor-core staging (FP32 only)
  TcCtx tc{TC ? 1 : 0, tcs, tcs + 2 * 128 * 32, 0, 0, 0};
  if constexpr (TC) tc_setup(tc, &s_taddr, &s_mbar);
  const int tid = threadIdx.x;
  for (;;) {
    __syncthreads();  // the previous task is done with shared memory and s_t
    if (tid == 0) s_t = atomicAdd(ticket, 1);
    __syncthreads();
    const int u = s_t;
    if (u >= ntasks) break;
    const DagTask t = tasks[u];
    owner_tile<T, TC, 255>(sd, big[t.b], t.k, t.j, t.p, flags + t.flags, CH, err, vals, D, sh, fronts, status, badcol,
                  Us, Ls, Bt, rinv, tc);
  }
  if constexpr (TC) tc_teardown(tc);
}

// ---------------------------------------------------------------------------
// The whole factorisation as ONE persistent launch over every level of the
// assembly forest, all K shifts and all instances of a batch.  Tasks, taken in
// ticket order (levels bottom-up; within a level the owner tiles first, then
// the shared-memory fronts, then the segments):
//   kFacSeg8/16/32: 256 / SEG (front, k) pairs with F <= SEG, one per segment
//              of SEG lanes (front_seg);
//   kFacCta  : one (front, k) pair of a front that fits in shared memory
//              (front_cta);
//   kFacOwner: one owner tile of a wider front (owner_tile).
// Before its assembly a task waits until its front's counter for its k,
// fdone[s * K + k], has reached need[s], the tasks of its children (one each for
// segment and shared-memory fronts, the tiles of an owner front); a finished task
// adds 1 to its parent's counter after its writes are visible.  Every wait is
// on a task with a smaller ticket (a child, or an earlier tile of the same
// front), which a running CTA already holds, so the schedule cannot deadlock
// whatever the residency, and every wait is bounded.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void fac_wait_children(const SymDev& sd, const int* fdone, const int* need, int s,
                                                  int k, int K, int* err, int64_t wait_ns) {
  const int want = need[s];
  if (want == 0) return;
  const int* f = fdone + ((int64_t)s * K + k) * kCtrStride;
  if (dag_ld_acquire(f) >= want) return;
  // the polls in between are relaxed: an acquiring one drops the SM's L1 lines
  // under the CTA beside it
  unsigned ns = 32;
  for (int64_t left = wait_ns; left > 0;) {
    __nanosleep(ns);
    int v;
    asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
    if (v >= want) break;
    left -= ns;
    ns += ns < 1024 ? ns >> 3 : 0;
  }
  if (dag_ld_acquire(f) < want) atomicExch(err, 1);
}

__device__ __forceinline__ void fac_publish(const SymDev& sd, int* fdone, int s, int k, int K) {
  const int p = sd.parent[s];
  if (p >= 0)
    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(fdone + ((int64_t)p * K + k) * kCtrStride) : "memory");
}

template <typename T, int SEG>
__device__ __forceinline__ void fac_segments(const SymDev& sd, const FactorTask& t, const int* need, int* fdone,
                                             int* err, int64_t wait_ns, const int32_t* __restrict__ wlist,
                                             const double* __restrict__ vals, const double* __restrict__ D,
                                             const Shifts& sh, T* __restrict__ fronts, int32_t* status,
                                             int32_t* badcol, T* sm) {
  const int q = t.q + (int)threadIdx.x / SEG, sl = threadIdx.x % SEG;
  const bool on = q < t.j;
  const int s = on ? wlist[t.s + q / sh.K] : 0, k = on ? q % sh.K : 0;
  if (on && sl == 0) fac_wait_children(sd, fdone, need, s, k, sh.K, err, wait_ns);
  __syncwarp();
  front_seg<T, SEG>(sd, s, k, on, sl, vals, D, sh, fronts, status, badcol, sm + threadIdx.x / SEG * SEG * SEG);
  __syncwarp();
  if (on && sl == 0) fac_publish(sd, fdone, s, k, sh.K);
}

template <typename T, bool TC, int MINB>
__global__ void __launch_bounds__(kOwnThreads, MINB)
k_factor_persistent(SymDev sd, const FactorTask* __restrict__ tasks, int ntasks, int* ticket, int* fdone,
                    const int* __restrict__ need, int* flags, int* err, const int32_t* __restrict__ wlist,
                    const double* __restrict__ vals, const double* __restrict__ D, const __grid_constant__ Shifts sh,
                    T* __restrict__ fronts, int32_t* status, int32_t* badcol, int CH, int64_t wait_ns,
                    size_t tc_off) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_t;
  __shared__ T rinv[32];
  __shared__ uint32_t s_taddr;
  __shared__ __align__(8) uint64_t s_mbar;
  T* sm = reinterpret_cast<T*>(smraw);
  float* tcs = reinterpret_cast<float*>(smraw + tc_off);  // tensor-core staging (FP32 owner tiles)
  TcCtx tc{TC ? 1 : 0, tcs, tcs + 2 * 128 * 32, 0, 0, 0};
  if constexpr (TC) tc_setup(tc, &s_taddr, &s_mbar);
  const int K = sh.K;
  const int tid = threadIdx.x;
  for (;;) {
    __syncthreads();  // the previous task is done with shared memory and s_t
    if (tid == 0) s_t = atomicAdd(ticket, 1);
    __syncthreads();
    const int u = s_t;
    if (u >= ntasks) break;
    const FactorTask t = tasks[u];
    if (t.kind == kFacSeg8) {
      fac_segments<T, 8>(sd, t, need, fdone, err, wait_ns, wlist, vals, D, sh, fronts, status, badcol, sm);
    } else if (t.kind == kFacSeg16) {
      fac_segments<T, 16>(sd, t, need, fdone, err, wait_ns, wlist, vals, D, sh, fronts, status, badcol, sm);
    } else if (t.kind == kFacSeg32) {
      fac_segments<T, 32>(sd, t, need, fdone, err, wait_ns, wlist, vals, D, sh, fronts, status, badcol, sm);
    } else {
      if (tid == 0) fac_wait_children(sd, fdone, need, t.s, t.k, K, err, wait_ns);
      __syncthreads();
      if (t.kind == kFacCta)
        front_cta<T, (MINB >= 3)>(sd, t.s, t.k, vals, D, sh, fronts, status, badcol, sm, rinv);
      else
        owner_tile<T, TC, MINB >= 3 ? 80 : 128>(sd, t.s, t.k, t.j, t.q, flags + t.flags, CH, err, vals, D, sh, fronts, status,
                          badcol, sm, sm + 32 * 32, sm + 32 * 32 + 32 * 33, rinv, tc);
      __syncthreads();
      if (tid == 0) fac_publish(sd, fdone, t.s, t.k, K);
    }
  }
  if constexpr (TC) tc_teardown(tc);
}

template <typename T, bool TC, int M>
int factor_persistent_launch(const SymDev& sd, const FactorTask* tasks, int ntasks, int* ticket, int* fdone,
                             const int* need, int* flags, int* err, const int32_t* wlist, const double* vals,
                             const double* D, const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol,
                             int CH, size_t smem, size_t tc_off, int64_t polls, cudaStream_t st) {
  static std::atomic<int> nsm_dev[kMaxDevices];
  const int dev = current_device();
  int nsm = nsm_dev[dev].load(std::memory_order_acquire);
  if (!nsm) {
    cudaFuncSetAttribute(k_factor_persistent<T, TC, M>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    nsm_dev[dev].store(nsm, std::memory_order_release);
  }
  int occ = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_factor_persistent<T, TC, M>, kOwnThreads, smem);
  const int grid = std::max(1, std::min(ntasks, std::max(1, occ) * std::max(nsm, 1)));
  k_factor_persistent<T, TC, M><<<grid, kOwnThreads, smem, st>>>(sd, tasks, ntasks, ticket, fdone, need, flags,
                                                                 err, wlist, vals, D, sh, (T*)fronts, status,
                                                                 badcol, CH, wait_limit_ns(polls),
                                                                 tc_off);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

// ctas: resident CTAs per SM the kernel is compiled for, 2 (128 registers per
// thread) or 3 (80; the owner tiles' register arrays then spill a little)
template <typename T>
int factor_persistent_impl(const SymDev& sd, const FactorTask* tasks, int ntasks, int* ticket, int* fdone,
                           const int* need, int* flags, int* err, const int32_t* wlist, const double* vals,
                           const double* D, const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol,
                           int CH, size_t smem, int64_t polls, int tc, int ctas, cudaStream_t st) {
  if (ntasks == 0) return 0;
  const int tc_on = tc && sizeof(T) == 4 ? 1 : 0;
  const size_t tc_off = smem;  // the staging follows everything the other task kinds use
  if (tc_on) smem += (size_t)kTcSmemFloats * sizeof(float);
  if (smem > (size_t)kSmemCap) return -1;
  if (tc_on)
    return factor_persistent_launch<T, true, 2>(sd, tasks, ntasks, ticket, fdone, need, flags, err, wlist, vals, D,
                                                sh, fronts, status, badcol, CH, smem, tc_off, polls, st);
  if (ctas >= 3)
    return factor_persistent_launch<T, false, 3>(sd, tasks, ntasks, ticket, fdone, need, flags, err, wlist, vals,
                                                 D, sh, fronts, status, badcol, CH, smem, tc_off, polls, st);
  return factor_persistent_launch<T, false, 2>(sd, tasks, ntasks, ticket, fdone, need, flags, err, wlist, vals, D,
                                               sh, fronts, status, badcol, CH, smem, tc_off, polls, st);
}

template <typename T>
int owner_impl(const SymDev& sd, const LevelPlan& lp, const int32_t* d_big, const DagTask* tasks,
               int* ticket, int* flags, int* err, const double* vals, const double* D,
               const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol, int tc, cudaStream_t st) {
  static std::atomic<int> nsm_dev[kMaxDevices];
  const int dev = current_device();
  int nsm = nsm_dev[dev].load(std::memory_order_acquire);
  if (!nsm) {
    cudaFuncSetAttribute(k_front_owner<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
    cudaFuncSetAttribute(k_front_owner<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    nsm_dev[dev].store(nsm, std::memory_order_release);
  }
  const int tc_on = tc && sizeof(T) == 4 ? 1 : 0;
  const size_t smem = ((size_t)(lp.own_ch + 1) * 32 + 32 * 32 + 32 * 33) * sizeof(T) +
                      (tc_on ? (size_t)kTcSmemFloats * sizeof(float) : 0);
  if (lp.own_ch < 32 || lp.own_ch % 32 || smem > (size_t)kSmemCap) return -1;
  int occ = 1;
  if (tc_on) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_front_owner<T, true>, kOwnThreads, smem);
  else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_front_owner<T, false>, kOwnThreads, smem);
  const int grid = std::max(1, std::min(lp.dag_tasks, std::max(1, occ) * std::max(nsm, 1)));
  if (tc_on)
    k_front_owner<T, true><<<grid, kOwnThreads, smem, st>>>(sd, d_big + lp.big_off, tasks + lp.dag_task_off,
                                                            lp.dag_tasks, ticket, flags, err, vals, D, sh,
                                                            (T*)fronts, status, badcol, lp.own_ch);
  else
    k_front_owner<T, false><<<grid, kOwnThreads, smem, st>>>(sd, d_big + lp.big_off, tasks + lp.dag_task_off,
                                                             lp.dag_tasks, ticket, flags, err, vals, D, sh,
                                                             (T*)fronts, status, badcol, lp.own_ch);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

template <typename T>
void set_smem_attrs() {
  static std::atomic<bool> done_dev[kMaxDevices];
  const int dev = current_device();
  if (done_dev[dev].load(std::memory_order_acquire)) return;
  cudaFuncSetAttribute(k_front_small<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_front_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_panel_big<T, 32>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_panel_big<T, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_panel_big<T, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  cudaFuncSetAttribute(k_panel_big<T, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemCap);
  done_dev[dev].store(true, std::memory_order_release);
}

template <typename T, int NB>
int run_panels(const SymDev& sd, const LevelPlan& lp, const int32_t* d_big,
               const BigFrontHost* bh, int K, T* fr, int32_t* status, int32_t* badcol,
               cudaStream_t st) {
  int launches = 0;
  for (int p0 = 0; p0 < lp.big_maxns; p0 += NB) {
    int maxMr = 0, mmax = 0;
    for (int b = 0; b < lp.big_count; ++b) {
      if (p0 >= bh[b].ns) continue;
      maxMr = std::max(maxMr, bh[b].F - p0);
      mmax = std::max(mmax, bh[b].F - p0 - std::min(NB, bh[b].ns - p0));
    }
    if (maxMr == 0) continue;
    const size_t smem = (size_t)(maxMr + 1) * NB * sizeof(T);
    k_panel_big<T, NB><<<dim3(lp.big_count, K), 512, smem, st>>>(sd, d_big, K, fr, p0, status, badcol);
    ++launches;
    if (mmax > 0) {
      const int tpd = (mmax + 63) / 64;
      k_update_big<T><<<dim3(tpd * tpd, lp.big_count, K), 256, 0, st>>>(sd, d_big, K, fr, p0, NB);
      ++launches;
    }
  }
  return launches;
}

template <typename T>
int factor_small_group(const SymDev& sd, const LevelPlan& lp, int g, const int32_t* d_small,
                       const double* vals, const double* D, const Shifts& sh, void* fronts,
                       int32_t* status, int32_t* badcol, cudaStream_t st) {
  set_smem_attrs<T>();
  T* fr = reinterpret_cast<T*>(fronts);
  const int K = sh.K;
  int launches = 0;
  {
    const auto& G = lp.groups[g];
    if (G.count == 0) return 0;
    if (G.cluster == 0) {
      const int32_t* lst = d_small + G.off;
      bool seg_class = false;
      // FP64 takes a CTA for the narrowest fronts too: its warps share the columns,
      // where rows as lanes leave some idle (118 buses 99 us, 136 with segments; 300
      // buses 154, 185)
      if constexpr (sizeof(T) == 4) {
        const int n = G.count * K;
        auto seg = [&](auto S) {
          constexpr int SEG = decltype(S)::value, per = 256 / SEG;
          k_front_seg<SEG><<<(n + per - 1) / per, 256, 0, st>>>(sd, lst, n, vals, D, sh, fr, status, badcol);
        };
        seg_class = G.maxF <= 32;
        if (G.maxF <= 8) seg(std::integral_constant<int, 8>{});
        else if (G.maxF <= 16) seg(std::integral_constant<int, 16>{});
        else if (G.maxF <= 32) seg(std::integral_constant<int, 32>{});
      }
      if (!seg_class)
        k_front_small<T><<<dim3(G.count, K), G.maxF <= 32 ? 128 : (G.maxF <= 96 ? 256 : 512),
                           (size_t)G.maxF * front_ld(G.maxF) * sizeof(T), st>>>(sd, lst, vals, D, sh, fr, status,
                                                                               badcol);
    } else {
      const int C = G.cluster;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(G.count * C, K, 1);
      cfg.blockDim = dim3(256, 1, 1);
      cfg.dynamicSmemBytes = cluster_smem<T>(G.maxF, C);
      cfg.stream = st;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = C;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      const int32_t* lst = d_small + G.off;
      if (cudaLaunchKernelEx(&cfg, k_front_cluster<T>, sd, lst, C, vals, D, sh, fr, status, badcol) !=
          cudaSuccess)
        return -1;
    }
    ++launches;
  }
  if (cudaGetLastError() != cudaSuccess) return -1;
  return launches;
}

template <typename T>
int factor_small_impl(const SymDev& sd, const LevelPlan& lp, const int32_t* d_small,
                      const double* vals, const double* D, const Shifts& sh, void* fronts,
                      int32_t* status, int32_t* badcol, cudaStream_t st) {
  int launches = 0;
  for (int g = 0; g < lp.n_groups; ++g) {
    const int n = factor_small_group<T>(sd, lp, g, d_small, vals, D, sh, fronts, status, badcol, st);
    if (n < 0) return -1;
    launches += n;
  }
  return launches;
}

template <typename T>
int factor_big_impl(const SymDev& sd, const LevelPlan& lp, const int32_t* d_big,
                    const BigFrontHost* bh, const double* vals, const double* D, const Shifts& sh,
                    void* fronts, int32_t* status, int32_t* badcol, cudaStream_t st) {
  set_smem_attrs<T>();
  T* fr = reinterpret_cast<T*>(fronts);
  const int K = sh.K;
  int launches = 0;
  if (lp.big_count > 0) {
    const int TW = 32;
    const int big = lp.big_count;
    const int32_t* lst = d_big + lp.big_off;
    k_assemble_big<T><<<dim3((lp.big_maxF + TW - 1) / TW, big, K), 256, 0, st>>>(
        sd, lst, vals, D, sh, fr, TW);
    ++launches;
    const BigFrontHost* b = bh + lp.big_off;
    if ((size_t)(lp.big_maxF + 1) * 32 * sizeof(T) <= (size_t)kSmemCap)
      launches += run_panels<T, 32>(sd, lp, lst, b, K, fr, status, badcol, st);
    else if ((size_t)(lp.big_maxF + 1) * 16 * sizeof(T) <= (size_t)kSmemCap)
      launches += run_panels<T, 16>(sd, lp, lst, b, K, fr, status, badcol, st);
    else if ((size_t)(lp.big_maxF + 1) * 8 * sizeof(T) <= (size_t)kSmemCap)
      launches += run_panels<T, 8>(sd, lp, lst, b, K, fr, status, badcol, st);
    else
      launches += run_panels<T, 4>(sd, lp, lst, b, K, fr, status, badcol, st);
  }
  if (cudaGetLastError() != cudaSuccess) return -1;
  return launches;
}

}  // namespace

int small_front_limit(int precision) { return precision == PISP_FP32 ? 224 : 160; }

int front_cluster_size(int F, int precision) {
  if (F <= 64) return 0;
  for (int C = 1; C <= 8; C *= 2) {
    const size_t need = precision == PISP_FP32 ? cluster_smem<float>(F, C) : cluster_smem<double>(F, C);
    if (need <= (size_t)kSmemCap) return C;
  }
  return -1;
}

int max_big_front(int precision) {
  return kSmemCap / (4 * (precision == PISP_FP32 ? 4 : 8)) - 1;
}

int launch_factor_small(int precision, const SymDev& sd, const LevelPlan& lp,
                        const int32_t* d_small, const double* vals, const double* D,
                        const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol,
                        cudaStream_t st) {
  if (precision == PISP_FP32)
    return factor_small_impl<float>(sd, lp, d_small, vals, D, sh, fronts, status, badcol, st);
  return factor_small_impl<double>(sd, lp, d_small, vals, D, sh, fronts, status, badcol, st);
}

int launch_factor_small_group(int precision, const SymDev& sd, const LevelPlan& lp, int g,
                              const int32_t* d_small, const double* vals, const double* D,
                              const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol,
                              cudaStream_t st) {
  if (precision == PISP_FP32)
    return factor_small_group<float>(sd, lp, g, d_small, vals, D, sh, fronts, status, badcol, st);
  return factor_small_group<double>(sd, lp, g, d_small, vals, D, sh, fronts, status, badcol, st);
}

int max_dag_front(int precision) { return kSmemCap / (32 * (precision == PISP_FP32 ? 4 : 8)) - 1; }

int owner_chunk_rows(int precision, int maxF, int tc) {
  // Rows per tile.  FP64 elimination runs at a small fraction of the FP32
  // rate on this part, so one SM per 32-column block is the bottleneck of a
  // panel step: 32-row tiles spread a block's update and elimination over
  // its chunks (1354-bus root: 0.66 ms against 0.82 with whole columns, when the
  // kernels inside were slower; 0.40 with 32-row tiles now).  In FP32 a tile is a
  // whole column block while it fits in shared memory: row chunks are handed
  // over from inside it (own_follow), without their reloads.
  const int full = (maxF + 31) / 32 * 32;
  if (precision != PISP_FP32) return std::min(32, full);
  // (CH + 1) * 32 + 2080 floats, plus the tensor-core staging when it is on
  const int fit = ((kSmemCap / 4 - 32 * 32 - 32 * 33 - (tc ? kTcSmemFloats : 0)) / 32 - 1) / 32 * 32;
  return std::min(full, fit);
}

void build_owner_tasks(const BigFrontHost* big, int32_t nbig, int32_t K, int32_t CH,
                       std::vector<DagTask>& out, int32_t& nflags) {
  out.clear();
  std::vector<int32_t> foff((size_t)nbig * K);
  nflags = 0;
  int maxJ = 0, maxQ = 0;
  for (int b = 0; b < nbig; ++b) {
    const int P = (big[b].ns + 31) / 32, J = (big[b].F + 31) / 32, Q = (big[b].F + CH - 1) / CH;
    maxJ = std::max(maxJ, J);
    maxQ = std::max(maxQ, Q);
    for (int k = 0; k < K; ++k) {
      foff[(size_t)b * K + k] = nflags;
      nflags += P * (Q + J);
    }
  }
  // (block, chunk) order: every wait of a tile is on a tile earlier in it
  for (int j = 0; j < maxJ; ++j)
    for (int q = 0; q < maxQ; ++q)
      for (int b = 0; b < nbig; ++b) {
        if (j >= (big[b].F + 31) / 32 || q >= (big[b].F + CH - 1) / CH) continue;
        for (int k = 0; k < K; ++k) out.push_back({kDagOwner, b, k, q, j, foff[(size_t)b * K + k]});
      }
}

void build_dag_tasks(const BigFrontHost* big, int32_t nbig, int32_t K, std::vector<DagTask>& out,
                     int32_t& nflags) {
  out.clear();
  std::vector<int32_t> foff((size_t)nbig * K);
  nflags = 0;
  int maxP = 0;
  for (int b = 0; b < nbig; ++b) {
    const int J = (big[b].F + 31) / 32, P = (big[b].ns + 31) / 32;
    maxP = std::max(maxP, P);
    for (int k = 0; k < K; ++k) {
      foff[(size_t)b * K + k] = nflags;
      nflags += J + P;
    }
  }
  for (int b = 0; b < nbig; ++b)
    for (int k = 0; k < K; ++k)
      for (int j = 0; j < (big[b].F + 31) / 32; ++j)
        out.push_back({kDagAsm, b, k, 0, j, foff[(size_t)b * K + k]});
  for (int p = 0; p < maxP; ++p) {
    for (int b = 0; b < nbig; ++b) {
      const int F = big[b].F, ns = big[b].ns;
      const int J = (F + 31) / 32, P = (ns + 31) / 32;
      if (p >= P) continue;
      const int nb = std::min(32, ns - 32 * p);
      for (int k = 0; k < K; ++k) {
        const int fo = foff[(size_t)b * K + k];
        if (p == 0) out.push_back({kDagPanel, b, k, 0, 0, fo});
        if (p + 1 < J) out.push_back({kDagUpdate, b, k, p, p + 1, fo});
        if (p + 1 < P) out.push_back({kDagPanel, b, k, p + 1, 0, fo});
        if (32 * p + nb < std::min(32 * p + 32, F)) out.push_back({kDagUpdate, b, k, p, p, fo});
        for (int j = p + 2; j < J; ++j) out.push_back({kDagUpdate, b, k, p, j, fo});
      }
    }
  }
}

int launch_factor_big_dag(int precision, const SymDev& sd, const LevelPlan& lp, const int32_t* d_big,
                          const DagTask* tasks, int* ticket, int* flags, int* err,
                          const double* vals, const double* D, const Shifts& sh, void* fronts,
                          int32_t* status, int32_t* badcol, int tc, cudaStream_t st) {
  if (lp.dag_owner) {
    if (precision == PISP_FP32)
      return owner_impl<float>(sd, lp, d_big, tasks, ticket, flags, err, vals, D, sh, fronts, status,
                               badcol, tc, st);
    return owner_impl<double>(sd, lp, d_big, tasks, ticket, flags, err, vals, D, sh, fronts, status,
                              badcol, tc, st);
  }
  if (precision == PISP_FP32)
    return big_dag_impl<float>(sd, lp, d_big, tasks, ticket, flags, err, vals, D, sh, fronts, status,
                               badcol, st);
  return big_dag_impl<double>(sd, lp, d_big, tasks, ticket, flags, err, vals, D, sh, fronts, status,
                              badcol, st);
}

int persistent_cta_front_limit(int precision) { return precision == PISP_FP32 ? 160 : 112; }

size_t factor_persistent_smem(int precision, int CH, bool has_owner, int maxCtaF) {
  const size_t es = precision == PISP_FP32 ? 4 : 8;
  size_t e = (size_t)(kOwnThreads / 32) * 32 * 32;                          // segments
  e = std::max(e, (size_t)maxCtaF * front_ld(maxCtaF));                      // shared-memory fronts
  if (has_owner) e = std::max(e, (size_t)(CH + 1) * 32 + 32 * 32 + 32 * 33);  // owner tiles
  return (e * es + 127) / 128 * 128;  // what follows it (the tensor-core staging) stays aligned
}

size_t tc_staging_bytes() { return (size_t)kTcSmemFloats * sizeof(float); }

int launch_factor_persistent(int precision, const SymDev& sd, const FactorTask* tasks, int ntasks, int* ticket,
                             int* fdone, const int* need, int* flags, int* err, const int32_t* wlist,
                             const double* vals, const double* D, const Shifts& sh, void* fronts,
                             int32_t* status, int32_t* badcol, int CH, size_t smem, int64_t polls, int tc,
                             int ctas, cudaStream_t st) {
  if (precision == PISP_FP32)
    return factor_persistent_impl<float>(sd, tasks, ntasks, ticket, fdone, need, flags, err, wlist, vals, D, sh,
                                         fronts, status, badcol, CH, smem, polls, tc, ctas, st);
  return factor_persistent_impl<double>(sd, tasks, ntasks, ticket, fdone, need, flags, err, wlist, vals, D, sh,
                                        fronts, status, badcol, CH, smem, polls, tc, ctas, st);
}

int launch_factor_big(int precision, const SymDev& sd, const LevelPlan& lp, const int32_t* d_big,
                      const BigFrontHost* big_host, const double* vals, const double* D,
                      const Shifts& sh, void* fronts, int32_t* status, int32_t* badcol,
                      cudaStream_t st) {
  if (precision == PISP_FP32)
    return factor_big_impl<float>(sd, lp, d_big, big_host, vals, D, sh, fronts, status, badcol, st);
  return factor_big_impl<double>(sd, lp, d_big, big_host, vals, D, sh, fronts, status, badcol, st);
}

}  // namespace pisp
