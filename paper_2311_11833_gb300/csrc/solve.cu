// The expansion-weighted combine (Eq. x_star / Remark 2), FP64 residuals, the
// adaptive residual sweeps' stopping test and the adjoint gradient.  The
// triangular solves are in solve_persistent.h.
//
// Vector layouts (T = factor precision; RV and RX: rhs_stride, rhs_stride64):
//   b, x    [N][R]      FP64, original row order (caller-owned)
//   X, Lam  [N][K][RX]  FP64, permuted row order, one slice per perturbation
//   Y, Rk   [N][K][RV]  T, permuted row order: corrections and residuals,
//                       which the solves compute and read in T
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>

#include "pisp_internal.h"

namespace pisp {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// x[perm[i]][r] = sum_k w_k X[i][k][r]   (Eq. x_star; FP64, k ascending)
__global__ void k_combine(SymDev sd, const double* __restrict__ X, Shifts sh, int R, int RX,
                          double* __restrict__ x) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= sd.N * R) return;
  const int64_t i = q / R;
  const int r = (int)(q % R);
  const int K = sh.K;
  double a = 0.0;
  for (int k = 0; k < K; ++k) a += sh.w[k] * X[(i * K + k) * RX + r];
  x[(int64_t)sd.perm[i] * R + r] = a;
}

// largest q in [0, n] with arow[q] <= a (arow[0] = 0 <= a)
__device__ __forceinline__ int active_slot(const int64_t* arow, int n, int64_t a) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (arow[mid] <= a) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// The FP64 residuals of the perturbed systems, in permuted row order (where
// an instance's rows keep its range), rounded to the precision of the solves
// that read them:
//   Rk[pi][k][r] = b[i][r] - sum_j A_ij X[pj][k][r] - t_k D_i X[pi][k][r],
// or with TRANS those of the transposed systems (A's columns through the CSC
// arrays).  GL = 2^lg lanes take one row, a lane its (k, r) columns, so that a
// few columns still fill a warp; the row's entries are read as broadcasts,
// four at a time, their values gathered before the four subtractions (entry
// order kept).  Bound by the FP64 pipe (2 multiply-adds per clock and SM):
// nnz K R of them, plus two and one conversion per row and column.
template <typename T, bool TRANS>
__global__ void __launch_bounds__(256) k_residual_per_k(SymDev sd, const double* __restrict__ vals,
                                                        const double* __restrict__ D,
                                                        const __grid_constant__ Shifts sh,
                                                        const double* __restrict__ b, const double* __restrict__ X,
                                                        int R, int RX, int RV, int lg, T* __restrict__ Rk,
                                                        ActiveSet as, int mode) {
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t ng = ((int64_t)gridDim.x * blockDim.x) >> lg;
  const int gl = 1 << lg, l = threadIdx.x & (gl - 1);
  const int K = sh.K, KR = K * R;
  int nact = 0;
  int64_t total = sd.N;
  if (mode == kResActive) {
    nact = *as.nact;
    total = as.arow[nact];
  }
  const int kl = l / R, rl = l - kl * R;  // (k, r) of this lane's first column
  const int64_t st = (int64_t)K * RX;
  for (int64_t a = t0 >> lg; a < total; a += ng) {
    int64_t pi = a;
    if (mode == kResActive && total < sd.N) {
      const int q = active_slot(as.arow, nact, a);
      pi = as.inst_off[as.ai[q]] + (a - as.arow[q]);
    }
    const int64_t i = sd.perm[pi];
    const bool zero = mode == kResZeroStopped && !as.act[sd.row_inst[i]];
    const int64_t* ptr = TRANS ? sd.at_ptr : sd.row_ptr;
    const int32_t* idx = TRANS ? sd.at_prow : sd.pcol;
    const int64_t e0 = ptr[i], e1 = ptr[i + 1];
    const double di = D[i];
    int k = kl, r = rl;
    for (int q = l; q < KR; q += gl) {
      if (q != l) {
        k = q / R;
        r = q - k * R;
      }
      const double* Xq = X + (int64_t)k * RX + r;
      double s = 0.0;
      if (!zero) {
        s = b[i * R + r] - sh.t[k] * di * Xq[pi * st];
        int64_t e = e0;
        for (; e + 4 <= e1; e += 4) {
          double v[4], x[4];
#pragma unroll
          for (int t = 0; t < 4; ++t) {
            v[t] = TRANS ? vals[sd.at_src[e + t]] : vals[e + t];
            x[t] = Xq[idx[e + t] * st];
          }
#pragma unroll
          for (int t = 0; t < 4; ++t) s -= v[t] * x[t];
        }
        for (; e < e1; ++e) s -= (TRANS ? vals[sd.at_src[e]] : vals[e]) * Xq[idx[e] * st];
      }
      Rk[(pi * K + k) * RV + r] = (T)s;
    }
  }
}

// r[i][c] = b[i][c] - sum_j A_ij x[j][c]  (FP64, original order), warp per row
__global__ void k_residual(SymDev sd, const double* __restrict__ vals, const double* __restrict__ b,
                           const double* __restrict__ x, int R, double* __restrict__ res) {
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= sd.N) return;
  const int64_t e0 = sd.row_ptr[i], e1 = sd.row_ptr[i + 1];
  for (int r = lane; r < R; r += 32) {
    double a = b[i * R + r];
    for (int64_t e = e0; e < e1; ++e) a -= vals[e] * x[(int64_t)sd.col[e] * R + r];
    res[i * R + r] = a;
  }
}

// ---- adaptive FP64 residual sweeps -----------------------------------------
// After the correction solves of sweep s, every instance g still iterating
// takes its correction, X += Y (FP64, one addition per entry: the sum the
// backward solve's accumulation would form), and gets the size of the
// correction d_s and of the new solution, per right-hand side r:
//   dmax[g][r] = max over its rows i and over k of |Y[pi][k][r]|,
//   xmax[g][r] = max over its rows i and over k of |X[pi][k][r]|.
// CTAs stride over chunks of kStatRows rows of the active set.  Within an
// instance the rows' (i, k) pairs form a matrix of R columns: thread t keeps
// column c = t % RB of a pass (RB = min(R, 256)) and every (256/RB)-th pair,
// so a warp's loads are contiguous; the per-column maxima meet in shared
// memory and then in one
// 64-bit atomicMax per (g, r) on the bit patterns (non-negative doubles
// order as their bit patterns, and a NaN orders above +inf, so a NaN never
// reads as converged).
constexpr int kStatThreads = 256;
constexpr int kStatRows = 64;

template <typename T>
__global__ void __launch_bounds__(kStatThreads)
k_refine_stats(SymDev sd, ActiveSet as, double* __restrict__ X, const T* __restrict__ Y, int K, int R, int RX, int RV,
               unsigned long long* __restrict__ dmax, unsigned long long* __restrict__ xmax) {
  __shared__ unsigned long long s_d[kStatThreads], s_x[kStatThreads];
  const int nact = *as.nact;
  const int64_t total = as.arow[nact];
  const int tid = threadIdx.x;
  const int RB = min(R, kStatThreads);
  const int nj = kStatThreads / RB;
  const int c = tid % RB, j = tid / RB;
  for (int64_t a0 = (int64_t)blockIdx.x * kStatRows; a0 < total; a0 += (int64_t)gridDim.x * kStatRows) {
    const int64_t a1 = min(total, a0 + kStatRows);
    // the instances overlapping active rows [a0, a1), in order (CTA-uniform)
    int q = active_slot(as.arow, nact, a0);
    for (;; ++q) {
      const int g = as.ai[q];
      const int64_t s0 = as.arow[q], s1 = as.arow[q + 1];
      const int64_t lo = max(a0, s0), hi = min(a1, s1);
      if (lo < hi) {
        // the instance's permuted rows are its original range: its (row, k)
        // pairs from i0 on are contiguous in X and Y
        const int64_t i0 = as.inst_off[g] + (lo - s0);
        const int64_t npair = (hi - lo) * K;
        for (int rb = 0; rb < R; rb += RB) {
          const int r = rb + c;
          unsigned long long md = 0, mx = 0;
          if (j < nj && r < R) {
            for (int64_t m = j; m < npair; m += nj) {
              const int64_t o = (i0 * K + m) * RX + r;
              const double y = (double)Y[(i0 * K + m) * RV + r];
              const double xn = X[o] + y;
              X[o] = xn;
              md = max(md, (unsigned long long)__double_as_longlong(fabs(y)));
              mx = max(mx, (unsigned long long)__double_as_longlong(fabs(xn)));
            }
          }
          s_d[tid] = md;
          s_x[tid] = mx;
          __syncthreads();
          if (j == 0 && r < R) {
            for (int t = 1; t < nj; ++t) {
              md = max(md, s_d[t * RB + c]);
              mx = max(mx, s_x[t * RB + c]);
            }
            atomicMax(dmax + (int64_t)g * R + r, md);
            atomicMax(xmax + (int64_t)g * R + r, mx);
          }
          __syncthreads();
        }
      }
      if (s1 >= a1) break;
    }
  }
}

// Exclusive prefix sum over the 1024 threads of a CTA (every thread calls);
// total = the sum of all v.
constexpr int kDecideThreads = 1024;

template <typename V>
__device__ V block_excl_scan(V v, V* sh, V& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  V x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const V y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[w] = x;
  __syncthreads();
  if (w == 0) {
    V y = sh[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const V z = __shfl_up_sync(kFull, y, o);
      if (lane >= o) y += z;
    }
    sh[lane] = y;
  }
  __syncthreads();
  total = sh[31];
  const V r = x - v + (w > 0 ? sh[w - 1] : V(0));
  __syncthreads();  // sh is reused by the next scan
  return r;
}

// One CTA, after sweep s = *sweep + 1 (the count of sweeps done is kept on
// the device, so that the same launch serves every sweep of a device-side
// loop).  For each instance g still iterating: the stopping test of
// extra-precise iterative refinement (Demmel, Hida, Kahan, Li, Mukherjee,
// Riedy, ACM TOMS 2006), with the contraction per sweep estimated from two
// successive corrections, so from the second sweep on.  Per right-hand side,
// rho = |d_s| / |d_{s-1}|: converged when |d_s| = 0, or (s >= 2) when rho <
// 1/2 and rho / (1 - rho) |d_s| <= tol |x| (the error that a contraction by
// rho per sweep leaves); stagnating when rho >= 1/2 (s >= 2: further sweeps
// no longer reduce the error).  After the first sweep only |d_1| = 0 stops:
// |d_1| / |x| is the first solve's error, which can understate the
// contraction by orders of magnitude.  The instance stops when every
// right-hand side has converged or stagnated, or after sweep S; nsw[g] = the
// sweeps it took.  dmax / xmax are zeroed for the next sweep.  Then the
// active set: pre[g] = the active instances before g (pre[G] = their number =
// *nact), ai and arow as in ActiveSet.  With a conditional handle (the sweeps
// as a device-side loop) the loop goes on while an instance is active and s <
// S: at most S sweeps whatever the data.
__global__ void __launch_bounds__(kDecideThreads)
k_refine_decide(int G, int R, double tol, int S, int* __restrict__ sweep, cudaGraphConditionalHandle cond,
                int has_cond, uint8_t* __restrict__ act, unsigned long long* __restrict__ dmax,
                unsigned long long* __restrict__ xmax, double* __restrict__ prevd, int* __restrict__ nsw,
                int* __restrict__ pre, int* __restrict__ nact, int* __restrict__ ai, int64_t* __restrict__ arow,
                const int64_t* __restrict__ inst_off) {
  __shared__ int sh[32];
  __shared__ long long sh64[32];
  const int s = *sweep + 1;
  const bool last = s >= S;
  for (int g = threadIdx.x; g < G; g += kDecideThreads) {
    if (!act[g]) continue;
    bool all = true;
    for (int r = 0; r < R; ++r) {
      const int64_t q = (int64_t)g * R + r;
      const double d = __longlong_as_double((long long)dmax[q]);
      const double x = __longlong_as_double((long long)xmax[q]);
      dmax[q] = 0;
      xmax[q] = 0;
      const double p = prevd[q];
      prevd[q] = d;
      bool done_r = d == 0.0;
      if (!done_r && s >= 2) {
        const double rho = d / p;  // NaN: neither test holds
        done_r = rho < 0.5 ? rho / (1.0 - rho) * d <= tol * x : rho >= 0.5;
      }
      all = all && done_r;
    }
    if (all || last) {
      act[g] = 0;
      nsw[g] = s;
    }
  }
  __syncthreads();
  const int64_t per = ((int64_t)G + kDecideThreads - 1) / kDecideThreads;
  const int64_t b = min((int64_t)G, (int64_t)threadIdx.x * per), e = min((int64_t)G, b + per);
  int c = 0;
  long long rows = 0;
  for (int64_t g = b; g < e; ++g)
    if (act[g]) {
      ++c;
      rows += inst_off[g + 1] - inst_off[g];
    }
  int total;
  long long total_rows;
  int o = block_excl_scan<int>(c, sh, total);
  long long ro = block_excl_scan<long long>(rows, sh64, total_rows);
  for (int64_t g = b; g < e; ++g) {
    pre[g] = o;
    if (act[g]) {
      ai[o] = (int)g;
      arow[o] = ro;
      ++o;
      ro += inst_off[g + 1] - inst_off[g];
    }
  }
  if (threadIdx.x == 0) {
    pre[G] = total;
    *nact = total;
    arow[total] = total_rows;
    *sweep = s;
    if (has_cond) cudaGraphSetConditional(cond, (!last && total > 0) ? 1u : 0u);
  }
}

// Every instance active before the first sweep: act = 1, pre[g] = g,
// *nact = G, ai[g] = g, arow = inst_off, no sweep done yet.
__global__ void k_refine_init(int G, uint8_t* __restrict__ act, int* __restrict__ pre, int* __restrict__ nact,
                              int* __restrict__ ai, int64_t* __restrict__ arow, const int64_t* __restrict__ inst_off,
                              int* __restrict__ sweep) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g < G) {
    act[g] = 1;
    ai[g] = g;
  }
  if (g <= G) {
    pre[g] = g;
    arow[g] = inst_off[g];
  }
  if (g == 0) {
    *nact = G;
    *sweep = 0;
  }
}

// In-order compaction of the persistent solves' unit lists (blockIdx.y = 0:
// forward, 1: backward) to the units whose instance range [rng.x, rng.y]
// holds an active instance (pre = running count of active instances), in two
// launches: CTA c counts its kCompactThreads units, then writes them at the
// sum of the counts of CTAs 0..c-1; the last CTA stores the length.
constexpr int kCompactThreads = 256;

__device__ __forceinline__ bool unit_active(const int2* rng, int n, int u, const int* pre) {
  return u < n && pre[rng[u].y + 1] > pre[rng[u].x];
}

__global__ void __launch_bounds__(kCompactThreads)
k_compact_count(const int2* __restrict__ rf, int nf, const int2* __restrict__ rb, int nb, const int* __restrict__ pre,
                int* __restrict__ cnt) {
  const int y = blockIdx.y;
  const int u = blockIdx.x * kCompactThreads + threadIdx.x;
  const int c = __syncthreads_count(unit_active(y ? rb : rf, y ? nb : nf, u, pre));
  if (threadIdx.x == 0) cnt[y * gridDim.x + blockIdx.x] = c;
}

__global__ void __launch_bounds__(kCompactThreads)
k_compact_write(const SolveUnit* __restrict__ uf, const int2* __restrict__ rf, int nf, SolveUnit* __restrict__ cf,
                const SolveUnit* __restrict__ ub, const int2* __restrict__ rb, int nb, SolveUnit* __restrict__ cb,
                const int* __restrict__ pre, const int* __restrict__ cnt, int* __restrict__ ucount) {
  __shared__ int s_part[kCompactThreads / 32], s_keep[kCompactThreads / 32];
  const int y = blockIdx.y;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // offset of this CTA: the kept units of the CTAs before it
  int part = 0;
  for (int c = threadIdx.x; c < (int)blockIdx.x; c += kCompactThreads) part += cnt[y * gridDim.x + c];
  part = __reduce_add_sync(kFull, part);
  const int u = blockIdx.x * kCompactThreads + threadIdx.x;
  const bool keep = unit_active(y ? rb : rf, y ? nb : nf, u, pre);
  const unsigned bal = __ballot_sync(kFull, keep);
  if (lane == 0) {
    s_part[w] = part;
    s_keep[w] = __popc(bal);
  }
  __syncthreads();
  int off = 0, before = 0, kept = 0;
  for (int q = 0; q < kCompactThreads / 32; ++q) {
    off += s_part[q];
    if (q < w) before += s_keep[q];
    kept += s_keep[q];
  }
  if (keep) {
    const int o = off + before + __popc(bal & ((1u << lane) - 1u));
    (y ? cb : cf)[o] = (y ? ub : uf)[u];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) ucount[y] = off + kept;
}

__global__ void k_axpy(int64_t n, const double* __restrict__ y, double* __restrict__ x) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) x[q] += y[q];
}

// grad[e] = - sum_k w_k sum_r Lam[pi][k][r] X[pj][k][r] for entry e = (i, j)
__global__ void k_grad_values(SymDev sd, const double* __restrict__ Lam,
                              const double* __restrict__ X, Shifts sh, int R, int RX,
                              double* __restrict__ grad) {
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (i >= sd.N) return;
  const int K = sh.K;
  const int KR = K * R;
  const int64_t pi = sd.iperm[i];
  const int64_t e0 = sd.row_ptr[i], e1 = sd.row_ptr[i + 1];
  for (int64_t eb = e0; eb < e1; eb += 32) {
    // permuted columns of up to 32 entries loaded at once, one per lane
    const int ne = (int)min((int64_t)32, e1 - eb);
    const int64_t pjl = lane < ne ? (int64_t)sd.iperm[sd.col[eb + lane]] : 0;
    for (int e = 0; e < ne; ++e) {
      const int64_t pj = __shfl_sync(0xffffffffu, pjl, e);
      double a = 0.0;
      for (int q = lane; q < KR; q += 32) {
        const int k = q / R;
        const int o = k * RX + (q - k * R);
        a += sh.w[k] * Lam[pi * K * RX + o] * X[pj * K * RX + o];
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) grad[eb + e] = -a;
    }
  }
}

__global__ void k_fill_nan_failed(SymDev sd, const int32_t* __restrict__ status, int K, int R,
                                  double* __restrict__ x) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= sd.N * R) return;
  const int g = sd.row_inst[q / R];
  int bad = 0;
  for (int k = 0; k < K; ++k) bad |= status[g * K + k];
  if (bad) x[q] = __longlong_as_double(0x7ff8000000000000LL);
}

inline unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// SMs of the current device (read once per device)
unsigned sm_count() {
  static std::atomic<int> nsm_dev[kMaxDevices];
  const int dev = current_device();
  int nsm = nsm_dev[dev].load(std::memory_order_acquire);
  if (!nsm) {
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    nsm = std::max(nsm, 1);
    nsm_dev[dev].store(nsm, std::memory_order_release);
  }
  return (unsigned)nsm;
}

}  // namespace

// The kernels hold no vector of a whole front; these are the widths accepted when
// they held one in 96 KB of shared memory, and no wider front has been run since.
int max_solve_front(int precision) { return precision == PISP_FP32 ? 24576 : 12288; }

int launch_combine(const SymDev& sd, const double* X, const Shifts& sh, int32_t R, double* x,
                   cudaStream_t st) {
  const int64_t n = sd.N * R;
  if (n == 0) return 0;
  k_combine<<<blocks_for(n, 256), 256, 0, st>>>(sd, X, sh, R, rhs_stride64(R), x);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

namespace {
template <typename T, bool TRANS>
int residual_impl(const SymDev& sd, const double* vals, const double* D, const Shifts& sh, const double* b,
                  const double* X, int32_t R, void* Rk, const ActiveSet& as, int mode, cudaStream_t st) {
  if (sd.N == 0) return 0;
  int lg = 0;
  while (lg < 5 && (1 << lg) < sh.K * R) ++lg;
  const int precision = sizeof(T) == 4 ? PISP_FP32 : PISP_FP64;
  unsigned grid = blocks_for(sd.N << lg, 256);
  if (mode == kResActive) grid = std::min<unsigned>(grid, 16u * sm_count());  // rows known on the device only
  k_residual_per_k<T, TRANS><<<grid, 256, 0, st>>>(sd, vals, D, sh, b, X, R, rhs_stride64(R),
                                                   rhs_stride(precision, R), lg, (T*)Rk, as, mode);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}
}  // namespace

int launch_residual_per_k(int precision, const SymDev& sd, const double* vals, const double* D,
                          const Shifts& sh, const double* b, const double* X, int32_t R,
                          void* Rk, const ActiveSet& as, int mode, cudaStream_t st) {
  if (precision == PISP_FP32) return residual_impl<float, false>(sd, vals, D, sh, b, X, R, Rk, as, mode, st);
  return residual_impl<double, false>(sd, vals, D, sh, b, X, R, Rk, as, mode, st);
}

int launch_refine_stats(int precision, const SymDev& sd, const ActiveSet& as, double* X, const void* Y, int32_t K,
                        int32_t R, unsigned long long* dmax, unsigned long long* xmax, cudaStream_t st) {
  if (sd.N == 0 || R < 1) return 0;
  const unsigned grid = std::min<unsigned>((unsigned)((sd.N + kStatRows - 1) / kStatRows), 32u * sm_count());
  const int RX = rhs_stride64(R), RV = rhs_stride(precision, R);
  if (precision == PISP_FP32)
    k_refine_stats<float><<<grid, kStatThreads, 0, st>>>(sd, as, X, (const float*)Y, K, R, RX, RV, dmax, xmax);
  else
    k_refine_stats<double><<<grid, kStatThreads, 0, st>>>(sd, as, X, (const double*)Y, K, R, RX, RV, dmax, xmax);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_refine_decide(int32_t G, int32_t R, double tol, int32_t S, int32_t* sweep,
                         cudaGraphConditionalHandle cond, int has_cond, uint8_t* act, unsigned long long* dmax,
                         unsigned long long* xmax, double* prevd, int32_t* nsw, int32_t* pre, int32_t* nact,
                         int32_t* ai, int64_t* arow, const int64_t* inst_off, cudaStream_t st) {
  if (G < 1) return 0;
  k_refine_decide<<<1, kDecideThreads, 0, st>>>(G, R, tol, S, sweep, cond, has_cond, act, dmax, xmax, prevd, nsw,
                                                pre, nact, ai, arow, inst_off);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_refine_init(int32_t G, uint8_t* act, int32_t* pre, int32_t* nact, int32_t* ai, int64_t* arow,
                       const int64_t* inst_off, int32_t* sweep, cudaStream_t st) {
  if (G < 1) return 0;
  k_refine_init<<<blocks_for((int64_t)G + 1, 256), 256, 0, st>>>(G, act, pre, nact, ai, arow, inst_off, sweep);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int compact_scratch(int32_t nf, int32_t nb) {
  return 2 * (int)((std::max(nf, nb) + kCompactThreads - 1) / kCompactThreads);
}

int launch_compact_units(const SolveUnit* uf, const int32_t* rf, int32_t nf, SolveUnit* cf, const SolveUnit* ub,
                         const int32_t* rb, int32_t nb, SolveUnit* cb, const int32_t* pre, int32_t* cnt,
                         int32_t* ucount, cudaStream_t st) {
  const int gx = compact_scratch(nf, nb) / 2;
  if (gx == 0) return 0;
  const dim3 grid(gx, 2);
  const int2* f2 = reinterpret_cast<const int2*>(rf);
  const int2* b2 = reinterpret_cast<const int2*>(rb);
  k_compact_count<<<grid, kCompactThreads, 0, st>>>(f2, nf, b2, nb, pre, cnt);
  if (cudaGetLastError() != cudaSuccess) return -1;
  k_compact_write<<<grid, kCompactThreads, 0, st>>>(uf, f2, nf, cf, ub, b2, nb, cb, pre, cnt, ucount);
  return cudaGetLastError() == cudaSuccess ? 2 : -1;
}

int launch_residual_T_per_k(int precision, const SymDev& sd, const double* vals, const double* D,
                            const Shifts& sh, const double* g, const double* Lam, int32_t R,
                            void* Rk, cudaStream_t st) {
  const ActiveSet none{};
  if (precision == PISP_FP32) return residual_impl<float, true>(sd, vals, D, sh, g, Lam, R, Rk, none, kResAll, st);
  return residual_impl<double, true>(sd, vals, D, sh, g, Lam, R, Rk, none, kResAll, st);
}

int launch_residual(const SymDev& sd, const double* vals, const double* b, const double* x,
                    int32_t R, double* r, cudaStream_t st) {
  if (sd.N == 0) return 0;
  k_residual<<<blocks_for(sd.N * 32, 256), 256, 0, st>>>(sd, vals, b, x, R, r);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_axpy(int64_t n, const double* y, double* x, cudaStream_t st) {
  if (n == 0) return 0;
  k_axpy<<<blocks_for(n, 256), 256, 0, st>>>(n, y, x);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_grad_values(const SymDev& sd, const double* Lam, const double* X, const Shifts& sh,
                       int32_t R, double* grad, cudaStream_t st) {
  if (sd.N == 0) return 0;
  k_grad_values<<<blocks_for(sd.N * 32, 256), 256, 0, st>>>(sd, Lam, X, sh, R, rhs_stride64(R), grad);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_fill_nan_failed(const SymDev& sd, const int32_t* status, int32_t K, int32_t R,
                           double* x, cudaStream_t st) {
  const int64_t n = sd.N * R;
  if (n == 0) return 0;
  k_fill_nan_failed<<<blocks_for(n, 256), 256, 0, st>>>(sd, status, K, R, x);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace pisp
