// FP64 solution of the generalized eigenproblem of Eq. 2,
//     sum_mn (H - E S) C = 0,
// for the eigenvalues inside an energy window, on the device:
//   1. Cholesky S = L L^T (blocked, right-looking, 32-wide panels with inverted
//      diagonal blocks) and, in the same sweep, X = L^-1 H;
//   2. A = L^-1 X^T, on and above the diagonal;
//   3. Householder reduction of A to a symmetric tridiagonal T (d, e);
//   4. Sturm-sequence counts and bisection on T, one thread per wanted
//      eigenvalue index.
// The paper solves this step with LAPACK on one CPU (Sec. II); this is a
// GPU route to the same numbers in the same (FP64) arithmetic.  The pivot
// check of step 1 reports a non-positive-definite S (OFM_ERR_NOT_POSDEF).
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

#include "fp64_util.h"
#include "ofm_internal.h"

namespace ofm {

constexpr int NB = 32;

// ------------------------------------------ Cholesky and reduction to A ------
//
// In blocks of NB rows.  With Q_j = L_jj^-1, block column j of the factor and
// block row j of X = L^-1 H come from the same two launches:
//   panel:  L_ij = S_ij Q_j^T (i > j),        X_j = Q_j H_j;
//   update: S_ik -= L_ij L_kj^T (i >= k > j), H_i -= L_ij X_j (i > j),
// and the CTA that updates the next diagonal block goes on to factor and invert
// it while the other CTAs work on the rest of the update.  The second half,
// A = L^-1 X^T, forms only the blocks on and above the diagonal (A_jc, c >= j,
// needs A_kc with k < j <= c only) and mirrors them: a third of the work of the
// full solve, one launch per block row, whose CTAs on row j + 1 multiply by
// Q_{j+1} right after their update.
// The panel's products with the explicit inverse are followed by one step of refinement
// against L_jj, Y += Q (B - L Y) (the last block's and the second half's need none; 11
// us a panel at n = 992).  Mean error of the levels against 60-digit arithmetic, n =
// 40 and 72, conditions of S of 1e4 to 1e10, relative to substitutions on the host:
// 2.3 without the step (3.1 at worst), 1.5 with it, 1.2 with substitutions here too
// (the rest is the square-root-free elimination of the diagonal blocks).
//
// FP64 issue bounds all of it (one warp instruction per 17 cycles and SM), so an
// item is a 32 x 16 strip, 512 of them (4.3 us), handed out by a counter to one
// CTA per SM, the next item's operands on their way while one is computed; one
// CTA per SM keeps the pipe of the factoring CTA free of other CTAs' work.
// n = 992: 1.95 (Cholesky) + 2.42 ms with substitutions, separate sweeps and
// the full second solve; 1.89 (factor and X) + 0.68 now.  n = 315: 0.58 + 0.35 ms;
// 0.36 + 0.14 now.

constexpr int ST_C = 16;               // columns of a strip
constexpr int ST_THREADS = 256;
constexpr size_t ST_SMEM = 120 * 1024; // more than half an SM's shared memory: one CTA per SM

struct StepSmem {
  double li[2][NB][NB + 1];   // L_ij of the item, double-buffered
  double b[2][NB][ST_C + 1];  // the strip of L_kj^T, X_j or A_j
  double q[NB][NB + 1];       // Q of the next diagonal block, or the block being factored
  double t[NB][NB + 1];       // a strip on its way through Q; unscaled columns of L
  double g[2][NB], h[2][NB], piv[NB];
  int item;
};
static_assert(sizeof(StepSmem) <= ST_SMEM, "strip buffers fit");

// Eight bytes into shared memory, asynchronously; zeros where !ok.
__device__ __forceinline__ void cpa8z(double* dst, const double* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"((unsigned long long)__cvta_generic_to_global(src)), "r"(ok ? 8 : 0)
               : "memory");
}

__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// 32 x 32 block at (r0, k0) of an n x n matrix into d.
__device__ __forceinline__ void fetch_block(double (*d)[NB + 1], const double* M, int n, int r0, int k0) {
  for (int e = threadIdx.x; e < NB * NB; e += ST_THREADS) {
    const int r = e >> 5, c = e & 31;
    const bool ok = r0 + r < n && k0 + c < n;
    cpa8z(&d[r][c], ok ? M + (size_t)(r0 + r) * n + k0 + c : M, ok);
  }
}
// strip d[t][c] = M(k0 + t, c0 + c), or M(c0 + c, k0 + t) when transposed
template <bool TR>
__device__ __forceinline__ void fetch_strip(double (*d)[ST_C + 1], const double* M, int n, int k0, int c0) {
  for (int e = threadIdx.x; e < NB * ST_C; e += ST_THREADS) {
    const int t = TR ? e & 31 : e >> 4, c = TR ? e >> 5 : e & 15;
    const bool ok = k0 + t < n && c0 + c < n;
    cpa8z(&d[t][c], ok ? (TR ? M + (size_t)(c0 + c) * n + k0 + t : M + (size_t)(k0 + t) * n + c0 + c) : M, ok);
  }
}

// Factor the symmetric block a (identity beyond kb) as L L^T and invert L, in
// one elimination without square roots: row y > j takes -(a_yj / d_j) times row
// j, whose entries left of j hold the inverse of the unit factor so far; the
// scaling by d^-1/2 follows for all columns at once.  A column costs one barrier
// and the chain update - reciprocal - scaling of the next pivot row, which warp 0
// works on with an FP64 sub-partition to itself (warp 4, its neighbour there, only
// waits).  The six warps on the others own the rows and hand row j + 2 over while
// warp 0 works on row j + 1.  Eight warps taking turns as the next pivot's
// owner, each step waiting for its neighbour's updates: 27 us a block; now 23.
__device__ void factor_block(StepSmem& sm, double (*a)[NB + 1], int kb, double* W, double* Qj, int n, int k0,
                             int* fail_col) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int own = warp == 0 || warp == 4 ? -1 : warp - (warp > 4 ? 2 : 1);   // 0..5: rows own, own + 6, ..
  double v[6];
  if (own >= 0)
#pragma unroll
    for (int q = 0; q < 6; ++q) v[q] = own + 6 * q < NB ? a[own + 6 * q][lane] : 0.0;
  // row y: subtract a_yj times the published row; column j turns into the inverse's
  auto update = [&](double row, double gx, int y, int j) {
    const double ay = __shfl_sync(0xffffffffu, row, j);
    if (lane == j) sm.t[y][j] = ay;
    return fma(-ay, gx, lane == j ? 0.0 : row);
  };
  auto publish = [&](double row, int j) {   // row j, all updates in
    double p = __shfl_sync(0xffffffffu, row, j);
    if (!(p > 0.0)) {
      if (lane == 0) atomicCAS(fail_col, -1, k0 + j);
      p = 1.0;   // keep going with finite numbers; the call reports failure
    }
    const double r = rcp64(p);
    sm.g[j & 1][lane] = lane == j ? r : row * r;
    if (lane == j) sm.piv[j] = p;
    a[j][lane] = row;
  };
  __syncthreads();   // the rows are in registers; a takes the finished ones
  if (warp == 0) publish(a[0][lane], 0);
  if (own == 1) sm.h[0][lane] = v[0];   // row 1 before any update
  __syncthreads();
  for (int j = 0; j + 1 < NB; ++j) {
    const double gx = sm.g[j & 1][lane];
    if (warp == 0) {
      publish(update(sm.h[j & 1][lane], gx, j + 1, j), j + 1);
    } else if (own >= 0) {
      const int y2 = j + 2;
#pragma unroll
      for (int q = 0; q < 6; ++q)
        if (own + 6 * q == y2 && y2 < NB) {
          v[q] = update(v[q], gx, y2, j);
          sm.h[(j + 1) & 1][lane] = v[q];
        }
#pragma unroll
      for (int q = 0; q < 6; ++q)
        if (own + 6 * q > y2 && own + 6 * q < NB) v[q] = update(v[q], gx, own + 6 * q, j);
    }
    __syncthreads();
  }
  const double d = sm.piv[lane], rs = rsqrt64(d);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int y = warp + 8 * q;
    const double ry = __shfl_sync(0xffffffffu, rs, y);
    Qj[y * NB + lane] = lane < y ? a[y][lane] * ry : lane == y ? ry : 0.0;
    if (y < kb && lane <= y)
      W[(size_t)(k0 + y) * n + k0 + lane] = lane < y ? sm.t[y][lane] * rs : d * rs;
  }
}

// acc of rows row and row + 16 (both at column col): sum over t of l[.][t] b[t][col]
__device__ __forceinline__ void strip_product(const double (*l)[NB + 1], const double (*b)[ST_C + 1], int row,
                                              int col, double& a0, double& a1) {
  a0 = a1 = 0.0;
#pragma unroll 8
  for (int t = 0; t < NB; ++t) {
    const double x = b[t][col];
    a0 = fma(l[row][t], x, a0);
    a1 = fma(l[row + 16][t], x, a1);
  }
}

// Rows row and row + 16 of the product of a lower triangular block with a strip.
__device__ __forceinline__ void lower_product(const double (*l)[NB + 1], const double (*b)[9], int row, int col,
                                              double& a0, double& a1) {
  a0 = a1 = 0.0;
#pragma unroll
  for (int t = 0; t < 16; ++t) {
    a0 = fma(l[row][t], b[t][col], a0);
    a1 = fma(l[row + 16][t], b[t][col], a1);
  }
#pragma unroll
  for (int t = 16; t < NB; ++t) a1 = fma(l[row + 16][t], b[t][col], a1);
}

// Diagonal block L_jj (zero above the diagonal, identity beyond the matrix).
__device__ __forceinline__ void load_diagonal(double (*d)[NB + 1], const double* L, int n, int k0) {
  for (int e = threadIdx.x; e < NB * NB; e += 128) {
    const int r = e >> 5, c = e & 31;
    d[r][c] = c <= r && k0 + r < n ? L[(size_t)(k0 + r) * n + k0 + c] : r == c ? 1.0 : 0.0;
  }
}

// Panel of block j: strips of eight rows of S_ij, then strips of eight columns
// of H_j, each multiplied by Q_j (lower triangular) in place, and refined but for the
// last block.
__global__ void __launch_bounds__(128) panel_kernel(double* W, double* B, const double* __restrict__ Q, int n,
                                                    int j) {
  __shared__ double q[NB][NB + 1], l[NB][NB + 1], b[NB][9];
  const int k0 = j * NB, below = n - k0 - NB, nl = below > 0 ? (below + 7) / 8 : 0;
  const bool isl = (int)blockIdx.x < nl;
  const int x0 = isl ? k0 + NB + 8 * blockIdx.x : 8 * (blockIdx.x - nl);
  for (int e = threadIdx.x; e < NB * NB; e += 128) q[e >> 5][e & 31] = Q[(size_t)j * NB * NB + e];
  if (below > 0) load_diagonal(l, W, n, k0);
  for (int e = threadIdx.x; e < NB * 8; e += 128) {
    const int t = isl ? e & 31 : e >> 3, c = isl ? e >> 5 : e & 7;
    const bool ok = k0 + t < n && x0 + c < n;
    b[t][c] = !ok ? 0.0 : isl ? W[(size_t)(x0 + c) * n + k0 + t] : B[(size_t)(k0 + t) * n + x0 + c];
  }
  __syncthreads();
  const int col = threadIdx.x & 7, row = threadIdx.x >> 3;
  const double s0 = b[row][col], s1 = b[row + 16][col];
  double a0, a1;
  lower_product(q, b, row, col, a0, a1);
  if (below > 0) {   // uniform
    double r0, r1;
    __syncthreads();
    b[row][col] = a0;
    b[row + 16][col] = a1;
    __syncthreads();
    lower_product(l, b, row, col, r0, r1);
    __syncthreads();
    b[row][col] = s0 - r0;
    b[row + 16][col] = s1 - r1;
    __syncthreads();
    lower_product(q, b, row, col, r0, r1);
    a0 += r0;
    a1 += r1;
  }
  if (x0 + col >= n) return;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = k0 + row + 16 * u;
    if (r >= n) continue;
    const double v = u ? a1 : a0;
    if (isl) W[(size_t)(x0 + col) * n + r] = v;
    else B[(size_t)r * n + x0 + col] = v;
  }
}

// Takes the CTA's next item (a uniform value; -1 when none is left).
__device__ __forceinline__ int claim(StepSmem& sm, int* next, int total) {
  __syncthreads();
  if (threadIdx.x == 0) {
    const int t = atomicAdd(next, 1);
    sm.item = t < total ? t : -1;
  }
  __syncthreads();
  return sm.item;
}

// Update after panel j; CTA 0 first updates, factors and inverts block j + 1
// (j = -1: factors block 0, with nothing to update).
__global__ void __launch_bounds__(ST_THREADS) factor_step_kernel(double* W, double* B, double* Q, int n, int j,
                                                                 int* next, int* fail_col) {
  extern __shared__ __align__(16) unsigned char raw[];
  StepSmem& sm = *reinterpret_cast<StepSmem*>(raw);
  const int nblk = (n + NB - 1) / NB, nstr = (n + ST_C - 1) / ST_C;
  const int R = nblk - 1 - j, k0 = j * NB, i0 = k0 + NB;
  const int tid = threadIdx.x, col = tid & 15, row = tid >> 4;
  if (blockIdx.x == 0) {
    const int kb = min(NB, n - i0);
    if (j >= 0) fetch_block(sm.li[0], W, n, i0, k0);
    cpa_commit();
    cpa_wait<0>();
    __syncthreads();
    for (int e = tid; e < NB * NB; e += ST_THREADS) {
      const int r = e >> 5, c = e & 31;
      double v = r == c ? 1.0 : 0.0;
      if (r < kb && c < kb) {
        v = W[(size_t)(i0 + max(r, c)) * n + i0 + min(r, c)];
        if (j >= 0) {
          double s = 0.0;
#pragma unroll 8
          for (int t = 0; t < NB; ++t) s = fma(sm.li[0][r][t], sm.li[0][c][t], s);
          v -= s;
        }
      }
      sm.q[r][c] = v;
    }
    __syncthreads();
    factor_block(sm, sm.q, kb, W, Q + (size_t)(j + 1) * NB * NB, n, i0, fail_col);
  }
  if (j < 0) return;
  // items: strips of the lower blocks of S but the two of block j + 1, then all of H
  const int ns = R * (R + 1) - 2, total = ns + R * nstr;
  auto place = [&](int t, int& r0, int& c0) {   // returns whether the item is one of S
    if (t < ns) {
      int r = (int)((sqrtf(4.f * (t + 2) + 1.f) - 1.f) * 0.5f);   // r (r + 1) <= t + 2
      while ((r + 1) * (r + 2) <= t + 2) ++r;
      while (r * (r + 1) > t + 2) --r;
      r0 = i0 + NB * r;
      c0 = i0 + ST_C * (t + 2 - r * (r + 1));
      return true;
    }
    const int r = (t - ns) / nstr;
    r0 = i0 + NB * r;
    c0 = ST_C * (t - ns - r * nstr);
    return false;
  };
  auto fetch = [&](int t, int buf) {
    if (t >= 0) {
      int r0, c0;
      const bool s = place(t, r0, c0);
      fetch_block(sm.li[buf], W, n, r0, k0);
      if (s) fetch_strip<true>(sm.b[buf], W, n, k0, c0);
      else fetch_strip<false>(sm.b[buf], B, n, k0, c0);
    }
    cpa_commit();
  };
  int cur = claim(sm, next, total), buf = 0;
  fetch(cur, 0);
  while (cur >= 0) {
    const int nxt = claim(sm, next, total);
    fetch(nxt, buf ^ 1);
    cpa_wait<1>();
    __syncthreads();
    int r0, c0;
    double* M = place(cur, r0, c0) ? W : B;
    double* o0 = M + (size_t)(r0 + row) * n + c0 + col;
    double* o1 = o0 + (size_t)16 * n;
    const bool w0 = c0 + col < n && r0 + row < n, w1 = c0 + col < n && r0 + row + 16 < n;
    const double p0 = w0 ? *o0 : 0.0, p1 = w1 ? *o1 : 0.0;
    double a0, a1;
    strip_product(sm.li[buf], sm.b[buf], row, col, a0, a1);
    if (w0) *o0 = p0 - a0;
    if (w1) *o1 = p1 - a1;
    cur = nxt;
    buf ^= 1;
  }
  cpa_wait<0>();
}

// Second half after block row j of A: T_i -= L_ij A_j on and right of the
// diagonal, and A_{j+1} = Q_{j+1} T_{j+1}, written to both triangles of A
// (j = -1: only A_0 = Q_0 T_0).
__global__ void __launch_bounds__(ST_THREADS) reduce_step_kernel(const double* __restrict__ L,
                                                                 const double* __restrict__ Q, double* T,
                                                                 double* A, int n, int j, int* next) {
  extern __shared__ __align__(16) unsigned char raw[];
  StepSmem& sm = *reinterpret_cast<StepSmem*>(raw);
  const int nblk = (n + NB - 1) / NB, nstr = (n + ST_C - 1) / ST_C;
  const int k0 = j * NB, i0 = k0 + NB;
  const int R = j < 0 ? 1 : nblk - 1 - j;      // block rows to update
  const int S0 = nstr - 2 * (j + 1);           // strips of the first; two fewer on each next
  const int tid = threadIdx.x, col = tid & 15, row = tid >> 4;
  const int total = R * S0 - R * (R - 1);
  for (int e = tid; e < NB * NB; e += ST_THREADS) sm.q[e >> 5][e & 31] = Q[(size_t)(j + 1) * NB * NB + e];
  auto place = [&](int t, int& r0, int& c0) {   // r: r S0 - r (r - 1) <= t
    const float h = 0.5f * (S0 + 1);
    int r = (int)(h - sqrtf(fmaxf(h * h - (float)t, 0.f)));
    r = max(0, min(r, R - 1));
    while (r + 1 < R && (r + 1) * S0 - (r + 1) * r <= t) ++r;
    while (r > 0 && r * S0 - r * (r - 1) > t) --r;
    r0 = i0 + NB * r;
    c0 = r0 + ST_C * (t - (r * S0 - r * (r - 1)));
  };
  auto fetch = [&](int t, int buf) {
    if (t >= 0 && j >= 0) {
      int r0, c0;
      place(t, r0, c0);
      fetch_block(sm.li[buf], L, n, r0, k0);
      fetch_strip<false>(sm.b[buf], A, n, k0, c0);
    }
    cpa_commit();
  };
  int cur = claim(sm, next, total), buf = 0;
  fetch(cur, 0);
  while (cur >= 0) {
    const int nxt = claim(sm, next, total);
    fetch(nxt, buf ^ 1);
    cpa_wait<1>();
    __syncthreads();
    int r0, c0;
    place(cur, r0, c0);
    double* o0 = T + (size_t)(r0 + row) * n + c0 + col;
    double* o1 = o0 + (size_t)16 * n;
    const bool w0 = c0 + col < n && r0 + row < n, w1 = c0 + col < n && r0 + row + 16 < n;
    const double p0 = w0 ? *o0 : 0.0, p1 = w1 ? *o1 : 0.0;
    double a0 = 0.0, a1 = 0.0;
    if (j >= 0) strip_product(sm.li[buf], sm.b[buf], row, col, a0, a1);
    a0 = p0 - a0;
    a1 = p1 - a1;
    if (r0 == i0) {
      __syncthreads();   // the strip of A_j is read
      sm.b[buf][row][col] = a0;
      sm.b[buf][row + 16][col] = a1;
      __syncthreads();
      strip_product(sm.q, sm.b[buf], row, col, a0, a1);
      const int c = c0 + col;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int r = r0 + row + 16 * u;
        if (r < n && c < n && c >= r) {
          A[(size_t)r * n + c] = u ? a1 : a0;
          A[(size_t)c * n + r] = u ? a1 : a0;
        }
      }
    } else {
      if (w0) *o0 = a0;
      if (w1) *o1 = a1;
    }
    cur = nxt;
    buf ^= 1;
  }
  cpa_wait<0>();
}

__global__ void transpose_kernel(const double* in, double* out, int n) {
  __shared__ double t[32][33];
  int x = blockIdx.x * 32 + threadIdx.x, y = blockIdx.y * 32 + threadIdx.y;
  if (x < n && y < n) t[threadIdx.y][threadIdx.x] = in[(long long)y * n + x];
  __syncthreads();
  x = blockIdx.y * 32 + threadIdx.x;
  y = blockIdx.x * 32 + threadIdx.y;
  if (x < n && y < n) out[(long long)y * n + x] = t[threadIdx.x][threadIdx.y];
}

// out = (in + in^T) / 2
__global__ void symmetrize_kernel(const double* __restrict__ in, double* __restrict__ out, int n) {
  __shared__ double t[32][33];
  int x = blockIdx.y * 32 + threadIdx.x, y = blockIdx.x * 32 + threadIdx.y;
  if (x < n && y < n) t[threadIdx.y][threadIdx.x] = in[(size_t)y * n + x];
  __syncthreads();
  x = blockIdx.x * 32 + threadIdx.x;
  y = blockIdx.y * 32 + threadIdx.y;
  if (x < n && y < n) out[(size_t)y * n + x] = 0.5 * (in[(size_t)y * n + x] + t[threadIdx.x][threadIdx.y]);
}

// ------------------------------------------------------- tridiagonalise ----

// Householder vector for column k: x = A[k+1:, k]; v = x - alpha e1 with
// alpha = -sign(x0) ||x||, tau = 2 / v^T v.  Stores v in vbuf[k+1:] and in
// A[k+1:, k] (for the back-transformation), d[k], e[k], tau[k].
__global__ void householder_kernel(double* A, int n, int k, double* vbuf, double* d, double* e,
                                   double* tau) {
  __shared__ double red[32];
  const int m = n - k - 1;
  double s = 0.0;
  for (int i = threadIdx.x + 1; i < m; i += blockDim.x) {
    double x = A[(long long)(k + 1 + i) * n + k];
    s += x * x;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) red[0] = s;
  }
  __syncthreads();
  const double sig = red[0];  // ||x[1:]||^2
  const double x0 = A[(long long)(k + 1) * n + k];
  double alpha, t, v0;
  if (sig == 0.0) {
    alpha = x0;
    t = 0.0;
    v0 = 1.0;
  } else {
    const double nrm = sqrt(x0 * x0 + sig);
    alpha = (x0 > 0.0) ? -nrm : nrm;
    v0 = x0 - alpha;
    t = 2.0 / (v0 * v0 + sig);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    double v = (i == 0) ? v0 : A[(long long)(k + 1 + i) * n + k];
    vbuf[k + 1 + i] = v;
    A[(long long)k * n + k + 1 + i] = v;  // row k keeps v for the back-transformation
  }
  if (threadIdx.x == 0) {
    d[k] = A[(long long)k * n + k];
    e[k] = alpha;
    tau[k] = t;
  }
}

// p = tau * A22 v over rows k+1.. (one warp per row).
__global__ void symv_kernel(const double* A, int n, int k, const double* vbuf, const double* tau,
                            double* p) {
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const int i = k + 1 + warp;
  if (i >= n) return;
  const double* row = A + (long long)i * n;
  double s = 0.0;
  for (int j = k + 1 + lane; j < n; j += 32) s += row[j] * vbuf[j];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) p[i] = tau[k] * s;
}

// A22 -= v w^T + w v^T with w = p - (tau/2)(v^T p) v; every CTA forms v^T p
// itself (a short read of two vectors) so the step needs no extra launch.
__global__ void rank2_kernel(double* A, int n, int k, const double* vbuf, const double* p,
                             const double* tau) {
  __shared__ double red[8];
  __shared__ double Ks;
  double s = 0.0;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  for (int j = k + 1 + tid; j < n; j += blockDim.x * blockDim.y) s += vbuf[j] * p[j];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if ((tid & 31) == 0) red[tid >> 5] = s;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x * blockDim.y) / 32; ++w) t += red[w];
    Ks = 0.5 * tau[k] * t;
  }
  __syncthreads();
  const double K = Ks;
  const int i = k + 1 + blockIdx.y * blockDim.y + threadIdx.y;
  const int j0 = k + 1 + blockIdx.x * 64;
  if (i >= n) return;
  const double vi = vbuf[i], wi = p[i] - K * vi;
  for (int jj = threadIdx.x; jj < 64; jj += blockDim.x) {
    const int j = j0 + jj;
    if (j >= n) break;
    const double vj = vbuf[j], wj = p[j] - K * vj;
    A[(long long)i * n + j] -= vi * wj + wi * vj;
  }
}

__global__ void tridiag_tail_kernel(const double* A, int n, double* d, double* e) {
  if (n >= 2) {
    d[n - 2] = A[(long long)(n - 2) * n + n - 2];
    e[n - 2] = A[(long long)(n - 1) * n + n - 2];
  }
  d[n - 1] = A[(long long)(n - 1) * n + n - 1];
}

// ---------------------------------------------------------------- bisection --

// Number of eigenvalues of T below x (negative pivots of T - x I).
__device__ int sturm_count(const double* d, const double* e, int n, double x, double pivmin) {
  int c = 0;
  double q = d[0] - x;
  if (fabs(q) < pivmin) q = -pivmin;
  if (q < 0) ++c;
  for (int j = 1; j < n; ++j) {
    q = d[j] - x - e[j - 1] * e[j - 1] / q;
    if (fabs(q) < pivmin) q = -pivmin;
    if (q < 0) ++c;
  }
  return c;
}

__device__ void gersh(const double* d, const double* e, int n, double* lo, double* hi) {
  double a = DBL_MAX, b = -DBL_MAX;
  for (int j = 0; j < n; ++j) {
    double r = (j > 0 ? fabs(e[j - 1]) : 0.0) + (j < n - 1 ? fabs(e[j]) : 0.0);
    a = fmin(a, d[j] - r);
    b = fmax(b, d[j] + r);
  }
  double w = fmax(fabs(a), fabs(b));
  *lo = a - 2.0 * DBL_EPSILON * w - 1e-300;
  *hi = b + 2.0 * DBL_EPSILON * w + 1e-300;
}

__device__ double pivmin_of(const double* e, int n) {
  double m = 0.0;
  for (int j = 0; j < n - 1; ++j) m = fmax(m, e[j] * e[j]);
  return fmax(DBL_MIN, DBL_MIN * m);
}

__global__ void count_kernel(const double* d, const double* e, int n, double x, int* out) {
  *out = sturm_count(d, e, n, x, pivmin_of(e, n));
}

__global__ void bisect_kernel(const double* d, const double* e, int n, int i_lo, int m, double* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m) return;
  const int idx = i_lo + t;
  double lo, hi;
  gersh(d, e, n, &lo, &hi);
  const double pm = pivmin_of(e, n);
  for (int it = 0; it < 200; ++it) {
    const double mid = 0.5 * (lo + hi);
    if (hi - lo <= 2.0 * DBL_EPSILON * fmax(fabs(lo), fabs(hi)) + 4.0 * DBL_MIN || mid == lo || mid == hi) break;
    if (sturm_count(d, e, n, mid, pm) > idx) hi = mid; else lo = mid;
  }
  out[t] = 0.5 * (lo + hi);
}

}  // namespace ofm

using namespace ofm;

static ofm_status sync_ctx(ofm_ctx* c, const char* what) {
  cudaError_t e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return ofm_cuda_check(c, e, what);
  return OFM_OK;
}

ofm_status ofm_window_factor(ofm_ctx* c) {
  const int n = c->dense_n;
  if (c->fault == OFM_FAULT_NOTPOSDEF) {
    c->window_fail_col = 0;
    return ofm_fail(c, OFM_ERR_NOT_POSDEF, "S is not positive definite: Cholesky pivot 0 is not positive (injected by OFM_FAULT=notposdef)");
  }
  const size_t bytes = sizeof(double) * (size_t)n * n;
  OFM_TRY(ofm_ensure(c, c->w_L, bytes, "window L"));
  OFM_TRY(ofm_ensure(c, c->w_A, bytes, "window A"));
  OFM_TRY(ofm_ensure(c, c->w_d, sizeof(double) * n, "window d"));
  OFM_TRY(ofm_ensure(c, c->w_e, sizeof(double) * n, "window e"));
  OFM_TRY(ofm_ensure(c, c->w_tau, sizeof(double) * n, "window tau"));
  OFM_TRY(ofm_ensure(c, c->w_tmp, sizeof(double) * 2 * n, "window vectors"));
  const int nblk = (n + NB - 1) / NB, nstr = (n + ST_C - 1) / ST_C;
  const size_t qbytes = sizeof(double) * (size_t)nblk * NB * NB;
  OFM_TRY(ofm_ensure(c, c->w_eval, bytes, "window scratch"));
  OFM_TRY(ofm_ensure(c, c->w_Q, qbytes + 2 * sizeof(int) * nblk, "window multipliers"));
  double* L = (double*)c->w_L.p;
  double* A = (double*)c->w_A.p;
  double* T = (double*)c->w_eval.p;
  double* Q = (double*)c->w_Q.p;
  int* next = (int*)((char*)c->w_Q.p + qbytes);   // item counters, one per launch
  int* flag = (int*)c->flag.p;
  cudaStream_t s = c->stream;
  OFM_CUDA(c, cudaFuncSetAttribute(factor_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ST_SMEM));
  OFM_CUDA(c, cudaFuncSetAttribute(reduce_step_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ST_SMEM));
  const int sms = 152;
  OFM_CUDA(c, cudaMemcpyAsync(L, c->dense_S.p, bytes, cudaMemcpyDeviceToDevice, s));
  const dim3 tg((n + 31) / 32, (n + 31) / 32);
  symmetrize_kernel<<<tg, dim3(32, 32), 0, s>>>((const double*)c->dense_H.p, A, n);
  OFM_CUDA(c, cudaMemsetAsync(flag, 0xff, sizeof(int), s));  // -1: no failure
  OFM_CUDA(c, cudaMemsetAsync(next, 0, 2 * sizeof(int) * nblk, s));
  // 1. S = L L^T, and H -> X = L^-1 H in w_A
  {
  KTimer kt(c, KC_CHOL, 2LL * nblk, 0.0, 4.0 / 3.0 * n * n * n);  // n^3/3 of the factor, n^3 of L^-1 H
  factor_step_kernel<<<1, ST_THREADS, ST_SMEM, s>>>(L, A, Q, n, -1, next, flag);
  for (int j = 0; j < nblk; ++j) {
    const int below = std::max(0, n - (j + 1) * NB);
    panel_kernel<<<(below + 7) / 8 + (n + 7) / 8, 128, 0, s>>>(L, A, Q, n, j);
    if (below == 0) break;
    const long long R = nblk - 1 - j, items = R * (R + 1) - 2 + R * nstr;
    factor_step_kernel<<<(int)std::min<long long>(sms, 1 + items), ST_THREADS, ST_SMEM, s>>>(L, A, Q, n, j, next + j,
                                                                                          flag);
  }
  }
  OFM_CUDA(c, cudaGetLastError());
  int fail = -1;
  OFM_CUDA(c, cudaMemcpyAsync(&fail, flag, sizeof(int), cudaMemcpyDeviceToHost, s));
  OFM_TRY(sync_ctx(c, "Cholesky of S"));
  if (fail >= 0) {
    c->window_fail_col = fail;
    char buf[160];
    snprintf(buf, sizeof buf, "S is not positive definite: Cholesky pivot %d is not positive", fail);
    return ofm_fail(c, OFM_ERR_NOT_POSDEF, buf);
  }
  // 2. A = L^-1 X^T, from the blocks on and above its diagonal
  {
  KTimer kt(c, KC_REDUCE, 1 + nblk, 0.0, 1.0 / 3.0 * n * n * n);
  transpose_kernel<<<tg, dim3(32, 32), 0, s>>>(A, T, n);
  for (int j = -1; j + 1 < nblk; ++j) {
    const long long R = j < 0 ? 1 : nblk - 1 - j, S0 = nstr - 2 * (j + 1), items = R * S0 - R * (R - 1);
    reduce_step_kernel<<<(int)std::min<long long>(sms, items), ST_THREADS, ST_SMEM, s>>>(L, Q, T, A, n, j,
                                                                                       next + nblk + j + 1);
  }
  }
  OFM_CUDA(c, cudaGetLastError());
  // 3. tridiagonalise
  double* d = (double*)c->w_d.p;
  double* e = (double*)c->w_e.p;
  double* tau = (double*)c->w_tau.p;
  double* vbuf = (double*)c->w_tmp.p;
  double* p = vbuf + n;
  {
  KTimer kt(c, KC_TRIDIAG, 0, 0.0, 4.0 / 3.0 * n * n * n);  // algorithmic (dsytrd) 4n^3/3 flops
  const ofm_status ps = ofm_tridiag_persistent(c, A, n, d, e, tau, p);
  if (ps == OFM_OK) {
    kt.add(1);
  } else if (ps != OFM_ERR_INVALID) {
    return ps;
  } else {
  kt.add(1 + 3LL * std::max(0, n - 2));
  for (int k = 0; k + 2 < n; ++k) {
    householder_kernel<<<1, 256, 0, s>>>(A, n, k, vbuf, d, e, tau);
    const int m = n - k - 1;
    symv_kernel<<<(m + 7) / 8, 256, 0, s>>>(A, n, k, vbuf, tau, p);
    rank2_kernel<<<dim3((m + 63) / 64, (m + 7) / 8), dim3(32, 8), 0, s>>>(A, n, k, vbuf, p, tau);
  }
  tridiag_tail_kernel<<<1, 1, 0, s>>>(A, n, d, e);
  }
  }
  OFM_CUDA(c, cudaGetLastError());
  OFM_TRY(sync_ctx(c, "tridiagonalisation"));
  c->factored = true;
  return OFM_OK;
}

ofm_status ofm_window_count(ofm_ctx* c, double lo, double hi, int* count_lo, int* count_hi) {
  const double hi_incl = std::nextafter(hi, HUGE_VAL);
  if (2 * (size_t)c->dense_n * sizeof(double) > 200 * 1024)
    return ofm_fail(c, OFM_ERR_INVALID, "dense window solve supports a basis of at most 12800");
  int* dc = (int*)c->flag.p + 2;   // two ints after the pivot flag
  int h[2] = {0, 0};
  KTimer kt(c, KC_BISECT);
  launch_count_below((const double*)c->w_d.p, (const double*)c->w_e.p, c->dense_n, lo, hi_incl, dc,
                     c->stream);
  OFM_CUDA(c, cudaGetLastError());
  OFM_CUDA(c, cudaMemcpyAsync(h, dc, 2 * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  OFM_TRY(sync_ctx(c, "Sturm count"));
  *count_lo = h[0];
  *count_hi = h[1];
  return OFM_OK;
}

// Upper estimate of one past the last index of [E_{i_lo}, E_{i_lo} + width]
// from FP32 counts (a guess; the caller checks it with FP64 eigenvalues).
ofm_status ofm_window_size_estimate(ofm_ctx* c, int i_lo, double width, int* i_end) {
  int* dv = (int*)c->flag.p + 4;   // after the pivot flag and the two counts
  KTimer kt(c, KC_BISECT);
  if (!launch_window_size((const double*)c->w_d.p, (const double*)c->w_e.p, c->dense_n, i_lo,
                          width, dv, c->stream)) {
    *i_end = c->dense_n;   // too long to stage: take everything above i_lo
    return OFM_OK;
  }
  OFM_CUDA(c, cudaGetLastError());
  OFM_CUDA(c, cudaMemcpyAsync(i_end, dv, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  return sync_ctx(c, "window size estimate");
}

ofm_status ofm_window_bisect(ofm_ctx* c, int i_lo, int i_hi, double* E_out) {
  const int m = i_hi - i_lo;
  double* out = (double*)c->w_tmp.p;  // 2n doubles, m <= n
  KTimer kt(c, KC_BISECT);
  if (!launch_multisection((const double*)c->w_d.p, (const double*)c->w_e.p, c->dense_n, i_lo, m,
                           out, c->stream))
    bisect_kernel<<<(m + 127) / 128, 128, 0, c->stream>>>((const double*)c->w_d.p,
                                                          (const double*)c->w_e.p, c->dense_n,
                                                          i_lo, m, out);
  OFM_CUDA(c, cudaGetLastError());
  OFM_CUDA(c, cudaMemcpyAsync(E_out, out, sizeof(double) * m, cudaMemcpyDeviceToHost, c->stream));
  return sync_ctx(c, "bisection");
}
