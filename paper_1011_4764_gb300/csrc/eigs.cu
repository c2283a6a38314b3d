// Batched fragment eigensolver: the lowest n_a eigenpairs of every fragment
// Hamiltonian (Sec. II, "calculation of basis wave functions"; the paper uses
// a preconditioned conjugate-gradient plane-wave solver per fragment).
//
// All fragments advance together through Chebyshev-filtered subspace
// iteration (Zhou, Saad, Tiago and Chelikowsky, "Self-consistent-field
// calculations using Chebyshev-filtered subspace iteration", J. Comput.
// Phys. 219 (2006)):
//   1. X: a block of m_a = n_a + guard vectors per fragment (random start
//      from a counter-based generator, SplitMix64 of Steele, Lea and Flood);
//   2. Y = p(H_a) X, p the degree-d Chebyshev polynomial of the first kind
//      mapped to the unwanted interval [b_lo, b_up] and scaled at the lowest
//      Ritz value (the scaled three-term recurrence; eigblk.cu);
//   3. Rayleigh-Ritz: G = Y^T Y and K = Y^T H Y (eigblk.cu), then per
//      fragment, in the storage precision: diagonal scaling, Cholesky of the
//      scaled G and one-sided Jacobi on the Cholesky factor of the shifted
//      L^-1 K L^-T when G is well conditioned, else Jacobi
//      eigendecomposition of G, canonical
//      orthogonalisation (directions with relative Gram eigenvalue below a
//      threshold are dropped) and Jacobi on the projected K -> Ritz values
//      and C;
//   4. X <- Y C, and residual norms ||(HY) C_i - theta_i X_i|| with (HY) C
//      formed on the fly (never stored: the next filter starts from X);
//   5. b_lo <- largest Ritz value, repeat until every wanted residual is
//      below tol.
// The Gershgorin bound b_up = 6/h^2 + max V holds for every fragment
// Hamiltonian (principal submatrix of the global one).
// The returned states are the first n_a Ritz vectors with the sign gauge
// "largest |component| positive, ties to the lowest box index".
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <cmath>
#include <cstdio>
#include <vector>

#include "fp64_util.h"
#include "ofm_internal.h"

using namespace ofm;

struct EigWork {
  std::vector<EigFrag> efr;           // block layout (eigblk.cu)
  long long elems = 0, vc_elems = 0;
  int mmax = 0;
  std::vector<long long> toff;        // per fragment offset into theta / res (m_a each)
  long long tsum = 0;
  EigFilterPlan filter;
  EigGramPlan gram;
  DevBuf d_efr, d_jobs, d_steps, buf[3], vc, coef, theta, res, Cm, work, blocks, partials, d_gitems, d_gpart,
      d_gfrag, d_gblk, d_toff, d_rank, d_vmax, rpart, sgn;
  double vlim[2] = {0.0, 0.0};        // max V, min V
  size_t rr_smem = 0, rot_smem = 0;   // dynamic shared memory of the two kernels
  int rr_threads = 256;                 // Rayleigh-Ritz CTA size
  int rot_blocks = 1;
  bool ready = false;
  // algorithmic traffic / work: a launch of the filter that advances S steps
  // reads one or two blocks and c0 + V and writes two, a single step ([1]) reads
  // two and writes one; ten flops per point, vector and step
  double filter_block[2] = {0, 0}, filter_vc[2] = {0, 0}, filter_flops = 0, gram_bytes = 0, gram_flops = 0,
         rot_bytes = 0, rot_flops = 0;
};

void ofm_eig_guards(const ofm_ctx* c, std::vector<GuardRef>& out) {
  if (!c->eig) return;
  const EigWork* w = c->eig;
  const struct { const DevBuf* b; const char* n; } bufs[] = {
      {&w->d_efr, "eigensolver fragment table"}, {&w->d_jobs, "filter work list"},
      {&w->d_steps, "filter step list"},
      {&w->buf[0], "eigensolver block 0"}, {&w->buf[1], "eigensolver block 1"},
      {&w->buf[2], "eigensolver block 2"}, {&w->vc, "filter potential"},
      {&w->coef, "filter coefficients"}, {&w->theta, "Ritz values"}, {&w->res, "residuals"},
      {&w->Cm, "Ritz coefficients"}, {&w->work, "Rayleigh-Ritz work"}, {&w->blocks, "Gram blocks"},
      {&w->partials, "Gram partials"}, {&w->d_gitems, "Gram items"}, {&w->d_gpart, "Gram partial offsets"},
      {&w->d_gfrag, "Gram fragments"}, {&w->d_gblk, "Gram block offsets"},
      {&w->d_toff, "eigensolver offsets"}, {&w->d_rank, "ranks"},
      {&w->d_vmax, "potential maxima"}, {&w->rpart, "residual partials"}, {&w->sgn, "export signs"}};
  for (const auto& x : bufs)
    if (x.b->p) out.push_back({x.b->p, x.b->cap, x.n});
}

void ofm_eig_free(ofm_ctx* c) {
  if (!c->eig) return;
  EigWork* w = c->eig;
  DevBuf* bufs[] = {&w->d_efr, &w->d_jobs, &w->d_steps, &w->buf[0], &w->buf[1], &w->buf[2], &w->vc, &w->coef,
                    &w->theta, &w->res, &w->Cm, &w->work, &w->blocks, &w->partials, &w->d_gitems,
                    &w->d_gpart, &w->d_gfrag, &w->d_gblk, &w->d_toff, &w->d_rank, &w->d_vmax,
                    &w->rpart, &w->sgn};
  for (DevBuf* b : bufs)
    if (b->p) cudaFree(b->p);
  delete w;
  c->eig = nullptr;
}

namespace {

// ---- per-fragment dense Rayleigh-Ritz (one CTA per fragment) -------------
//
// T is the arithmetic of the small dense problems: FP64 for FP64 storage;
// FP32 for FP32 storage, where the states themselves carry FP32 rounding
// (the FP64 pipe of one SM issues about 2 FMA per clock on this part, so
// FP64 here would make the eigensolver bound by a handful of SMs).

// Round-robin schedule (circle method): index ne-1 stays, the others
// rotate; round r pairs (r, ne-1) and ((r+k) mod (ne-1), (r-k) mod (ne-1)).
// Every pair meets once per sweep and the pairs of a round are disjoint.

template <typename T> struct Eps;
template <> struct Eps<float> { static constexpr double v = 6.0e-8; };
template <> struct Eps<double> { static constexpr double v = 1.1e-16; };

// Cyclic parallel Jacobi on the symmetric n x n matrix A (leading dim lda),
// accumulating the rotations into V (which must hold the identity or a
// start basis).  Round-robin pairing: n_even/2 disjoint rotations per round.
// A and V live in shared memory when they fit, so a round costs two CTA
// barriers (after the rows, after the columns) and no global-memory round
// trips.  Stops when the off-diagonal
// mass is at the rounding level of an n x n matrix or a sweep rotated
// nothing (elements below rounding relative to their diagonal pair are
// left alone).
template <typename T>
__device__ void cta_jacobi(T* A, T* V, int n, int lda, int* perm, T* cs, double* red) {
  const int tid = threadIdx.x, nt = blockDim.x;
  const int ne = n + (n & 1);
  const int half = ne / 2;
  const double eps = Eps<T>::v;
  const T eps_t = (T)Eps<T>::v;
  // norms, reductions and thresholds in the working precision T: the FP64
  // units of this part are few, and a stopping test needs no more
  for (int sweep = 0; sweep < 40; ++sweep) {
    T off = 0, tot = 0;
    for (int e = tid; e < n * n; e += nt) {
      const int i = e / n, j = e - (e / n) * n;
      const T a = A[i * lda + j];
      tot += a * a;
      if (i != j) off += a * a;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_down_sync(0xffffffffu, off, o);
      tot += __shfl_down_sync(0xffffffffu, tot, o);
    }
    if ((tid & 31) == 0) {
      red[2 * (tid >> 5)] = (double)off;
      red[2 * (tid >> 5) + 1] = (double)tot;
    }
    __syncthreads();
    if (tid == 0) {
      double so = 0.0, st = 0.0;
      for (int w = 0; w < nt / 32; ++w) {
        so += red[2 * w];
        st += red[2 * w + 1];
      }
      const double tol = 4.0 * n * eps;
      red[64] = (so <= tol * tol * st || so == 0.0 || (sweep > 0 && red[65] == 0.0)) ? 1.0 : 0.0;
      red[65] = 0.0;                      // rotations applied in the coming sweep
      red[66] = 2.0 * eps * sqrt(st / n);  // absolute floor: rounding level of an element
    }
    __syncthreads();
    const bool done = red[64] != 0.0;
    const T floor_t = (T)red[66];
    __syncthreads();
    if (done) break;
    const int lane = tid & 31, warp = tid >> 5, nwarps = nt >> 5;
    for (int r = 0; r < ne - 1; ++r) {
      // rows p, q: one warp per pair.  The warp forms its pair's angle itself
      // (every lane the same arithmetic) and goes on to the row update, so
      // the angle needs no phase or barrier of its own; perm[] and cs[] carry
      // the pairs and angles to the column phase.  With d = a_qq - a_pp,
      //   t = sgn(d) 2 a_pq / (|d| + sqrt(d^2 + 4 a_pq^2))
      // is the smaller root of t^2 + 2 theta t - 1 = 0, theta = d / (2 a_pq)
      // (the classical cyclic-Jacobi tangent), with one division and one
      // square root fewer than forming theta first.
      for (int k = warp; k < half; k += nwarps) {
        int p, q;
        {   // the round-robin pairing without integer division
          const int M = ne - 1;
          if (k == 0) {
            p = r;
            q = M;
          } else {
            p = r + k;
            if (p >= M) p -= M;
            q = r - k;
            if (q < 0) q += M;
          }
        }
        T c = 1, s = 0;
        if (p < n && q < n) {
          const T apq = A[p * lda + q];
          const T app = A[p * lda + p], aqq = A[q * lda + q];
          const T thr = fmax(T(4) * eps_t * eps_t * fabs(app * aqq), floor_t * floor_t);
          if (apq * apq > thr) {
            if (lane == 0) red[65] = 1.0;
            const T d = aqq - app;
            const T t = (d >= T(0) ? T(2) : T(-2)) * apq / (fabs(d) + sqrt(d * d + T(4) * apq * apq));
            c = T(1) / sqrt(t * t + T(1));
            s = t * c;
          }
        }
        if (lane == 0) {
          perm[k] = p | (q << 16);
          cs[2 * k] = c;
          cs[2 * k + 1] = s;
        }
        __syncwarp();   // every lane has read a_pq, a_pp, a_qq before the rows change
        if (p >= n || q >= n || s == T(0)) continue;   // uniform over the warp
        for (int j = lane; j < n; j += 32) {
          const T ap = A[p * lda + j], aq = A[q * lda + j];
          A[p * lda + j] = c * ap - s * aq;
          A[q * lda + j] = s * ap + c * aq;
        }
      }
      __syncthreads();
      // columns p, q of A and V: one warp per pair, lanes down the column
      for (int k = warp; k < half; k += nwarps) {
        const int pq = perm[k], p = pq & 0xffff, q = pq >> 16;
        const T c = cs[2 * k], s = cs[2 * k + 1];
        if (p >= n || q >= n || s == T(0)) continue;
        for (int i = lane; i < n; i += 32) {
          const T ap = A[i * lda + p], aq = A[i * lda + q];
          A[i * lda + p] = c * ap - s * aq;
          A[i * lda + q] = s * ap + c * aq;
          const T vp = V[i * lda + p], vq = V[i * lda + q];
          V[i * lda + p] = c * vp - s * vq;
          V[i * lda + q] = s * vp + c * vq;
        }
      }
      __syncthreads();
    }
  }
}

// 1 / sqrt(x) to about an ulp: the approximate FP32 reciprocal square root and one
// Newton step; rsqrt64 in FP64.
__device__ __forceinline__ float rsqrt1(float x) {
  const float y = rsqrtf(x);
  return y * fmaf(-0.5f * x * y, y, 1.5f);
}
__device__ __forceinline__ double rsqrt1(double x) { return rsqrt64(x); }
// A pivot's square root and its reciprocal.  In FP32 by correctly rounded
// operations: Ritz values and vectors of a block with a level tens of Ha deep carry the
// pivots' relative error (2 u of 88 Ha is 1e-5).
__device__ __forceinline__ float pivot_root(float x, float& inv) {
  const float s = __fsqrt_rn(x);
  inv = __frcp_rn(s);
  return s;
}
__device__ __forceinline__ double pivot_root(double x, double& inv) {
  inv = rsqrt64(x);
  return x * inv;
}
__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double madd(double a, double b, double c) { return fma(a, b, c); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One-sided Jacobi (Hestenes; on a Cholesky factor, Veselic and Hari, "A note
// on a one-sided Jacobi algorithm", Numer. Math. 56 (1989)): B = G G^T with G
// the lower Cholesky factor, right rotations make G's columns orthogonal, G J =
// Q diag(sqrt(lambda)); the columns' directions are the eigenvectors and their
// squared norms the eigenvalues, with no rotation matrix to accumulate.  Row j
// of g holds column j of G.  One SM works on a fragment, so a round is bound by
// its issue slots (FP64: by the FP64 pipe): two columns read and written
// instead of the two-sided form's two rows and four columns, one barrier
// instead of two, GW lanes per pair (32 / GW pairs share an instruction; NE
// elements per lane, n <= GW NE), and the rotation's tangent in FP32 arithmetic:
// it only steers convergence, the cosine and sine belong to that tangent to
// full precision.
// A pair is rotated while the cosine between its columns is above 4 eps;
// squared norms are formed anew in every sweep and updated by t d within it.
// Ends after a sweep whose largest squared cosine was below eps / 1000 (the
// next one's would be of the order of its square).  Returns false when 30
// sweeps did not suffice.  The whole Rayleigh-Ritz step, 27 blocks of 120 vectors
// in FP32: 2.1 ms with the two-sided form, 1.0 ms; blocks of 8 to 30 in FP64:
// 0.75 ms, 0.47 ms.
template <typename T, int GW, int NE>
__device__ bool cta_jacobi1(T* g, int n, int ld, T* nrm, int* rotated) {
  const int tid = threadIdx.x, ln = tid & (GW - 1), grp = tid / GW, ngrp = blockDim.x / GW;
  const int ne = n + (n & 1), half = ne / 2, M = ne - 1;
  const T tol2 = T(16) * (T)Eps<T>::v * (T)Eps<T>::v, big2 = T(1e-3) * (T)Eps<T>::v;
  auto group_sum = [](T v) {
#pragma unroll
    for (int o = GW / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  for (int sweep = 0; sweep < 30; ++sweep) {
    for (int j0 = 0; j0 < n; j0 += ngrp) {
      const int j = min(j0 + grp, n - 1);
      T v = T(0);
#pragma unroll
      for (int u = 0; u < NE; ++u) {
        const T a = ln + GW * u < n ? g[j * ld + ln + GW * u] : T(0);
        v = madd(a, a, v);
      }
      v = group_sum(v);
      if (ln == 0 && j0 + grp < n) nrm[j] = v;
    }
    if (tid == 0) *rotated = 0;
    __syncthreads();
    for (int r = 0; r < M; ++r) {
      for (int k0 = 0; k0 < half; k0 += ngrp) {
        const int k = k0 + grp;
        int p = r, q = M;   // the round-robin pairing without integer division
        if (k != 0) {
          p = r + k;
          if (p >= M) p -= M;
          q = r - k;
          if (q < 0) q += M;
        }
        const bool valid = k < half && p < n && q < n;
        if (!valid) p = q = 0;
        T* gp = g + p * ld + ln;
        T* gq = g + q * ld + ln;
        T a[NE], b[NE], d = T(0);
#pragma unroll
        for (int u = 0; u < NE; ++u) {
          const bool in = ln + GW * u < n;
          a[u] = in ? gp[GW * u] : T(0);
          b[u] = in ? gq[GW * u] : T(0);
          d = madd(a[u], b[u], d);
        }
        const T np = nrm[p], nq = nrm[q];
        d = group_sum(d);
        const T d2 = d * d, nn = np * nq;
        const bool rot = valid && d2 > tol2 * nn;
        if (!__any_sync(0xffffffffu, rot)) continue;
        // the smaller root t of t^2 + 2 z t - 1 = 0, z = (nq - np) / (2 d)
        const float df = (float)d, ddf = (float)(nq - np);
        const float x = fmaf(4.0f * df, df, ddf * ddf);
        const float tf = __fdividef(ddf >= 0.0f ? 2.0f * df : -2.0f * df, fabsf(ddf) + x * rsqrtf(fmaxf(x, 1e-37f)));
        const T t = rot ? (T)tf : T(0);
        const T c = rsqrt1(madd(t, t, T(1))), s = t * c;
        if (rot) {
#pragma unroll
          for (int u = 0; u < NE; ++u) {
            if (ln + GW * u < n) {
              gp[GW * u] = madd(c, a[u], -s * b[u]);
              gq[GW * u] = madd(s, a[u], c * b[u]);
            }
          }
        }
        __syncwarp();   // every lane has read both norms
        if (rot && ln == 0) {
          nrm[p] = madd(-t, d, np);
          nrm[q] = madd(t, d, nq);
          if (d2 > big2 * nn) *rotated = 1;
        }
      }
      __syncthreads();
    }
    const bool again = *rotated != 0;
    __syncthreads();
    if (!again) return true;
  }
  return false;
}

// Lanes per pair: 16 in FP32, 8 in FP64 (where an instruction costs the pipe the
// same whatever its lanes do).
template <typename T>
__device__ bool jacobi1(T* g, int n, int ld, T* nrm, int* rotated) {
  constexpr int GW = sizeof(T) == 8 ? 8 : 16;
  const int ne = (n + GW - 1) / GW;
  if (ne <= 1) return cta_jacobi1<T, GW, 1>(g, n, ld, nrm, rotated);
  if (ne <= 2) return cta_jacobi1<T, GW, 2>(g, n, ld, nrm, rotated);
  if (ne <= 3) return cta_jacobi1<T, GW, 3>(g, n, ld, nrm, rotated);
  if (ne <= 4) return cta_jacobi1<T, GW, 4>(g, n, ld, nrm, rotated);
  if (ne <= 5) return cta_jacobi1<T, GW, 5>(g, n, ld, nrm, rotated);
  if (ne <= 6) return cta_jacobi1<T, GW, 6>(g, n, ld, nrm, rotated);
  if (ne <= 8) return cta_jacobi1<T, GW, 8>(g, n, ld, nrm, rotated);
  if (ne <= 10) return cta_jacobi1<T, GW, 10>(g, n, ld, nrm, rotated);
  if (ne <= 12) return cta_jacobi1<T, GW, 12>(g, n, ld, nrm, rotated);
  if (ne <= 15) return cta_jacobi1<T, GW, 15>(g, n, ld, nrm, rotated);
  return false;
}

// Cholesky factor of the symmetric matrix in M, in place: row j of M becomes
// column j of L (zero before the diagonal), rinv[j] = 1 / L_jj.  A pivot that is
// not above tol clears *ok (and counts as one).
// By panels of 32 rows: one warp factors the 32 x 32 diagonal block in
// registers (lane k holds column k, the pivot row goes round by shuffles), each
// warp then finishes 32 columns of the panel's rows against it, and all warps
// take the panel's products off the rest: three barriers a panel instead of
// one per column.
template <typename T>
__device__ void cta_cholesky(T* M, int m, int ld, T tol, T* rinv, int* ok) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  for (int j0 = 0; j0 < m; j0 += 32) {
    const int nb = min(32, m - j0);
    if (warp == 0) {
      T a[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) a[i] = i < nb && lane < nb ? M[(j0 + i) * ld + j0 + lane] : T(0);
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        if (j < nb) {
          T piv = __shfl_sync(0xffffffffu, a[j], j);
          const bool bad = !(piv > tol);
          if (bad) piv = T(1);
          T r;
          const T d = pivot_root(piv, r);
          const T x = lane == j ? d : a[j] * r;   // row j of the factor
          if (lane == 0) {
            if (bad) *ok = 0;
            rinv[j0 + j] = r;
          }
          a[j] = lane < j ? T(0) : x;
#pragma unroll
          for (int i = j + 1; i < 32; ++i) a[i] = madd(-__shfl_sync(0xffffffffu, x, i), x, a[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i < nb && lane < nb) M[(j0 + i) * ld + j0 + lane] = a[i];
    }
    __syncthreads();
    // columns past the panel: x_i = (a_i - sum_{j<i} R_ji x_j) / R_ii down the rows
    for (int k0 = j0 + 32 + 32 * warp; k0 < m; k0 += 32 * nw) {
      const int k = k0 + lane;
      T a[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) a[i] = k < m ? M[(j0 + i) * ld + k] : T(0);
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        a[j] *= rinv[j0 + j];
#pragma unroll
        for (int i = j + 1; i < 32; ++i) a[i] = madd(-M[(j0 + j) * ld + j0 + i], a[j], a[i]);
      }
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (k < m) M[(j0 + i) * ld + k] = a[i];
    }
    __syncthreads();
    // the rest: row i loses sum_j R_ji R_jk, k >= i
    for (int i = j0 + 32 + warp; i < m; i += nw)
      for (int k = i + lane; k < m; k += 32) {
        T v = M[i * ld + k];
#pragma unroll 8
        for (int j = 0; j < 32; ++j) v = madd(-M[(j0 + j) * ld + i], M[(j0 + j) * ld + k], v);
        M[i * ld + k] = v;
      }
    // the panel's rows before the diagonal block
    for (int e = tid; e < nb * j0; e += blockDim.x) M[(j0 + e / j0) * ld + e % j0] = T(0);
    __syncthreads();
  }
}

// Row solves in place: every row x of X (m rows of m) becomes L^-1 x
// (BACK: L^-T x), row j of R = column j of L, rinv = 1 / diagonal.  A warp takes
// RB rows at a time into registers (lane i + 32 u) and needs no barrier: each
// solved entry is broadcast by a shuffle and its multiple of L's column (row)
// taken from the remaining ones; a column of L is read once per RB rows.
template <typename T, int NU, bool BACK>
__device__ void row_solves(const T* R, const T* rinv, T* X, int m, int ld) {
  constexpr int RB = sizeof(T) == 8 ? 2 : 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int r0 = warp * RB; r0 < m; r0 += nw * RB) {
    T v[RB][NU];
#pragma unroll
    for (int r = 0; r < RB; ++r)
#pragma unroll
      for (int u = 0; u < NU; ++u)
        v[r][u] = r0 + r < m && lane + 32 * u < m ? X[(r0 + r) * ld + lane + 32 * u] : T(0);
#pragma unroll
    for (int uu = 0; uu < NU; ++uu) {
      const int u = BACK ? NU - 1 - uu : uu;
      const int nj = min(32, m - 32 * u);
      for (int q = 0; q < nj; ++q) {
        const int jj = BACK ? nj - 1 - q : q, j = 32 * u + jj;
        const T ri = rinv[j];
        T x[RB];
#pragma unroll
        for (int r = 0; r < RB; ++r) x[r] = __shfl_sync(0xffffffffu, v[r][u], jj) * ri;
#pragma unroll
        for (int w = 0; w < NU; ++w) {
          if (BACK ? w > u : w < u) continue;
          const int i = lane + 32 * w;
          // L_ij below the diagonal (forward), L_ji before it (backward)
          T l = T(0);
          if (BACK ? i < j : (i > j && i < m)) l = BACK ? R[i * ld + j] : R[j * ld + i];
#pragma unroll
          for (int r = 0; r < RB; ++r) v[r][w] = madd(-l, x[r], v[r][w]);
        }
#pragma unroll
        for (int r = 0; r < RB; ++r)
          if (lane == jj) v[r][u] = x[r];
      }
    }
#pragma unroll
    for (int r = 0; r < RB; ++r)
#pragma unroll
      for (int u = 0; u < NU; ++u)
        if (r0 + r < m && lane + 32 * u < m) X[(r0 + r) * ld + lane + 32 * u] = v[r][u];
  }
}

template <typename T, bool BACK>
__device__ void rr_row_solves(const T* R, const T* rinv, T* X, int m, int ld) {
  const int nu = (m + 31) / 32;
  if (nu == 1) row_solves<T, 1, BACK>(R, rinv, X, m, ld);
  else if (nu == 2) row_solves<T, 2, BACK>(R, rinv, X, m, ld);
  else if (nu == 3) row_solves<T, 3, BACK>(R, rinv, X, m, ld);
  else if (nu == 4) row_solves<T, 4, BACK>(R, rinv, X, m, ld);
  else if (nu == 5) row_solves<T, 5, BACK>(R, rinv, X, m, ld);
  else if (nu == 6) row_solves<T, 6, BACK>(R, rinv, X, m, ld);
  else row_solves<T, 8, BACK>(R, rinv, X, m, ld);   // m <= 256
}

// val_j = q_j^T B q_j / q_j^T q_j of the rows q_j of Q (m rows of m): a warp takes RB
// rows at a time, lanes along B's columns.  B need not be symmetric to the last bit.
template <typename T>
__device__ void rayleigh_values(const T* B, const T* Q, T* val, int m, int ld) {
  constexpr int RB = sizeof(T) == 8 ? 2 : 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int r0 = warp * RB; r0 < m; r0 += nw * RB) {
    const T* q[RB];
    T s[RB], d[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      q[r] = Q + min(r0 + r, m - 1) * ld;
      s[r] = d[r] = T(0);
    }
    for (int k0 = 0; k0 < m; k0 += 32) {
      const int k = min(k0 + lane, m - 1);
      T w[RB];
#pragma unroll
      for (int r = 0; r < RB; ++r) w[r] = T(0);
#pragma unroll 4
      for (int i = 0; i < m; ++i) {
        const T b = B[i * ld + k];
#pragma unroll
        for (int r = 0; r < RB; ++r) w[r] = madd(b, q[r][i], w[r]);
      }
      if (k0 + lane < m)
#pragma unroll
        for (int r = 0; r < RB; ++r) {
          s[r] = madd(w[r], q[r][k], s[r]);
          d[r] = madd(q[r][k], q[r][k], d[r]);
        }
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      s[r] = warp_sum(s[r]);
      d[r] = warp_sum(d[r]);
      if (lane == 0 && r0 + r < m) val[r0 + r] = s[r] / d[r];
    }
  }
}

// At least 256 and at most this many threads (the reduction scratch holds 32
// warps' partials; the FP64 form needs the registers), one warp per rotation pair of a round where that fits.
template <typename T>
constexpr int rr_max_threads() { return sizeof(T) == 8 ? 640 : 1024; }

// Inputs: blocks of the self pair of fragment f, [K | G] with K = Y^T H Y
// and G = Y^T Y (m x m each, symmetrised).  Outputs: C (m x m row-major,
// columns = Ritz vectors in the Y basis, ascending Ritz values; dropped
// directions give zero columns), theta (m; dropped directions repeat the
// largest kept value), rank (number of kept directions).
// Work matrices A, U, W (row stride ld) and vectors D, sig, idx live in
// dynamic shared memory (ld = the odd one of m + 1, m + 2: column walks across
// the warp hit distinct banks) or, for large m, in `work` (ld = m).
template <typename T>
__global__ void __launch_bounds__(rr_max_threads<T>()) rayleigh_ritz_kernel(const EigFrag* efr, const long long* blk_off,
                                                            const double* blocks, T* work,
                                                            long long wstride, double* Cm,
                                                            long long cstride, double* theta,
                                                            const long long* toff, double rank_tol,
                                                            int* rank_out, int use_smem, double v_min, double tol) {
  extern __shared__ __align__(16) unsigned char rr_raw[];
  __shared__ int perm[520];
  __shared__ T cs[520];
  __shared__ double red[80];
  __shared__ int nkeep;
  const int f = blockIdx.x;
  const int m = efr[f].n;
  const int tid = threadIdx.x, nt = blockDim.x;
  const double* Kb = blocks + blk_off[f];
  const double* Gb = Kb + (long long)m * m;
  const int ld = use_smem ? m + 1 + (m & 1) : m;
  T* A = use_smem ? reinterpret_cast<T*>(rr_raw) : work + f * wstride;
  T* U = A + (long long)m * ld;
  T* W = U + (long long)m * ld;
  T* D = W + (long long)m * ld;           // m
  T* sig = D + m;                         // m
  T* rinv = sig + m;                      // m
  int* idx = reinterpret_cast<int*>(rinv + m);   // m
  double* C = Cm + f * cstride;
  double* th = theta + toff[f];

  for (int i = tid; i < m; i += nt) {
    const double g = Gb[(long long)i * m + i];
    D[i] = g > 0.0 ? (T)(1.0 / sqrt(g)) : T(0);
  }
  __syncthreads();
  // entry (i, j) of D M D; a diagonal one is rounded once (see pivot_root)
  auto scaled = [&](double v, int i, int j) {
    return i == j ? (T)((double)D[i] * D[i] * v) : D[i] * (T)v * D[j];
  };
  for (int e = tid; e < m * m; e += nt) {
    const int i = e / m, j = e - (e / m) * m;
    A[i * ld + j] = scaled(Gb[e], i, j);
    U[i * ld + j] = (i == j) ? T(1) : T(0);
  }
  __syncthreads();
  // Fast path: when the scaled Gram is well conditioned (every Cholesky
  // pivot above chol_tol, the usual case once the iteration has started to
  // converge), G_s = L L^T, B = L^-1 K_s L^-T, one Jacobi on the nearly
  // diagonal B, C = D L^-T Q.  Otherwise the canonical orthogonalisation
  // below drops the near-dependent directions.
  {
    __shared__ int chol_ok;
    __shared__ T sigma_s;
    const T chol_tol = sizeof(T) == 8 ? T(1e-8) : T(1e-3);
    if (tid == 0) chol_ok = 1;
    for (int e = tid; e < m * m; e += nt) {
      const int i = e / m, j = e - (e / m) * m;
      W[i * ld + j] = A[i * ld + j];
    }
    __syncthreads();
    cta_cholesky<T>(W, m, ld, chol_tol, rinv, &chol_ok);   // row j = column j of L
    if (chol_ok) {
      // U <- L^-1 (D K D): D K D is symmetric, so its rows are the columns to
      // solve for; row c of U is then column c of L^-1 (D K D)
      for (int e = tid; e < m * m; e += nt) {
        const int i = e / m, j = e - (e / m) * m;
        U[i * ld + j] = scaled(Kb[e], i, j);
      }
      __syncthreads();
      rr_row_solves<T, false>(W, rinv, U, m, ld);
      __syncthreads();
      // A <- its transpose, then B = L^-1 (D K D) L^-T row by row
      for (int e = tid; e < m * m; e += nt) {
        const int i = e / m, j = e - (e / m) * m;
        A[i * ld + j] = U[j * ld + i];
      }
      __syncthreads();
      rr_row_solves<T, false>(W, rinv, A, m, ld);
      // sigma: B + sigma I is positive definite.  The larger of two lower bounds
      // of B's spectrum, Gershgorin's and min V (H_f >= min V), less a tenth of B's
      // largest diagonal entry for the rounding of K.  The vectors' error is of the
      // order of u sigma, so sigma follows B, not the potential: with min V alone, a
      // well anywhere in the grid left its depth times u in every fragment.
      __syncthreads();
      for (int i = tid >> 5; i < m; i += nt >> 5) {
        T s = T(0);
        for (int j = tid & 31; j < m; j += 32) s += j == i ? T(0) : fabs(A[i * ld + j]);
        s = warp_sum(s);
        if ((tid & 31) == 0) sig[i] = A[i * ld + i] - s;
      }
      __syncthreads();
      if (tid < 32) {
        T mx = T(0), low = T(3e38), rad = T(0);
        for (int i = tid; i < m; i += 32) {
          const T b = A[i * ld + i];
          mx = fmax(mx, fabs(b));
          low = fmin(low, sig[i]);
          rad = fmax(rad, b - sig[i]);
        }
        for (int o = 16; o > 0; o >>= 1) {
          mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          low = fmin(low, __shfl_xor_sync(0xffffffffu, low, o));
          rad = fmax(rad, __shfl_xor_sync(0xffffffffu, rad, o));
        }
        if (tid == 0) {
          sigma_s = T(0.1) * mx - fmax(low, (T)v_min);
          // The two-sided form instead where sigma is far above B, and on a nearly
          // diagonal B with a level so deep that the one-sided form's angles, 4 u
          // each, leave a residual of the order of the tolerance: the two-sided
          // form's are u |B| over the gap.
          const bool deep = T(16) * (T)Eps<T>::v * mx > (T)tol && rad <= T(0.05) * mx;
          chol_ok = sigma_s <= T(4) * mx && !deep;
        }
      }
      __syncthreads();
      const T sigma = sigma_s;
      const bool shifted = chol_ok != 0;   // uniform
      // U <- the Cholesky factor of B + sigma I (symmetrised), row j = column j
      for (int e = tid; e < m * m; e += nt) {
        const int i = e / m, j = e - (e / m) * m;
        U[i * ld + j] = T(0.5) * (A[i * ld + j] + A[j * ld + i]) + (i == j ? sigma : T(0));
      }
      __syncthreads();
      if (shifted) cta_cholesky<T>(U, m, ld, T(1e-30), sig, &chol_ok);
      bool one = chol_ok != 0;
      if (one) one = jacobi1<T>(U, m, ld, sig, perm);
      if (one) {
        // Q_j = row j / |row j|, lambda_j its Rayleigh quotient of B (|row j|^2 - sigma
        // carries the rounding of every rotation, relative to sigma)
        for (int j = tid >> 5; j < m; j += nt >> 5) {
          T v = T(0);
          for (int i = tid & 31; i < m; i += 32) v = madd(U[j * ld + i], U[j * ld + i], v);
          v = warp_sum(v);
          const T r = rsqrt1(v);
          for (int i = tid & 31; i < m; i += 32) U[j * ld + i] *= r;
        }
        __syncthreads();
        rayleigh_values<T>(A, U, sig, m, ld);
      } else {
        // the two-sided form on B; its vectors, transposed, into U's rows
        for (int e = tid; e < m * m; e += nt) {
          const int i = e / m, j = e - (e / m) * m;
          if (i < j) {
            const T v = T(0.5) * (A[i * ld + j] + A[j * ld + i]);
            A[i * ld + j] = v;
            A[j * ld + i] = v;
          }
          U[i * ld + j] = (i == j) ? T(1) : T(0);
        }
        __syncthreads();
        cta_jacobi<T>(A, U, m, ld, perm, cs, red);   // A -> diag(theta), U -> Q
        for (int e = tid; e < m * m; e += nt) {
          const int i = e / m, j = e - (e / m) * m;
          if (i < j) {
            const T v = U[i * ld + j];
            U[i * ld + j] = U[j * ld + i];
            U[j * ld + i] = v;
          }
        }
        for (int j = tid; j < m; j += nt) sig[j] = A[j * ld + j];
      }
      __syncthreads();
      for (int j = tid; j < m; j += nt) {
        const T t = sig[j];
        int rk = 0;
        for (int i = 0; i < m; ++i) {
          const T ti = sig[i];
          rk += (ti < t || (ti == t && i < j)) ? 1 : 0;
        }
        idx[j] = rk;
      }
      rr_row_solves<T, true>(W, rinv, U, m, ld);   // row j of U <- L^-T Q_j
      __syncthreads();
      for (int e = tid; e < m * m; e += nt) {
        const int k = e / m, j = e - (e / m) * m;
        C[(long long)k * m + idx[j]] = (double)(D[k] * U[j * ld + k]);
      }
      for (int j = tid; j < m; j += nt) th[idx[j]] = (double)sig[j];
      if (tid == 0) rank_out[f] = m;
      return;
    }
  }
  cta_jacobi<T>(A, U, m, ld, perm, cs, red);
  // rank decision on the scaled Gram spectrum
  if (tid == 0) {
    T smax = 0;
    for (int i = 0; i < m; ++i) smax = fmax(smax, A[i * ld + i]);
    int r = 0;
    for (int i = 0; i < m; ++i) {
      const T s = A[i * ld + i];
      if ((double)s > rank_tol * (double)smax) {
        idx[r] = i;
        sig[r] = s;
        ++r;
      }
    }
    nkeep = r;
  }
  __syncthreads();
  const int r = nkeep;
  // W = D U_keep sig^-1/2  (m x r)
  for (int e = tid; e < m * r; e += nt) {
    const int k = e / r, j = e - (e / r) * r;
    W[k * ld + j] = D[k] * U[k * ld + idx[j]] / sqrt(sig[j]);
  }
  __syncthreads();
  // A <- K W (m x r), then U <- W^T (K W) (r x r), symmetrised
  for (int e = tid; e < m * r; e += nt) {
    const int k = e / r, j = e - (e / r) * r;
    T s = 0;
    for (int l = 0; l < m; ++l) s += (T)Kb[(long long)k * m + l] * W[l * ld + j];
    A[k * ld + j] = s;
  }
  __syncthreads();
  for (int e = tid; e < r * r; e += nt) {
    const int i = e / r, j = e - (e / r) * r;
    if (j < i) continue;
    T s = 0, t = 0;
    for (int l = 0; l < m; ++l) {
      s += W[l * ld + i] * A[l * ld + j];
      t += W[l * ld + j] * A[l * ld + i];
    }
    U[i * ld + j] = T(0.5) * (s + t);
    U[j * ld + i] = T(0.5) * (s + t);
  }
  __syncthreads();
  for (int e = tid; e < r * r; e += nt) {
    const int i = e / r, j = e - (e / r) * r;
    A[i * ld + j] = (i == j) ? T(1) : T(0);
  }
  __syncthreads();
  cta_jacobi<T>(U, A, r, ld, perm, cs, red);     // U -> diag(theta), A -> Q
  // ascending order: rank of each Ritz value
  for (int j = tid; j < r; j += nt) {
    const T t = U[j * ld + j];
    int rk = 0;
    for (int i = 0; i < r; ++i) {
      const T ti = U[i * ld + i];
      rk += (ti < t || (ti == t && i < j)) ? 1 : 0;
    }
    idx[j] = rk;
  }
  __syncthreads();
  // C[:, rank(j)] = W Q[:, j]
  for (int e = tid; e < m * m; e += nt) C[e] = 0.0;
  __syncthreads();
  for (int e = tid; e < m * r; e += nt) {
    const int k = e / r, j = e - (e / r) * r;
    T s = 0;
    for (int l = 0; l < r; ++l) s += W[k * ld + l] * A[l * ld + j];
    C[(long long)k * m + idx[j]] = (double)s;
  }
  double tmax = -DBL_MAX;
  for (int j = 0; j < r; ++j) tmax = fmax(tmax, (double)U[j * ld + j]);
  for (int j = tid; j < m; j += nt) {
    if (j < r) th[idx[j]] = (double)U[j * ld + j];
    else th[j] = tmax;
  }
  if (tid == 0) rank_out[f] = r;
}

constexpr int VMAX_BLOCKS = 152;

// max and min of V: per-block partials in the storage type (FP32 compares
// are cheap, FP64 ones are not on this part), then one block combines them
// into out[0] = max, out[1] = min; part holds 2 * VMAX_BLOCKS doubles.
template <typename T>
__global__ void __launch_bounds__(256) vmax_partial_kernel(const T* V, long long n, double* part) {
  __shared__ T red[8], redm[8];
  T m = V[0], mn = V[0];
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += 256LL * gridDim.x) {
    m = max(m, V[i]);
    mn = min(mn, V[i]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  }
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5] = m;
    redm[threadIdx.x >> 5] = mn;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) {
      m = max(m, red[w]);
      mn = min(mn, redm[w]);
    }
    part[2 * blockIdx.x] = (double)m;
    part[2 * blockIdx.x + 1] = (double)mn;
  }
}

__global__ void vmax_final_kernel(const double* part, int nb, double* out) {
  if (threadIdx.x != 0) return;
  double m = part[0], mn = part[1];
  for (int b = 1; b < nb; ++b) {
    m = fmax(m, part[2 * b]);
    mn = fmin(mn, part[2 * b + 1]);
  }
  out[0] = m;
  out[1] = mn;
}

}  // namespace

// Range of V (max, min) for the filter's bounds: taken at every solve,
// since V may change while the fragment layout (and the workspace) stays.
static ofm_status eig_vlim(ofm_ctx* c) {
  EigWork* w = c->eig;
  cudaStream_t s = c->stream;
  const long long npts = (long long)c->grid.n[0] * c->grid.n[1] * c->grid.n[2];
  KTimer kt(c, KC_EIG_INIT);
  double* part = (double*)w->d_vmax.p + 2;
  if (c->storage == OFM_STORE_FP64)
    vmax_partial_kernel<double><<<VMAX_BLOCKS, 256, 0, s>>>((const double*)c->V.p, npts, part);
  else
    vmax_partial_kernel<float><<<VMAX_BLOCKS, 256, 0, s>>>((const float*)c->V.p, npts, part);
  vmax_final_kernel<<<1, 32, 0, s>>>(part, VMAX_BLOCKS, (double*)w->d_vmax.p);
  OFM_CUDA(c, cudaGetLastError());
  OFM_CUDA(c, cudaMemcpyAsync(w->vlim, w->d_vmax.p, 2 * sizeof(double), cudaMemcpyDeviceToHost, s));
  OFM_CUDA(c, cudaStreamSynchronize(s));
  return OFM_OK;
}

static ofm_status eig_setup(ofm_ctx* c, int guard_opt) {
  if (!c->eig) c->eig = new EigWork();
  EigWork* w = c->eig;
  w->ready = false;
  const bool fp64 = c->storage == OFM_STORE_FP64;
  const size_t es = fp64 ? 8 : 4;
  const int nf = c->nfrag;
  w->mmax = 0;
  w->toff.resize(nf);
  w->tsum = 0;
  std::vector<int> m(nf);
  for (int a = 0; a < nf; ++a) {
    const DevFrag& F = c->frags[a];
    const long long P = (long long)F.ext[0] * F.ext[1] * F.ext[2];
    const int g = guard_opt > 0 ? guard_opt : std::max(4, F.n / 4);
    m[a] = std::min((int)std::min<long long>((long long)F.n + g, P - 1), 256);
    w->mmax = std::max(w->mmax, m[a]);
    w->toff[a] = w->tsum;
    w->tsum += m[a];
  }
  // the widest block the solver takes: 184 vectors in FP32, 117 in FP64 (at that
  // width the Gram's stages take 124 KB and the rotation's coefficients and
  // stages 154 KB)
  if (w->mmax > (fp64 ? 117 : 184))
    return ofm_fail(c, OFM_ERR_INVALID, "block size too large for the rotation kernel");
  eig_layout(c->frags, m, w->efr, w->elems, w->vc_elems);
  eig_filter_plan(w->efr, fp64, w->filter);
  OFM_CUDA(c, eig_gram_plan(w->efr, fp64, w->gram));
  OFM_CUDA(c, eig_rotate_plan(w->efr, fp64, w->rot_blocks, w->rot_smem));
  if (w->gram.smem > (size_t)SMEM_PLAN_MAX || w->rot_smem > (size_t)SMEM_PLAN_MAX)
    return ofm_fail(c, OFM_ERR_INVALID, "block size too large for the rotation kernel");
  w->filter_block[0] = w->filter_block[1] = w->filter_vc[0] = w->filter_vc[1] = 0;
  std::vector<char> step(nf, 0);
  for (int a : w->filter.steps) step[a] = 1;
  w->filter_flops = w->gram_bytes = w->gram_flops = w->rot_bytes = w->rot_flops = 0;
  for (int a = 0; a < nf; ++a) {
    const DevFrag& F = c->frags[a];
    const double P = (double)F.ext[0] * F.ext[1] * F.ext[2];
    w->filter_block[(int)step[a]] += P * m[a] * es;
    w->filter_vc[(int)step[a]] += P * es;
    w->filter_flops += 10.0 * P * m[a];
    w->gram_bytes += P * 2.0 * m[a] * es;
    w->gram_flops += 2.0 * P * m[a] * 2.0 * m[a];
    w->rot_bytes += P * 3.0 * m[a] * es;   // Y and H Y in, X out
    w->rot_flops += 2.0 * 2.0 * P * m[a] * m[a];
  }
  cudaStream_t s = c->stream;
  for (int i = 0; i < 3; ++i) {
    OFM_TRY(ofm_ensure(c, w->buf[i], w->elems * es, "eigensolver block"));
    OFM_CUDA(c, cudaMemsetAsync(w->buf[i].p, 0, w->elems * es, s));   // the padding stays zero
  }
  OFM_TRY(ofm_ensure(c, w->vc, w->vc_elems * es, "filter potential"));
  OFM_TRY(ofm_ensure(c, w->theta, sizeof(double) * w->tsum, "Ritz values"));
  OFM_TRY(ofm_ensure(c, w->res, sizeof(double) * w->tsum, "residuals"));
  OFM_TRY(ofm_ensure(c, w->d_rank, sizeof(int) * nf, "ranks"));
  OFM_TRY(ofm_ensure(c, w->d_vmax, (2 + 2 * VMAX_BLOCKS) * sizeof(double), "max and min V"));
  const long long mm = (long long)w->mmax * w->mmax;
  OFM_TRY(ofm_ensure(c, w->Cm, sizeof(double) * mm * nf, "Ritz coefficients"));
  OFM_TRY(ofm_ensure(c, w->work, sizeof(double) * (3 * mm + 4 * w->mmax + 8) * nf, "Rayleigh-Ritz work"));
  OFM_TRY(ofm_ensure(c, w->blocks, sizeof(double) * w->gram.blk_elems, "Gram blocks"));
  OFM_TRY(ofm_ensure(c, w->partials, es * w->gram.part_elems, "Gram partials"));
  OFM_TRY(ofm_ensure(c, w->rpart, sizeof(double) * (size_t)nf * w->rot_blocks * w->mmax, "residual partials"));
  OFM_TRY(ofm_ensure(c, w->sgn, es * (size_t)nf * w->mmax, "export signs"));
  const struct { DevBuf* b; const void* p; size_t n; const char* what; } tabs[] = {
      {&w->d_efr, w->efr.data(), sizeof(EigFrag) * nf, "eigensolver table"},
      {&w->d_jobs, w->filter.jobs.data(), sizeof(int4) * w->filter.jobs.size(), "filter work list"},
      {&w->d_steps, w->filter.steps.data(), sizeof(int) * w->filter.steps.size(), "filter step list"},
      {&w->d_gitems, w->gram.items.data(), sizeof(int4) * w->gram.items.size(), "Gram items"},
      {&w->d_gpart, w->gram.part_off.data(), sizeof(long long) * w->gram.part_off.size(), "Gram partial offsets"},
      {&w->d_gfrag, w->gram.fitems.data(), sizeof(int2) * nf, "Gram fragments"},
      {&w->d_gblk, w->gram.blk_off.data(), sizeof(long long) * nf, "Gram block offsets"},
      {&w->d_toff, w->toff.data(), sizeof(long long) * nf, "eigensolver offsets"}};
  for (const auto& t : tabs) {
    OFM_TRY(ofm_ensure(c, *t.b, t.n, t.what));
    if (t.n) OFM_CUDA(c, cudaMemcpyAsync(t.b->p, t.p, t.n, cudaMemcpyHostToDevice, s));
  }
  w->rr_threads = std::min(fp64 ? rr_max_threads<double>() : rr_max_threads<float>(),
                           std::max(256, 32 * ((w->mmax + 1) / 2)));
  const size_t rr = (3 * (size_t)w->mmax * (w->mmax + 1 + (w->mmax & 1)) + 4 * (size_t)w->mmax) * es;
  w->rr_smem = rr <= (size_t)SMEM_PLAN_MAX ? rr : 0;
  if (w->rr_smem) {
    if (fp64) OFM_CUDA(c, cudaFuncSetAttribute(rayleigh_ritz_kernel<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_PLAN_MAX));
    else OFM_CUDA(c, cudaFuncSetAttribute(rayleigh_ritz_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_PLAN_MAX));
  }
  w->ready = true;
  return OFM_OK;
}

// Gram blocks of (Y, HY), Rayleigh-Ritz, rotation of Y into xo, residuals.
// H X = (H Y) C is formed only for the residual norms, in registers: the
// next filter starts from X alone and the export reads X, so it is never
// stored.
static ofm_status eig_rr(ofm_ctx* c, int y, int hy, int xo, unsigned long long salt, double tol) {
  EigWork* w = c->eig;
  const bool fp64 = c->storage == OFM_STORE_FP64;
  const int nf = c->nfrag;
  cudaStream_t s = c->stream;
  const EigFrag* ef = (const EigFrag*)w->d_efr.p;
  {
    KTimer kt(c, KC_GRAM, 2, w->gram_bytes, w->gram_flops);
    launch_eig_gram(w->gram, ef, nf, (const int4*)w->d_gitems.p, (const long long*)w->d_gpart.p,
                    (const int2*)w->d_gfrag.p, (const long long*)w->d_gblk.p, w->buf[y].p, w->buf[hy].p,
                    w->partials.p, (double*)w->blocks.p, fp64, s);
  }
  const long long mm = (long long)w->mmax * w->mmax;
  { KTimer kt(c, KC_RR);
  if (fp64)
    rayleigh_ritz_kernel<double><<<nf, w->rr_threads, w->rr_smem, s>>>(
        ef, (const long long*)w->d_gblk.p, (const double*)w->blocks.p,
        (double*)w->work.p, 3 * mm + 4 * w->mmax + 8, (double*)w->Cm.p, mm, (double*)w->theta.p,
        (const long long*)w->d_toff.p, 1e-13, (int*)w->d_rank.p, w->rr_smem > 0 ? 1 : 0, w->vlim[1], tol);
  else
    rayleigh_ritz_kernel<float><<<nf, w->rr_threads, w->rr_smem, s>>>(
        ef, (const long long*)w->d_gblk.p, (const double*)w->blocks.p,
        (float*)w->work.p, 3 * mm + 4 * w->mmax + 8, (double*)w->Cm.p, mm, (double*)w->theta.p,
        (const long long*)w->d_toff.p, 1e-5, (int*)w->d_rank.p, w->rr_smem > 0 ? 1 : 0, w->vlim[1], tol);
  }
  KTimer kt(c, KC_ROTATE, 2, w->rot_bytes, w->rot_flops);
  launch_eig_rotate(ef, (const DevFrag*)c->d_frags.p, nf, w->rot_blocks, w->rot_smem, w->buf[y].p, w->buf[hy].p,
                    w->buf[xo].p, (const double*)w->Cm.p, mm, (const int*)w->d_rank.p, (const double*)w->theta.p,
                    (const long long*)w->d_toff.p, (double*)w->rpart.p, w->mmax, salt, (double*)w->res.p, fp64, s);
  OFM_CUDA(c, cudaGetLastError());
  return OFM_OK;
}

// The filter of degree deg on block xb (workspace wb), then H Y: y and hy
// receive the blocks that hold Y and H Y.
static ofm_status eig_filter(ofm_ctx* c, int xb, int wb, int deg, int plain_slot, int& y, int& hy) {
  EigWork* w = c->eig;
  const int L = deg + 1;
  const int passes = eig_filter_passes(w->filter, L), steps = w->filter.steps.empty() ? 0 : L;
  // the first launch reads one block, the others two; every one writes two
  // (one, when it makes a single step)
  const double blocks = (2.0 * passes - 1.0) + (w->filter.S > 1 ? 2.0 : 1.0) * passes;
  KTimer kt(c, KC_FILTER, passes + steps,
            blocks * w->filter_block[0] + passes * w->filter_vc[0] + (3.0 * L - 1.0) * w->filter_block[1] +
                L * w->filter_vc[1],
            L * w->filter_flops);
  const int r = launch_eig_filter(w->filter, (const EigFrag*)w->d_efr.p, w->efr, (const int4*)w->d_jobs.p,
                                  (const int*)w->d_steps.p, w->buf[xb].p, w->buf[wb].p, w->vc.p,
                                  (const double*)w->coef.p, deg, plain_slot, c->storage == OFM_STORE_FP64,
                                  c->grid.h, c->stream);
  hy = r ? wb : xb;
  y = r ? xb : wb;
  OFM_CUDA(c, cudaGetLastError());
  return OFM_OK;
}

static ofm_status ofm_fragment_eigs_impl(ofm_ctx* c, const ofm_eig_opts* opts, double* eps_out,
                                        double* resid_out) {
  OFM_RANGE("ofm_fragment_eigs");
  if (!c) return OFM_ERR_INVALID;
  if (!c->built) return ofm_fail(c, OFM_ERR_STATE, "ofm_build_fragments must come first");
  if (!eps_out) return ofm_fail(c, OFM_ERR_INVALID, "eps_out must not be NULL");
  ofm_eig_opts o{};
  if (opts) o = *opts;
  const bool fp64 = c->storage == OFM_STORE_FP64;
  const double tol = o.tol > 0 ? o.tol : (fp64 ? 1e-9 : 1e-5);
  // 240: uneven FP32 blocks of 32-49 states in 16-24 point boxes once needed
  // 176 outer iterations (14 since the spread cap holds for whole blocks);
  // converged blocks stop early, so the bound costs nothing
  const int max_iter = o.max_iter > 0 ? o.max_iter : 240;
  const int degree = o.degree > 0 ? o.degree : 32;
  if (o.tol < 0 || o.max_iter < 0 || o.degree < 0 || o.extra_states < 0 || degree > 200)
    return ofm_fail(c, OFM_ERR_INVALID, "bad eigensolver options");
  if (!c->eig || !c->eig->ready || c->eig->efr.size() != (size_t)c->nfrag || o.extra_states > 0) {
    OFM_TRY(eig_setup(c, o.extra_states));
  }
  OFM_TRY(eig_vlim(c));
  EigWork* w = c->eig;
  const int nf = c->nfrag;
  cudaStream_t s = c->stream;
  c->assembled = c->dense_ready = c->factored = false;

  // c0 + V in the blocks' layout, and the start block in buffer 0
  {
    KTimer kt(c, KC_EIG_INIT, 2);
    launch_eig_vc((const EigFrag*)w->d_efr.p, (const DevFrag*)c->d_frags.p, w->efr, c->V.p, c->grid.n,
                  c->grid.h, w->vc.p, fp64, s);
    launch_eig_init((const EigFrag*)w->d_efr.p, (const DevFrag*)c->d_frags.p, w->efr, w->buf[0].p, o.seed, fp64, s);
  }
  OFM_CUDA(c, cudaGetLastError());
  // coefficient table: degree steps x fragments x (alpha, beta, shift)
  OFM_TRY(ofm_ensure(c, w->coef, sizeof(double) * 3 * nf * (degree + 1), "filter coefficients"));
  std::vector<double> coef(3 * (size_t)nf * (degree + 1));
  // plain H (alpha 1, beta 0, shift 0) sits in slot `degree`
  for (int f = 0; f < nf; ++f) {
    double* cf = &coef[3 * ((size_t)degree * nf + f)];
    cf[0] = 1.0; cf[1] = 0.0; cf[2] = 0.0;
  }
  OFM_CUDA(c, cudaMemcpyAsync(w->coef.p, coef.data(), sizeof(double) * coef.size(), cudaMemcpyHostToDevice, s));

  // initial Rayleigh-Ritz of the random block; xb holds the current block X
  int xb = 0, y = 0, hy = 0;
  OFM_TRY(eig_filter(c, 0, 1, 0, degree, y, hy));
  OFM_TRY(eig_rr(c, y, hy, 2, 0x1234ULL + o.seed, tol));
  xb = 2;
  std::vector<double> th(w->tsum), rs(w->tsum);
  const double bup = 6.0 / (c->grid.h * c->grid.h) + w->vlim[0];
  // The filter may spread the wanted part of the block by at most a factor
  // s: a component shrunk by s relative to the largest one in its vector
  // carries rounding of unit roundoff u x s.  For a random block every
  // vector mixes every state, so s <= 0.1 tol / u keeps that floor below
  // the tolerance (FP32: 1e2, FP64: 1e6).  Once the block holds Ritz
  // vectors, the lower states enter vector i only through its error,
  // about the largest residual r of the fragment, so the floor is u s r
  // and s may grow to 0.1 tol / (u r), up to 1e6 (FP32) / 1e12 (FP64).
  const double u_round = fp64 ? 1.1e-16 : 6e-8;
  const double s_min = fp64 ? 1e6 : 1e2, s_max = fp64 ? 1e12 : 1e6;
  // A spread that is too much for a fragment shows as a residual that grows
  // (boxes a few points thick: the rounding of the lower states comes back
  // larger than what the filter removed); its cap then falls tenfold, and from
  // then on it holds for the whole block: few wanted states next to each other
  // leave the degree free, and a guard vector swamped by the lowest state is lost
  // to the Gram's rank in every pass (one state with four guards in FP32, 48
  // random starts: 6 ended at 240 passes, all in 7 or fewer now).
  std::vector<double> cap(nf, s_max), rlast(nf, HUGE_VAL);
  bool converged = false;
  int it = 0;
  for (; it <= max_iter; ++it) {
    OFM_CUDA(c, cudaMemcpyAsync(th.data(), w->theta.p, sizeof(double) * w->tsum, cudaMemcpyDeviceToHost, s));
    OFM_CUDA(c, cudaMemcpyAsync(rs.data(), w->res.p, sizeof(double) * w->tsum, cudaMemcpyDeviceToHost, s));
    OFM_CUDA(c, cudaStreamSynchronize(s));
    converged = true;
    for (int f = 0; f < nf && converged; ++f)
      for (int i = 0; i < c->frags[f].n; ++i)
        if (!(rs[w->toff[f] + i] <= tol)) {
          converged = false;
          break;
        }
    if (converged || it == max_iter) break;
    // degree of this iteration: T_d grows like exp(d acosh(t)) below the
    // damped interval, so the ratio between the bottom of the spectrum
    // (min V on the first pass, the lowest Ritz value after) and the last
    // wanted Ritz value is about exp(d (acosh(t_low) - acosh(t_want)));
    // keep it within the fragment's spread cap for every fragment
    int deg = degree;
    for (int f = 0; f < nf; ++f) {
      const int m = w->efr[f].n;
      const double* t = &th[w->toff[f]];
      double rmax = 0.0;
      for (int i = 0; i < c->frags[f].n; ++i) rmax = std::max(rmax, rs[w->toff[f] + i]);
      if (it > 1 && rmax > 3.0 * rlast[f]) cap[f] = std::max(s_min, 0.1 * cap[f]);
      rlast[f] = rmax;
      const double smax = (it == 0 || !(rmax > 0.0))
                              ? s_min
                              : std::min(cap[f], std::max(s_min, 0.1 * tol / (u_round * rmax)));
      const double spread_max = std::log(smax);
      double blo = t[m - 1], a0 = t[0];
      double bu = std::max(bup, blo + 1e-3);
      if (!(blo > a0)) blo = a0 + 1e-3 * (bu - a0);
      const double e = 0.5 * (bu - blo), cc = 0.5 * (bu + blo);
      const double low = (it == 0) ? std::min(w->vlim[1], a0) : a0;
      const int top = cap[f] < s_max ? m - 1 : c->frags[f].n - 1;
      const double tl = (cc - low) / e, tw = (cc - t[top]) / e;
      if (tl > 1.0) {
        const double gap = std::acosh(tl) - (tw > 1.0 ? std::acosh(tw) : 0.0);
        if (gap > 0.0) deg = std::min(deg, std::max(4, (int)(spread_max / gap)));
      }
    }
    // filter coefficients from the current Ritz values
    for (int f = 0; f < nf; ++f) {
      const int m = w->efr[f].n;
      const double* t = &th[w->toff[f]];
      double blo = t[m - 1], a0 = t[0];
      double bu = std::max(bup, blo + 1e-3);
      if (!(blo > a0)) blo = a0 + 1e-3 * (bu - a0);
      const double e = 0.5 * (bu - blo), cc = 0.5 * (bu + blo);
      const double sigma1 = e / (a0 - cc);
      double sigma = sigma1;
      const double tau = 2.0 / sigma1;
      for (int k = 0; k < deg; ++k) {
        double* cf = &coef[3 * ((size_t)k * nf + f)];
        if (k == 0) {
          cf[0] = sigma1 / e;
          cf[1] = 0.0;
        } else {
          const double sn = 1.0 / (tau - sigma);
          cf[0] = 2.0 * sn / e;
          cf[1] = -sigma * sn;
          sigma = sn;
        }
        cf[2] = cc;
      }
    }
    OFM_CUDA(c, cudaMemcpyAsync(w->coef.p, coef.data(), sizeof(double) * 3 * nf * deg, cudaMemcpyHostToDevice, s));
    const int wb = (xb + 1) % 3, xo = (xb + 2) % 3;
    OFM_TRY(eig_filter(c, xb, wb, deg, degree, y, hy));
    OFM_TRY(eig_rr(c, y, hy, xo, 0x9876ULL * (it + 1) + o.seed, tol));
    xb = xo;
  }
  // export the first n_a Ritz vectors with the sign gauge
  {
    int nmax = 1;
    for (const DevFrag& F : c->frags) nmax = std::max(nmax, F.n);
    KTimer kt(c, KC_EXPORT, 2);
    launch_eig_export((const EigFrag*)w->d_efr.p, (const DevFrag*)c->d_frags.p, w->efr, nmax, w->buf[xb].p,
                      w->sgn.p, w->mmax, c->states.p, fp64, s);
  }
  OFM_CUDA(c, cudaGetLastError());
  OFM_CUDA(c, cudaStreamSynchronize(s));
  double worst = 0.0;
  for (int f = 0; f < nf; ++f)
    for (int i = 0; i < c->frags[f].n; ++i) {
      eps_out[c->frags[f].basis0 + i] = th[w->toff[f] + i];
      if (resid_out) resid_out[c->frags[f].basis0 + i] = rs[w->toff[f] + i];
      worst = std::max(worst, rs[w->toff[f] + i]);
    }
  OFM_TRY(ofm_wait_status(c));
  std::fill(c->frag_set.begin(), c->frag_set.end(), 1);
  c->have_states = true;
  c->last_eig_iters = it;
  const bool injected = c->fault == OFM_FAULT_NONCONV;
  if (injected) converged = false;
  if (!converged) {
    char buf[192];
    if (injected)
      snprintf(buf, sizeof buf, "fragment eigensolver: not converged (injected by OFM_FAULT=nonconv; "
               "largest residual %.3e after %d iterations)", worst, it);
    else
      snprintf(buf, sizeof buf, "fragment eigensolver: largest residual %.3e > tol %.3e after %d iterations",
               worst, tol, it);
    return ofm_fail(c, OFM_ERR_NOT_CONVERGED, buf);
  }
  return OFM_OK;
}

extern "C" ofm_status ofm_fragment_eigs(ofm_ctx* c, const ofm_eig_opts* opts, double* eps_out, double* resid_out) {
  const ofm_status st = ofm_fragment_eigs_impl(c, opts, eps_out, resid_out);
  if ((st != OFM_OK && st != OFM_ERR_NOT_CONVERGED) || !c || !c->checks) return st;
  const ofm_status g = ofm_check_guards_now(c, "ofm_fragment_eigs");
  return g != OFM_OK ? g : st;
}
