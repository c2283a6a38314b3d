// Eigenvectors of Eq. 2 for the eigenvalues of an energy window (the
// optional C of the window solve), from the factorisation the eigenvalues
// came from:
//   1. inverse iteration on the tridiagonal T: for each eigenvalue lambda
//      (accurate to a few ulps from the Sturm multisection), solve
//      (T - lambda I) y = b three times from a pseudo-random b, with
//      Gaussian elimination with partial pivoting on the tridiagonal matrix
//      (the row exchanges fill one extra superdiagonal); y grows along the
//      eigenvector by 1/|lambda - lambda_true| per solve.  Eigenvalues
//      closer than 1e-5 ||T||_1 form a cluster, whose vectors are computed
//      in order by one warp and orthogonalised against each other (modified
//      Gram-Schmidt) after every solve; separate clusters run in parallel.
//   2. back-transformation x = Q y with the Householder reflectors of the
//      tridiagonal reduction, Q = H_0 H_1 ... H_{n-3}, H_k = I - tau_k v_k v_k^T
//      (v_k kept in row k of the reduced matrix), applied from k = n-3 down;
//   3. C = L^-T x (back substitution with the Cholesky factor), so that
//      H C = S C diag(E) and C^T S C = I.
// Steps 2 and 3 run in one CTA per eigenvector.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <vector>

#include "fp64_util.h"
#include "ofm_internal.h"

namespace ofm {

namespace {

__device__ __forceinline__ double warp_sum(double s) {
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Deterministic start vector entry in [-1, 1): SplitMix64 of (index, row).
__device__ __forceinline__ double start_entry(unsigned long long j, unsigned long long i) {
  unsigned long long z = (j << 32) ^ i ^ 0x5851F42D4C957F2DULL;
  z += 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  z ^= z >> 31;
  return (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

// One warp per cluster of eigenvalues [cl[c], cl[c+1]).  Scratch per cluster:
// dd, du, du2, dl (n each) and a byte of pivoting per row, in shared memory
// with the current vector where they fit (scratch == nullptr), else in global
// memory.  Lane 0 runs the sequential factorisation and solves with the running
// entry in a register: the chain per row is one FMA (forward) and one FMA (back
// substitution, with U's rows scaled by their reciprocal diagonals
// beforehand); the warp does the vector work.  315 rows, 31 vectors with the
// back-transformation below: 1126 us with scratch in global memory and rows of
// R and L read when they are due, 742 us now.
__global__ void __launch_bounds__(32) stein_kernel(const double* __restrict__ d,
                                                    const double* __restrict__ e, int n,
                                                    const double* __restrict__ lam,
                                                    const int* __restrict__ cl, double tnorm,
                                                    double* scratch, unsigned char* piv_scratch,
                                                    double* __restrict__ Y) {
  extern __shared__ __align__(16) double st_smem[];
  const int c = blockIdx.x, lane = threadIdx.x;
  double* dd = scratch ? scratch + (size_t)c * 5 * n : st_smem;
  double* du = dd + n;
  double* du2 = du + n;
  double* dl = du2 + n;
  double* y = dl + n;
  unsigned char* swp = scratch ? piv_scratch + (size_t)c * n : reinterpret_cast<unsigned char*>(y + n);
  const double pert = DBL_EPSILON * tnorm;   // replaces an exactly singular pivot
  auto mag = [](double x) { return __double_as_longlong(x) & 0x7fffffffffffffffLL; };   // |x| as ordered bits
  for (int j = cl[c]; j < cl[c + 1]; ++j) {
    double* yj = Y + (size_t)j * n;
    const double shift = lam[j];
    for (int i = lane; i < n; i += 32) {
      dd[i] = d[i] - shift;
      dl[i] = i + 1 < n ? e[i] : 0.0;
      y[i] = start_entry((unsigned long long)j, (unsigned long long)i);
    }
    __syncwarp();
    if (lane == 0) {
      // LU of T - shift I with partial pivoting, rows i and i + 1 in registers:
      // (p, u): the current row's diagonal and superdiagonal; dd becomes U's
      // reciprocal diagonal, du and du2 its superdiagonals, dl the multipliers
      double p = dd[0], u = n > 1 ? dl[0] : 0.0;
      for (int i = 0; i + 1 < n; ++i) {
        const double l = dl[i], pn = dd[i + 1], un = i + 2 < n ? dl[i + 1] : 0.0;
        if (mag(p) >= mag(l)) {
          if (p == 0.0) p = pert;
          const double r = rcp64(p), f = l * r;
          swp[i] = 0;
          dd[i] = r;
          du[i] = u;
          du2[i] = 0.0;
          dl[i] = f;
          p = fma(-f, u, pn);
          u = un;
        } else {
          const double r = rcp64(l), f = p * r;
          swp[i] = 1;
          dd[i] = r;
          du[i] = pn;
          du2[i] = un;
          dl[i] = f;
          p = fma(-f, pn, u);
          u = -f * un;
        }
      }
      if (p == 0.0) p = pert;
      dd[n - 1] = rcp64(p);
      du[n - 1] = du2[n - 1] = 0.0;
    }
    __syncwarp();
    for (int i = lane; i < n; i += 32) {
      du[i] *= -dd[i];
      du2[i] *= -dd[i];
    }
    __syncwarp();
    for (int it = 0; it < 3; ++it) {
      if (lane == 0) {
        // forward: apply the row exchanges and L
        double t = y[0];
        for (int i = 0; i + 1 < n; ++i) {
          const double b = y[i + 1], l = dl[i];
          const bool sw = swp[i] != 0;
          y[i] = sw ? b : t;
          t = sw ? fma(-l, b, t) : fma(-l, t, b);
        }
        y[n - 1] = t;
      }
      __syncwarp();
      for (int i = lane; i < n; i += 32) y[i] *= dd[i];
      __syncwarp();
      if (lane == 0) {
        // back substitution with U's scaled rows
        double y1 = y[n - 1], y2 = 0.0;
        for (int i = n - 2; i >= 0; --i) {
          const double t = fma(du[i], y1, fma(du2[i], y2, y[i]));
          y[i] = t;
          y2 = y1;
          y1 = t;
        }
      }
      __syncwarp();
      // orthogonalise against the cluster's earlier vectors
      for (int q = cl[c]; q < j; ++q) {
        const double* yq = Y + (size_t)q * n;
        double s = 0.0;
        for (int i = lane; i < n; i += 32) s += yq[i] * y[i];
        s = warp_sum(s);
        for (int i = lane; i < n; i += 32) y[i] -= s * yq[i];
        __syncwarp();
      }
      double s = 0.0;
      for (int i = lane; i < n; i += 32) s += y[i] * y[i];
      s = warp_sum(s);
      const double inv = s > 0.0 ? 1.0 / sqrt(s) : 1.0;
      for (int i = lane; i < n; i += 32) y[i] *= inv;
      __syncwarp();
    }
    for (int i = lane; i < n; i += 32) yj[i] = y[i];
    __syncwarp();
  }
}

// Eight bytes into shared memory, asynchronously.
__device__ __forceinline__ void cpa8(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"((unsigned long long)__cvta_generic_to_global(src))
               : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One CTA of four warps (one per FP64 sub-partition: more only queue) per
// eigenvector: x = Q y, then C(:, j) = L^-T x.  Both are chains of n steps of
// one dot product or one multiple; a step costs one barrier, and its row of R or
// L arrives through a ring of shared-memory rows filled three steps ahead (each
// thread copies the entries i = tid mod 128 that it also uses, so no barrier
// guards the ring).  RING 0: no ring (the rows do not fit), read in place.
constexpr int BT_THREADS = 128;
template <int RING>
__global__ void __launch_bounds__(BT_THREADS) backtransform_kernel(const double* __restrict__ R,
                                                                   const double* __restrict__ tau,
                                                                   const double* __restrict__ L, int n,
                                                                   const double* __restrict__ Y,
                                                                   double* __restrict__ C) {
  extern __shared__ double sx[];
  double* x = sx;         // n
  double* dinv = sx + n;  // n
  double* ring = dinv + n;   // RING rows of n
  __shared__ double red[2][4];
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < n; i += BT_THREADS) {
    x[i] = Y[(size_t)j * n + i];
    dinv[i] = rcp64(L[(size_t)i * n + i]);
  }
  // entries [lo, hi) of row r of M into ring slot q, the thread's own ones
  auto fetch = [&](const double* M, int r, int lo, int hi, int q) {
    if (RING > 0) {
      if (r >= 0 && r < n)
        for (int i = lo + ((tid - lo) & (BT_THREADS - 1)); i < hi; i += BT_THREADS)
          cpa8(ring + (size_t)q * n + i, M + (size_t)r * n + i);
      cpa_commit();
    }
  };
  constexpr int AHEAD = RING > 0 ? RING - 1 : 0;
  // x = H_0 (H_1 (... (H_{n-3} y))): thread tid owns the entries i = tid mod 128
  int buf = 0, q = 0;
  for (int a = 0; a < AHEAD; ++a) fetch(R, n - 3 - a, n - 2 - a, n, a);
  for (int k = n - 3; k >= 0; --k) {
    fetch(R, k - AHEAD, k - AHEAD + 1, n, RING > 0 ? (q + AHEAD) % RING : 0);
    cpa_wait<AHEAD>();
    const double* v = RING > 0 ? ring + (size_t)q * n : R + (size_t)k * n;
    if (RING > 0) q = (q + 1) % RING;
    const double t = tau[k];
    if (t == 0.0) continue;   // uniform over the CTA
    double s = 0.0;
    const int i0 = k + 1 + ((tid - k - 1) & (BT_THREADS - 1));   // first owned entry > k
    for (int i = i0; i < n; i += BT_THREADS) s = fma(v[i], x[i], s);
    s = warp_sum(s);
    if (lane == 0) red[buf][warp] = s;
    __syncthreads();
    const double f = -t * ((red[buf][0] + red[buf][1]) + (red[buf][2] + red[buf][3]));
    buf ^= 1;
    for (int i = i0; i < n; i += BT_THREADS) x[i] = fma(f, v[i], x[i]);
  }
  cpa_wait<0>();
  __syncthreads();
  // L^T c = x, from the last row up: c_i = x_i / L_ii, then x_p -= L_ip c_i (p < i)
  q = 0;
  for (int a = 0; a < AHEAD; ++a) fetch(L, n - 1 - a, 0, n - 1 - a, a);
  for (int i = n - 1; i >= 0; --i) {
    fetch(L, i - AHEAD, 0, i - AHEAD, RING > 0 ? (q + AHEAD) % RING : 0);
    cpa_wait<AHEAD>();
    const double* Li = RING > 0 ? ring + (size_t)q * n : L + (size_t)i * n;
    if (RING > 0) q = (q + 1) % RING;
    const double cv = x[i] * dinv[i];
    for (int p = tid; p < i; p += BT_THREADS) x[p] = fma(-Li[p], cv, x[p]);
    __syncthreads();
    if (tid == 0) C[(size_t)j * n + i] = cv;
  }
}

}  // namespace

}  // namespace ofm

using namespace ofm;

// m eigenvectors for the eigenvalues E (host copy, ascending) that the last
// ofm_window_bisect left on the device in w_tmp[0..m).
ofm_status ofm_window_vectors(ofm_ctx* c, int m, const double* E, double* C_out) {
  const int n = c->dense_n;
  cudaStream_t s = c->stream;
  // ||T||_1 from d and e for the cluster threshold and the pivot guard
  std::vector<double> hd(n), he(std::max(1, n - 1));
  OFM_CUDA(c, cudaMemcpyAsync(hd.data(), c->w_d.p, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
  if (n > 1)
    OFM_CUDA(c, cudaMemcpyAsync(he.data(), c->w_e.p, sizeof(double) * (n - 1), cudaMemcpyDeviceToHost, s));
  OFM_CUDA(c, cudaStreamSynchronize(s));
  double tnorm = 0.0;
  for (int i = 0; i < n; ++i) {
    const double r = std::fabs(hd[i]) + (i > 0 ? std::fabs(he[i - 1]) : 0.0) +
                     (i + 1 < n ? std::fabs(he[i]) : 0.0);
    tnorm = std::max(tnorm, r);
  }
  if (!(tnorm > 0.0)) tnorm = 1.0;
  std::vector<int> cl{0};
  for (int j = 1; j < m; ++j)
    if (E[j] - E[j - 1] > 1e-5 * tnorm) cl.push_back(j);
  cl.push_back(m);
  const int nc = (int)cl.size() - 1;
  // device scratch: eigenvalues stay in w_tmp; Y, C, LU arrays, cluster table
  const size_t ybytes = sizeof(double) * (size_t)n * m;
  // the factorisations live in shared memory where they fit
  const size_t stmem = (5 * sizeof(double) + 1) * (size_t)n;
  const bool in_smem = stmem <= (size_t)SMEM_PLAN_MAX;
  const size_t lubytes = in_smem ? 0 : sizeof(double) * 5 * (size_t)n * nc;
  const size_t pivbytes = in_smem ? 0 : ((size_t)n * nc + 15) / 16 * 16;
  const size_t clbytes = sizeof(int) * (size_t)(nc + 1);
  const size_t total = 2 * ybytes + lubytes + pivbytes + clbytes + 1024;
  OFM_TRY(ofm_ensure(c, c->staging, total, "window eigenvector scratch"));
  unsigned char* base = (unsigned char*)c->staging.p;
  double* Y = (double*)base;
  double* Cd = (double*)(base + ybytes);
  double* lu = (double*)(base + 2 * ybytes);
  unsigned char* piv = base + 2 * ybytes + lubytes;
  int* dcl = (int*)(base + 2 * ybytes + lubytes + pivbytes);
  OFM_CUDA(c, cudaMemcpyAsync(dcl, cl.data(), clbytes, cudaMemcpyHostToDevice, s));
  {
    KTimer kt(c, KC_VECTORS, 2, 0.0, 4.0 * n * (double)n * m);
    if (in_smem && stmem > 48 * 1024)
      OFM_CUDA(c, cudaFuncSetAttribute(stein_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_PLAN_MAX));
    stein_kernel<<<nc, 32, in_smem ? stmem : 0, s>>>((const double*)c->w_d.p, (const double*)c->w_e.p, n,
                                                    (const double*)c->w_tmp.p, dcl, tnorm,
                                                    in_smem ? nullptr : lu, piv, Y);
    const size_t row = sizeof(double) * (size_t)n;
    const bool ring = 6 * row <= (size_t)SMEM_PLAN_MAX;
    const size_t smem = (ring ? 6 : 2) * row;
    const void* bt = ring ? (const void*)backtransform_kernel<4> : (const void*)backtransform_kernel<0>;
    if (smem > 48 * 1024) OFM_CUDA(c, cudaFuncSetAttribute(bt, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_PLAN_MAX));
    const double *R = (const double*)c->w_A.p, *tau = (const double*)c->w_tau.p, *L = (const double*)c->w_L.p;
    if (ring) backtransform_kernel<4><<<m, BT_THREADS, smem, s>>>(R, tau, L, n, Y, Cd);
    else backtransform_kernel<0><<<m, BT_THREADS, smem, s>>>(R, tau, L, n, Y, Cd);
  }
  OFM_CUDA(c, cudaGetLastError());
  OFM_CUDA(c, cudaMemcpyAsync(C_out, Cd, ybytes, cudaMemcpyDeviceToHost, s));
  OFM_CUDA(c, cudaStreamSynchronize(s));
  return OFM_OK;
}
