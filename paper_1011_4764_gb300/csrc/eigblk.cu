// Block operations of the fragment eigensolver (a0): start vectors, the
// Chebyshev filter, the Gram matrices, the rotation by the Ritz coefficients
// and the export of the states.
//
// Layout.  A fragment's block is state-major: state j is one contiguous vector
// of the box's points (EigFrag: the layout's axes are a permutation of the
// grid's, slowest the longest one the box does not span, its extent along the
// fastest axis padded to a multiple of four with zeros).  Each operation then streams whole
// vectors: the filter keeps planes on chip, the Gram and the
// rotation read and write points with 16-byte accesses and no transposition.
// The library's states are point-major; init and export convert once per solve.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>
#include <vector>

#include "ofm_internal.h"

namespace ofm {
namespace {

__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ULL;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
  return x ^ (x >> 31);
}

// Box coordinates of layout point t; false for the padding of the fastest axis.
__device__ __forceinline__ bool box_coords(const EigFrag& E, int t, int (&q)[3]) {
  const int c0 = t % E.e0p, r = t / E.e0p;
  const int c1 = r % E.e[1], c2 = r / E.e[1];
  q[E.ax[0]] = c0;
  q[E.ax[1]] = c1;
  q[E.ax[2]] = c2;
  return c0 < E.e[0] && c2 < E.e[2];
}

// Index of box point q in the fragment's dilated storage box.
__device__ __forceinline__ int dilated_index(const DevFrag& F, const int (&q)[3]) {
  return ((q[2] + F.lo[2]) * F.dext[1] + q[1] + F.lo[1]) * F.dext[0] + q[0] + F.lo[0];
}

__device__ __forceinline__ double uniform53(unsigned long long r) {
  return (double)(r >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

__device__ __forceinline__ void cpa16z(void* dst, const void* src, bool ok) {
  const int n = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"((unsigned long long)__cvta_generic_to_global(src)), "r"(n)
               : "memory");
}
__device__ __forceinline__ void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cpa_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// ------------------------------------------------------------------ start --

// Uniform(-1, 1) start vectors on the box points (53 random bits for FP64
// storage, 24 for FP32: FP32 arithmetic there), zero in the padding.
template <typename T>
__global__ void __launch_bounds__(256) eig_init_kernel(const EigFrag* ef, const DevFrag* fr, T* X,
                                                       unsigned long long seed) {
  const int f = blockIdx.z, j = blockIdx.y;
  const EigFrag E = ef[f];
  if (j >= E.n) return;
  const DevFrag F = fr[f];
  const unsigned long long s0 = splitmix64(seed);
  for (int t = blockIdx.x * 256 + threadIdx.x; t < E.Ps; t += 256 * gridDim.x) {
    int q[3];
    T v = T(0);
    if (box_coords(E, t, q) && j < E.n) {
      const unsigned long long key = ((unsigned long long)f << 44) ^ ((unsigned long long)j << 32) ^
                                     (unsigned long long)dilated_index(F, q);
      const unsigned long long r = splitmix64(key + s0);
      if (sizeof(T) == 8) v = (T)uniform53(r);
      else v = (T)((float)(r >> 40) * (2.0f / 16777216.0f) - 1.0f);
    }
    X[E.off + (long long)j * E.Ps + t] = v;
  }
}

// c0 + V on every box point, in the layout's order.
template <typename T>
__global__ void __launch_bounds__(256) eig_vc_kernel(const EigFrag* ef, const DevFrag* fr, const T* V,
                                                     T c0, int gx, int gy, int gz, T* vc) {
  const EigFrag E = ef[blockIdx.y];
  const DevFrag F = fr[blockIdx.y];
  for (int t = blockIdx.x * 256 + threadIdx.x; t < E.Ps; t += 256 * gridDim.x) {
    int q[3];
    T v = T(0);
    if (box_coords(E, t, q)) {
      const int x = (F.doff[0] + F.lo[0] + q[0]) % gx, y = (F.doff[1] + F.lo[1] + q[1]) % gy,
                z = (F.doff[2] + F.lo[2] + q[2]) % gz;
      v = c0 + V[(long long)x + (long long)gx * (y + (long long)gy * z)];
    }
    vc[E.voff + t] = v;
  }
}

// ----------------------------------------------------------------- filter --
//
// One step of the scaled three-term recurrence is
//     u_{k+1} = al (H u_k - sh u_k) + be u_{k-1},
// three blocks through HBM.  In FP32 a launch advances S steps: a CTA owns
// whole planes (every point of the two fastest axes) of one or more vectors and
// marches along the third axis; at tick t level s computes plane t - s of
// u_{k+s}, from the plane level s - 1 computed one tick earlier (in-plane
// neighbours through shared memory), the planes before and after it
// (registers) and u_{k+s-2} (the register level s - 2 kept for its own lower
// neighbour).  No point is computed twice, and S steps read two blocks and
// write two: 4 / S blocks a step instead of three.  The last launch ends with
// H u_d (al 1, be 0, sh 0), so its two outputs are Y and H Y.  In place: a launch
// reads planes t + 1 and t of two blocks and writes planes t - S + 1 and t - S of
// the same two, each thread its own points only.
// A thread owns 4 x 2 points of the plane.  What its neighbours read lies in
// shared memory by patch: both rows (16 bytes each) and the left and right
// columns (8 bytes each), so every access of a warp is contiguous: 34
// wavefronts per warp, level and 256 points (12 of them writes, 8 for c0 + V).
// The arithmetic is packed FP32 pairs along x.  The bound is shared memory and
// instruction issue instead of HBM.  FP64 goes one step per launch: it is bound
// by the FP64 pipe (8 instructions per point), which a CTA per vector spreads
// worse over the SMs than a thread per point.
// Measured per step (27 boxes of 40^3, 120 vectors, FP32): 250 us against 432 us for one
// launch per step.

// the type's own fused multiply-add (an unqualified fma of floats may be the
// FP64 one)
__device__ __forceinline__ float fma1(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma1(double a, double b, double c) { return ::fma(a, b, c); }

// threads of a filter CTA at most: 14 warps at 128 registers, 12 at 168 (S = 4)
__host__ __device__ constexpr int ft_max(int S) { return S == 4 ? 384 : 448; }

template <typename T> struct Pk;
template <> struct Pk<float> {
  using E = unsigned long long;
  static constexpr int NS = 2;
  static __device__ __forceinline__ E zero() { return 0ULL; }
  static __device__ __forceinline__ E dup(float a) {
    E r;
    asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
    return r;
  }
  static __device__ __forceinline__ E pack(float a, float b) {
    E r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
  }
  static __device__ __forceinline__ float2 unpack(E a) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a));
    return r;
  }
  static __device__ __forceinline__ E add(E a, E b) {
    E r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
  }
  static __device__ __forceinline__ E mul(E a, E b) {
    E r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
  }
  static __device__ __forceinline__ E fma(E a, E b, E c) {
    E r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
  }
};
template <> struct Pk<double> {
  using E = double;
  static constexpr int NS = 1;
  static __device__ __forceinline__ E zero() { return 0.0; }
  static __device__ __forceinline__ E dup(double a) { return a; }
  static __device__ __forceinline__ E add(E a, E b) { return a + b; }
  static __device__ __forceinline__ E mul(E a, E b) { return a * b; }
  static __device__ __forceinline__ E fma(E a, E b, E c) { return ::fma(a, b, c); }
};

template <typename E>
struct alignas(16) E2 {
  E a, b;
};

__device__ __forceinline__ void cpa16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"((unsigned long long)__cvta_generic_to_global(src))
               : "memory");
}

// Words of a level's exchange area for tp patches: top rows, bottom rows, left
// and right columns, each with one more entry that stays zero.
__host__ __device__ constexpr int filter_area(int tp) { return 12 * (tp + 1); }

// job: fragment, first vector, vectors of this CTA.  A holds u_k and receives
// level S - 1 (untouched when S is 1), B holds u_{k-1} (has_prev) and receives
// level S.  Coefficients of level s: slot k0 + s - 1, or plain_slot for level S
// when plain_last.  EVEN: every box has e[0] a multiple of 4 and e[1] even, so
// every patch is whole (the tests of ragged patches are half the instructions).
template <int S, bool EVEN>
__global__ void __launch_bounds__(ft_max(S), 1) eig_filter_kernel(
    const EigFrag* __restrict__ ef, const int4* __restrict__ jobs, float* A, float* B,
    const float* __restrict__ vc, const double* __restrict__ coef, int nfrag, int k0, int plain_last,
    int plain_slot, int has_prev, float c1) {
  using P = Pk<float>;
  using E = P::E;
  constexpr int RING = S + 2;
  extern __shared__ __align__(16) float fsm[];
  __shared__ ulonglong2 cf[2 * S];   // {al, al} {-al sh, ..}, {-al c1, ..} {be, be}
  const int4 job = jobs[blockIdx.x];
  const EigFrag* Fp = ef + job.x;
  const int e0 = Fp->e[0], e1 = Fp->e[1], e2 = Fp->e[2], e0p = Fp->e0p;
  const int hx = e0p / 4, hy = (e1 + 1) / 2, tp = hx * hy;   // patches of a plane
  const int vplane = e0p * e1;                               // points of a plane
  const int area = filter_area(tp);
  const int np = job.z, tid = threadIdx.x;
  float* vring = fsm + np * 2 * S * area;                    // RING planes of c0 + V
  for (int i = tid; i < np * 2 * S * area; i += blockDim.x) fsm[i] = 0.f;
  if (tid < S) {
    const int slot = (plain_last && tid + 1 == S) ? plain_slot : k0 + tid;
    const double* c = coef + 3 * ((size_t)slot * nfrag + job.x);
    const float al = (float)c[0];
    cf[2 * tid] = make_ulonglong2(P::dup(al), P::dup(-al * (float)c[2]));
    cf[2 * tid + 1] = make_ulonglong2(P::dup(-al * c1), P::dup((float)c[1]));
  }
  const int pi = tid / tp;
  const bool live = pi < np;
  const int pt = tid - pi * tp, px = pt % hx, py = pt / hx;
  const int nv = EVEN ? 4 : min(4, e0 - 4 * px);   // valid columns of the patch
  const bool vy = EVEN || 2 * py + 1 < e1;
  // exchange area: entry words of the neighbours (tp: the zero entry)
  const int oT = 0, oB = 4 * (tp + 1), oL = 8 * (tp + 1), oR = 10 * (tp + 1);
  const bool f0 = Fp->full[0] != 0, f1 = Fp->full[1] != 0;
  const int up = py > 0 ? oB + 4 * (pt - hx)
                 : !f1  ? 4 * tp
                        : ((e1 & 1) ? oT : oB) + 4 * (pt + (hy - 1) * hx);
  const int dn = py + 1 < hy ? oT + 4 * (pt + hx) : f1 ? oT + 4 * px : 4 * tp;
  const int lf = px > 0 ? oR + 2 * (pt - 1) : f0 ? oR + 2 * (pt + hx - 1) : 4 * tp;
  const int rg = px + 1 < hx ? oL + 2 * (pt + 1) : f0 ? oL + 2 * (pt - px) : 4 * tp;
  const int vo = 2 * py * e0p + 4 * px, vo1 = vy ? e0p : 0;
  float* my = fsm + (live ? pi : 0) * 2 * S * area;
  const long long g0 = Fp->off + (long long)(job.y + (live ? pi : 0)) * Fp->Ps + vo;
  float* pa = A + g0;
  float* pb = B + g0;
  const float* vg = vc + Fp->voff;

  E bel[S][4], vin[4], pin[4];   // pairs: row 0 columns 01, 23, row 1 columns 01, 23
#pragma unroll
  for (int s = 0; s < S; ++s)
#pragma unroll
    for (int i = 0; i < 4; ++i) bel[s][i] = 0ULL;
#pragma unroll
  for (int i = 0; i < 4; ++i) vin[i] = pin[i] = 0ULL;
  auto ldrow = [](const float* p, E& a, E& b) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    a = v.x;
    b = v.y;
  };
  // plane t of u_k, plane t - 1 of u_{k-1} into registers
  auto fetch = [&](int t) {
    if (has_prev && t > 0 && t <= e2) {
      const float* p = pb + (t - 1) * vplane;
      ldrow(p, pin[0], pin[1]);
      if (vy) ldrow(p + e0p, pin[2], pin[3]);
    }
    if (t < e2) {
      const float* p = pa + t * vplane;
      ldrow(p, vin[0], vin[1]);
      if (vy) ldrow(p + e0p, vin[2], vin[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) vin[i] = 0ULL;
    }
  };
  // plane t of c0 + V into its ring slot
  auto fetch_v = [&](int t, int slot) {
    if (t < e2)
      for (int i = 4 * tid; i < vplane; i += 4 * blockDim.x)
        cpa16(vring + slot * vplane + i, vg + (long long)t * vplane + i);
    cpa_commit();
  };
  // a patch into a level's exchange area; its last valid column is the right one
  auto put = [&](float* o, const E (&v)[4]) {
    *reinterpret_cast<ulonglong2*>(o + oT + 4 * pt) = make_ulonglong2(v[0], v[1]);
    *reinterpret_cast<ulonglong2*>(o + oB + 4 * pt) = make_ulonglong2(v[2], v[3]);
    const float2 a = P::unpack(v[0]), b = P::unpack(v[1]), c = P::unpack(v[2]), d = P::unpack(v[3]);
    *reinterpret_cast<float2*>(o + oL + 2 * pt) = make_float2(a.x, c.x);
    float2 r = make_float2(b.y, d.y);
    if (nv < 4) r = nv == 3 ? make_float2(b.x, d.x) : nv == 2 ? make_float2(a.y, c.y) : make_float2(a.x, c.x);
    *reinterpret_cast<float2*>(o + oR + 2 * pt) = r;
  };
  fetch_v(0, 0);
  if (live) fetch(0);
  __syncthreads();   // the zeroed areas, the coefficients
  int vslot = 0;     // ring slot of plane t
  for (int t = 0; t < e2 + S; ++t) {
    const int vnext = vslot + 1 == RING ? 0 : vslot + 1;
    fetch_v(t + 1, vnext);
    if (live) {
      E ab[4], pv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ab[i] = vin[i];    // plane t of u_k: above level 1's plane
        pv[i] = pin[i];    // plane t - 1 of u_{k-1}
      }
      float* wr = my + (t & 1) * S * area;
      const float* rd = my + ((t & 1) ^ 1) * S * area;
      if (t < e2) put(wr, ab);
#pragma unroll
      for (int s = 1; s <= S; ++s) {
        const int p = t - s;
        E nw[4];
        if (p >= 0 && p < e2) {
          const float* pl = rd + (s - 1) * area;
          int vs = vslot - s;
          if (vs < 0) vs += RING;
          const float* v = vring + vs * vplane + vo;
          E c[4];
          ldrow(pl + oT + 4 * pt, c[0], c[1]);
          ldrow(pl + oB + 4 * pt, c[2], c[3]);
          const ulonglong2 q0 = cf[2 * s - 2], q1 = cf[2 * s - 1];
          const float2 l = *reinterpret_cast<const float2*>(pl + lf);
          const float2 r = *reinterpret_cast<const float2*>(pl + rg);
          E d0, d1;
          ldrow(pl + dn, d0, d1);
          // right neighbours come from the patch, or after its last valid column
          // from the loaded one
          {   // row 0
            E u0, u1, w0, w1;
            ldrow(pl + up, u0, u1);
            ldrow(v, w0, w1);
            const float2 a = P::unpack(c[0]), b = P::unpack(c[1]);
            float xa = a.y, xb = b.x, xc = b.y;
            E m0 = c[2], m1 = c[3];
            if constexpr (!EVEN) {
              if (nv == 1) xa = r.x;
              if (nv == 2) xb = r.x;
              if (nv == 3) xc = r.x;
              if (!vy) { m0 = d0; m1 = d1; }
            }
            const E s0 = P::add(P::add(P::add(u0, m0), P::pack(l.x + xa, a.x + xb)), P::add(bel[s - 1][0], ab[0]));
            const E s1 = P::add(P::add(P::add(u1, m1), P::pack(a.y + xc, b.x + r.x)), P::add(bel[s - 1][1], ab[1]));
            nw[0] = P::fma(q1.x, s0, P::fma(P::fma(q0.x, w0, q0.y), c[0], P::mul(q1.y, pv[0])));
            nw[1] = P::fma(q1.x, s1, P::fma(P::fma(q0.x, w1, q0.y), c[1], P::mul(q1.y, pv[1])));
          }
          {   // row 1
            E w0, w1;
            ldrow(v + vo1, w0, w1);
            const float2 a = P::unpack(c[2]), b = P::unpack(c[3]);
            float xa = a.y, xb = b.x, xc = b.y;
            if constexpr (!EVEN) {
              if (nv == 1) xa = r.y;
              if (nv == 2) xb = r.y;
              if (nv == 3) xc = r.y;
            }
            const E s0 = P::add(P::add(P::add(c[0], d0), P::pack(l.y + xa, a.x + xb)), P::add(bel[s - 1][2], ab[2]));
            const E s1 = P::add(P::add(P::add(c[1], d1), P::pack(a.y + xc, b.x + r.y)), P::add(bel[s - 1][3], ab[3]));
            nw[2] = P::fma(q1.x, s0, P::fma(P::fma(q0.x, w0, q0.y), c[2], P::mul(q1.y, pv[2])));
            nw[3] = P::fma(q1.x, s1, P::fma(P::fma(q0.x, w1, q0.y), c[3], P::mul(q1.y, pv[3])));
          }
          if constexpr (!EVEN) {   // padding stays zero
            if (nv < 4) {
              float2 a0 = P::unpack(nw[0]), a1 = P::unpack(nw[1]), a2 = P::unpack(nw[2]), a3 = P::unpack(nw[3]);
              a1.y = a3.y = 0.f;
              if (nv < 3) a1.x = a3.x = 0.f;
              if (nv < 2) a0.y = a2.y = 0.f;
              nw[0] = P::pack(a0.x, a0.y);
              nw[1] = P::pack(a1.x, a1.y);
              nw[2] = P::pack(a2.x, a2.y);
              nw[3] = P::pack(a3.x, a3.y);
            }
            if (!vy) nw[2] = nw[3] = 0ULL;
          }
          if (s < S) put(wr + s * area, nw);
          if (s >= S - 1) {
            float* g = (s == S ? pb : pa) + p * vplane;
            *reinterpret_cast<ulonglong2*>(g) = make_ulonglong2(nw[0], nw[1]);
            if (vy) *reinterpret_cast<ulonglong2*>(g + e0p) = make_ulonglong2(nw[2], nw[3]);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            pv[i] = bel[s - 1][i];     // u_{k+s-1}, the plane level s + 1 computes next
            bel[s - 1][i] = c[i];
            ab[i] = nw[i];
          }
        } else {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            pv[i] = bel[s - 1][i];
            ab[i] = 0ULL;
          }
        }
        // the next planes, once level 1 has used these (in their registers)
        if (s == 1) fetch(t + 1);
      }
    }
    vslot = vnext;
    cpa_wait<0>();
    __syncthreads();
  }
}

// One step over HBM, for boxes the kernel above does not take (all three axes
// spanned, or a large plane; FP64): a thread owns W consecutive points of the
// fastest axis and eight states, two at a time; out may be prev (each thread
// reads its own points of it only).  list: the fragments it is for.  W = 4 in FP32
// (16-byte accesses: nine per four points and state, one point per thread made
// that many per point), 1 in FP64, which is bound by the FP64 pipe.
template <typename T, int W>
__global__ void __launch_bounds__(256) eig_step_kernel(const EigFrag* __restrict__ ef, const int* __restrict__ list,
                                                       const T* __restrict__ in, const T* prev, T* out,
                                                       const T* __restrict__ vc,
                                                       const double* __restrict__ coef, T c1) {
  struct alignas(W * sizeof(T)) Row {
    T v[W];
  };
  const int f = list[blockIdx.z];
  const EigFrag E = ef[f];
  const int t = (blockIdx.x * 256 + threadIdx.x) * W;
  const int j0 = blockIdx.y * 8;
  if (t >= E.Ps || j0 >= E.n) return;
  const int c0 = t % E.e0p, r = t / E.e0p;
  const int c[3] = {c0, r % E.e[1], r / E.e[1]};
  const int nv = min(W, E.e[0] - c0);   // valid points; the padding stays zero
  if (nv <= 0) return;
  // neighbours: the row before and after along the slower axes, the point before
  // and after the thread's own along the fastest
  int nb[6];
  nb[0] = c0 + W < E.e[0] ? t + W : E.full[0] ? t - c0 : -1;
  nb[1] = c0 > 0 ? t - 1 : E.full[0] ? t + E.e[0] - 1 : -1;
  const int st[3] = {1, E.e0p, E.e0p * E.e[1]};
#pragma unroll
  for (int d = 1; d < 3; ++d)
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const int q = c[d] + (s ? -1 : 1);
      nb[2 * d + s] = q >= 0 && q < E.e[d] ? t + (s ? -st[d] : st[d])
                      : E.full[d]          ? t + (s ? (E.e[d] - 1) : (1 - E.e[d])) * st[d]
                                           : -1;
    }
  const double* cf = coef + 3 * f;
  const T al = (T)cf[0], be = (T)cf[1], mc = -al * c1;
  T w[W];
  {
    const Row v = *reinterpret_cast<const Row*>(vc + E.voff + t);
#pragma unroll
    for (int i = 0; i < W; ++i) w[i] = al * (v.v[i] - (T)cf[2]);
  }
  auto row = [](const T* p, bool ok) {
    if (ok) return *reinterpret_cast<const Row*>(p);
    Row z;
#pragma unroll
    for (int i = 0; i < W; ++i) z.v[i] = T(0);
    return z;
  };
  constexpr int JB = 2;
  for (int j = j0; j < min(j0 + 8, E.n); j += JB) {
    Row x[JB], yp[JB], ym[JB], zp[JB], zm[JB], pv[JB];
    T xr[JB], xl[JB];
#pragma unroll
    for (int u = 0; u < JB; ++u) {
      const bool on = j + u < E.n;
      const long long b = E.off + (long long)(on ? j + u : j) * E.Ps;
      const T* p = in + b;
      x[u] = row(p + t, true);
      yp[u] = row(p + nb[2], nb[2] >= 0);
      ym[u] = row(p + nb[3], nb[3] >= 0);
      zp[u] = row(p + nb[4], nb[4] >= 0);
      zm[u] = row(p + nb[5], nb[5] >= 0);
      xr[u] = nb[0] >= 0 ? p[nb[0]] : T(0);
      xl[u] = nb[1] >= 0 ? p[nb[1]] : T(0);
      pv[u] = row(prev + b + t, prev != nullptr);
    }
#pragma unroll
    for (int u = 0; u < JB; ++u) {
      if (j + u >= E.n) break;
      Row o;
#pragma unroll
      for (int i = 0; i < W; ++i) {
        const T rt = i + 1 < W && i + 1 < nv ? x[u].v[i + 1 < W ? i + 1 : i] : xr[u];
        const T lt = i > 0 ? x[u].v[i > 0 ? i - 1 : 0] : xl[u];
        T v = w[i] * x[u].v[i];
        if (prev) v = fma1(be, pv[u].v[i], v);
        v = fma1(mc, ((rt + lt) + (yp[u].v[i] + ym[u].v[i])) + (zp[u].v[i] + zm[u].v[i]), v);
        o.v[i] = i < nv ? v : T(0);
      }
      *reinterpret_cast<Row*>(out + E.off + (long long)(j + u) * E.Ps + t) = o;
    }
  }
}

// ------------------------------------------------------------------- Gram --
//
// G = Y^T Y and K = Y^T (H Y) of every fragment, upper halves.  The m vectors
// are dealt to Tn = ceil(m / MI) groups, group i holding the vectors i, i + Tn,
// i + 2 Tn, ...; a register tile is the MI x MI products of two groups (i <= j)
// of one of the two matrices, one tile per thread.  Vector rows of consecutive
// groups are adjacent in shared memory with a pitch of 4 mod 32 words, so a
// warp's 16-byte reads hit distinct banks.  Fewer tiles than threads: the
// threads form groups that take other points, summed in order at the end; more:
// the tiles are cut into sets, one per CTA.  Items are (fragment, chunk of
// points, set); the finalize sums the chunks in FP64.
// FP32 pipe bound: MI = 8 reads 16 x 16 bytes per 256 FMAs.  27 blocks of
// 64000 x 120 FP32: 1.8 ms against 9.2 ms
// for 64 x 64 tiles of all products.
constexpr int GR_THREADS = 256;

template <typename T> struct GrT;
template <> struct GrT<float> { static constexpr int MI = 8, U = 4; using V = float4; };
template <> struct GrT<double> { static constexpr int MI = 2, U = 2; using V = double2; };

__device__ __forceinline__ void gr_fma(float& acc, const float4& a, const float4& b) {
  acc = fmaf(a.x, b.x, acc);
  acc = fmaf(a.y, b.y, acc);
  acc = fmaf(a.z, b.z, acc);
  acc = fmaf(a.w, b.w, acc);
}
__device__ __forceinline__ void gr_fma(double& acc, const double2& a, const double2& b) {
  acc = fma(a.x, b.x, acc);
  acc = fma(a.y, b.y, acc);
}

// item: fragment, first point, points, set
template <typename T>
__global__ void __launch_bounds__(GR_THREADS, sizeof(T) == 4 ? 2 : 3) eig_gram_kernel(
    const EigFrag* __restrict__ ef, const int4* __restrict__ items,
    const long long* __restrict__ part_off, const T* __restrict__ Y, const T* __restrict__ HY,
    T* __restrict__ partials, int KP) {
  constexpr int MI = GrT<T>::MI, U = GrT<T>::U;
  using V = typename GrT<T>::V;
  extern __shared__ __align__(16) unsigned char gsm[];
  const int4 it = items[blockIdx.x];
  const EigFrag F = ef[it.x];
  const int m = F.n, Tn = (m + MI - 1) / MI, TT = Tn * (Tn + 1) / 2;
  const int nsets = (2 * TT + GR_THREADS - 1) / GR_THREADS, per = (2 * TT + nsets - 1) / nsets;
  const int i0 = it.w * per, T_ = min(per, 2 * TT - i0);   // tiles of this set
  const int G = GR_THREADS / per;
  const int tid = threadIdx.x;
  const int g = tid / per, lt = tid - g * per;
  const bool act = g < G && lt < T_;
  const int pitch = KP + (sizeof(T) == 4 ? 4 : 2);
  T* S = reinterpret_cast<T*>(gsm);   // [2][2 m][pitch]
  const int stage = 2 * m * pitch;
  int ra[MI], rb[MI];   // shared row offsets of the tile's vectors (clamped past m)
  {
    const int id = act ? i0 + lt : 0;
    const int hf = id / TT;
    int u = id - hf * TT, ti = 0;
    while (u >= Tn - ti) {
      u -= Tn - ti;
      ++ti;
    }
    const int tj = ti + u;
#pragma unroll
    for (int r = 0; r < MI; ++r) {
      ra[r] = min(ti + Tn * r, m - 1) * pitch;
      rb[r] = (min(tj + Tn * r, m - 1) + hf * m) * pitch;
    }
  }
  T acc[MI][MI];
#pragma unroll
  for (int r = 0; r < MI; ++r)
#pragma unroll
    for (int c = 0; c < MI; ++c) acc[r][c] = T(0);
  const int units = KP / U;   // 16-byte units of a row
  const int nst = (it.z + KP - 1) / KP;
  auto issue = [&](int st) {
    if (st < nst) {
      T* d = S + (st & 1) * stage;
      const int p0 = it.y + st * KP, pend = it.y + it.z;   // points past the chunk read zero
      for (int e = tid; e < 2 * m * units; e += GR_THREADS) {
        const int r = e / units, q = e - r * units;
        const int p = p0 + q * U;
        const bool ok = p < pend;
        const T* src = (r < m ? Y + F.off + (long long)r * F.Ps : HY + F.off + (long long)(r - m) * F.Ps);
        cpa16z(d + r * pitch + q * U, src + (ok ? p : 0), ok);
      }
    }
    cpa_commit();
  };
  issue(0);
  for (int st = 0; st < nst; ++st) {
    issue(st + 1);
    cpa_wait<1>();
    __syncthreads();
    if (act) {
      const T* d = S + (st & 1) * stage;
      for (int q = g; q < units; q += G) {
        const T* b = d + q * U;
        V a[MI];
#pragma unroll
        for (int r = 0; r < MI; ++r) a[r] = *reinterpret_cast<const V*>(b + ra[r]);
#pragma unroll
        for (int c = 0; c < MI; ++c) {
          const V v = *reinterpret_cast<const V*>(b + rb[c]);
#pragma unroll
          for (int r = 0; r < MI; ++r) gr_fma(acc[r][c], a[r], v);
        }
      }
    }
    __syncthreads();   // the stage is consumed
  }
  cpa_wait<0>();
  T* out = partials + part_off[blockIdx.x];   // [r][c][tile]
  if (G == 1) {
    if (act)
#pragma unroll
      for (int r = 0; r < MI; ++r)
#pragma unroll
        for (int c = 0; c < MI; ++c) out[(r * MI + c) * per + lt] = acc[r][c];
    return;
  }
  __syncthreads();
  if (act)
#pragma unroll
    for (int r = 0; r < MI; ++r)
#pragma unroll
      for (int c = 0; c < MI; ++c) S[(g * MI * MI + r * MI + c) * per + lt] = acc[r][c];
  __syncthreads();
  for (int e = tid; e < MI * MI * per; e += GR_THREADS) {
    // four sums side by side: a quarter of the roundings on a large term's sum
    T v[4] = {T(0), T(0), T(0), T(0)};
    int q = 0;
    for (; q + 4 <= G; q += 4)
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] += S[(q + u) * MI * MI * per + e];
    for (; q < G; ++q) v[0] += S[q * MI * MI * per + e];
    if (e % per < T_) out[e] = (v[0] + v[1]) + (v[2] + v[3]);
  }
}

// blocks of fragment f: K then G, m x m each, symmetric; chunks summed in order.
template <typename T>
__global__ void __launch_bounds__(256) eig_gram_sum_kernel(const EigFrag* __restrict__ ef,
                                                           const int2* __restrict__ fitems,
                                                           const long long* __restrict__ part_off,
                                                           const T* __restrict__ partials,
                                                           const long long* __restrict__ blk_off,
                                                           double* __restrict__ blocks) {
  constexpr int MI = GrT<T>::MI;
  const int f = blockIdx.x;
  const EigFrag F = ef[f];
  const int m = F.n, Tn = (m + MI - 1) / MI, TT = Tn * (Tn + 1) / 2;
  const int nsets = (2 * TT + GR_THREADS - 1) / GR_THREADS, per = (2 * TT + nsets - 1) / nsets;
  const int2 fi = fitems[f];   // first item, chunks (items ordered chunk, set)
  double* Kb = blocks + blk_off[f];
  double* Gb = Kb + (long long)m * m;
  const long long cstep = (long long)nsets * per * MI * MI;   // partials of one chunk
  for (int e = blockIdx.y * 256 + threadIdx.x; e < m * m; e += 256 * gridDim.y) {
    const int i = e / m, j = e - (e / m) * m;
    if (j < i) continue;
    int ti = i % Tn, r = i / Tn, tj = j % Tn, c = j / Tn;
    if (ti > tj) {
      const int a = ti, b = r;
      ti = tj; r = c;
      tj = a; c = b;
    }
    const int id = ti * Tn - ti * (ti - 1) / 2 + tj - ti;
    double s[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = h * TT + id, set = q / per, lt = q - set * per;
      const T* p = partials + part_off[fi.x + set] + (r * MI + c) * per + lt;
      double v = 0.0;
#pragma unroll 4
      for (int k = 0; k < fi.y; ++k) v += (double)p[k * cstep];
      s[h] = v;
    }
    Gb[i * m + j] = Gb[j * m + i] = s[0];
    Kb[i * m + j] = Kb[j * m + i] = s[1];
  }
}

// --------------------------------------------------------------- rotation --
//
// X = Y C and, for the residual norms only, H X = (H Y) C (never stored); the
// columns >= rank get fresh random values (their H X counts as zero).  A CTA
// keeps the coefficients in shared memory and takes tiles of points; thread
// (column group, point group) accumulates RC columns x RP points of both
// products, the points as packed pairs in FP32.  Rows of Y and H Y come in
// chunks of 16 vectors through two stages of asynchronous copies.  FP32 pipe
// bound: 6 shared 16-byte reads per 128 FMAs.  27 blocks of 64000 x 120 FP32:
// 2.7 ms against 13.1 ms
// for 64-point tiles with one point per thread.
constexpr int RT_THREADS = 256;
constexpr int RT_KC = 16;   // vectors per stage

// point groups of a CTA with cg column groups (64 at most: the staged rows)
__host__ __device__ constexpr int rt_groups(int cg) { return RT_THREADS / cg < 64 ? RT_THREADS / cg : 64; }

template <typename T> struct RtT;
template <> struct RtT<float> { static constexpr int RP = 8, RC = 8, U = 4; };
template <> struct RtT<double> { static constexpr int RP = 4, RC = 4, U = 2; };

template <typename T>
__global__ void __launch_bounds__(RT_THREADS, 1) eig_rotate_kernel(
    const EigFrag* __restrict__ ef, const DevFrag* __restrict__ fr, const T* __restrict__ Y,
    const T* __restrict__ HY, T* __restrict__ Xo, const double* __restrict__ Cm, long long cstride,
    const int* __restrict__ rank, const double* __restrict__ theta, const long long* __restrict__ toff,
    double* __restrict__ partial, int mstride, unsigned long long salt) {
  using P = Pk<T>;
  using E = typename P::E;
  constexpr int RP = RtT<T>::RP, RC = RtT<T>::RC, U = RtT<T>::U, NP = RP / P::NS, NV = RP / U;
  extern __shared__ __align__(16) unsigned char rsm[];
  const int f = blockIdx.y;
  const EigFrag F = ef[f];
  const int m = F.n, r = rank[f];
  const int cg = (m + RC - 1) / RC, mc = cg * RC;   // column groups, coefficient row length
  const int PG = rt_groups(cg), pts = PG * RP;      // point groups, points of a tile
  const int tid = threadIdx.x;
  const int jg = tid / PG, pg = tid - jg * PG;
  const bool act = jg < cg;
  T* Cs = reinterpret_cast<T*>(rsm);                // m x mc
  T* St = Cs + (size_t)m * mc;                      // [2][2][RT_KC][pts]
  const int stage = 2 * RT_KC * pts;
  for (int e = tid; e < m * mc; e += RT_THREADS) {
    const int k = e / mc, j = e - k * mc;
    Cs[e] = j < m ? (T)Cm[f * cstride + (long long)k * m + j] : T(0);
  }
  T th[RC], rsum[RC];
#pragma unroll
  for (int c = 0; c < RC; ++c) {
    const int j = jg * RC + c;
    th[c] = act && j < m ? (T)theta[toff[f] + j] : T(0);
    rsum[c] = T(0);
  }
  const int ntile = ((int)F.Ps + pts - 1) / pts, nch = (m + RT_KC - 1) / RT_KC;
  const int upr = pts / U;   // 16-byte units of a staged row
  const int ntot = blockIdx.x < ntile ? ((ntile - 1 - (int)blockIdx.x) / (int)gridDim.x + 1) * nch : 0;
  auto issue = [&](int n) {   // chunk n of the CTA's sequence of (tile, chunk)
    if (n < ntot) {
      const int tile = blockIdx.x + (n / nch) * gridDim.x, k0 = (n % nch) * RT_KC;
      T* d = St + (n & 1) * stage;
      const int nk = min(RT_KC, m - k0);
      for (int e = tid; e < 2 * nk * upr; e += RT_THREADS) {
        const int row = e / upr, q = e - row * upr;
        const int h = row >= nk, k = row - h * nk;
        const int p = tile * pts + q * U;
        const bool ok = p < F.Ps;
        const T* src = (h ? HY : Y) + F.off + (long long)(k0 + k) * F.Ps;
        cpa16z(d + (h * RT_KC + k) * pts + q * U, src + (ok ? p : 0), ok);
      }
    }
    cpa_commit();
  };
  E ax[RC][NP], ah[RC][NP];
  issue(0);
  for (int n = 0; n < ntot; ++n) {
    const int ch = n % nch;
    issue(n + 1);
    cpa_wait<1>();
    __syncthreads();
    if (ch == 0) {
#pragma unroll
      for (int c = 0; c < RC; ++c)
#pragma unroll
        for (int q = 0; q < NP; ++q) ax[c][q] = ah[c][q] = P::zero();
    }
    if (act) {
      const int k0 = ch * RT_KC, nk = min(RT_KC, m - k0);
      const T* dy = St + (n & 1) * stage + pg * U;   // unit v of the points: v PG U + pg U
      const T* dh = dy + RT_KC * pts;
      const T* cs = Cs + (size_t)k0 * mc + jg * RC;
#pragma unroll 2
      for (int k = 0; k < nk; ++k) {
        E y[NP], h[NP];
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const E2<E> a = *reinterpret_cast<const E2<E>*>(dy + k * pts + v * PG * U);
          const E2<E> b = *reinterpret_cast<const E2<E>*>(dh + k * pts + v * PG * U);
          y[2 * v] = a.a; y[2 * v + 1] = a.b;
          h[2 * v] = b.a; h[2 * v + 1] = b.b;
        }
        T cc[RC];
#pragma unroll
        for (int c = 0; c < RC; c += U) {
          const E2<E> a = *reinterpret_cast<const E2<E>*>(cs + (size_t)k * mc + c);
          if constexpr (sizeof(T) == 4) {
            const float2 u = Pk<float>::unpack(a.a), w = Pk<float>::unpack(a.b);
            cc[c] = u.x; cc[c + 1] = u.y; cc[c + 2] = w.x; cc[c + 3] = w.y;
          } else {
            cc[c] = a.a; cc[c + 1] = a.b;
          }
        }
#pragma unroll
        for (int c = 0; c < RC; ++c) {
          const E d = P::dup(cc[c]);
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            ax[c][q] = P::fma(y[q], d, ax[c][q]);
            ah[c][q] = P::fma(h[q], d, ah[c][q]);
          }
        }
      }
    }
    if (ch == nch - 1 && act) {
      // the tile's results: X out, residual sums
      const int tile = blockIdx.x + (n / nch) * gridDim.x;
#pragma unroll
      for (int c = 0; c < RC; ++c) {
        const int j = jg * RC + c;
        if (j >= m) continue;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
          const int t = tile * pts + v * PG * U + pg * U;
          if (t >= F.Ps) continue;
          T xv[U], hv[U];
          if constexpr (sizeof(T) == 4) {
            const float2 a = Pk<float>::unpack(ax[c][2 * v]), b = Pk<float>::unpack(ax[c][2 * v + 1]);
            const float2 p = Pk<float>::unpack(ah[c][2 * v]), q = Pk<float>::unpack(ah[c][2 * v + 1]);
            xv[0] = a.x; xv[1] = a.y; xv[2] = b.x; xv[3] = b.y;
            hv[0] = p.x; hv[1] = p.y; hv[2] = q.x; hv[3] = q.y;
          } else {
            xv[0] = ax[c][2 * v]; xv[1] = ax[c][2 * v + 1];
            hv[0] = ah[c][2 * v]; hv[1] = ah[c][2 * v + 1];
          }
          if (j >= r) {   // dropped direction: a fresh random vector
            const DevFrag D = fr[f];
            const T inv = (T)(1.0 / sqrt((double)F.e[0] * F.e[1] * F.e[2]));
            const unsigned long long s0 = splitmix64(salt);
            for (int i = 0; i < U; ++i) {
              int q[3];
              hv[i] = T(0);
              xv[i] = T(0);
              if (box_coords(F, t + i, q)) {
                const unsigned long long key = ((unsigned long long)f << 44) ^ ((unsigned long long)j << 32) ^
                                               (unsigned long long)dilated_index(D, q);
                xv[i] = (T)uniform53(splitmix64(key + s0)) * inv;
              }
            }
          }
#pragma unroll
          for (int i = 0; i < U; ++i) {
            const T d = hv[i] - th[c] * xv[i];
            rsum[c] = fma1(d, d, rsum[c]);
          }
          T* o = Xo + F.off + (long long)j * F.Ps + t;
          if constexpr (sizeof(T) == 4)
            *reinterpret_cast<float4*>(o) = make_float4(xv[0], xv[1], xv[2], xv[3]);
          else
            *reinterpret_cast<double2*>(o) = make_double2(xv[0], xv[1]);
        }
      }
    }
    __syncthreads();   // the stage is consumed
  }
  cpa_wait<0>();
  __syncthreads();
  // residual partials of the CTA: per column over the point groups, in order
  T* red = St;   // [column][PG]
  if (act)
#pragma unroll
    for (int c = 0; c < RC; ++c) red[(jg * RC + c) * PG + pg] = rsum[c];
  __syncthreads();
  for (int j = tid; j < m; j += RT_THREADS) {
    double s = 0.0;
    for (int q = 0; q < PG; ++q) s += (double)red[j * PG + q];
    partial[((long long)f * gridDim.x + blockIdx.x) * mstride + j] = s;
  }
}

__global__ void eig_residual_kernel(const EigFrag* ef, const double* partial, int nblocks, int mstride,
                                    const long long* toff, double* res) {
  const int f = blockIdx.x;
  const int m = ef[f].n;
  for (int j = threadIdx.x; j < m; j += blockDim.x) {
    double s = 0.0;
#pragma unroll 4
    for (int b = 0; b < nblocks; ++b) s += partial[((long long)f * nblocks + b) * mstride + j];
    res[toff[f] + j] = sqrt(s);
  }
}

// ----------------------------------------------------------------- export --

// Sign gauge of the first n_a vectors: the largest |component| positive, ties
// to the lowest box index (x fastest).  One CTA per (vector, fragment).
template <typename T>
__global__ void __launch_bounds__(256) eig_sign_kernel(const EigFrag* ef, const DevFrag* fr, const T* X,
                                                       T* sgn, int mstride) {
  __shared__ T bv[8];
  __shared__ int bi[8], bs[8];
  const int f = blockIdx.y, j = blockIdx.x;
  const EigFrag E = ef[f];
  if (j >= fr[f].n) return;   // uniform
  const T* x = X + E.off + (long long)j * E.Ps;
  int st[3];   // box index strides of the layout's axes
  {
    int ext[3];
    for (int a = 0; a < 3; ++a) ext[E.ax[a]] = E.e[a];
    const int bst[3] = {1, ext[0], ext[0] * ext[1]};
    for (int a = 0; a < 3; ++a) st[a] = bst[E.ax[a]];
  }
  T best = T(-1);
  int idx = 0x7fffffff, sign = 0;
  for (int t = threadIdx.x; t < E.Ps; t += 256) {
    const T v = x[t];
    const T a = fabs(v);
    if (a > best || a == best) {
      const int c0 = t % E.e0p, r = t / E.e0p, c1 = r % E.e[1], c2 = r / E.e[1];
      if (c0 >= E.e[0] || c2 >= E.e[2]) continue;
      const int b = c0 * st[0] + c1 * st[1] + c2 * st[2];
      if (a > best || b < idx) {
        best = a;
        idx = b;
        sign = v < T(0);
      }
    }
  }
  auto take = [&](T v, int i, int s) {
    if (v > best || (v == best && i < idx)) {
      best = v;
      idx = i;
      sign = s;
    }
  };
  for (int o = 16; o > 0; o >>= 1) {
    const T v = __shfl_xor_sync(0xffffffffu, best, o);
    const int i = __shfl_xor_sync(0xffffffffu, idx, o), s = __shfl_xor_sync(0xffffffffu, sign, o);
    take(v, i, s);
  }
  if ((threadIdx.x & 31) == 0) {
    bv[threadIdx.x >> 5] = best;
    bi[threadIdx.x >> 5] = idx;
    bs[threadIdx.x >> 5] = sign;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) take(bv[w], bi[w], bs[w]);
    sgn[(long long)f * mstride + j] = sign ? T(-1) : T(1);
  }
}

// State-major block -> the library's point-major dilated storage, 32 points x
// 32 states per CTA through shared memory (both sides coalesced).
template <typename T>
__global__ void __launch_bounds__(256) eig_export_kernel(const EigFrag* ef, const DevFrag* fr, const T* X,
                                                         const T* sgn, int mstride, T* states) {
  __shared__ T tile[32][33];
  const int f = blockIdx.z, j0 = blockIdx.y * 32, t0 = blockIdx.x * 32;
  const EigFrag E = ef[f];
  const DevFrag D = fr[f];
  if (j0 >= D.n || t0 >= E.Ps) return;   // uniform
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int i = w; i < 32; i += 8) {
    const int j = j0 + i, t = t0 + lane;
    T v = T(0);
    if (j < D.n && t < E.Ps) v = sgn[(long long)f * mstride + j] * X[E.off + (long long)j * E.Ps + t];
    tile[i][lane] = v;
  }
  __syncthreads();
  for (int i = w; i < 32; i += 8) {
    const int t = t0 + i, j = j0 + lane;
    int q[3];
    if (t < E.Ps && box_coords(E, t, q) && j < D.n)
      states[D.off + (long long)dilated_index(D, q) * D.ld + j] = tile[lane][i];
  }
}

}  // namespace

// ------------------------------------------------------------------ host ----

// Layout of blocks of m[a] vectors: axes permuted so that the slowest is the
// longest axis the box does not span (the filter marches along it and its
// plane is the smallest), the other two in the order that pads fewer points
// (a box two points wide is not padded to four), in grid order among equals.
void eig_layout(const std::vector<DevFrag>& fr, const std::vector<int>& m,
                std::vector<EigFrag>& out, long long& elems, long long& vc_elems) {
  out.resize(fr.size());
  elems = vc_elems = 0;
  for (size_t a = 0; a < fr.size(); ++a) {
    const DevFrag& F = fr[a];
    EigFrag& E = out[a];
    int march = 2;
    for (int d = 2; d >= 0; --d)
      if (!F.full[d] && (F.full[march] || F.ext[d] > F.ext[march])) march = d;
    int k = 0;
    for (int d = 0; d < 3; ++d)
      if (d != march) E.ax[k++] = d;
    E.ax[2] = march;
    auto padded = [&](int fast, int next) { return (long long)((F.ext[fast] + 3) / 4 * 4) * F.ext[next]; };
    if (padded(E.ax[1], E.ax[0]) < padded(E.ax[0], E.ax[1])) std::swap(E.ax[0], E.ax[1]);
    for (int i = 0; i < 3; ++i) {
      E.e[i] = F.ext[E.ax[i]];
      E.full[i] = F.full[E.ax[i]];
    }
    E.e0p = (E.e[0] + 3) / 4 * 4;
    E.Ps = E.e0p * E.e[1] * E.e[2];
    E.n = m[a];
    E.off = elems;
    E.voff = vc_elems;
    elems += ((long long)E.Ps * E.n + 63) / 64 * 64;
    vc_elems += ((long long)E.Ps + 63) / 64 * 64;
  }
}

// Bytes of shared memory of a filter CTA with np vectors and S levels.
static int filter_patches(const EigFrag& E) { return (E.e0p / 4) * ((E.e[1] + 1) / 2); }
static long long filter_smem(const EigFrag& E, int np, int S) {
  return 4LL * ((long long)np * 2 * S * filter_area(filter_patches(E)) + (long long)(S + 2) * E.e0p * E.e[1]);
}

using FilterFn = void (*)(const EigFrag*, const int4*, float*, float*, const float*, const double*, int, int, int,
                          int, int, float);
static FilterFn filter_entry(int S, bool even) {
  if (even)
    return S == 1 ? eig_filter_kernel<1, true> : S == 2 ? eig_filter_kernel<2, true>
         : S == 3 ? eig_filter_kernel<3, true> : eig_filter_kernel<4, true>;
  return S == 1 ? eig_filter_kernel<1, false> : S == 2 ? eig_filter_kernel<2, false>
       : S == 3 ? eig_filter_kernel<3, false> : eig_filter_kernel<4, false>;
}

// Work list of the on-chip filter: FP32, boxes that leave an axis to march
// along and whose plane has at most 448 patches (3584 points); the others go
// one step per launch (plan.steps), beside them, and all of them do where that is
// faster (filter_prefers_steps).  Four levels per launch where two CTAs of
// one vector fit an SM (planes of up to about 1400 points), else three, fewer
// where the shared memory asks for it: per step of 20e6 point-vectors in
// planes of 32 x 32, S = 4 takes 23 us, S = 3 26 us, S = 2 35 us; of 207e6 in
// planes of 40 x 40, 275, 250 and 340 us.  Vectors per CTA: the count that keeps
// the most vectors resident on an SM, the smallest of those (separate CTAs do
// not wait at each other's barriers).
//
// Whether single steps over HBM beat the on-chip filter.  A launch of the latter
// is a chain of e[2] + S ticks per wave of CTAs, about 0.7 us + 2.3 ns for every
// thread on the SM each, S steps; a single step is about 6 us and 1.7 us per
// million point-vectors, 2.7 us past the 8.5 million whose three blocks fit L2.
// So a few vectors of a long box go by steps: us per step on chip / by steps, 1 box
// 12 x 12 x 200, 25 vectors 42.6 / 6.3; 100 x 90 x 30, 30 vectors 52 / 20; 8 boxes
// 24^3, 16 vectors 10.7 / 8.3; but 4 boxes 16 x 12 x 12, 10 vectors 4.5 / 6.3; 8
// boxes 40^3, 16 vectors 14.6 / 20; 31 boxes 16 x 32 x 32, 40 vectors 25.7 / 55.6.
static bool filter_prefers_steps(const EigFilterPlan& plan, const std::vector<EigFrag>& ef, long long per_sm) {
  double total = 0.0;
  int ticks = 0;
  for (const int4& j : plan.jobs) {
    total += 1e-6 * j.z * ef[j.x].Ps;
    ticks = std::max(ticks, ef[j.x].e[2] + plan.S);
  }
  const double ctas = plan.jobs.size() / 152.0, waves = std::max(1.0, ctas / per_sm);
  const double on_sm = std::max(1.0, std::min(ctas, (double)per_sm));
  const double chip = waves * ticks / plan.S * (0.7 + 0.0023 * plan.threads * on_sm);
  return 6.0 + 1.7 * std::min(total, 8.5) + 2.7 * std::max(0.0, total - 8.5) < chip;
}

void eig_filter_plan(const std::vector<EigFrag>& ef, bool fp64, EigFilterPlan& plan) {
  plan = EigFilterPlan();
  const long long cap = 226 * 1024;
  int S = 4;
  std::vector<char> fits(ef.size(), 0);
  for (size_t a = 0; a < ef.size(); ++a) {
    const EigFrag& E = ef[a];
    const long long tp = (long long)(E.e0p / 4) * ((E.e[1] + 1) / 2);
    fits[a] = !fp64 && !E.full[2] && tp <= ft_max(1) && filter_smem(E, 1, 1) <= cap;
    if (!fits[a]) {
      plan.steps.push_back((int)a);
      continue;
    }
    if (2 * ((tp + 31) / 32 * 32) > ft_max(4) || 2 * (filter_smem(E, 1, 4) + 1024) > cap) S = std::min(S, 3);
    while (filter_smem(E, 1, S) > cap) --S;
    plan.even = plan.even && E.e[0] % 4 == 0 && E.e[1] % 2 == 0;
  }
  if (plan.steps.size() == ef.size()) return;
  struct J { int4 j; long long cost; };
  std::vector<J> jobs;
  int threads = 32;
  long long smem = 0;
  for (size_t a = 0; a < ef.size(); ++a) {
    if (!fits[a]) continue;
    const EigFrag& E = ef[a];
    const int tp = filter_patches(E);
    int np = 1, best = 0;
    for (int k = 1; k <= E.n && k * tp <= ft_max(S) && filter_smem(E, k, S) <= cap; ++k) {
      const int res = k * (int)std::min<long long>(cap / (filter_smem(E, k, S) + 1024), ft_max(S) / ((k * tp + 31) / 32 * 32));
      if (res > best) {
        best = res;
        np = k;
      }
    }
    const int cnt = (E.n + np - 1) / np;
    np = (E.n + cnt - 1) / cnt;   // even shares
    threads = std::max(threads, (np * tp + 31) / 32 * 32);
    smem = std::max(smem, filter_smem(E, np, S));
    for (int q = 0; q < E.n; q += np) {
      const int k = std::min(np, E.n - q);
      jobs.push_back({make_int4((int)a, q, k, 0), (long long)k * tp * E.e[2]});
    }
  }
  std::stable_sort(jobs.begin(), jobs.end(), [](const J& x, const J& y) { return x.cost > y.cost; });
  plan.S = S;
  plan.threads = threads;
  plan.smem = (size_t)smem;
  for (const J& j : jobs) plan.jobs.push_back(j.j);
  const long long per_sm = std::min<long long>(cap / (smem + 1024), ft_max(S) / threads);
  if (filter_prefers_steps(plan, ef, std::max(1LL, per_sm))) {
    plan = EigFilterPlan();
    for (size_t a = 0; a < ef.size(); ++a) plan.steps.push_back((int)a);
    return;
  }
  for (int q = 1; q <= S; ++q)
    if (cudaFuncSetAttribute((const void*)filter_entry(q, plan.even), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap) != cudaSuccess) {
      cudaGetLastError();
      plan = EigFilterPlan();
      for (size_t a = 0; a < ef.size(); ++a) plan.steps.push_back((int)a);
      return;
    }
}

// Launches of the on-chip filter over L steps.  Every launch, and every single
// step of the others, swaps the two blocks: where both run, their numbers have
// the same parity, so that all fragments end in the same block.
int eig_filter_passes(const EigFilterPlan& plan, int L) {
  if (plan.S == 0) return 0;
  const int np = (L + plan.S - 1) / plan.S;
  return plan.steps.empty() || (np - L) % 2 == 0 ? np : np + 1;   // np + 1 <= L there
}

static void filter_pass(const EigFilterPlan& plan, const EigFrag* ef, int nfrag, void* A, void* B,
                        const void* vc, const double* coef, int k0, int S, bool plain_last,
                        int plain_slot, bool has_prev, double h, cudaStream_t s, const int4* jobs) {
  const float c1 = (float)(0.5 / (h * h));
  filter_entry(S, plan.even)<<<(unsigned)plan.jobs.size(), plan.threads, plan.smem, s>>>(
      ef, jobs, (float*)A, (float*)B, (const float*)vc, coef, nfrag, k0, plain_last, plain_slot, has_prev, c1);
}

int launch_eig_filter(const EigFilterPlan& plan, const EigFrag* d_ef, const std::vector<EigFrag>& ef,
                      const int4* d_jobs, const int* d_steps, void* A, void* B, const void* vc, const double* coef,
                      int deg, int plain_slot, bool fp64, double h, cudaStream_t s) {
  const int nf = (int)ef.size(), L = deg + 1;   // deg steps and H u_deg
  int swaps = 0;
  if (plan.S > 0) {
    void *cur = A, *prev = B;   // u_k, u_{k-1}
    bool hp = false;
    const int np = eig_filter_passes(plan, L);
    for (int i = 0, k = 0; i < np; ++i) {
      const int S = (L - k + (np - i) - 1) / (np - i);
      const bool last = i == np - 1;
      filter_pass(plan, d_ef, nf, cur, prev, vc, coef, k, S, last, plain_slot, hp, h, s, d_jobs);
      std::swap(cur, prev);   // level S went to prev's block, level S - 1 to cur's
      hp = true;
      k += S;
    }
    swaps = np;
  }
  if (!plan.steps.empty()) {
    void *cur = A, *prev = B;
    int psmax = 1, rows = 1;
    for (int a : plan.steps) {
      psmax = std::max(psmax, ef[a].Ps);
      rows = std::max(rows, ef[a].n);
    }
    const int W = fp64 ? 1 : 4;
    const dim3 g((psmax / W + 255) / 256, (rows + 7) / 8, (unsigned)plan.steps.size());
    for (int k = 0; k <= deg; ++k) {
      const double* cf = coef + 3 * (size_t)(k == deg ? plain_slot : k) * nf;
      const bool p = k > 0 && k < deg;
      if (fp64)
        eig_step_kernel<double, 1><<<g, 256, 0, s>>>(d_ef, d_steps, (const double*)cur, p ? (const double*)prev : nullptr,
                                                     (double*)prev, (const double*)vc, cf, 0.5 / (h * h));
      else
        eig_step_kernel<float, 4><<<g, 256, 0, s>>>(d_ef, d_steps, (const float*)cur, p ? (const float*)prev : nullptr,
                                                    (float*)prev, (const float*)vc, cf, (float)(0.5 / (h * h)));
      std::swap(cur, prev);
    }
    swaps = L;
  }
  return swaps & 1;   // H Y is in A (0) or B (1), Y in the other
}

void launch_eig_init(const EigFrag* d_ef, const DevFrag* d_fr, const std::vector<EigFrag>& ef, void* X,
                     unsigned long long seed, bool fp64, cudaStream_t s) {
  int psmax = 1, rows = 1;
  for (const EigFrag& E : ef) {
    psmax = std::max(psmax, E.Ps);
    rows = std::max(rows, E.n);
  }
  const dim3 g(std::min((psmax + 255) / 256, 16), rows, (unsigned)ef.size());
  if (fp64) eig_init_kernel<double><<<g, 256, 0, s>>>(d_ef, d_fr, (double*)X, seed);
  else eig_init_kernel<float><<<g, 256, 0, s>>>(d_ef, d_fr, (float*)X, seed);
}

void launch_eig_vc(const EigFrag* d_ef, const DevFrag* d_fr, const std::vector<EigFrag>& ef, const void* V,
                   const int gn[3], double h, void* vc, bool fp64, cudaStream_t s) {
  int psmax = 1;
  for (const EigFrag& E : ef) psmax = std::max(psmax, E.Ps);
  const dim3 g(std::min((psmax + 255) / 256, 64), (unsigned)ef.size());
  const double c0 = 3.0 / (h * h);
  if (fp64) eig_vc_kernel<double><<<g, 256, 0, s>>>(d_ef, d_fr, (const double*)V, c0, gn[0], gn[1], gn[2], (double*)vc);
  else eig_vc_kernel<float><<<g, 256, 0, s>>>(d_ef, d_fr, (const float*)V, (float)c0, gn[0], gn[1], gn[2], (float*)vc);
}

// Gram plan: items of about `chunk` points (a multiple of 256).
template <typename T>
static void gram_plan(const std::vector<EigFrag>& ef, EigGramPlan& g) {
  constexpr int MI = GrT<T>::MI, U = GrT<T>::U;
  g = EigGramPlan();
  long long pts = 0;
  int mmax = 1, gmax = 1;
  for (const EigFrag& E : ef) {
    pts += E.Ps;
    mmax = std::max(mmax, E.n);
  }
  // about four items per SM, 256 to 1024 points: a chunk's sums are in the
  // working precision, the chunks are added in FP64
  const int chunk = (int)std::min<long long>(1024, std::max<long long>(256, (pts / (4 * 152) + 255) / 256 * 256));
  for (size_t a = 0; a < ef.size(); ++a) {
    const EigFrag& E = ef[a];
    const int Tn = (E.n + MI - 1) / MI, TT = Tn * (Tn + 1) / 2;
    const int nsets = (2 * TT + GR_THREADS - 1) / GR_THREADS, per = (2 * TT + nsets - 1) / nsets;
    gmax = std::max(gmax, GR_THREADS / per);
    g.fitems.push_back(make_int2((int)g.items.size(), (E.Ps + chunk - 1) / chunk));
    for (int p = 0; p < E.Ps; p += chunk)
      for (int st = 0; st < nsets; ++st) {
        g.items.push_back(make_int4((int)a, p, std::min(chunk, E.Ps - p), st));
        g.part_off.push_back(g.part_elems);
        g.part_elems += (long long)per * MI * MI;
      }
    g.blk_off.push_back(g.blk_elems);
    g.blk_elems += 2LL * E.n * E.n;
  }
  // points per stage: enough 16-byte units for every thread group, two stages
  // within 100 KB (two CTAs per SM)
  auto bytes = [&](int KP) { return 2LL * 2 * mmax * (KP + (sizeof(T) == 4 ? 4 : 2)) * (long long)sizeof(T); };
  g.KP = 32;
  while (g.KP < 128 && g.KP / U < 2 * gmax && bytes(2 * g.KP) <= 100 * 1024) g.KP *= 2;
  g.smem = (size_t)std::max<long long>(bytes(g.KP), gmax > 1 ? (long long)GR_THREADS * MI * MI * sizeof(T) : 0);
}

cudaError_t eig_gram_plan(const std::vector<EigFrag>& ef, bool fp64, EigGramPlan& g) {
  if (fp64) gram_plan<double>(ef, g);
  else gram_plan<float>(ef, g);
  const void* k = fp64 ? (const void*)eig_gram_kernel<double> : (const void*)eig_gram_kernel<float>;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_PLAN_MAX);
}

void launch_eig_gram(const EigGramPlan& g, const EigFrag* d_ef, int nfrag, const int4* d_items,
                     const long long* d_part_off, const int2* d_fitems, const long long* d_blk_off,
                     const void* Y, const void* HY, void* partials, double* blocks, bool fp64, cudaStream_t s) {
  const dim3 fg(nfrag, std::max(1, std::min(16, 16 * 152 / nfrag)));
  if (fp64) {
    eig_gram_kernel<double><<<(unsigned)g.items.size(), GR_THREADS, g.smem, s>>>(
        d_ef, d_items, d_part_off, (const double*)Y, (const double*)HY, (double*)partials, g.KP);
    eig_gram_sum_kernel<double><<<fg, 256, 0, s>>>(d_ef, d_fitems, d_part_off, (const double*)partials, d_blk_off, blocks);
  } else {
    eig_gram_kernel<float><<<(unsigned)g.items.size(), GR_THREADS, g.smem, s>>>(
        d_ef, d_items, d_part_off, (const float*)Y, (const float*)HY, (float*)partials, g.KP);
    eig_gram_sum_kernel<float><<<fg, 256, 0, s>>>(d_ef, d_fitems, d_part_off, (const float*)partials, d_blk_off, blocks);
  }
}

// Rotation: CTAs per fragment (a whole number of waves of one CTA per SM, at
// most one per tile) and shared memory of the largest block.
template <typename T>
static void rotate_plan(const std::vector<EigFrag>& ef, int& blocks, size_t& smem) {
  constexpr int RP = RtT<T>::RP, RC = RtT<T>::RC;
  smem = 0;
  int tiles = 1;
  for (const EigFrag& E : ef) {
    const int cg = (E.n + RC - 1) / RC, PG = rt_groups(cg), pts = PG * RP;
    smem = std::max(smem, ((size_t)E.n * cg * RC + 4 * (size_t)RT_KC * pts) * sizeof(T));
    tiles = std::max(tiles, (E.Ps + pts - 1) / pts);
  }
  const int nf = (int)ef.size();
  blocks = std::max(1, std::min(tiles, 4 * 152 / nf));
}

cudaError_t eig_rotate_plan(const std::vector<EigFrag>& ef, bool fp64, int& blocks, size_t& smem) {
  if (fp64) rotate_plan<double>(ef, blocks, smem);
  else rotate_plan<float>(ef, blocks, smem);
  const void* k = fp64 ? (const void*)eig_rotate_kernel<double> : (const void*)eig_rotate_kernel<float>;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_PLAN_MAX);
}

void launch_eig_rotate(const EigFrag* d_ef, const DevFrag* d_fr, int nfrag, int blocks, size_t smem,
                       const void* Y, const void* HY, void* Xo, const double* Cm, long long cstride,
                       const int* rank, const double* theta, const long long* toff, double* partial,
                       int mstride, unsigned long long salt, double* res, bool fp64, cudaStream_t s) {
  const dim3 g(blocks, nfrag);
  if (fp64)
    eig_rotate_kernel<double><<<g, RT_THREADS, smem, s>>>(d_ef, d_fr, (const double*)Y, (const double*)HY, (double*)Xo,
                                                         Cm, cstride, rank, theta, toff, partial, mstride, salt);
  else
    eig_rotate_kernel<float><<<g, RT_THREADS, smem, s>>>(d_ef, d_fr, (const float*)Y, (const float*)HY, (float*)Xo, Cm,
                                                        cstride, rank, theta, toff, partial, mstride, salt);
  eig_residual_kernel<<<nfrag, 128, 0, s>>>(d_ef, partial, blocks, mstride, toff, res);
}

void launch_eig_export(const EigFrag* d_ef, const DevFrag* d_fr, const std::vector<EigFrag>& ef, int nmax,
                       const void* X, void* sgn, int mstride, void* states, bool fp64, cudaStream_t s) {
  int psmax = 1;
  for (const EigFrag& E : ef) psmax = std::max(psmax, E.Ps);
  const dim3 gs(nmax, (unsigned)ef.size()), ge((psmax + 31) / 32, (nmax + 31) / 32, (unsigned)ef.size());
  if (fp64) {
    eig_sign_kernel<double><<<gs, 256, 0, s>>>(d_ef, d_fr, (const double*)X, (double*)sgn, mstride);
    eig_export_kernel<double><<<ge, 256, 0, s>>>(d_ef, d_fr, (const double*)X, (const double*)sgn, mstride, (double*)states);
  } else {
    eig_sign_kernel<float><<<gs, 256, 0, s>>>(d_ef, d_fr, (const float*)X, (float*)sgn, mstride);
    eig_export_kernel<float><<<ge, 256, 0, s>>>(d_ef, d_fr, (const float*)X, (const float*)sgn, mstride, (float*)states);
  }
}

}  // namespace ofm
