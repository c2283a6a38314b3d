// H phi on the dilated fragment boxes (Eq. 1 with the 7-point stencil), and
// the layout conversions between the caller's column-major states and the
// library's point-major storage.
//
// H phi(r) = (3/h^2) phi(r) - (1/(2 h^2)) sum_{6 neighbours} phi + V(r) phi(r)
// with phi zero outside its box (Sec. II: H phi_i^(j) with the whole-system
// H).  It is evaluated on every point of the dilated box, where it can be
// non-zero.  Storage is point-major (the n states of one point are adjacent),
// so one thread owns 16 bytes of states of one point and every neighbour
// access of a warp is a contiguous run: the kernel is a streaming stencil,
// bound by HBM bandwidth.  The launch grid is 3-D: blockIdx.y is the
// fragment, blockIdx.x a chunk of its (x, y, 16-byte column group) elements
// and blockIdx.z a chunk of z planes that each thread marches through.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "ofm_internal.h"
#include "ptx_util.h"

namespace ofm {

template <typename T> struct Vec16;
template <> struct Vec16<float> { using type = float4; static constexpr int n = 4; };
template <> struct Vec16<double> { using type = double2; static constexpr int n = 2; };

__device__ __forceinline__ float4 fma4(float a, float4 x, float4 y) {
  return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}
__device__ __forceinline__ double2 fma4(double a, double2 x, double2 y) {
  return make_double2(fma(a, x.x, y.x), fma(a, x.y, y.y));
}
__device__ __forceinline__ float4 add4(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}
__device__ __forceinline__ double2 add4(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ float4 zero4(float) { return make_float4(0.f, 0.f, 0.f, 0.f); }
__device__ __forceinline__ double2 zero4(double) { return make_double2(0.0, 0.0); }

// Neighbour index along one dimension in the storage box: +/-1 step of
// `stride` points; in a full-span dimension it wraps, otherwise a step out
// of the storage box reads zero (returns -1).
__device__ __forceinline__ int nb_index(int p, int c, int ext, int full, int dir, int stride) {
  int c2 = c + dir;
  if (c2 < 0 || c2 >= ext) {
    if (!full) return -1;
    c2 = (c2 + ext) % ext;
  }
  return p + (c2 - c) * stride;
}

// z-marching form: a thread owns one (x, y, 16-byte column)
// of a fragment and walks along z, keeping the planes z-1, z, z+1 of its
// column in registers; only the plane ahead, the four in-plane neighbours
// (cache hits: the neighbouring threads load them as their own centre),
// and V are loaded per output.
template <typename T>
__global__ void __launch_bounds__(256) apply_zmarch_kernel(
    const DevFrag* __restrict__ fr, const T* __restrict__ V, const T* __restrict__ in,
    T* __restrict__ out, int gx, int gy, int gz, T c0, T c1, int zc) {
  using V16 = typename Vec16<T>::type;
  constexpr int VN = Vec16<T>::n;
  __shared__ DevFrag Fs;
  if (threadIdx.x == 0) Fs = fr[blockIdx.y];
  __syncthreads();
  const DevFrag& F = Fs;
  const int qpp = F.ld / VN;
  const int ex = F.dext[0], ey = F.dext[1], ez = F.dext[2];
  const int e = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (e >= ex * ey * qpp) return;
  const int pxy = e / qpp, q = e - pxy * qpp;
  const int x = pxy % ex, y = pxy / ex;
  const int plane = ex * ey;
  // in-plane neighbours (branch-free: outside the storage box -> self, weight 0)
  int nb[4];
  nb[0] = nb_index(pxy, x, ex, F.full[0], +1, 1);
  nb[1] = nb_index(pxy, x, ex, F.full[0], -1, 1);
  nb[2] = nb_index(pxy, y, ey, F.full[1], +1, ex);
  nb[3] = nb_index(pxy, y, ey, F.full[1], -1, ex);
  T w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    w[i] = nb[i] >= 0 ? T(1) : T(0);
    if (nb[i] < 0) nb[i] = pxy;
  }
  const V16* S = reinterpret_cast<const V16*>(in + F.off);
  V16* O = reinterpret_cast<V16*>(out + F.off);
  // this CTA's chunk of planes (blockIdx.z): zc planes
  const int z0 = (int)blockIdx.z * zc;
  const int z1 = min(ez, z0 + zc);
  if (z0 >= z1) return;
  const int X = (F.doff[0] + x) % gx, Y = (F.doff[1] + y) % gy;
  const T* Vrow = V + (long long)Y * gx + X;
  const long long vstride = (long long)gx * gy;
  // planes below and at the start
  auto plane_val = [&](int z) -> V16 {
    int zz = z;
    if (zz < 0 || zz >= ez) {
      if (!F.full[2]) return zero4(T());
      zz = (zz + ez) % ez;
    }
    return S[(zz * plane + pxy) * qpp + q];
  };
  V16 below = plane_val(z0 - 1);
  V16 ctr = plane_val(z0);
  for (int z = z0; z < z1; ++z) {
    const V16 above = plane_val(z + 1);
    const int base = z * plane;
    V16 sum = add4(below, above);
#pragma unroll
    for (int i = 0; i < 4; ++i) sum = fma4(w[i], S[(base + nb[i]) * qpp + q], sum);
    const T v = Vrow[(long long)((F.doff[2] + z) % gz) * vstride];
    V16 hy = fma4(c0 + v, ctr, zero4(T()));
    O[(base + pxy) * qpp + q] = fma4(-c1, sum, hy);
    below = ctr;
    ctr = above;
  }
}

// Shared-memory staged form (the default where a tile fits): a CTA owns
// rows [y0, y1) of one fragment (every x) for a chunk of z planes.  For each
// plane it needs, one thread issues at most three bulk copies (the staged
// rows y0-1 .. y1 are contiguous in storage except where a full-span
// dimension wraps) into a ring of STG_BUF plane buffers, completing on the
// buffer's mbarrier; a slot is refilled as soon as its plane is no longer
// needed, so up to three planes per CTA are in flight while it computes.  All six neighbours then
// come from shared memory; V streams from global memory into registers one
// plane ahead of its use.  Staged rows outside a non-periodic storage box are zeroed
// once; planes outside it complete their barrier phase without a copy and
// are skipped in the sum.
constexpr int STG_BUF = 5;
constexpr int STG_THREADS = 256;
constexpr int STG_EPT = 4;   // tile elements per thread (16 bytes each)

template <typename T>
__global__ void __launch_bounds__(STG_THREADS) apply_staged_kernel(
    const DevFrag* __restrict__ fr, const T* __restrict__ V, const T* __restrict__ in,
    T* __restrict__ out, int gx, int gy, int gz, T c0, T c1, int ty, int zc, int* flag) {
  using namespace ptx;
  using V16 = typename Vec16<T>::type;
  constexpr int VN = Vec16<T>::n;
  extern __shared__ __align__(128) unsigned char stg_smem[];
  __shared__ DevFrag Fs;
  __shared__ __align__(8) unsigned long long mbar[STG_BUF];
  const int tid = threadIdx.x;
  if (tid == 0) Fs = fr[blockIdx.y];
  __syncthreads();
  const DevFrag& F = Fs;
  const int ex = F.dext[0], ey = F.dext[1], ez = F.dext[2];
  const int y0 = (int)blockIdx.x * ty, y1 = min(ey, y0 + ty);
  const int z0 = (int)blockIdx.z * zc, z1 = min(ez, z0 + zc);
  if (y0 >= y1 || z0 >= z1) return;   // uniform over the CTA
  const int qpp = F.ld / VN;
  const int rows = y1 - y0 + 2;                 // staged rows y0-1 .. y1
  const long long rowE = (long long)ex * F.ld;  // elements of one storage row
  const long long planeE = rows * rowE;         // elements of one staged plane
  T* buf = reinterpret_cast<T*>(stg_smem);
  if (tid == 0) {
    for (int i = 0; i < STG_BUF; ++i) mbar_init(smem_u32(&mbar[i]), 1);
    fence_mbar_init();
  }
  // Staged row r holds storage row y0-1+r (wrapped in a full-span dimension);
  // only the first and the last staged row can fall outside the storage box.
  auto srow = [&](int r) { return ((y0 - 1 + r) % ey + ey) % ey; };
  auto zero_row = [&](int r) { return !F.full[1] && (y0 - 1 + r < 0 || y0 - 1 + r >= ey); };
  // those rows read zero: written once, never the target of a copy
  for (int k = 0; k < 2; ++k) {
    const int r = k ? rows - 1 : 0;
    if (zero_row(r))
      for (int i = 0; i < STG_BUF; ++i)
        for (long long e = tid; e < rowE; e += STG_THREADS) buf[i * planeE + r * rowE + e] = T(0);
  }
  fence_async_smem();
  __syncthreads();

  const T* src = in + F.off;
  // end of the run of staged rows from r that is contiguous in storage
  auto run_end = [&](int r) {
    int r2 = r + 1;
    if (zero_row(r)) return r2;
    while (r2 < rows && !zero_row(r2) && srow(r2) == srow(r2 - 1) + 1) ++r2;
    return r2;
  };
  auto plane_ok = [&](int p) { return F.full[2] || (p >= 0 && p < ez); };
  // thread 0: fetch plane p (z0-1 <= p <= z1) into ring slot (p-z0+1) % STG_BUF
  auto issue = [&](int p) {
    const int j = p - (z0 - 1);
    const uint32_t mb = smem_u32(&mbar[j % STG_BUF]);
    if (!plane_ok(p)) {
      mbar_arrive(mb);   // the phase completes without a copy; the plane is skipped
      return;
    }
    const int zz = (p % ez + ez) % ez;
    T* dst = buf + (long long)(j % STG_BUF) * planeE;
    uint32_t bytes = 0;
    for (int r = 0; r < rows; ++r)
      if (!zero_row(r)) bytes += (uint32_t)(rowE * sizeof(T));
    mbar_arrive_expect(mb, bytes);
    for (int r = 0; r < rows;) {
      const int r2 = run_end(r);
      if (!zero_row(r))
        bulk_g2s(smem_u32(dst + r * rowE), src + ((long long)zz * ey + srow(r)) * rowE,
                 (uint32_t)((r2 - r) * rowE * sizeof(T)), mb);
      r = r2;
    }
  };
  auto wait_plane = [&](int p) {
    const int j = p - (z0 - 1);
    return mbar_wait(smem_u32(&mbar[j % STG_BUF]), (uint32_t)((j / STG_BUF) & 1), flag);
  };
  // prologue: fill the ring with planes z0-1 .. z0+STG_BUF-2; afterwards the
  // end of iteration z refills the slot of plane z-1 with plane z+STG_BUF-1
  const int plast = z1;   // last plane needed
  int pnext = min(plast, z0 + STG_BUF - 2) + 1;   // next plane to issue
  if (tid == 0)
    for (int p = z0 - 1; p < pnext; ++p) issue(p);
  int pwait = z0 - 1;     // planes < pwait have been waited for

  const int per_row = ex * qpp;
  const int nel = (y1 - y0) * per_row;   // <= STG_THREADS * STG_EPT (host's tile choice)
  V16* O = reinterpret_cast<V16*>(out + F.off);
  const long long vplane = (long long)gx * gy;
  const int rowq = ex * qpp;   // 16-byte elements of one staged row
  // per element of this thread: staged index, global index within a plane, V index within a plane
  int sidx[STG_EPT], xs[STG_EPT], gidx[STG_EPT], vidx[STG_EPT];   // all < 2^31 (planner)
#pragma unroll
  for (int u = 0; u < STG_EPT; ++u) {
    const int e = tid + u * STG_THREADS;
    const int ee = e < nel ? e : 0;
    const int yl = ee / per_row;
    const int rem = ee - yl * per_row;
    const int x = rem / qpp, q = rem - x * qpp;
    const int y = y0 + yl;
    xs[u] = x;
    sidx[u] = (yl + 1) * rowq + x * qpp + q;
    gidx[u] = (y * ex + x) * qpp + q;
    vidx[u] = ((F.doff[1] + y) % gy) * gx + (F.doff[0] + x) % gx;
  }
  const long long gplane = (long long)ey * ex * qpp;   // 16-byte elements of one storage plane
  // V of the plane being computed, loaded one iteration ahead
  T vv[STG_EPT];
  auto prefetch = [&](int z) {
    const long long zv = (long long)((F.doff[2] + z) % gz) * vplane;
#pragma unroll
    for (int u = 0; u < STG_EPT; ++u) {
      if (tid + u * STG_THREADS < nel) vv[u] = V[zv + vidx[u]];
    }
  };
  prefetch(z0);
  bool ok = true;
  for (int z = z0; z < z1; ++z) {
    T vc[STG_EPT];
#pragma unroll
    for (int u = 0; u < STG_EPT; ++u) vc[u] = vv[u];
    if (z + 1 < z1) prefetch(z + 1);
    // planes z-1, z, z+1 must have landed
    while (ok && pwait <= z + 1) {
      ok = wait_plane(pwait);
      if (ok) ++pwait;
    }
    if (!__syncthreads_and(ok)) {
      ok = false;
      break;
    }
    const int jb = z - 1 - (z0 - 1), jc = jb + 1, ja = jb + 2;
    const V16* Bb = reinterpret_cast<const V16*>(buf + (long long)(jb % STG_BUF) * planeE);
    const V16* Bc = reinterpret_cast<const V16*>(buf + (long long)(jc % STG_BUF) * planeE);
    const V16* Ba = reinterpret_cast<const V16*>(buf + (long long)(ja % STG_BUF) * planeE);
    const bool has_b = plane_ok(z - 1), has_a = plane_ok(z + 1);
    const long long zo = (long long)z * gplane;
#pragma unroll
    for (int u = 0; u < STG_EPT; ++u) {
      if (tid + u * STG_THREADS >= nel) continue;
      const int sc = sidx[u], x = xs[u];
      V16 sum = add4(Bc[sc + rowq], Bc[sc - rowq]);
      const int xp = nb_index(x, x, ex, F.full[0], +1, 1), xm = nb_index(x, x, ex, F.full[0], -1, 1);
      if (xp >= 0) sum = add4(sum, Bc[sc + (xp - x) * qpp]);
      if (xm >= 0) sum = add4(sum, Bc[sc + (xm - x) * qpp]);
      if (has_b) sum = add4(sum, Bb[sc]);
      if (has_a) sum = add4(sum, Ba[sc]);
      V16 hy = fma4(c0 + vc[u], Bc[sc], zero4(T()));
      O[zo + gidx[u]] = fma4(-c1, sum, hy);
    }
    __syncthreads();   // slot of plane z-1 is free
    if (tid == 0 && pnext <= plast) issue(pnext);
    ++pnext;
  }
  if (!ok) {
    // drain: every issued copy must land before the CTA's shared memory is released
    for (; pwait < min(pnext, plast + 1); ++pwait) wait_plane(pwait);
    __syncthreads();
  }
}

// Launch shape of the stencils.  Staged form: x = row tiles of ty rows, y =
// fragments, z = chunks of zc planes; ty minimises the staged rows (tile plus
// two halo rows) per output row within the shared-memory budget (two CTAs per
// SM, else one) and at most STG_EPT elements per thread, and the chunk count
// fills about two resident waves of the GB300 (152 SMs).  Register form (fallback when even one row does not fit):
// x covers the (x, y, column group) elements of the largest plane.
ApplyGrid apply_grid(const std::vector<DevFrag>& fr, bool fp64, int form) {
  const int vn = fp64 ? 2 : 4;
  const int es = fp64 ? 8 : 4;
  const int sms = 152;
  long long mx = 1, threads = 0, rowB = 0, rowQ = 0;
  int zmax = 1, ymax = 1;
  for (const DevFrag& f : fr) {
    const long long xy = (long long)f.dext[0] * f.dext[1] * (f.ld / vn);
    mx = std::max(mx, xy);
    threads += xy;
    zmax = std::max(zmax, f.dext[2]);
    ymax = std::max(ymax, f.dext[1]);
    rowB = std::max(rowB, (long long)f.dext[0] * f.ld * es);
    rowQ = std::max(rowQ, (long long)f.dext[0] * (f.ld / vn));
  }
  ApplyGrid g;
  // staged form where the caller (form 2), or with form 0 OFM_STENCIL=staged,
  // asks for it
  const char* env = std::getenv("OFM_STENCIL");
  const bool try_staged =
      form == 2 || (form == 0 && env != nullptr && std::strcmp(env, "staged") == 0);
  const long long budgets[2] = {110 * 1024, 200 * 1024};
  for (int bi = 0; bi < 2 && try_staged && !g.staged; ++bi) {
    int best = 0;
    long long best_cost = 0;
    for (int ty = 1; ty <= ymax; ++ty) {
      if ((long long)STG_BUF * (ty + 2) * rowB > budgets[bi]) break;
      if ((long long)ty * rowQ > (long long)STG_THREADS * STG_EPT) break;
      const long long cost = (long long)((ymax + ty - 1) / ty) * (ty + 2);
      if (best == 0 || cost <= best_cost) {
        best = ty;
        best_cost = cost;
      }
    }
    if (best > 0) {
      g.staged = true;
      g.ty = best;
      g.smem = (int)((long long)STG_BUF * (best + 2) * rowB);
      const int per_sm = bi == 0 ? 2 : 1;
      long long per_chunk = 0;
      for (const DevFrag& f : fr) per_chunk += (f.dext[1] + best - 1) / best;
      const long long nch = std::max(1LL, std::min<long long>(zmax, (2LL * sms * per_sm + per_chunk - 1) / per_chunk));
      g.zc = (int)((zmax + nch - 1) / nch);
      g.z = (zmax + g.zc - 1) / g.zc;
      g.x = (ymax + best - 1) / best;
    }
  }
  if (g.staged) {
    // once per plan (the call is not free: kept out of the launch path)
    const void* k = fp64 ? (const void*)apply_staged_kernel<double> : (const void*)apply_staged_kernel<float>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_PLAN_MAX) == cudaSuccess)
      return g;
    cudaGetLastError();   // not available: the register form below
    g = ApplyGrid();
  }
  // register form
  g.x = (int)((mx + 255) / 256);
  const long long want = 2LL * sms * 2048;
  const long long nch = std::max(1LL, std::min<long long>(zmax, (want + threads - 1) / std::max(1LL, threads)));
  g.zc = (int)((zmax + nch - 1) / nch);
  g.z = (zmax + g.zc - 1) / g.zc;
  return g;
}

template <typename T>
static void zmarch(const ApplyGrid& ag, int nfrag, const DevFrag* d_fr, const void* V,
                   const void* in, void* out, const int gn[3], double h, int* flag, cudaStream_t s) {
  const double c0 = 3.0 / (h * h), c1 = 0.5 / (h * h);
  dim3 g(ag.x, nfrag, ag.z);
  if (ag.staged)
    apply_staged_kernel<T><<<g, STG_THREADS, ag.smem, s>>>(d_fr, (const T*)V, (const T*)in, (T*)out, gn[0], gn[1],
                                                          gn[2], (T)c0, (T)c1, ag.ty, ag.zc, flag);
  else
    apply_zmarch_kernel<T><<<g, 256, 0, s>>>(d_fr, (const T*)V, (const T*)in, (T*)out, gn[0], gn[1], gn[2],
                                             (T)c0, (T)c1, ag.zc);
}

void launch_apply_global(const DevFrag* d_fr, int nfrag, const ApplyGrid& g, const void* V,
                         const void* states, void* hphi, const int gn[3], double h, bool fp64,
                         int* flag, cudaStream_t s) {
  if (fp64) zmarch<double>(g, nfrag, d_fr, V, states, hphi, gn, h, flag, s);
  else zmarch<float>(g, nfrag, d_fr, V, states, hphi, gn, h, flag, s);
}

// ------------------------------------------------------------ conversions --

// Columns [first, first + Fn.n) of one fragment's stored states (every
// storage point, halo included) into the layout Fn; pad columns zero.
template <typename T>
__global__ void select_states_kernel(DevFrag Fo, DevFrag Fn, int first, const T* __restrict__ src,
                                     T* __restrict__ dst) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Fn.Pd * Fn.ld) return;
  const long long p = i / Fn.ld;
  const int j = (int)(i - p * Fn.ld);
  dst[Fn.off + i] = (j < Fn.n) ? src[Fo.off + p * Fo.ld + first + j] : T(0);
}

void launch_select_states(const DevFrag& Fo, const DevFrag& Fn, int first, const void* src,
                          void* dst, bool fp64, cudaStream_t s) {
  const long long n = Fn.Pd * Fn.ld;
  const int blocks = (int)((n + 255) / 256);
  if (fp64)
    select_states_kernel<double><<<blocks, 256, 0, s>>>(Fo, Fn, first, (const double*)src, (double*)dst);
  else
    select_states_kernel<float><<<blocks, 256, 0, s>>>(Fo, Fn, first, (const float*)src, (float*)dst);
}

template <typename T>
__global__ void convert_V_kernel(const double* __restrict__ src, T* __restrict__ dst, long long n) {
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = (T)src[i];
}

void launch_convert_V(const double* src, void* dst, long long n, bool fp64, cudaStream_t s) {
  int blocks = (int)((n + 255) / 256);
  if (fp64) convert_V_kernel<double><<<blocks, 256, 0, s>>>(src, (double*)dst, n);
  else convert_V_kernel<float><<<blocks, 256, 0, s>>>(src, (float*)dst, n);
}

// Column-major box states (P x n, box order) -> point-major dilated storage.
// Writes every interior point and every state column < ld (pad columns get 0).
template <typename T>
__global__ void import_kernel(DevFrag F, const double* __restrict__ src, T* __restrict__ dst) {
  const long long P = (long long)F.ext[0] * F.ext[1] * F.ext[2];
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P * F.ld) return;
  const int s = (int)(i / P);
  const long long p = i - (long long)s * P;
  const int x = (int)(p % F.ext[0]);
  const int y = (int)((p / F.ext[0]) % F.ext[1]);
  const int z = (int)(p / ((long long)F.ext[0] * F.ext[1]));
  const long long pd = ((long long)(z + F.lo[2]) * F.dext[1] + (y + F.lo[1])) * F.dext[0] + (x + F.lo[0]);
  dst[F.off + pd * F.ld + s] = (s < F.n) ? (T)src[(long long)s * P + p] : (T)0;
}

void launch_import_states(const DevFrag* /*d_fr*/, int /*a*/, const DevFrag& fa, const double* src,
                          void* states, bool fp64, cudaStream_t s) {
  const long long P = (long long)fa.ext[0] * fa.ext[1] * fa.ext[2];
  const long long tot = P * fa.ld;
  int blocks = (int)((tot + 255) / 256);
  if (fp64) import_kernel<double><<<blocks, 256, 0, s>>>(fa, src, (double*)states);
  else import_kernel<float><<<blocks, 256, 0, s>>>(fa, src, (float*)states);
}

// Point-major storage -> column-major doubles.  dilated=false: box points
// (P_a x n); dilated=true: every point of the dilated box (Pd x n).
template <typename T>
__global__ void export_kernel(DevFrag F, const T* __restrict__ srcbuf, double* __restrict__ dst,
                              int dilated) {
  const int ex = dilated ? F.dext[0] : F.ext[0];
  const int ey = dilated ? F.dext[1] : F.ext[1];
  const int ez = dilated ? F.dext[2] : F.ext[2];
  const long long P = (long long)ex * ey * ez;
  long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P * F.n) return;
  const int s = (int)(i / P);
  const long long p = i - (long long)s * P;
  const int x = (int)(p % ex);
  const int y = (int)((p / ex) % ey);
  const int z = (int)(p / ((long long)ex * ey));
  const int ox = dilated ? 0 : F.lo[0], oy = dilated ? 0 : F.lo[1], oz = dilated ? 0 : F.lo[2];
  const long long pd = ((long long)(z + oz) * F.dext[1] + (y + oy)) * F.dext[0] + (x + ox);
  dst[(long long)s * P + p] = (double)srcbuf[F.off + pd * F.ld + s];
}

void launch_export_states(const DevFrag& fa, const void* buf, double* dst, bool fp64,
                          bool dilated, cudaStream_t s) {
  const long long P = dilated ? fa.Pd : (long long)fa.ext[0] * fa.ext[1] * fa.ext[2];
  const long long tot = P * fa.n;
  int blocks = (int)((tot + 255) / 256);
  if (fp64) export_kernel<double><<<blocks, 256, 0, s>>>(fa, (const double*)buf, dst, dilated ? 1 : 0);
  else export_kernel<float><<<blocks, 256, 0, s>>>(fa, (const float*)buf, dst, dilated ? 1 : 0);
}

}  // namespace ofm
