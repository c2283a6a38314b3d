// Block-sparse products with the assembled pencil of Eq. 2: Y = H X or
// Y = S X over the pair list, H and S taken from the FP64 pair blocks (the
// block a <= b is stored, the block b > a is its transpose).  This is the
// operation a window solver that never forms the dense n x n matrices is
// built from, for bases too large for the dense FP64 path.
//
// One CTA per (fragment a, R of its rows, up to 16 columns of X), R = 8 or 16:
// the output tile accumulates over the row's blocks in a fixed order (the pair
// list's), so the result is deterministic.  FP64 throughout, and FP64 bound:
// a product of 16 columns does 8 FMAs per byte of the blocks.  The tile is
// cut into 2 x MJ register tiles; the CTA's threads form G groups that take
// every G-th point of the inner index, so a product with one column keeps all
// lanes busy too, and the groups' sums are added in group order.  Block and X
// panels go through two shared-memory stages of asynchronous copies, either
// orientation of a block read along its stored rows.  64 fragments of 96
// states, H X and S X: k = 16: 2.59 ms with one CTA per (fragment, 8 columns)
// and a shuffle reduction per output, 0.83 ms now (1.2 TFLOP/s).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include "ofm_internal.h"

namespace ofm {
namespace {

constexpr int SP_C = 16;         // columns of X per CTA at most
constexpr int SP_R = 16;         // rows per CTA at most
constexpr int SP_KB = 64;        // inner points per stage
constexpr int SP_LD = 18;        // shared row stride: even (16-byte reads), 2 mod 16 banks
constexpr int SP_THREADS = 128;

struct SpEnt {
  long long off;   // arena offset of the stored pair's H block (its S block follows)
  int b;           // column fragment
  int tr;          // 1: the stored block is M_ba (the pair is (b, a)), read transposed
};

__device__ __forceinline__ void cpa8(double* dst, const double* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"((unsigned long long)__cvta_generic_to_global(src))
               : "memory");
}

// MJ: columns of a register tile (1 for a single column, else 2)
template <int MJ>
__global__ void __launch_bounds__(SP_THREADS) pencil_apply_kernel(
    const double* __restrict__ blocks, const DevFrag* __restrict__ fr, const int* __restrict__ rowptr,
    const SpEnt* __restrict__ ents, int which, const double* __restrict__ X, long long ldx,
    double* __restrict__ Y, long long ldy, int k, int R) {
  __shared__ __align__(16) double Ms[2][SP_KB * SP_LD], Xs[2][SP_KB * SP_LD];   // [point][row / column]
  const int a = blockIdx.x, r0 = blockIdx.y * R, c0 = blockIdx.z * SP_C;
  const int na = fr[a].n, ra = fr[a].basis0;
  if (r0 >= na) return;   // uniform
  const int mr = min(R, na - r0), kc = min(SP_C, k - c0);
  const int q0 = rowptr[a], q1 = rowptr[a + 1];
  const int tid = threadIdx.x;
  const int tm = (mr + 1) / 2, tn = (kc + MJ - 1) / MJ, T = tm * tn;   // T <= 64
  const int G = SP_THREADS / T, g = tid / T, t = tid - g * T;
  const int i0 = 2 * (t / tn), j0 = MJ * (t % tn);
  double acc[2][MJ];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < MJ; ++j) acc[i][j] = 0.0;
  // pad rows and columns of the tile are read by the last register tiles
  for (int e = tid; e < 2 * SP_KB * SP_LD; e += SP_THREADS) {
    (&Ms[0][0])[e] = 0.0;
    (&Xs[0][0])[e] = 0.0;
  }
  __syncthreads();
  // stages of (block q, points p0 .. p0 + SP_KB), in order
  int iq = q0, ip = 0;   // next stage to issue
  auto issue = [&](int buf) {
    if (iq < q1) {
      const SpEnt E = ents[iq];
      const int nb = fr[E.b].n;
      const int nk = min(SP_KB, nb - ip);
      // the stored block holds n_a n_b entries whichever way it is stored
      const double* m = blocks + E.off + (which ? (long long)na * nb : 0);
      if (E.tr) {   // M_ba: row j, columns r0 ..
        for (int e = tid; e < nk * SP_R; e += SP_THREADS) {
          const int j = e / SP_R, i = e % SP_R;
          if (i < mr) cpa8(&Ms[buf][j * SP_LD + i], m + (long long)(ip + j) * na + r0 + i);
        }
      } else {
        for (int e = tid; e < mr * SP_KB; e += SP_THREADS) {
          const int i = e / SP_KB, j = e % SP_KB;
          if (j < nk) cpa8(&Ms[buf][j * SP_LD + i], m + (long long)(r0 + i) * nb + ip + j);
        }
      }
      const double* xb = X + (long long)c0 * ldx + fr[E.b].basis0 + ip;
      for (int e = tid; e < kc * SP_KB; e += SP_THREADS) {
        const int c = e / SP_KB, j = e % SP_KB;
        if (j < nk) cpa8(&Xs[buf][j * SP_LD + c], xb + c * ldx + j);
      }
      ip += SP_KB;
      if (ip >= nb) {
        ip = 0;
        ++iq;
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  issue(0);
  int buf = 0;
  for (int q = q0; q < q1; ++q) {
    const int nb = fr[ents[q].b].n;
    for (int p0 = 0; p0 < nb; p0 += SP_KB, buf ^= 1) {
      issue(buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
      __syncthreads();
      const int nk = min(SP_KB, nb - p0);
      if (g < G) {
#pragma unroll 4
        for (int j = g; j < nk; j += G) {
          const double2 m = *reinterpret_cast<const double2*>(&Ms[buf][j * SP_LD + i0]);
          double x[MJ];
          if constexpr (MJ == 2) {
            const double2 x2 = *reinterpret_cast<const double2*>(&Xs[buf][j * SP_LD + j0]);
            x[0] = x2.x;
            x[1] = x2.y;
          } else {
            x[0] = Xs[buf][j * SP_LD + j0];
          }
#pragma unroll
          for (int c = 0; c < MJ; ++c) {
            acc[0][c] = fma(m.x, x[c], acc[0][c]);
            acc[1][c] = fma(m.y, x[c], acc[1][c]);
          }
        }
      }
      __syncthreads();   // the stage is consumed
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // the groups' sums in group order: [g][tile][2][MJ], at most 4 values a thread
  double* red = &Ms[0][0];
  static_assert(SP_THREADS * 4 <= 2 * SP_KB * SP_LD, "the groups' sums fit the stages");
  if (g < G)
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < MJ; ++j) red[(g * T + t) * 2 * MJ + i * MJ + j] = acc[i][j];
  __syncthreads();
  for (int e = tid; e < T * 2 * MJ; e += SP_THREADS) {
    const int tt = e / (2 * MJ), ij = e % (2 * MJ);
    const int i = 2 * (tt / tn) + ij / MJ, c = MJ * (tt % tn) + ij % MJ;
    double v = 0.0;
    for (int q = 0; q < G; ++q) v += red[q * T * 2 * MJ + e];
    if (i < mr && c < kc) Y[(long long)(c0 + c) * ldy + ra + r0 + i] = v;
  }
}

}  // namespace

// Block rows of the pencil for the current pair list: for every fragment its
// pairs in the pair list's order, the stored block a <= b as is, the mirror
// b > a transposed.  Rebuilt only after the pair list or the plan changes.
static ofm_status pencil_tables(ofm_ctx* c) {
  if (!c->sp_stale) return OFM_OK;
  const int nf = c->nfrag;
  std::vector<std::vector<SpEnt>> rows(nf);
  for (size_t p = 0; p < c->pairs.size(); ++p) {
    const int a = c->pairs[p].a, b = c->pairs[p].b;
    const long long off = c->simt_pairs[p].blk_off;
    rows[a].push_back({off, b, 0});
    if (b != a) rows[b].push_back({off, a, 1});
  }
  std::vector<int> rowptr(nf + 1, 0);
  std::vector<SpEnt> ents;
  for (int a = 0; a < nf; ++a) {
    ents.insert(ents.end(), rows[a].begin(), rows[a].end());
    rowptr[a + 1] = (int)ents.size();
  }
  OFM_TRY(ofm_ensure(c, c->sp_rowptr, sizeof(int) * (nf + 1), "pencil block rows"));
  OFM_TRY(ofm_ensure(c, c->sp_ents, sizeof(SpEnt) * std::max<size_t>(1, ents.size()), "pencil blocks"));
  OFM_CUDA(c, cudaMemcpyAsync(c->sp_rowptr.p, rowptr.data(), sizeof(int) * (nf + 1),
                              cudaMemcpyHostToDevice, c->stream));
  OFM_CUDA(c, cudaMemcpyAsync(c->sp_ents.p, ents.data(), sizeof(SpEnt) * ents.size(),
                              cudaMemcpyHostToDevice, c->stream));
  OFM_CUDA(c, cudaStreamSynchronize(c->stream));   // the host tables are released
  c->sp_flops_per_col = 0.0;
  c->sp_bytes_fixed = 0.0;
  for (size_t p = 0; p < c->pairs.size(); ++p) {
    const double nn = (double)c->frags[c->pairs[p].a].n * c->frags[c->pairs[p].b].n;
    c->sp_flops_per_col += (c->pairs[p].a == c->pairs[p].b ? 2.0 : 4.0) * nn;
    c->sp_bytes_fixed += 8.0 * nn;   // one of the pair's two blocks is read per product
  }
  c->sp_stale = false;
  return OFM_OK;
}

}  // namespace ofm

using namespace ofm;

static ofm_status ofm_pencil_apply_impl(ofm_ctx* c, int which, const double* X, long long ldx,
                                       double* Y, long long ldy, int k) {
  OFM_RANGE("ofm_pencil_apply");
  if (!c) return OFM_ERR_INVALID;
  if (!c->assembled) return ofm_fail(c, OFM_ERR_STATE, "ofm_assemble_HS must come first");
  if (which != 0 && which != 1) return ofm_fail(c, OFM_ERR_INVALID, "which must be 0 (H) or 1 (S)");
  if (!X || !Y) return ofm_fail(c, OFM_ERR_INVALID, "X and Y must not be NULL");
  if (k < 1) return ofm_fail(c, OFM_ERR_INVALID, "k must be >= 1");
  const long long n = c->basis;
  if (ldx < n || ldy < n) return ofm_fail(c, OFM_ERR_INVALID, "leading dimensions must be >= the basis size");
  {   // Y must not overlap X (the kernel reads X while it writes Y)
    const char* x0 = (const char*)X;
    const char* x1 = (const char*)(X + (k - 1) * ldx + n);
    const char* y0 = (const char*)Y;
    const char* y1 = (const char*)(Y + (k - 1) * ldy + n);
    if (x0 < y1 && y0 < x1) return ofm_fail(c, OFM_ERR_INVALID, "X and Y overlap");
  }
  OFM_TRY(ofm_wait_status(c));
  OFM_TRY(pencil_tables(c));
  {
    // algorithmic traffic: every stored block once, X read and Y written once
    KTimer kt(c, KC_PENCIL, 1, c->sp_bytes_fixed + 16.0 * (double)n * k, c->sp_flops_per_col * k);
    int namax = 1;
    for (const DevFrag& f : c->frags) namax = std::max(namax, f.n);
    // 16 rows per CTA (less X traffic) where that leaves 8 CTAs per SM, else 8
    const long long z = (k + SP_C - 1) / SP_C;
    const int R = (long long)c->nfrag * ((namax + 15) / 16) * z >= 8 * 152 ? 16 : 8;
    // grid.z is limited to 65535: very wide X goes in slices of columns
    for (long long z0 = 0; z0 < z; z0 += 65535) {
      const dim3 g(c->nfrag, (namax + R - 1) / R, (unsigned)std::min<long long>(65535, z - z0));
      const double* x = X + z0 * SP_C * ldx;
      double* y = Y + z0 * SP_C * ldy;
      const int kk = (int)(k - z0 * SP_C);
      const double* blk = (const double*)c->blocks.p;
      const DevFrag* f = (const DevFrag*)c->d_frags.p;
      const int* rp = (const int*)c->sp_rowptr.p;
      const SpEnt* en = (const SpEnt*)c->sp_ents.p;
      if (k == 1) pencil_apply_kernel<1><<<g, SP_THREADS, 0, c->stream>>>(blk, f, rp, en, which, x, ldx, y, ldy, kk, R);
      else pencil_apply_kernel<2><<<g, SP_THREADS, 0, c->stream>>>(blk, f, rp, en, which, x, ldx, y, ldy, kk, R);
    }
  }
  OFM_CUDA(c, cudaGetLastError());
  return OFM_OK;
}

extern "C" ofm_status ofm_pencil_apply(ofm_ctx* c, int which, const double* X, long long ldx, double* Y, long long ldy, int k) {
  const ofm_status st = ofm_pencil_apply_impl(c, which, X, ldx, Y, ldy, k);
  if (st != OFM_OK || !c || !c->checks) return st;
  return ofm_check_guards_now(c, "ofm_pencil_apply");
}
