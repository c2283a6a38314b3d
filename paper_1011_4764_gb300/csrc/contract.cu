// Pair-block contraction on CUDA cores (FP64 and FP32 arithmetic), the
// deterministic reduction of K-chunk partials into FP64 blocks, and the
// scatter of blocks into dense basis-ordered H and S.
//
// For a pair a <= b the blocks are (Sec. II)
//     S_ab = Phi_a^T Phi_b       over B_a ∩ B_b,
//     H_ab = Phi_a^T (H Phi_b)   over B_a ∩ B_b+.
// States are stored on dilated boxes with a zero halo, so both sums run over
// the same region R = B_a ∩ B_b+ and become one GEMM
//     [S_ab | H_ab] = Phi_a[R]^T [Phi_b[R] | HPhi_b[R]]
// with M = n_a, N = 2 n_b and K = |R|.  R is cut into pieces (boxes that are
// contiguous in both storages) and each piece into chunks of whole x-rows; a
// CTA gathers the rows of its chunk into shared memory and accumulates one
// output tile of at most TILE x TILE, written as a partial.  The finalize kernel sums
// the partials of each pair in a fixed order, so results are bitwise
// reproducible run to run.
#include <cuda_runtime.h>

#include <algorithm>

#include "ofm_internal.h"

namespace ofm {

constexpr int TILE = 64;   // output tile edge
constexpr int NT = 256;    // threads per CTA
constexpr int STAGE_BYTES = 32 * 1024;   // staged rows of both operands
constexpr int KT_MAX = 256;              // points per stage at most

// MI adjacent values, read from shared memory as one 16-byte word
template <typename T, int MI>
struct alignas(16) MiVec {
  T v[MI];
};

// The products of the points g, g + G, ... of a stage for a thread's first NV
// register tiles.  NV is a compile-time count: a predicated-off FP64 FMA takes
// its slot in the FP64 pipe all the same (a run-time test of each of four
// tiles measured like four tiles: 1170 us instead of 285 us on a chain
// of 15 fragments of 21 states).  An absent tile reads the row's first columns and
// its sums are dropped.
template <typename Tacc, int MI, int NU, int NV>
__device__ __forceinline__ void simt_products(const Tacc* S, int w, int g, int nk, int G,
                                              const int (&ra)[NU], const int (&cb)[NU],
                                              Tacc (&acc)[NU][MI][MI]) {
#pragma unroll 2
  for (int kk = g; kk < nk; kk += G) {
    const Tacc* row = S + kk * w;
#pragma unroll
    for (int u = 0; u < NV; ++u) {
      const MiVec<Tacc, MI> a = *reinterpret_cast<const MiVec<Tacc, MI>*>(row + max(ra[u], 0));
      const MiVec<Tacc, MI> b = *reinterpret_cast<const MiVec<Tacc, MI>*>(row + cb[u]);
#pragma unroll
      for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < MI; ++j) acc[u][i][j] = fma(a.v[i], b.v[j], acc[u][i][j]);
    }
  }
}

// A CTA takes one item: the valid part (mr x nc, at most TILE x TILE) of an
// output tile over one K chunk.  The valid part is cut into MI x MI register
// tiles; T of them.  With T >= NT a thread owns up to NU of them and walks
// every point; with fewer, the CTA's threads form G = NT / T groups, group g
// takes the points g, g + G, ... of a stage, and the groups' sums are added
// in group order at the end (deterministic).  So no thread multiplies the
// padding of a 64 x 64 tile: the FP64 pipe (about 1.9 FMA per clock and SM) is
// the bound, and with 6-state fragments the padded tile does 57 times the
// useful products (tiny chain: 290 us padded, 19 us with these groups).
// FP64 takes MI = 2 (the finest split, its FMAs hide any shared-memory read),
// FP32 MI = 4 (2 shared reads per 4 FMAs).
template <typename Tin, typename Tacc, int MI, int NU>
__global__ void __launch_bounds__(NT) contract_simt_kernel(
    const DevFrag* __restrict__ fr, const DevPair* __restrict__ prs, const Piece* __restrict__ pcs,
    const WorkItem* __restrict__ items, const Tin* __restrict__ states,
    const Tin* __restrict__ hphi, Tacc* __restrict__ partials) {
  __shared__ __align__(16) unsigned char stage[STAGE_BYTES];
  __shared__ long long pa_s[KT_MAX], pb_s[KT_MAX];

  const WorkItem it = items[blockIdx.x];
  const DevPair pr = prs[it.pair];
  const DevFrag A = fr[pr.a];
  const DevFrag B = fr[pr.b];
  const Piece pc = pcs[it.piece];
  const int m0 = it.mt * TILE, n0 = it.nt * TILE;
  const Tin* Pa = states + A.off;
  const Tin* Pb = states + B.off;
  const Tin* Hb = hphi + B.off;
  const int tid = threadIdx.x;
  const int lenx = pc.len[0], leny = pc.len[1];
  const int npts = (it.r1 - it.r0) * lenx;
  const int mr = min(TILE, A.n - m0), nc = min(TILE, 2 * B.n - n0);
  const int tm = (mr + MI - 1) / MI, tn = (nc + MI - 1) / MI;
  const int T = tm * tn;   // register tiles of the item, row-major
  const int mrp = tm * MI, ncp = tn * MI, w = mrp + ncp;
  const int ktmax = min(KT_MAX, STAGE_BYTES / (w * (int)sizeof(Tacc)));
  const int G = T >= NT ? 1 : min(NT / T, ktmax);   // at most one group per staged point
  const int g = G > 1 ? tid / T : 0;   // >= G: idle in the products
  const int KT = G == 1 ? min(32, ktmax) : G * max(1, min(128, ktmax) / G);
  Tacc* S = reinterpret_cast<Tacc*>(stage);   // [point][A columns, then B columns]

  int ra[NU], cb[NU];   // shared-memory columns of this thread's register tiles (-1: none)
#pragma unroll
  for (int u = 0; u < NU; ++u) {
    const int q = G > 1 ? (u == 0 && g < G ? tid - g * T : T) : tid + u * NT;
    const int t = q < T ? q : 0;
    ra[u] = q < T ? (t / tn) * MI : -1;
    cb[u] = mrp + (t % tn) * MI;
  }
  Tacc acc[NU][MI][MI];
#pragma unroll
  for (int u = 0; u < NU; ++u)
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
      for (int j = 0; j < MI; ++j) acc[u][i][j] = Tacc(0);

  // staging: L lanes per point (a power of two covering w up to 32), four
  // points' loads in flight per lane group
  const int L = w > 16 ? 32 : w > 8 ? 16 : 8;
  const int lc = tid % L, lp = tid / L, np = NT / L;
  for (int k0 = 0; k0 < npts; k0 += KT) {
    const int nk = min(KT, npts - k0);
    for (int q = tid; q < nk; q += NT) {
      const int k = k0 + q;
      const int r = it.r0 + k / lenx, x = k % lenx;
      const int y = r % leny, z = r / leny;
      pa_s[q] = (((long long)(pc.la[2] + z) * A.dext[1] + (pc.la[1] + y)) * A.dext[0] + pc.la[0] + x) * A.ld;
      pb_s[q] = (((long long)(pc.lb[2] + z) * B.dext[1] + (pc.lb[1] + y)) * B.dext[0] + pc.lb[0] + x) * B.ld;
    }
    __syncthreads();
    for (int q0 = lp; q0 < nk; q0 += 4 * np)
      for (int c = lc; c < w; c += L) {
        // column c of a staged row: A state, Phi_b state or H Phi_b state
        const Tin* src = nullptr;
        bool isA = c < mrp;
        if (isA) {
          if (c < mr) src = Pa + m0 + c;
        } else {
          const int nn = n0 + c - mrp;
          if (c - mrp < nc) src = nn < B.n ? Pb + nn : Hb + (nn - B.n);
        }
        Tin v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int q = q0 + u * np;
          v[u] = Tin(0);
          if (src != nullptr && q < nk) v[u] = src[isA ? pa_s[q] : pb_s[q]];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int q = q0 + u * np;
          if (q < nk) S[q * w + c] = (Tacc)v[u];
        }
      }
    __syncthreads();
    if (g < G) {
      if (NU == 1 || T <= NT) simt_products<Tacc, MI, NU, 1>(S, w, g, nk, G, ra, cb, acc);
      else if (T <= 2 * NT) simt_products<Tacc, MI, NU, 2>(S, w, g, nk, G, ra, cb, acc);
      else simt_products<Tacc, MI, NU, NU>(S, w, g, nk, G, ra, cb, acc);
    }
    __syncthreads();
  }
  Tacc* out = partials + it.part_off;
  if (G == 1) {
#pragma unroll
    for (int u = 0; u < NU; ++u) {
      if (ra[u] < 0) continue;
#pragma unroll
      for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < MI; ++j) out[(ra[u] + i) * TILE + cb[u] - mrp + j] = acc[u][i][j];
    }
    return;
  }
  // the groups' sums, [g][i][j][tile] (NT MI^2 values at most), added in group order
  if (ra[0] >= 0)
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
      for (int j = 0; j < MI; ++j) S[((g * MI + i) * MI + j) * T + tid - g * T] = acc[0][i][j];
  __syncthreads();
  for (int e = tid; e < T * MI * MI; e += NT) {
    Tacc v = Tacc(0);
    for (int q = 0; q < G; ++q) v += S[q * T * MI * MI + e];
    const int t = e % T, ij = e / T;
    out[((t / tn) * MI + ij / MI) * TILE + (t % tn) * MI + ij % MI] = v;
  }
}

void launch_contract_simt(int prec, bool store_fp64, const DevFrag* d_fr, const DevPair* d_pairs,
                          const Piece* d_pieces, const WorkItem* d_items, int nitems,
                          const void* states, const void* hphi, void* partials, int tile,
                          cudaStream_t s) {
  (void)tile;
  if (nitems <= 0) return;
  static_assert(NT * 2 * 2 * sizeof(double) <= STAGE_BYTES && NT * 4 * 4 * sizeof(float) <= STAGE_BYTES,
                "the groups' sums fit the staging buffer");
  if (prec == OFM_PREC_FP64) {
    if (store_fp64)
      contract_simt_kernel<double, double, 2, 4><<<nitems, NT, 0, s>>>(
          d_fr, d_pairs, d_pieces, d_items, (const double*)states, (const double*)hphi,
          (double*)partials);
    else
      contract_simt_kernel<float, double, 2, 4><<<nitems, NT, 0, s>>>(
          d_fr, d_pairs, d_pieces, d_items, (const float*)states, (const float*)hphi,
          (double*)partials);
  } else {
    contract_simt_kernel<float, float, 4, 1><<<nitems, NT, 0, s>>>(
        d_fr, d_pairs, d_pieces, d_items, (const float*)states, (const float*)hphi,
        (float*)partials);
  }
}

// Sum of the partials of output (i, c) of pair pr, chunks in plan order (a
// tile's chunks are consecutive items with consecutive partial tiles).
template <typename Tacc>
__device__ __forceinline__ double sum_partials(const DevPair& pr, const WorkItem* items,
                                               const Tacc* partials, int i, int c) {
  const int mt = i / TILE, nt = c / TILE;
  const int base = pr.item0 + (mt * pr.ntiles + nt) * pr.nchunk;
  const Tacc* p = partials + items[base].part_off + (i % TILE) * TILE + (c % TILE);
  double s = 0.0;
#pragma unroll 4
  for (int k = 0; k < pr.nchunk; ++k) s += (double)p[(long long)k * TILE * TILE];
  return s;
}

// Block layout: H_ab then S_ab, each n_a x n_b row-major; blockIdx.y cuts a
// pair's outputs (one CTA per pair left the FP64 sums of a few pairs on as
// many SMs).
template <typename Tacc>
__global__ void finalize_simt_kernel(const DevFrag* __restrict__ fr, const DevPair* __restrict__ prs,
                                     const WorkItem* __restrict__ items,
                                     const Tacc* __restrict__ partials, double* __restrict__ blocks) {
  const DevPair pr = prs[blockIdx.x];
  const int na = fr[pr.a].n, nb = fr[pr.b].n;
  double* Hblk = blocks + pr.blk_off;
  double* Sblk = Hblk + (long long)na * nb;
  const bool diag = (pr.a == pr.b);
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < na * nb; e += gridDim.y * blockDim.x) {
    const int i = e / nb, m = e % nb;
    double s = sum_partials(pr, items, partials, i, m);
    double h = sum_partials(pr, items, partials, i, nb + m);
    if (diag) {
      s = 0.5 * (s + sum_partials(pr, items, partials, m, i));
      h = 0.5 * (h + sum_partials(pr, items, partials, m, nb + i));
    }
    Sblk[e] = s;
    Hblk[e] = h;
  }
}

void launch_finalize_simt(int prec, const DevFrag* d_fr, const DevPair* d_pairs, int npairs,
                          const WorkItem* d_items, const void* partials, int tile, double* blocks,
                          cudaStream_t s) {
  (void)tile;
  if (npairs <= 0) return;
  // about 16 CTAs per SM over all pairs, at most 16 per pair
  const int y = std::min(16, std::max(1, 16 * 152 / npairs));
  if (prec == OFM_PREC_FP64)
    finalize_simt_kernel<double><<<dim3(npairs, y), 256, 0, s>>>(
        d_fr, d_pairs, d_items, (const double*)partials, blocks);
  else
    finalize_simt_kernel<float><<<dim3(npairs, y), 256, 0, s>>>(
        d_fr, d_pairs, d_items, (const float*)partials, blocks);
}

// Dense basis-ordered matrices from the blocks; the lower block of a pair
// a < b is the transpose of its upper block.  Hd, Sd must be zeroed first.
__global__ void scatter_dense_kernel(const DevFrag* __restrict__ fr, const DevPair* __restrict__ prs,
                                     const double* __restrict__ blocks, int n,
                                     double* __restrict__ Hd, double* __restrict__ Sd) {
  const DevPair pr = prs[blockIdx.x];
  const DevFrag A = fr[pr.a], B = fr[pr.b];
  const double* Hblk = blocks + pr.blk_off;
  const double* Sblk = Hblk + (long long)A.n * B.n;
  for (int e = threadIdx.x; e < A.n * B.n; e += blockDim.x) {
    const int i = e / B.n, m = e % B.n;
    const long long r = A.basis0 + i, c = B.basis0 + m;
    Hd[r * n + c] = Hblk[e];
    Sd[r * n + c] = Sblk[e];
    if (pr.a != pr.b) {
      Hd[c * n + r] = Hblk[e];
      Sd[c * n + r] = Sblk[e];
    }
  }
}

void launch_scatter_dense(const DevFrag* d_fr, const DevPair* d_pairs, int npairs,
                          const double* blocks, int n, double* Hd, double* Sd, cudaStream_t s) {
  if (npairs <= 0) return;
  scatter_dense_kernel<<<npairs, 256, 0, s>>>(d_fr, d_pairs, blocks, n, Hd, Sd);
}

}  // namespace ofm
