// Pair-block contraction on the 5th-generation tensor cores (tcgen05), the
// "pair" schedule:
//     [S_ab | H_ab] = Phi_a[R]^T [Phi_b[R] | HPhi_b[R]]   (Sec. II),
// M = n_a (padded to 128), N = 2 n_b (each half padded to 8), K = |R|.
//
// Operands.  pack_kernel (region.cu) writes every fragment's states and H phi
// once per assembly, over its storage box with one axis widened to whole
// 8-point units of the grid: a unit (8 points along that axis) of a fragment is
// one contiguous block of rows_pad x 8 points in the K-major no-swizzle operand
// layout (core matrices of 8 states x 16 bytes; TF32 two cores per 8-state
// group, BF16 one), the rows of phi and of H phi one after the other (BF16 hi+lo:
// both hi, then both lo): one operand of 2 rows_pad MMA columns, since an MMA of 128
// rows takes about the same 33 ns for any number of them.  Both fragments of a pair share
// the grid's units and are zero outside their own boxes, so the pair sums over the
// units that both touch, and a run of units along the axis is one bulk copy: no
// conversion stands between the copies and the MMAs.  Of a only phi is wanted: its
// units come whole, H phi too (one copy a run, some 40 ns each, instead of one or two
// a unit), where they are small; a pair of a fragment with itself takes a's rows
// from b's copy.  56 uneven boxes with 826 pairs: contraction 2.13 ms in TF32 and 1.69
// in BF16 hi+lo with a conversion of FP32 rows in shared memory for every pair, 0.58
// and 0.74 ms with phi and H phi as separate planes and MMAs, 0.51 and 0.54 ms now.
//
// A persistent CTA per SM takes items (pair, rows of units of a piece) from a
// global counter, the largest first, through a warp-specialised pipeline: a
// producer warp issues the copies of a stage (one run of units per lane), one
// thread issues the MMAs into two alternating TMEM accumulators (a K step is one
// unit in TF32, two in BF16; hi*hi + hi*lo + lo*hi for the split), four warps
// drain an accumulator into the item's FP32 partial tile.  Operand rows past a
// fragment's own (M to 128) are whatever follows in shared memory: they reach
// only accumulator rows that nobody reads.  A finalize
// kernel sums the partials of each pair in a fixed order.  Every wait is
// bounded: on timeout the CTA sets an error flag, drains its copies and MMAs,
// frees its tensor memory and returns.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <vector>

#include "ofm_internal.h"
#include "ptx_util.h"

using namespace ofm;
using namespace ofm::ptx;

namespace {

struct TcFrag {
  int nux, dext1;     // units along the unit axis, extent along the next axis of the storage box
  int n, rows;        // states, padded to 8
  long long base;     // byte offset in the plane arena
};

struct TcPair {
  int a, b;
  int item0, nitem;
  long long blk_off;    // block arena offset (same layout as the CUDA-core path)
};

struct TcItem {
  int pair;
  int la[3], lb[3];     // start of the piece in both storage boxes, unit axis first (in units)
  int m, leny;          // units per row, rows per plane of the piece
  int r0, r1;           // rows of the item
  long long part_off;   // FP32 partial tile of n_a x 2 n_b
};

enum { TC_TF32 = 0, TC_BF16 = 1, TC_BF16X3 = 2, TC_NKIND = 3 };
template <int KIND> struct TcKind {
  static constexpr int UB = KIND == TC_TF32 ? 32 : 16;   // bytes of a unit per state
  static constexpr int NPL = KIND == TC_BF16X3 ? 2 : 1;  // parts of an operand (hi, lo)
  static constexpr int KU = KIND == TC_TF32 ? 1 : 2;     // units per MMA
  static constexpr int SHARE = KIND == TC_BF16 ? 2 : 1;  // BF16 takes half the plan's bytes
};

// ----------------------------------------------------------- PTX helpers --

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor, no swizzle: start address, leading
// (K-direction core) byte offset, stride (8-row group) byte offset,
// descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// Instruction descriptor: FP32 accumulator, A/B format (1 = BF16, 2 = TF32),
// both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t instr_desc(uint32_t fmt, uint32_t M, uint32_t N) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

template <int KIND>
__device__ __forceinline__ void mma(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                    uint32_t accum) {
  if constexpr (KIND == TC_TF32) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
        : "memory");
  } else {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
        : "memory");
  }
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
               : "memory");
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// ----------------------------------------------------------- the kernel ---

constexpr int TS_THREADS = 192;       // warp 0 copies, 1 MMA, 2-5 epilogue
constexpr int TS_NSTAGE = 4;
constexpr int TS_STAGE = 48 * 1024;
constexpr int TS_UMAX = 32;           // units of a stage at most (one run per lane)
constexpr int TS_NQ = 4;              // work-item ring between the roles
constexpr int TS_ACC_COLS = 256;      // TMEM columns of one accumulator; two of them
// stages, then room for the operand rows read past the last one, then 4 KB of
// zeros: the second half of a BF16 K step whose item ends with a single unit, 16
// bytes for each of up to 256 rows
constexpr int TS_NZERO = 256 * 16;
constexpr int TS_SLACK = 8 * 1024, TS_ZERO = TS_NSTAGE * TS_STAGE + TS_SLACK, TS_SMEM = TS_ZERO + TS_NZERO;

// Units per stage of a pair: a stage holds the units of both operands' planes;
// even, so that only an item's last stage can end with half a BF16 K step.
constexpr int TS_MINUNITS = 256;       // units an item may take whatever part of them is padding

// A pair's units in shared memory: bytes of a unit of b (phi, H phi), of a (the
// same, phi alone, or none of its own) and a's lo rows after its hi rows.  a comes
// whole where a stage still holds four units of both (BF16 hi+lo: 8 boxes 40^3, 96
// states, 612 us whole, 687 by parts; 27 boxes 24^3, 128 states, two units a stage,
// 926 and 836).
template <int KIND> struct TcShape {
  int pa, wa, wb, sa, lo_a, units;
  bool self, whole;
  __host__ __device__ constexpr TcShape(int ra, int rb, bool same)
      : pa(ra * TcKind<KIND>::UB), wa(2 * TcKind<KIND>::NPL * pa), wb(2 * TcKind<KIND>::NPL * rb * TcKind<KIND>::UB),
        sa(0), lo_a(0), units(0), self(same), whole(same || TS_STAGE / (wa + wb) >= 4) {
    sa = whole ? wa : TcKind<KIND>::NPL * pa;
    lo_a = whole ? 2 * pa : pa;
    const int u = TS_STAGE / (wb + (self ? 0 : sa));
    units = u > TS_UMAX ? TS_UMAX : u / 2 * 2;
  }
};
static_assert(TcShape<TC_TF32>(128, 128, false).units >= 4 && TcShape<TC_BF16X3>(128, 128, false).units >= 4,
              "four units fit a stage");

template <int KIND>
__global__ void __launch_bounds__(TS_THREADS, 1) tc_contract_kernel(
    const TcFrag* __restrict__ fr, const TcPair* __restrict__ prs, const TcItem* __restrict__ items,
    const int* __restrict__ order, int nitems, const unsigned char* __restrict__ planes,
    float* __restrict__ partials, int* flag, int* next) {
  using KT = TcKind<KIND>;
  constexpr int UB = KT::UB, NPL = KT::NPL, KU = KT::KU;
  constexpr uint32_t SBO = 8 * UB;     // next 8-state group of a unit
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) unsigned long long full[TS_NSTAGE], empty[TS_NSTAGE], acc_full[2], acc_empty[2];
  __shared__ __align__(8) unsigned long long q_full[TS_NQ], q_empty[TS_NQ];
  __shared__ int q_item[TS_NQ];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_s, issued_s, mma_steps_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid == 0) {
    for (int i = 0; i < TS_NSTAGE; ++i) {
      mbar_init(smem_u32(&full[i]), 1);
      mbar_init(smem_u32(&empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&acc_full[i]), 1);
      mbar_init(smem_u32(&acc_empty[i]), 4);
    }
    for (int i = 0; i < TS_NQ; ++i) {
      mbar_init(smem_u32(&q_full[i]), 1);
      mbar_init(smem_u32(&q_empty[i]), 5);   // the MMA thread and the four epilogue warps
    }
    fence_mbar_init();
    abort_s = 0;
    issued_s = 0;
    mma_steps_s = 0;
  }
  for (int i = tid; i < TS_NZERO / 16; i += TS_THREADS)
    reinterpret_cast<uint4*>(smem + TS_ZERO)[i] = make_uint4(0, 0, 0, 0);
  fence_async_smem();   // the zeros are read by the tensor cores
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(2 * TS_ACC_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  // bounded wait that also ends when another role gave up
  auto wait = [&](unsigned long long* bar, uint32_t parity) -> bool {
    const uint32_t a = smem_u32(bar);
    for (int i = 0; i < (1 << 20); ++i) {
      if (mbar_try(a, parity)) return true;
      if (*(volatile int*)&abort_s) return false;
    }
    atomicExch(flag, 1);
    *(volatile int*)&abort_s = 1;
    return false;
  };

  if (warp == 0) {
    // ---------------------------------------------------------- producer
    int g = 0;
    bool ok = true;
    for (int item_no = 0; ok; ++item_no) {
      const int qs = item_no % TS_NQ, qu = item_no / TS_NQ;
      int ii = 0;
      if (lane == 0) {
        const bool w = qu == 0 || wait(&q_empty[qs], (uint32_t)((qu - 1) & 1));
        ii = w ? atomicAdd(next, 1) : nitems;
        ii = ii < nitems ? order[ii] : -1;
        q_item[qs] = ii;
        mbar_arrive(smem_u32(&q_full[qs]));   // release: the index is visible to the waiters
        ok = w;
      }
      ii = __shfl_sync(0xffffffffu, ii, 0);
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
      if (!ok || ii < 0) break;
      const TcItem it = items[ii];
      const TcPair pr = prs[it.pair];
      const TcFrag A = fr[pr.a], B = fr[pr.b];
      const TcShape<KIND> sh(A.rows, B.rows, pr.a == pr.b);
      const int U = sh.units;
      const int nu = (it.r1 - it.r0) * it.m;
      for (int k0 = 0; k0 < nu; k0 += U, ++g) {
        const int s = g % TS_NSTAGE, u = g / TS_NSTAGE;
        if (u > 0) {
          bool w = true;
          if (lane == 0) w = wait(&empty[s], (uint32_t)((u - 1) & 1));
          ok = __shfl_sync(0xffffffffu, w ? 1 : 0, 0) != 0;
          if (!ok) break;
        }
        const int nk = min(U, nu - k0);
        const uint32_t mb = smem_u32(&full[s]);
        if (lane == 0) mbar_arrive_expect(mb, (uint32_t)(nk * (sh.wb + (sh.self ? 0 : sh.sa))));
        __syncwarp();
        const int row0 = k0 / it.m, x0 = k0 - row0 * it.m;
        const int nruns = (k0 + nk - 1) / it.m - row0 + 1;   // <= U <= 32
        if (lane < nruns) {
          const int x = lane == 0 ? x0 : 0;
          const int ks = lane == 0 ? k0 : (row0 + lane) * it.m;
          const int run = min(it.m - x, k0 + nk - ks);
          const int r = it.r0 + row0 + lane;
          const int y = r % it.leny, z = r / it.leny;
          const long long qa = ((long long)(it.la[2] + z) * A.dext1 + it.la[1] + y) * A.nux + it.la[0] + x;
          const long long qb = ((long long)(it.lb[2] + z) * B.dext1 + it.lb[1] + y) * B.nux + it.lb[0] + x;
          const unsigned char* sa = planes + A.base / KT::SHARE + qa * sh.wa;
          const unsigned char* sb = planes + B.base / KT::SHARE + qb * sh.wb;
          const uint32_t dB = smem_u32(smem + (size_t)s * TS_STAGE), dA = dB + (uint32_t)(U * sh.wb);
          bulk_g2s(dB + (uint32_t)((ks - k0) * sh.wb), sb, (uint32_t)(run * sh.wb), mb);
          const uint32_t oa = dA + (uint32_t)((ks - k0) * sh.sa);
          if (sh.whole && !sh.self) {
            bulk_g2s(oa, sa, (uint32_t)(run * sh.wa), mb);
          } else if (!sh.self) {
            for (int k = 0; k < run; ++k)
#pragma unroll
              for (int pl = 0; pl < NPL; ++pl)
                bulk_g2s(oa + (uint32_t)(k * sh.sa + pl * sh.pa), sa + k * sh.wa + pl * 2 * sh.pa, (uint32_t)sh.pa, mb);
          }
        }
        if (lane == 0) *(volatile int*)&issued_s = g + 1;
      }
    }
  } else if (warp == 1) {
    // -------------------------------------------------------------- MMAs
    if (lane == 0) {
      constexpr uint32_t FMT = KIND == TC_TF32 ? 2u : 1u;
      int g = 0;
      bool ok = true;
      for (int item_no = 0; ok; ++item_no) {
        const int qs = item_no % TS_NQ, qu = item_no / TS_NQ;
        if (!(ok = wait(&q_full[qs], (uint32_t)(qu & 1)))) break;
        const int ii = *(volatile int*)&q_item[qs];
        mbar_arrive(smem_u32(&q_empty[qs]));
        if (ii < 0) break;
        const TcItem it = items[ii];
        const TcPair pr = prs[it.pair];
        const int ra = fr[pr.a].rows, rb = fr[pr.b].rows;
        const TcShape<KIND> sh(ra, rb, pr.a == pr.b);
        const int U = sh.units;
        const int nu = (it.r1 - it.r0) * it.m;
        const uint32_t idesc = instr_desc(FMT, 128, (uint32_t)(2 * rb));
        const int b = item_no & 1, ubar = item_no >> 1;
        if (ubar > 0 && !(ok = wait(&acc_empty[b], (uint32_t)((ubar - 1) & 1)))) break;
        tc_fence_after();
        const uint32_t dst = tmem + (uint32_t)(b * TS_ACC_COLS);   // S, then H
        for (int k0 = 0; k0 < nu; k0 += U, ++g) {
          const int s = g % TS_NSTAGE, u = g / TS_NSTAGE;
          if (!(ok = wait(&full[s], (uint32_t)(u & 1)))) break;
          tc_fence_after();
          const int nk = min(U, nu - k0);
          const uint32_t zero = smem_u32(smem + TS_ZERO);
          uint32_t p = smem_u32(smem + (size_t)s * TS_STAGE);
          uint32_t a = sh.self ? p : p + (uint32_t)(U * sh.wb);
          const uint32_t la = (uint32_t)sh.lo_a, lb = (uint32_t)(sh.wb / 2);   // hi -> lo
          for (int q = 0; q < nk; q += KU) {
            // TF32: both cores of the unit; BF16: this unit's core and the next
            // unit's (zeros after the last)
            const bool two = KU == 1 || q + 1 < nk;
            auto desc = [&](uint32_t addr, uint32_t ustep) {
              return smem_desc(addr, KU == 1 ? 128u : two ? ustep : zero - addr, SBO);
            };
            const uint64_t a0 = desc(a, (uint32_t)sh.sa), p0 = desc(p, (uint32_t)sh.wb);
            const uint32_t acc = (k0 > 0 || q > 0) ? 1u : 0u;
            mma<KIND>(dst, a0, p0, idesc, acc);
            if constexpr (NPL == 2) {
              const uint64_t a1 = desc(a + la, (uint32_t)sh.sa), p1 = desc(p + lb, (uint32_t)sh.wb);
              mma<KIND>(dst, a0, p1, idesc, 1u);
              mma<KIND>(dst, a1, p0, idesc, 1u);
            }
            a += (uint32_t)(KU * sh.sa);
            p += (uint32_t)(KU * sh.wb);
          }
          mma_commit(smem_u32(&empty[s]));
          *(volatile int*)&mma_steps_s = g + 1;
        }
        if (!ok) break;
        mma_commit(smem_u32(&acc_full[b]));
      }
    }
  } else {
    // ---------------------------------------------------------- epilogue
    const int q = warp & 3;   // tensor-memory lane quadrant of this warp
    bool ok = true;
    for (int item_no = 0; ok; ++item_no) {
      const int qs = item_no % TS_NQ, qu = item_no / TS_NQ;
      ok = __all_sync(0xffffffffu, wait(&q_full[qs], (uint32_t)(qu & 1)));
      if (!ok) break;
      const int ii = *(volatile int*)&q_item[qs];
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&q_empty[qs]));
      if (ii < 0) break;
      const TcItem it = items[ii];
      const TcPair pr = prs[it.pair];
      const int na = fr[pr.a].n, nb = fr[pr.b].n, N = fr[pr.b].rows;
      const int b = item_no & 1, ubar = item_no >> 1;
      ok = __all_sync(0xffffffffu, wait(&acc_full[b], (uint32_t)(ubar & 1)));
      if (!ok) break;
      tc_fence_after();
      const int row = q * 32 + lane;
      float* out = partials + it.part_off + (long long)row * 2 * nb;
      if (q * 32 < na) {
        for (int hf = 0; hf < 2; ++hf)
          for (int c0 = 0; c0 < nb; c0 += 8) {
            float v[8];
            tmem_ld8(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * TS_ACC_COLS + hf * N + c0), v);
            if (row < na) {
              float* o = out + hf * nb + c0;
              if (c0 + 8 <= nb && (reinterpret_cast<uintptr_t>(o) & 15) == 0) {
                *reinterpret_cast<float4*>(o) = make_float4(v[0], v[1], v[2], v[3]);
                *reinterpret_cast<float4*>(o + 4) = make_float4(v[4], v[5], v[6], v[7]);
              } else {
#pragma unroll
                for (int j = 0; j < 8; ++j)
                  if (c0 + j < nb) o[j] = v[j];
              }
            }
          }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&acc_empty[b]));
    }
  }

  __syncthreads();
  if (abort_s && tid == 0) {
    // drain before the shared and tensor memory are released: the copies of
    // the last issued stages and the MMAs of the last committed stage
    auto drain = [&](unsigned long long* bar, uint32_t parity) {
      const uint32_t a = smem_u32(bar);
      for (int i = 0; i < (1 << 24) && !mbar_test(a, parity); ++i)
        if (i > 64) __nanosleep(64);
    };
    const int issued = issued_s;
    for (int g = max(0, issued - TS_NSTAGE); g < issued; ++g)
      drain(&full[g % TS_NSTAGE], (uint32_t)((g / TS_NSTAGE) & 1));
    const int ms = mma_steps_s;
    if (ms > 0) drain(&empty[(ms - 1) % TS_NSTAGE], (uint32_t)(((ms - 1) / TS_NSTAGE) & 1));
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(2 * TS_ACC_COLS)
                 : "memory");
}

// Sum of the partial tiles of each pair in plan order -> FP64 blocks
// (H_ab then S_ab, n_a x n_b row-major); diagonal blocks symmetrised.  A pair's
// partial tiles are consecutive; the FP32 terms are summed error-free (the
// rounding error of every addition carried in a second word), without FP64
// arithmetic per term.
__global__ void __launch_bounds__(256) tc_finalize_kernel(const TcFrag* __restrict__ fr,
                                                          const TcPair* __restrict__ prs,
                                                          const TcItem* __restrict__ items,
                                                          const float* __restrict__ partials,
                                                          double* __restrict__ blocks) {
  const TcPair pr = prs[blockIdx.x];
  const int na = fr[pr.a].n, nb = fr[pr.b].n, N = 2 * nb;
  double* Hblk = blocks + pr.blk_off;
  double* Sblk = Hblk + (long long)na * nb;
  const float* base = pr.nitem > 0 ? partials + items[pr.item0].part_off : partials;
  const long long step = (long long)na * N;
  auto sum = [&](int i, int c) {
    const float* p = base + (long long)i * N + c;
    float s = 0.f, e = 0.f;
#pragma unroll 4
    for (int k = 0; k < pr.nitem; ++k) {
      const float x = p[k * step];
      const float t = s + x, bp = t - s;
      e += (s - (t - bp)) + (x - bp);
      s = t;
    }
    return (double)s + (double)e;
  };
  // blockIdx.y: a chunk of outputs
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < na * nb; e += gridDim.y * blockDim.x) {
    const int i = e / nb, m = e % nb;
    double s = sum(i, m), h = sum(i, nb + m);
    if (pr.a == pr.b) {
      s = 0.5 * (s + sum(m, i));
      h = 0.5 * (h + sum(m, nb + i));
    }
    Sblk[e] = s;
    Hblk[e] = h;
  }
}

// First unit and number of units (cyclic, NU units of 8 points) that the points
// [s, s + len) of a periodic axis of n points touch.
void unit_range(int n, int NU, int s, int len, int& us, int& cnt) {
  us = s / 8;
  if (len >= n) {
    cnt = NU;
    return;
  }
  const int e = s + len - 1;   // < 2 n
  cnt = e < n ? e / 8 - us + 1 : NU - us + (e - n) / 8 + 1;
  cnt = std::min(cnt, NU);
}

// Touched units of the boxes along axis d: of the storage box from us (nux of
// them), of the fragment's own points from us + iu (ic).
struct UnitAxis {
  std::vector<int> us, nux, iu, ic;
  UnitAxis(const std::vector<DevFrag>& fr, int n, int d) {
    const int NU = (n + 7) / 8;
    us.resize(fr.size());
    nux = iu = ic = us;
    for (size_t f = 0; f < fr.size(); ++f) {
      const DevFrag& F = fr[f];
      unit_range(n, NU, F.doff[d], F.dext[d], us[f], nux[f]);
      iu[f] = 0;
      ic[f] = NU;
      if (nux[f] == NU) continue;   // the whole axis: units outside the box hold zeros
      int s = 0;
      unit_range(n, NU, (F.doff[d] + F.lo[d]) % n, F.ext[d], s, ic[f]);
      iu[f] = (s - us[f] + NU) % NU;
    }
  }
};

}  // namespace

struct TcPlan {
  std::vector<TcFrag> frags;
  std::vector<RUnit> units;
  std::vector<int4> pack_cta;
  std::vector<TcPair> pairs;
  std::vector<TcItem> items;
  std::vector<int> order;       // items, the largest first
  long long part_elems = 0, plane_bytes = 0;
  int axis = 0;                 // of the units
  DevBuf d_frags, d_units, d_pcta, d_pairs, d_items, d_order, partials;
  bool ok = false, uploaded = false;
  std::string why;
};

void ofm_tc_guards(const TcPlan* t, std::vector<GuardRef>& out) {
  if (!t) return;
  const struct { const DevBuf* b; const char* n; } bufs[] = {
      {&t->d_frags, "tensor-core fragments"}, {&t->d_units, "tensor-core pack units"},
      {&t->d_pcta, "tensor-core pack table"}, {&t->d_pairs, "tensor-core pairs"},
      {&t->d_items, "tensor-core items"}, {&t->d_order, "tensor-core item order"},
      {&t->partials, "tensor-core partials"}};
  for (const auto& x : bufs)
    if (x.b->p) out.push_back({x.b->p, x.b->cap, x.n});
}

void ofm_tc_plan_free(TcPlan* t) {
  if (!t) return;
  DevBuf* bufs[] = {&t->d_frags, &t->d_units, &t->d_pcta, &t->d_pairs, &t->d_items, &t->d_order, &t->partials};
  for (DevBuf* b : bufs)
    if (b->p) cudaFree(b->p);
  delete t;
}

void ofm_tc_free(ofm_ctx* c) {
  ofm_tc_plan_free(c->tc);
  c->tc = nullptr;
}

// Host plan of the pair contraction after a build: one item per row chunk of a
// piece, chunks of about asm_chunk points (0: sized for about four items per
// SM).  Not usable (with the reason) for FP64 storage or more than 128 states.
ofm_status ofm_plan_extra(ofm_ctx* c) {
  if (!c->tc) c->tc = new TcPlan();
  TcPlan* t = c->tc;
  t->frags.clear(); t->units.clear(); t->pack_cta.clear(); t->pairs.clear(); t->items.clear(); t->order.clear();
  t->part_elems = t->plane_bytes = 0;
  t->ok = t->uploaded = false;
  if (c->storage != OFM_STORE_FP32) {
    t->why = "tensor-core contraction needs FP32 storage";
    return OFM_OK;
  }
  for (const DevFrag& F : c->frags)
    if (F.n > 128) {
      t->why = "tensor-core contraction supports at most 128 states per fragment";
      return OFM_OK;
    }
  // The axis of the units: the one along which the pairs' operand units and the
  // planes come to the fewest bytes (x among equals).  A box of 18 points at an odd
  // offset touches four units, 32 points; along an axis that it spans whole, or
  // shares whole with its neighbours, hardly any point is padding.  Chains along
  // x in BF16 hi+lo, units always along x and along the axis taken: 31 boxes of 16 x
  // 32 x 32, 32 states, 314 and 201 us; 64 of 16 x 20 x 32, 16 states, 328 and 216 us;
  // 4 of 16 x 12 x 12, 6 states, 67 and 58 us.
  const int* gn = c->grid.n;
  const UnitAxis uax[3] = {UnitAxis(c->frags, gn[0], 0), UnitAxis(c->frags, gn[1], 1), UnitAxis(c->frags, gn[2], 2)};
  double cost_of[3] = {0, 0, 0};
  auto rows_of = [&](int f) { return (c->frags[f].n + 7) / 8 * 8; };
  for (size_t f = 0; f < c->frags.size(); ++f)
    for (int d = 0; d < 3; ++d)
      cost_of[d] += 2.0 * rows_of((int)f) * uax[d].nux[f] * c->frags[f].dext[(d + 1) % 3] * c->frags[f].dext[(d + 2) % 3];
  for (const HostPair& hp : c->pairs) {
    const DevFrag &A = c->frags[hp.a], &B = c->frags[hp.b];
    double pts[3], un[3];
    for (int d = 0; d < 3; ++d) {
      const UnitAxis& U = uax[d];
      pts[d] = (double)dim_count(gn[d], A.doff[d] + A.lo[d], A.ext[d], B.doff[d], B.dext[d]);
      un[d] = (double)dim_count((gn[d] + 7) / 8, U.us[hp.a] + U.iu[hp.a], U.ic[hp.a], U.us[hp.b], U.nux[hp.b]);
    }
    for (int d = 0; d < 3; ++d)
      cost_of[d] += (rows_of(hp.a) + 2.0 * rows_of(hp.b)) * un[d] * pts[(d + 1) % 3] * pts[(d + 2) % 3];
  }
  const int ux = cost_of[1] < cost_of[0] ? (cost_of[2] < cost_of[1] ? 2 : 1) : (cost_of[2] < cost_of[0] ? 2 : 0);
  const int ax[3] = {ux, ux == 0 ? 1 : 0, ux == 2 ? 1 : 2};   // the K order's axes, fastest first
  t->axis = ux;
  const std::vector<int>&us = uax[ux].us, &iu = uax[ux].iu, &ic = uax[ux].ic;
  const int n0 = gn[ux], NU = (n0 + 7) / 8;
  long long tiles = 0;
  for (size_t f = 0; f < c->frags.size(); ++f) {
    const DevFrag& F = c->frags[f];
    TcFrag q;
    q.nux = uax[ux].nux[f];
    q.dext1 = F.dext[ax[1]];
    q.n = F.n;
    q.rows = rows_of((int)f);
    RUnit u;
    u.frag = (int)f;
    for (int d = 0; d < 3; ++d) u.s0[d] = d == ux ? 8 * us[f] : F.doff[d];
    u.L[0] = 8 * q.nux; u.L[1] = F.dext[ax[1]]; u.L[2] = F.dext[ax[2]];
    u.p8 = u.L[0] * u.L[1];
    u.ntiles = (int)(((long long)u.p8 * u.L[2] + 63) / 64);
    u.tile0 = tiles;
    u.base = t->plane_bytes;
    q.base = u.base;
    tiles += u.ntiles;
    t->plane_bytes += (long long)u.ntiles * 64 * q.rows * 8;
    t->frags.push_back(q);
    t->units.push_back(u);
    for (int t0 = 0; t0 < u.ntiles; t0 += 4)
      t->pack_cta.push_back(make_int4((int)f, t0, std::min(4, u.ntiles - t0), 0));
  }
  const long long target = c->asm_chunk > 0 ? c->asm_chunk : std::max<long long>(1024, c->kh / (4 * 152));
  for (size_t p = 0; p < c->pairs.size(); ++p) {
    const HostPair& hp = c->pairs[p];
    const DevFrag &A = c->frags[hp.a], &B = c->frags[hp.b];
    const TcFrag& TB = t->frags[hp.b];
    TcPair tq;
    tq.a = hp.a;
    tq.b = hp.b;
    tq.blk_off = c->simt_pairs[p].blk_off;
    tq.item0 = (int)t->items.size();
    // the unit axis in units, the others in points
    std::vector<Run> runs[3];
    runs[0] = dim_runs(NU, (us[hp.a] + iu[hp.a]) % NU, ic[hp.a], us[hp.b], TB.nux);
    for (int k = 1; k < 3; ++k) {
      const int d = ax[k];
      runs[k] = dim_runs(gn[d], (A.doff[d] + A.lo[d]) % gn[d], A.ext[d], B.doff[d], B.dext[d]);
    }
    // shared points per row, and units they take
    const long long xpts = dim_count(n0, A.doff[ux] + A.lo[ux], A.ext[ux], B.doff[ux], B.dext[ux]);
    long long xunits = 0;
    for (const Run& r : runs[0]) xunits += r.len;
    for (const Run& rz : runs[2])
      for (const Run& ry : runs[1])
        for (const Run& rx : runs[0]) {
          const int rows = ry.len * rz.len;
          // The FP32 accumulation in tensor memory drops bits at every step, so an
          // item has as many units as its shared points fill (above a minimum): units
          // padded with zeros must not lengthen the sum.
          const long long pts = rx.len * xpts * rows / xunits;
          const long long units = std::max(std::min<long long>(TS_MINUNITS, target / 8), std::min(target, pts) / 8);
          const int per = (int)std::max<long long>(1, units / rx.len);
          for (int r0 = 0; r0 < rows; r0 += per) {
            TcItem it;
            it.pair = (int)p;
            it.la[0] = iu[hp.a] + rx.ta; it.la[1] = A.lo[ax[1]] + ry.ta; it.la[2] = A.lo[ax[2]] + rz.ta;
            it.lb[0] = rx.lb; it.lb[1] = ry.lb; it.lb[2] = rz.lb;
            it.m = rx.len;
            it.leny = ry.len;
            it.r0 = r0;
            it.r1 = std::min(rows, r0 + per);
            it.part_off = t->part_elems;
            t->part_elems += (long long)A.n * 2 * B.n;
            t->items.push_back(it);
          }
        }
    tq.nitem = (int)t->items.size() - tq.item0;
    t->pairs.push_back(tq);
  }
  t->order.resize(t->items.size());
  for (size_t i = 0; i < t->order.size(); ++i) t->order[i] = (int)i;
  auto cost = [&](int i) {
    const TcItem& it = t->items[i];
    const TcPair& q = t->pairs[it.pair];
    return (long long)(it.r1 - it.r0) * it.m * (t->frags[q.a].rows + 2 * t->frags[q.b].rows);
  };
  std::stable_sort(t->order.begin(), t->order.end(), [&](int x, int y) { return cost(x) > cost(y); });
  t->ok = true;
  return OFM_OK;
}

template <typename T>
static ofm_status put(ofm_ctx* c, DevBuf& b, const std::vector<T>& v, const char* what) {
  OFM_TRY(ofm_ensure(c, b, sizeof(T) * std::max<size_t>(1, v.size()), what));
  if (!v.empty()) OFM_CUDA(c, cudaMemcpyAsync(b.p, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice, c->stream));
  return OFM_OK;
}

// Bytes of the operand planes: 8 per value of the widened boxes (TF32, BF16
// hi+lo), 4 in BF16.
static long long arena_bytes(const TcPlan* t, ofm_precision prec) {
  return std::max<long long>(16, prec == OFM_PREC_BF16 ? t->plane_bytes / 2 : t->plane_bytes);
}

// Device tables (after a re-plan) and buffers, made before any capture.
ofm_status ofm_tc_prepare(ofm_ctx* c, ofm_precision prec) {
  TcPlan* t = c->tc;
  if (!t || !t->ok) return ofm_fail(c, OFM_ERR_INVALID, t ? t->why : "no tensor-core plan");
  void* arena = nullptr;
  OFM_TRY(ofm_pair_planes(c, arena_bytes(t, prec), &arena));
  OFM_TRY(ofm_ensure_big(c, t->partials, sizeof(float) * (size_t)std::max<long long>(1, t->part_elems), "tc partials"));
  if (t->uploaded) return OFM_OK;
  OFM_TRY(put(c, t->d_frags, t->frags, "tc fragments"));
  OFM_TRY(put(c, t->d_units, t->units, "tc pack units"));
  OFM_TRY(put(c, t->d_pcta, t->pack_cta, "tc pack table"));
  OFM_TRY(put(c, t->d_pairs, t->pairs, "tc pairs"));
  OFM_TRY(put(c, t->d_items, t->items, "tc items"));
  OFM_TRY(put(c, t->d_order, t->order, "tc item order"));
  static bool attr = false;   // the kernels' shared-memory limit, once per process
  if (!attr) {
    cudaFuncSetAttribute(tc_contract_kernel<TC_TF32>, cudaFuncAttributeMaxDynamicSharedMemorySize, TS_SMEM);
    cudaFuncSetAttribute(tc_contract_kernel<TC_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, TS_SMEM);
    cudaFuncSetAttribute(tc_contract_kernel<TC_BF16X3>, cudaFuncAttributeMaxDynamicSharedMemorySize, TS_SMEM);
    OFM_CUDA(c, cudaGetLastError());
    attr = true;
  }
  t->uploaded = true;
  return OFM_OK;
}

// a1 (H phi and the operand planes), a3/a4 (contraction into FP32 partials) and
// a5 (the fixed-order sum into the FP64 block arena) on the context stream.
ofm_status ofm_contract_tc(ofm_ctx* c, ofm_precision prec) {
  TcPlan* t = c->tc;
  if (!t || !t->ok) return ofm_fail(c, OFM_ERR_INVALID, t ? t->why : "no tensor-core plan");
  if (!t->uploaded) return ofm_fail(c, OFM_ERR_STATE, "tensor-core plan not prepared");
  const int kind = prec == OFM_PREC_TF32 ? TC_TF32 : prec == OFM_PREC_BF16 ? TC_BF16 : TC_BF16X3;
  void* arena = nullptr;
  OFM_TRY(ofm_pair_planes(c, arena_bytes(t, prec), &arena));
  OFM_TRY(ofm_pair_pack(c, kind, t->axis, (const RUnit*)t->d_units.p, (const int4*)t->d_pcta.p, (int)t->pack_cta.size(), arena,
                        arena_bytes(t, prec)));
  int* fl = (int*)c->flag.p + OFM_FLAG_TC;
  int* next = (int*)c->flag.p + OFM_FLAG_QUEUE;
  OFM_CUDA(c, cudaMemsetAsync(next, 0, sizeof(int), c->stream));
  const TcFrag* fr = (const TcFrag*)t->d_frags.p;
  const TcPair* pr = (const TcPair*)t->d_pairs.p;
  const TcItem* it = (const TcItem*)t->d_items.p;
  {
    KTimer kt(c, KC_CONTRACT, 1, c->contract_bytes, (double)c->flops);
    const int ni = (int)t->items.size(), grid = std::min(ni, 152);   // one persistent CTA per SM
    const int* od = (const int*)t->d_order.p;
    const unsigned char* pl = (const unsigned char*)arena;
    float* pa = (float*)t->partials.p;
    if (ni > 0) {
      if (kind == TC_TF32) tc_contract_kernel<TC_TF32><<<grid, TS_THREADS, TS_SMEM, c->stream>>>(fr, pr, it, od, ni, pl, pa, fl, next);
      else if (kind == TC_BF16) tc_contract_kernel<TC_BF16><<<grid, TS_THREADS, TS_SMEM, c->stream>>>(fr, pr, it, od, ni, pl, pa, fl, next);
      else tc_contract_kernel<TC_BF16X3><<<grid, TS_THREADS, TS_SMEM, c->stream>>>(fr, pr, it, od, ni, pl, pa, fl, next);
    }
    OFM_CUDA(c, cudaGetLastError());
  }
  {
    KTimer kt(c, KC_FINALIZE, 1, (double)t->part_elems * 4);
    int amax = 1, bmax = 1;
    for (const TcPair& q : t->pairs) {
      amax = std::max(amax, t->frags[q.a].n);
      bmax = std::max(bmax, t->frags[q.b].n);
    }
    if (!t->pairs.empty())
      tc_finalize_kernel<<<dim3((int)t->pairs.size(), (amax * bmax + 255) / 256), 256, 0, c->stream>>>(
          fr, pr, it, (const float*)t->partials.p, (double*)c->blocks.p);
    OFM_CUDA(c, cudaGetLastError());
  }
  c->tc_check = true;
  return OFM_OK;
}

// Reports a bounded-wait timeout of an earlier tensor-core or staged-stencil
// launch (each sets its flag word; the flags are read once and cleared).
ofm_status ofm_wait_status(ofm_ctx* c) {
  if (c->fault_due) {
    c->fault_due = false;
    c->tc_check = c->stencil_check = false;
    return ofm_fail(c, OFM_ERR_TIMEOUT, "a bounded device wait exceeded its bound (injected by OFM_FAULT=timeout)");
  }
  if (c->tc_check) {
    int h = 0;
    int* f = (int*)c->flag.p + OFM_FLAG_TC;
    OFM_CUDA(c, cudaMemcpyAsync(&h, f, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    OFM_CUDA(c, cudaStreamSynchronize(c->stream));
    c->tc_check = false;
    if (h) {
      cudaMemsetAsync(f, 0, sizeof(int), c->stream);
      return ofm_fail(c, OFM_ERR_TIMEOUT, "tensor-core contraction: an mbarrier wait exceeded its bound");
    }
  }
  if (c->stencil_check) {
    int h = 0;
    int* f = (int*)c->flag.p + OFM_FLAG_STENCIL;
    OFM_CUDA(c, cudaMemcpyAsync(&h, f, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    OFM_CUDA(c, cudaStreamSynchronize(c->stream));
    c->stencil_check = false;
    if (h) {
      cudaMemsetAsync(f, 0, sizeof(int), c->stream);
      return ofm_fail(c, OFM_ERR_TIMEOUT, "stencil: a staged-plane wait exceeded its bound");
    }
  }
  return OFM_OK;
}

