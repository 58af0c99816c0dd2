// Split-precision dense GEMM core on the 5th-generation tensor cores (tcgen05, sm_103a), shared by
// the forward Chebyshev chain (dense_split.cu) and the adjoint (adjoint_split.cu).
//
// One product on a block of state rows: Y^T = Psi^T Omega~^T with Omega~ = S + i A (S real
// symmetric, A real antisymmetric), i.e. with X.B := sum_k X[j][k] B[i][k]
//   Yr = Psi_r.S - Psi_i.A,   Yi = Psi_r.A + Psi_i.S       (HAS_A; A = 0 drops two streams).
// Each K stage loads the Psi_r, Psi_i tiles and one S (and one A) tile, and every tile is used twice
// (split_issue_stage).  Every operand
// is held as NS BF16 slices (x = x_0 + x_1 + ..., x_s = bf16 of the remainder), and the products
// x_a y_b with a + b < NS (3 for NS = 2, 6 for NS = 3) are summed in FP32 in tensor memory.
// The epilogue (epi_block) is one of: the Chebyshev term (recurrence psi_{l+1} = -2i Y +
// psi_{l-1}, Bessel accumulation and step phase on FP32 masters, Eqs. 10 and 12), the adjoint
// term, or the gradient dot; the first two also write the next product's slices.
//
// k_split_persist: one CTA per SM walks its tiles with a dedicated TMA warp, MMA warp and eight epilogue warps, and two
// tensor-memory buffers so that a tile's epilogue overlaps the next tile's MMAs.  Tiles are
// rasterized in groups of 8 row blocks so that co-running CTAs share operands in L2.  TMA loads
// are K-major with 128- or 64-byte swizzle; stages and buffers are handed over by mbarriers.
// Every wait is bounded; a wait that gives up records FQ_BIT_TIMEOUT, drains this CTA's own
// copies and MMAs, frees tensor memory and returns.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>

#include <algorithm>
#include <mutex>

#include "internal.h"

namespace {


constexpr int BM = 128;      // state rows per tile (tcgen05 M)
constexpr int RASTER_GROUP = 8;
// Epilogue warps of the persistent kernels: two per tensor-memory lane quarter, each taking half of
// the tile's columns, with a transposing stage (epi_transpose) of its own.
constexpr int EPI_WARPS = 8;
constexpr int EPI_STAGE_BYTES = 4096;
constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz

// ------------------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait: false if the phase did not complete within kWaitCycles.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try(bar, parity)) {
    if (clock64() - t0 > kWaitCycles) return false;
  }
  return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(
          dst),
      "l"((uint64_t)map), "r"(bar), "r"(x), "r"(y)
      : "memory");
}

// Shared-memory matrix descriptor: K-major rows of ROWB bytes (128 or 64) with the matching
// swizzle, 8-row atoms of 8 * ROWB bytes.
template <int ROWB>
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);           // start address
  d |= (uint64_t)1 << 16;                             // leading-dimension offset (unused, swizzled K-major)
  d |= (uint64_t)((8 * ROWB) >> 4) << 32;             // stride between 8-row atoms
  d |= (uint64_t)1 << 46;                             // descriptor version for tcgen05
  d |= (uint64_t)(ROWB == 128 ? 2 : 4) << 61;         // 128-byte or 64-byte swizzle
  return d;
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = __uint_as_float(r[q]);
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = __uint_as_float(r[q]);
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* v) {
  uint32_t r[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) r[q] = __float_as_uint(v[q]);
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ------------------------------------------------------------------------- slices
template <int NS>
__device__ __forceinline__ void split_f32(float x, __nv_bfloat16 (&s)[NS]) {
  float r = x;
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    s[q] = __float2bfloat16_rn(r);
    r -= __bfloat162float(s[q]);
  }
}

// NS slices of two values, packed (a's in the low half): the slices of split_f32, two to a conversion
// (a conversion takes as long as eight FP32 instructions; with one per slice they were a third of the
// epilogue's arithmetic).  With this and SplitTerm a BF16X3 / X6 product of 64-wide tiles went from
// 13.9 / 17.7 to 13.5 / 16.7 us at N = 200 and from 27.2 / 43.6 to 26.1 / 42.4 us at N = 1000, a gradient
// step at N = 1024 from 589 to 576 us (X3).
template <int NS>
__device__ __forceinline__ void split_pair(float a, float b, uint32_t (&s)[NS]) {
#pragma unroll
  for (int t = 0; t < NS; ++t) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    s[t] = (uint32_t)__bfloat16_as_ushort(h.x) | ((uint32_t)__bfloat16_as_ushort(h.y) << 16);
    a -= __uint_as_float(s[t] << 16);
    b -= __uint_as_float(s[t] & 0xffff0000u);
  }
}

template <int NS>
__device__ __forceinline__ void split_f64(double x, __nv_bfloat16 (&s)[NS]) {
  double r = x;
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    s[q] = __double2bfloat16(r);
    r -= (double)__bfloat162float(s[q]);
  }
}

// Entry (i, c) of Omega~_m = S + i A with S = sa H0 + sb H1 - sbeta 1 and A = sc [H0, H1]
// (Eqs. 11 and 14), formed in FP32 from the FP64 operators: the split paths keep at most 24 bits
// of an entry (three BF16 slices), and FP64 arithmetic runs at a small fraction of the FP32 rate
// on this GPU.  The multiply-adds are spelt out so that every kernel forming it rounds alike.
__device__ __forceinline__ void omega_entry(double h0, double h1, double k, bool diag, float sa, float sb,
                                            float sc, float sbeta, float& S, float& A) {
  S = fmaf(sa, (float)h0, fmaf(sb, (float)h1, diag ? -sbeta : 0.f));
  A = sc * (float)k;
}

// Left operand and FP32 masters of the initial block: identity rows (build_UT) or given states.
template <int NS>
__global__ void k_split_init(const double2* __restrict__ x0, int n, int nc, int ldm, int np, int kp, float* mre,
                             float* mim, __nv_bfloat16* sl, size_t slice_stride) {
  const size_t total = (size_t)nc * kp;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total; q += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(q / kp), c = (int)(q % kp);
    const bool im_half = c >= np;
    const int i = im_half ? c - np : c;
    float v = 0.f;
    if (i < n) {
      double2 z = x0 ? x0[(size_t)j * n + i] : make_double2(i == j ? 1.0 : 0.0, 0.0);
      v = (float)(im_half ? z.y : z.x);
      if (im_half) mim[(size_t)j * ldm + i] = v;
      else mre[(size_t)j * ldm + i] = v;
    }
    __nv_bfloat16 s[NS];
    split_f32<NS>(v, s);
#pragma unroll
    for (int t = 0; t < NS; ++t) sl[t * slice_stride + q] = s[t];
  }
}

// Products kept for NS slices: (a, b) with a + b < NS, ordered smallest first.
template <int NS> struct Pairs;
template <> struct Pairs<2> {
  static constexpr int N = 3;
  static __device__ __forceinline__ int a(int p) { return p == 0 ? 1 : 0; }  // (1,0), (0,1), (0,0)
  static __device__ __forceinline__ int b(int p) { return p == 1 ? 1 : 0; }
};
template <> struct Pairs<3> {
  static constexpr int N = 6;
  static __device__ __forceinline__ int a(int p) { const int t[6] = {1, 0, 2, 1, 0, 0}; return t[p]; }
  static __device__ __forceinline__ int b(int p) { const int t[6] = {1, 2, 0, 0, 1, 0}; return t[p]; }
};

// Workspace of the split chain (dense_split.cu's fq_split_workspace): the right operand's slices
// (S, A), two left-operand slice buffers (ping-pong across terms), three FP32 master state buffers
// (planar) for psi_l / psi_{l-1} / acc, and the chain counters.
struct SplitWs {
  __nv_bfloat16* os;  // S slices
  __nv_bfloat16* oa;  // A slices
  __nv_bfloat16* a[2];
  float* m[3][2];
  unsigned int* flags;  // chain counters: [CHAIN_MAXP][row blocks]
  int np, kp, ldm, ncp;
  size_t bstride, astride;
};

struct SplitMaps {
  CUtensorMap a[3];   // left operand slices [ncp][2 Np]: Psi_r in columns [0, Np), Psi_i in [Np, 2 Np)
  CUtensorMap os[3];  // S slices [Np][Np]
  CUtensorMap oa[3];  // A slices [Np][Np]
};

// Epilogue of one split GEMM (Y = left . right^T on a 128 x BN tile, FP32 in tensor memory).
enum SplitMode {
  EPI_FWD = 0,  // Chebyshev term: psi_{l+1} = -2i Y + psi_{l-1}, acc += a psi_{l+1}, phase at the last term
  EPI_ADJ = 1,  // adjoint term: out = cpa g + i cw Y + b2
  EPI_DOT = 2,  // gradient dot: partial[tile][epilogue warp] = sum of conj(b) Y over the warp's part of the tile
};

// A Chebyshev term's scalars in FP32 (converted once: FP64 conversions run at the FP64 rate, five of them
// took 600 cycles of every 32 x 32 block).
struct SplitTerm {
  int first, last;
  float coef0, coef, ph_re, ph_im, bound2;
  unsigned int* status;
};

SplitTerm split_term(const fq_term& t) {
  return SplitTerm{t.first,          t.last,           (float)t.coef0,   (float)t.coef,
                   (float)t.ph_re,   (float)t.ph_im,   (float)t.bound2,  t.status};
}

struct SplitEpi {
  int n, nc, ldm, np;          // dims; ldm: FP32 master row stride; np: real part width in K'
  const float* cur_re;         // FWD: psi_l masters (first term: psi_0); ADJ: g; DOT: b
  const float* cur_im;
  const float* prev_re;        // FWD: psi_{l-1}; ADJ: b2 (NULL: absent)
  const float* prev_im;
  float* acc_re;
  float* acc_im;
  float* out_re;               // FWD: psi_{l+1} (in place of psi_{l-1}) or X at the last term; ADJ: out
  float* out_im;
  __nv_bfloat16* slice_out;    // next left operand: NS slices, each [nc][Kp]
  size_t slice_stride;         // elements between slices
  int kp;
  float cpa_re, cpa_im, cw;    // ADJ coefficients
  double2* partial;            // DOT output, EPI_WARPS a tile
  SplitTerm t;
};

template <int NS, int BN, int BKE, bool HAS_A>
struct SplitCfg {
  static constexpr int ROWB = BKE * 2;                // bytes per K row of a stage (swizzle span)
  static constexpr int A_BYTES = BM * ROWB;           // one slice of Psi_r or Psi_i, one stage
  static constexpr int B_BYTES = BN * ROWB;           // one slice of S or A, one stage
  static constexpr int STAGE_BYTES = 2 * NS * A_BYTES + (HAS_A ? 2 : 1) * NS * B_BYTES;
  static constexpr int STAGES = (198000 / STAGE_BYTES) > 4 ? 4 : (198000 / STAGE_BYTES);
  // 64-wide complex tiles multiply each left tile by the stacked [S; A] rows in one N = 128 MMA
  // (split_issue_stage); other tiles take S and A in MMAs of their own
  static constexpr bool STACKED = HAS_A && BN == 64;
  // 64-wide real tiles multiply a left slice by the stacked rows of the two leading right slices
  static constexpr bool SLICED = !HAS_A && BN == 64;
  static constexpr int ACC_COLS = STACKED || SLICED ? 4 * BN : 2 * BN;  // tensor-memory columns of one tile's sums
  // stages, their alignment, barriers, then the epilogue warps' transposing stages
  static constexpr size_t TAIL = 256;
  static constexpr size_t SMEM = (size_t)STAGES * STAGE_BYTES + 1024 + TAIL + EPI_WARPS * EPI_STAGE_BYTES;
  static_assert(SMEM <= 232448, "shared memory of one CTA");
  // one stage in shared memory: Psi_r slices, Psi_i slices, then S_q (and A_q) of slice q side by side
  static __device__ __forceinline__ uint32_t right(uint32_t st, int q, int part) {
    return st + 2 * NS * A_BYTES + ((HAS_A ? 2 : 1) * q + part) * B_BYTES;
  }
};

// TMA loads of one stage (columns kx .. kx + BKE of the left rows j0 .. and the right rows i0 ..).
template <int NS, int BN, int BKE, bool HAS_A>
__device__ __forceinline__ void split_load_stage(uint32_t st, uint32_t bar, const CUtensorMap* left,
                                                 const CUtensorMap* os, const CUtensorMap* oa, int kx, int np, int j0,
                                                 int i0) {
  using Cfg = SplitCfg<NS, BN, BKE, HAS_A>;
#pragma unroll
  for (int q = 0; q < NS; ++q) {
    tma_load_2d(st + q * Cfg::A_BYTES, left + q, bar, kx, j0);              // Psi_r
    tma_load_2d(st + (NS + q) * Cfg::A_BYTES, left + q, bar, np + kx, j0);  // Psi_i
    tma_load_2d(Cfg::right(st, q, 0), os + q, bar, kx, i0);                 // S
    if (HAS_A) tma_load_2d(Cfg::right(st, q, 1), oa + q, bar, kx, i0);      // A
  }
}

// The MMAs of one stage into the accumulators at acc (fresh: the tile's first stage overwrites them).
//  STACKED: Psi_r.[S; A] -> columns [0, 2 BN) and Psi_i.[S; A] -> columns [2 BN, 4 BN), two MMAs of
//    N = 128 per slice pair and 16 values of k: an MMA's operands then cost 8 KB of shared-memory
//    reads per 64 tensor cycles.  Four MMAs of N = 64 read 6 KB per 32 cycles, more than the 128
//    bytes a cycle of shared memory: 43 -> 35 us a product at N = 1000 (BF16X3, K stages of 64).
//    split_load_y forms Yr and Yi from the four sums.
//  other complex tiles: Yr += Psi_r.S - Psi_i.A, Yi += Psi_r.A + Psi_i.S (negate-A bit);
//  SLICED (real): a left slice that goes with both S_0 and S_1 takes them stacked, in one MMA of N = 128 onto
//    2 BN columns (Psi_0, and Psi_1 in BF16X6); Psi_{NS-1}.S_0 and, in BF16X6, Psi_0.S_2 go onto one half, for
//    Psi_r and, 2 BN columns on, for Psi_i; split_load_y adds the halves.  An MMA of N = 64 takes about 60
//    cycles for its 6 KB of operands, one of N = 128 about 80: a gradient step at N = 1024 552 -> 496 us
//    (BF16X3) and 890 -> 770 us (BF16X6).
//  other real right operands: Yr += Psi_r.S, Yi += Psi_i.S.
template <int NS, int BN, int BKE, bool HAS_A>
__device__ __forceinline__ void split_issue_stage(uint32_t acc, uint32_t st, bool fresh) {
  using Cfg = SplitCfg<NS, BN, BKE, HAS_A>;
  constexpr int MN = Cfg::STACKED ? 2 * BN : BN;
  constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(MN >> 3) << 17) |
                             ((uint32_t)(BM >> 4) << 24);
  constexpr uint32_t idesc_neg = idesc | (1u << 13);  // negate the left operand
  if constexpr (Cfg::SLICED) {
    constexpr uint32_t idesc2 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * BN) >> 3) << 17) |
                                ((uint32_t)(BM >> 4) << 24);
#pragma unroll
    for (int kk = 0; kk < BKE / 16; ++kk) {
      const uint64_t ds = smem_desc<Cfg::ROWB>(Cfg::right(st, 0, 0) + 32 * kk);
      const uint32_t first = (fresh && kk == 0) ? 0u : 1u;
#pragma unroll
      for (int a = 0; a < NS; ++a)
#pragma unroll
        for (int part = 0; part < 2; ++part)
          mma_bf16(acc + part * 2 * BN, smem_desc<Cfg::ROWB>(st + (part * NS + a) * Cfg::A_BYTES + 32 * kk), ds,
                   a < NS - 1 ? idesc2 : idesc, a == 0 ? first : 1u);
      if (NS == 3) {
#pragma unroll
        for (int part = 0; part < 2; ++part)
          mma_bf16(acc + part * 2 * BN + BN, smem_desc<Cfg::ROWB>(st + part * NS * Cfg::A_BYTES + 32 * kk),
                   smem_desc<Cfg::ROWB>(Cfg::right(st, NS - 1, 0) + 32 * kk), idesc, 1u);
      }
    }
    return;
  }
#pragma unroll
  for (int p = 0; p < Pairs<NS>::N; ++p) {
    const uint32_t pr = st + Pairs<NS>::a(p) * Cfg::A_BYTES;
    const uint32_t pi = st + (NS + Pairs<NS>::a(p)) * Cfg::A_BYTES;
    const uint32_t os = Cfg::right(st, Pairs<NS>::b(p), 0), oa = Cfg::right(st, Pairs<NS>::b(p), 1);
#pragma unroll
    for (int kk = 0; kk < BKE / 16; ++kk) {
      const uint32_t first = (fresh && p == 0 && kk == 0) ? 0u : 1u;
      const uint64_t dpr = smem_desc<Cfg::ROWB>(pr + 32 * kk), dpi = smem_desc<Cfg::ROWB>(pi + 32 * kk);
      const uint64_t dos = smem_desc<Cfg::ROWB>(os + 32 * kk);
      if constexpr (Cfg::STACKED) {
        mma_bf16(acc, dpr, dos, idesc, first);
        mma_bf16(acc + 2 * BN, dpi, dos, idesc, first);
      } else if constexpr (HAS_A) {
        const uint64_t doa = smem_desc<Cfg::ROWB>(oa + 32 * kk);
        mma_bf16(acc, dpr, dos, idesc, first);
        mma_bf16(acc, dpi, doa, idesc_neg, 1u);
        mma_bf16(acc + BN, dpr, doa, idesc, first);
        mma_bf16(acc + BN, dpi, dos, idesc, 1u);
      } else {
        mma_bf16(acc, dpr, dos, idesc, first);
        mma_bf16(acc + BN, dpi, dos, idesc, first);
      }
    }
  }
}

__device__ __forceinline__ void store_f4(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void load_f4(const float* p, float* v) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}

__device__ __forceinline__ void store4(float* p, size_t idx, int cnt, const float (&v)[4]) {
  if (cnt >= 4) {
    store_f4(p + idx, v);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (q < cnt) p[idx + q] = v[q];
  }
}

// NS BF16 slices of 4 new complex entries into the next left operand (row j, columns ib..ib+cnt):
// the real parts at column ib, the imaginary parts at column np + ib of each slice.
template <int NS>
__device__ __forceinline__ void store_slices(const SplitEpi& e, int j, int ib, int cnt, const float (&o_r)[4],
                                             const float (&o_i)[4]) {
  const size_t srow = (size_t)j * e.kp + ib;
#pragma unroll
  for (int part = 0; part < 2; ++part) {
    uint32_t lo[NS], hi[NS];  // two bf16 per word
    split_pair<NS>(part ? o_i[0] : o_r[0], part ? o_i[1] : o_r[1], lo);
    split_pair<NS>(part ? o_i[2] : o_r[2], part ? o_i[3] : o_r[3], hi);
#pragma unroll
    for (int t = 0; t < NS; ++t) {
      __nv_bfloat16* d = e.slice_out + t * e.slice_stride + srow + (part ? e.np : 0);
      if (cnt >= 4) {
        *reinterpret_cast<uint2*>(d) = make_uint2(lo[t], hi[t]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (q < cnt) d[q] = __ushort_as_bfloat16((unsigned short)((q < 2 ? lo[t] : hi[t]) >> (16 * (q & 1))));
      }
    }
  }
}

// Epilogue stage of a warp: 32 rows x 32 columns of FP32 (4 KB), 16-byte units XOR-swizzled by row.
static_assert(EPI_STAGE_BYTES == 32 * 32 * sizeof(float), "one 32 x 32 block a warp");

// Turns a warp's 32 x 32 block from the tensor-memory layout (lane = row, v = its 32 columns) into
// rows spread over lanes: out[4 p .. 4 p + 3] = columns 4 (lane % 8) .. of row 4 p + lane / 8, so that
// the warp's global accesses cover four rows of 128 contiguous bytes.  Without it every lane walks a
// row of its own: 32 lines an instruction, and the load/store unit (one line a cycle) set the
// epilogue's time, 5.5 us per 16 columns of a 128-row tile at N = 200.  A BF16X3 product with it, 128 /
// 64-wide tiles: N = 200 34 -> 24 / 20 -> 15 us, N = 1000 60 -> 48 / 35 -> 28 us, N = 2048 145 -> 127 /
// 148 -> 136 us.
__device__ __forceinline__ void epi_transpose(float* stage, int lane, const float (&v)[32], float (&out)[32]) {
#pragma unroll
  for (int c = 0; c < 8; ++c) store_f4(stage + lane * 32 + 4 * (c ^ (lane & 7)), v + 4 * c);
  __syncwarp();
#pragma unroll
  for (int p = 0; p < 8; ++p) {
    const int row = 4 * p + (lane >> 3);
    load_f4(stage + row * 32 + 4 * ((lane & 7) ^ (row & 7)), out + 4 * p);
  }
  __syncwarp();
}

// Yr and Yi of 32 columns at c0 of this warp's 32 rows (trow: the tile's sums at the warp's lanes), in
// the row-contiguous layout of epi_transpose.
template <int NS, int BN, int BKE, bool HAS_A>
__device__ __forceinline__ void split_load_y(uint32_t trow, int c0, float* stage, int lane, float (&yr)[32],
                                             float (&yi)[32]) {
  using Cfg = SplitCfg<NS, BN, BKE, HAS_A>;
#pragma unroll
  for (int part = 0; part < 2; ++part) {
    float v[2][16];
#pragma unroll
    for (int h = 0; h < 2; ++h) tmem_ld16(trow + (Cfg::SLICED ? 2 * part : part) * BN + c0 + 16 * h, v[h]);
    if constexpr (Cfg::STACKED || Cfg::SLICED) {
      float w[2][16];  // STACKED: Psi_i.A for Yr, Psi_i.S for Yi; SLICED: the products with S_1
#pragma unroll
      for (int h = 0; h < 2; ++h)
        tmem_ld16(trow + (Cfg::SLICED ? 2 * part + 1 : part ? 2 : 3) * BN + c0 + 16 * h, w[h]);
      tmem_wait_ld();
#pragma unroll
      for (int q = 0; q < 32; ++q)
        v[q >> 4][q & 15] += part || Cfg::SLICED ? w[q >> 4][q & 15] : -w[q >> 4][q & 15];
    } else {
      tmem_wait_ld();
    }
    float u[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) u[q] = v[q >> 4][q & 15];
    epi_transpose(stage, lane, u, part ? yi : yr);
  }
}

// A Chebyshev term at one entry of Y: psi_{l+1} = -2i Y + psi_{l-1} (x; the first term, psi_1 = -i Y, has sg = 1
// and x = 0) and z += a_{l+1} psi_{l+1} (the first term's z is a_0 psi_0).  Spelt out in FMAs so that every kernel
// rounds alike.
__device__ __forceinline__ void fwd_entry(float sg, float c, float yr, float yi, float xr, float xi, float& zr,
                                          float& zi, float& nr, float& ni) {
  nr = fmaf(sg, yi, xr);
  ni = fmaf(-sg, yr, xi);
  zr = fmaf(c, nr, zr);
  zi = fmaf(c, ni, zi);
}

// X = e^{-i beta h} acc of one entry, the phase (pr, pi).
__device__ __forceinline__ void fwd_phase(float pr, float pi, float ar, float ai, float& o_r, float& o_i) {
  o_r = fmaf(pr, ar, -__fmul_rn(pi, ai));
  o_i = fmaf(pr, ai, __fmul_rn(pi, ar));
}

// Epilogue of one 32-row x 32-column block (rows jb .., columns ib0 ..) in the layout of
// epi_transpose; BATCH row groups' operands are loaded together.
template <int NS, int EPI, int BATCH>
__device__ __forceinline__ void epi_block(const SplitEpi& e, const float (&yr)[32], const float (&yi)[32], int jb,
                                          int ib0, int lane, bool& bad, double& dsr, double& dsi) {
  const float c0f = e.t.coef0, cf = e.t.coef, sg = e.t.first ? 1.f : 2.f;
  const float b2 = e.t.bound2;
  const int ib = ib0 + 4 * (lane & 7), cnt = min(4, e.n - ib);
  if (cnt <= 0) return;
  // The operands are loaded without a branch: rows are clamped to the block, a row's four entries at ib
  // lie within its stride (ldm is a multiple of 4), and a pointer that a term does not have is another
  // one's.  With a branch per load (a vector, scalars at the edge, zero) the warp waited for each load
  // by itself: a BF16X3 / X6 product of 64-wide tiles took 14.5 / 18.9 us at N = 200 and 27.7 / 44.8 us
  // at N = 1000, now 13.9 / 17.7 and 27.2 / 43.6; a gradient step at N = 1024 615 -> 589 us (X3).
  const bool first = EPI == EPI_FWD && e.t.first;
  const float* x_re = EPI == EPI_FWD && !first ? e.prev_re : e.cur_re;
  const float* x_im = EPI == EPI_FWD && !first ? e.prev_im : e.cur_im;
  const float* z_re = EPI == EPI_FWD ? (first ? x_re : e.acc_re) : (e.prev_re ? e.prev_re : x_re);
  const float* z_im = EPI == EPI_FWD ? (first ? x_im : e.acc_im) : (e.prev_re ? e.prev_im : x_im);
#pragma unroll
  for (int g = 0; g < 8; g += BATCH) {
    float x_r[BATCH][4], x_i[BATCH][4], z_r[BATCH][4], z_i[BATCH][4];
    float sr = 0.f, si = 0.f;
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int j = jb + 4 * (g + u) + (lane >> 3);
      const size_t idx = (size_t)min(j, e.nc - 1) * e.ldm + ib;
      load_f4(x_re + idx, x_r[u]);
      load_f4(x_im + idx, x_i[u]);
      if (EPI != EPI_DOT) {
        load_f4(z_re + idx, z_r[u]);
        load_f4(z_im + idx, z_i[u]);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (j >= e.nc || q >= cnt) x_r[u][q] = x_i[u][q] = 0.f;
      }
      if (EPI == EPI_ADJ && !e.prev_re) {
#pragma unroll
        for (int q = 0; q < 4; ++q) z_r[u][q] = z_i[u][q] = 0.f;
      }
      if (first) {  // z holds psi_0
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          z_r[u][q] = __fmul_rn(c0f, z_r[u][q]);
          z_i[u][q] = __fmul_rn(c0f, z_i[u][q]);
          x_r[u][q] = x_i[u][q] = 0.f;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int j = jb + 4 * (g + u) + (lane >> 3);
      const size_t idx = (size_t)j * e.ldm + ib;
      const float* vr = yr + 4 * (g + u);
      const float* vi = yi + 4 * (g + u);
      if (EPI == EPI_DOT) {  // conj(b) Y; entries beyond the block are zero in b
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          sr = fmaf(x_r[u][q], vr[q], fmaf(x_i[u][q], vi[q], sr));
          si = fmaf(x_r[u][q], vi[q], fmaf(-x_i[u][q], vr[q], si));
        }
        continue;
      }
      if (j >= e.nc) continue;
      float o_r[4], o_i[4];
      if (EPI == EPI_ADJ) {  // out = cpa g + i cw Y + b2
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          o_r[q] = e.cpa_re * x_r[u][q] - e.cpa_im * x_i[u][q] - e.cw * vi[q] + z_r[u][q];
          o_i[q] = e.cpa_re * x_i[u][q] + e.cpa_im * x_r[u][q] + e.cw * vr[q] + z_i[u][q];
          bad |= q < cnt && !(o_r[q] * o_r[q] + o_i[q] * o_i[q] <= b2);
        }
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          fwd_entry(sg, cf, vr[q], vi[q], x_r[u][q], x_i[u][q], z_r[u][q], z_i[u][q], o_r[q], o_i[q]);
          bad |= q < cnt && !(o_r[q] * o_r[q] + o_i[q] * o_i[q] <= b2);
        }
        if (e.t.last) {  // X in place of psi_L
#pragma unroll
          for (int q = 0; q < 4; ++q) fwd_phase(e.t.ph_re, e.t.ph_im, z_r[u][q], z_i[u][q], o_r[q], o_i[q]);
        }
        if (!e.t.last) {
          store4(e.acc_re, idx, cnt, z_r[u]);
          store4(e.acc_im, idx, cnt, z_i[u]);
        }
      }
      store4(e.out_re, idx, cnt, o_r);
      store4(e.out_im, idx, cnt, o_i);
      store_slices<NS>(e, j, ib, cnt, o_r, o_i);
    }
    if (EPI == EPI_DOT) {
      dsr += (double)sr;
      dsi += (double)si;
    }
  }
}

// One split GEMM Y = left . right^T on 128-row x BN-column tiles:
//   HAS_A:  Yr = Psi_r.S - Psi_i.A,  Yi = Psi_r.A + Psi_i.S   (right = S + i A)
//   !HAS_A: Yr = Psi_r.S,            Yi = Psi_i.S             (right = S real)
// followed by the epilogue EPI.  One CTA per SM walks the tiles blockIdx.x, blockIdx.x + gridDim.x, ...
// Warp 0 (one thread) streams TMA stages, warp 1 (one thread) issues the MMAs of tile i into
// tensor-memory buffer i & 1, and the epilogue warps run the epilogue of tile i from its buffer while
// tile i + 1 accumulates in the other one.  Buffers are handed over by mbarriers (tfull: MMAs of a tile
// done; tempty: its accumulators read).  Every wait is bounded; one that gives up sets the abort flag
// and FQ_BIT_TIMEOUT, and the CTA drains its own copies and MMAs before it returns.
constexpr int PTHREADS = 64 + 32 * EPI_WARPS;
// column range [begin, end) of epilogue warp `warp` (2 .. 1 + EPI_WARPS) of a BN-wide tile
template <int BN>
__device__ __forceinline__ int epi_begin(int warp) { return ((warp - 2) >> 2) * (BN * 4 / EPI_WARPS); }

template <int NS, int BN, int BKE, int EPI, bool HAS_A>
__global__ void __launch_bounds__(PTHREADS, 1)
k_split_persist(const __grid_constant__ SplitMaps maps, int nk, int tiles_j, int tiles_i, SplitEpi e) {
  using Cfg = SplitCfg<NS, BN, BKE, HAS_A>;
  constexpr int STAGES = Cfg::STAGES;
  constexpr uint32_t BUF_COLS = Cfg::ACC_COLS;      // one tile's sums
  constexpr uint32_t TMEM_COLS = 2 * BUF_COLS;      // two buffers (<= 512)
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* gbase = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + STAGES * Cfg::STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 5);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES);
  const uint32_t tfull0 = smem_u32(bars + 2 * STAGES), tempty0 = smem_u32(bars + 2 * STAGES + 2);
  const uint32_t done = smem_u32(bars + 2 * STAGES + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ntiles = tiles_i * tiles_j;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, EPI_WARPS);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto coords = [&](int t, int& j0, int& i0) {
    const int per = RASTER_GROUP * tiles_i, g = t / per;
    const int gj = min(RASTER_GROUP, tiles_j - g * RASTER_GROUP), r = t - g * per;
    j0 = (g * RASTER_GROUP + r % gj) * BM;
    i0 = (r / gj) * BN;
  };

  if (warp == 0) {
    if (lane == 0) {  // ---------------- TMA producer
      int g = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        int j0, i0;
        coords(t, j0, i0);
        for (int kb = 0; kb < nk; ++kb) {
          const int s = g % STAGES;
          if (g >= STAGES && !(ok = mbar_wait(empty0 + 8 * s, ((g / STAGES) - 1) & 1))) break;
          if (*(volatile int*)abort_flag) {
            ok = false;
            break;
          }
          const uint32_t st = base + s * Cfg::STAGE_BYTES;
          const uint32_t bar = full0 + 8 * s;
          mbar_expect_tx(bar, Cfg::STAGE_BYTES);
          const int kx = kb * BKE;
          split_load_stage<NS, BN, BKE, HAS_A>(st, bar, maps.a, maps.os, maps.oa, kx, e.np, j0, i0);
          ++g;
        }
      }
      if (!ok) {
        atomicExch(abort_flag, 1);
        atomicOr(e.t.status, FQ_BIT_TIMEOUT);
      }
      // every copy issued must have landed before the CTA may exit
      for (int q = max(0, g - STAGES); q < g; ++q) mbar_wait(full0 + 8 * (q % STAGES), (q / STAGES) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ---------------- MMA issuer
      int g = 0, i = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++i) {
        const int b = i & 1;
        if (i >= 2 && !(ok = mbar_wait(tempty0 + 8 * b, ((i >> 1) - 1) & 1))) break;
        const uint32_t acc = tmem + (uint32_t)b * BUF_COLS;
        for (int kb = 0; kb < nk; ++kb, ++g) {
          const int s = g % STAGES;
          ok = mbar_wait(full0 + 8 * s, (g / STAGES) & 1);
          if (!ok || *(volatile int*)abort_flag) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t st = base + s * Cfg::STAGE_BYTES;
          split_issue_stage<NS, BN, BKE, HAS_A>(acc, st, kb == 0);
          mma_commit(empty0 + 8 * s);
        }
        if (!ok) break;
        mma_commit(tfull0 + 8 * b);  // this tile's accumulators are complete once its MMAs are
      }
      if (!ok) {
        atomicExch(abort_flag, 1);
        atomicOr(e.t.status, FQ_BIT_TIMEOUT);
      }
      mma_commit(done);  // every MMA issued above has completed once this arrives
      mbar_wait(done, 0);
    }
  } else {  // ---------------- epilogue warps: tensor-memory lane quarter warp % 4
    const int quarter = warp & 3;
    float* stage =
        reinterpret_cast<float*>(gbase + STAGES * Cfg::STAGE_BYTES + Cfg::TAIL + (warp - 2) * EPI_STAGE_BYTES);
    bool bad = false, ok = true;
    double dsr = 0.0, dsi = 0.0;
    int i = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
      const int b = i & 1;
      bool go = mbar_wait(tfull0 + 8 * b, (i >> 1) & 1);
      tc_fence_after();
      go = __all_sync(0xffffffffu, go && !*(volatile int*)abort_flag);  // warp-uniform: tcgen05.ld is .aligned
      if (!go) {
        ok = false;
        break;
      }
      int j0, i0;
      coords(t, j0, i0);
      const uint32_t trow = tmem + (uint32_t)b * BUF_COLS + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
      for (int c0 = epi_begin<BN>(warp), c1 = c0 + BN * 4 / EPI_WARPS; c0 < c1; c0 += 32) {
        float yr[32], yi[32];
        split_load_y<NS, BN, BKE, HAS_A>(trow, c0, stage, lane, yr, yi);
        if (c0 + 32 >= c1) {  // this warp's sums are read: the buffer's next MMAs may start
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(tempty0 + 8 * b);
        }
        if (i0 + c0 < e.n) epi_block<NS, EPI, 4>(e, yr, yi, j0 + quarter * 32, i0 + c0, lane, bad, dsr, dsi);
      }
      if (EPI == EPI_DOT) {  // a sum per warp: no barrier that a warp giving up could miss
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) {
          dsr += __shfl_xor_sync(0xffffffffu, dsr, w);
          dsi += __shfl_xor_sync(0xffffffffu, dsi, w);
        }
        if (lane == 0)
          e.partial[((size_t)(j0 / BM) * tiles_i + i0 / BN) * EPI_WARPS + warp - 2] = make_double2(dsr, dsi);
        dsr = dsi = 0.0;
      }
    }
    if (!ok) {
      atomicExch(abort_flag, 1);
      atomicOr(e.t.status, FQ_BIT_TIMEOUT);
    }
    if (bad) atomicOr(e.t.status, FQ_BIT_BOUND);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------------- chained products
// A chain of dependent products Y_p = left_p . right^T, p = 0 .. nprod-1, with one right operand
// (a step's Omega~_m) and product p's left operand written by product p-1's epilogue: the L
// Chebyshev terms of a step (forward or adjoint).  One cooperative launch runs the whole chain:
// work unit u = p * tiles + t (tiles in row-block-major order), CTA c takes the units c, c + G, ...
// in increasing order.  Product p's tiles of state-row block tj need exactly the rows tj of its left
// operand, i.e. the epilogues of product p-1's tiles (tj, *): a counter per (p - 1, tj) counts their
// epilogue warps, and the TMA producer waits for it (bounded) before loading.  A unit waits only on units with a
// smaller index, and all CTAs are resident (cooperative launch), so the chain always advances; the
// epilogue of one unit overlaps the MMAs of the next as in k_split_persist.
constexpr int CHAIN_MAXP = 12;

struct ChainArgs {
  SplitMaps rmaps;                 // right operand (os, oa); its a[] is unused
  CUtensorMap left[CHAIN_MAXP][3]; // left operand slices of product p
  SplitEpi epi[CHAIN_MAXP];        // epilogue of product p (slice_out = product p+1's left operand)
  int nprod, nk, tiles_j, tiles_i;
  unsigned int* flags;             // [nprod][tiles_j]: finished epilogue warps (EPI_WARPS a tile) of product p in
                                   // row block tj (zeroed before the launch)
};

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add(unsigned int* p, unsigned int v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
// bounded wait until *p >= target (acquire); false if it gave up
__device__ __forceinline__ bool wait_count(const unsigned int* p, unsigned int target) {
  const long long t0 = clock64();
  while (ld_acquire_u32(p) < target) {
    if (clock64() - t0 > kWaitCycles) return false;
    __nanosleep(64);
  }
  return true;
}

// The FP32 side of a kept tile (KEEP chains): this warp's 32 rows (lane = row) x 32 columns of psi_l,
// psi_{l-1} and acc over the products of a chain.  The two states stay in tensor memory, columns
// KEEP_COL + 128 slot + 64 part (psi_l in slot l & 1), and acc in registers.
constexpr uint32_t KEEP_COL = 256;
template <int NS> constexpr int KEEP_STAGE_BYTES = 2 * NS * 1024;  // 16 columns of a warp's slices
template <int NS, bool STACKED>
struct KeptTile {
  float ar[32], ai[32];
  int row, col;    // this lane's row, the warp's first column
  uint32_t trow;   // the warp's tensor-memory lanes
  unsigned char* stage;

  // psi_0 from the masters of the first product (slot 0; slot 1 is the first term's zero), acc = a_0 psi_0
  __device__ __forceinline__ void load(const SplitEpi& e, int half) {
    const size_t base = (size_t)min(row, e.nc - 1) * e.ldm;
#pragma unroll
    for (int q = 0; q < 32; q += 4) {
      float v[4] = {}, w[4] = {};
      if (col + q < e.n) {  // ldm is a multiple of 4
        load_f4(e.cur_re + base + col + q, v);
        load_f4(e.cur_im + base + col + q, w);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ar[q + u] = row < e.nc && col + q + u < e.n ? v[u] : 0.f;
        ai[q + u] = row < e.nc && col + q + u < e.n ? w[u] : 0.f;
      }
    }
#pragma unroll
    for (int c = 0; c < 32; c += 8) {
      const float zero[8] = {};
      const uint32_t at = trow + KEEP_COL + 32 * half + c;
      tmem_st8(at, ar + c);
      tmem_st8(at + 64, ai + c);
      tmem_st8(at + 128, zero);
      tmem_st8(at + 192, zero);
    }
    tmem_wait_st();
#pragma unroll
    for (int q = 0; q < 32; ++q) {
      ar[q] = __fmul_rn(e.t.coef0, ar[q]);
      ai[q] = __fmul_rn(e.t.coef0, ai[q]);
    }
  }

  // product p of the chain from the tile's sums (64 columns each: Psi_r.S, Psi_r.A, Psi_i.S, Psi_i.A when
  // STACKED; the two parts of Yr, then of Yi, when the right operand is real): the new state, acc and the slices; `tempty` is signalled once the sums are read.
  __device__ __forceinline__ void term(const SplitEpi& e, int p, int half, int lane, uint32_t tempty, bool& bad) {
    const float cf = e.t.coef, sg = e.t.first ? 1.f : 2.f, b2 = e.t.bound2;
    const bool last = e.t.last, edge = col + 32 > e.n;
    const uint32_t psi = trow + KEEP_COL + 128 * ((p + 1) & 1) + 32 * half;  // psi_{l-1}, then psi_{l+1}
#pragma unroll
    for (int c = 0; c < 32; c += 8) {
      float y[2][8], w[2][8], x[2][8];
      const uint32_t sums = trow + 32 * half + c;
      tmem_ld8(sums, y[0]);
      tmem_ld8(sums + (STACKED ? 192 : 64), w[0]);
      tmem_ld8(sums + (STACKED ? 64 : 128), y[1]);
      tmem_ld8(sums + (STACKED ? 128 : 192), w[1]);
      tmem_ld8(psi + c, x[0]);
      tmem_ld8(psi + 64 + c, x[1]);
      tmem_wait_ld();
      if (c == 24) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float o_r, o_i;
        const float yr = STACKED ? y[0][q] - w[0][q] : y[0][q] + w[0][q];
        fwd_entry(sg, cf, yr, y[1][q] + w[1][q], x[0][q], x[1][q], ar[c + q], ai[c + q], o_r, o_i);
        bad |= !(o_r * o_r + o_i * o_i <= b2);  // zero beyond the block
        y[0][q] = o_r;
        y[1][q] = o_i;
      }
      if (last) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          fwd_phase(e.t.ph_re, e.t.ph_im, ar[c + q], ai[c + q], y[0][q], y[1][q]);
          ar[c + q] = y[0][q];
          ai[c + q] = y[1][q];
        }
      }
      if (edge) {  // the slices' padding stays zero, also beside an entry that is not finite
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (col + c + q >= e.n) y[0][q] = y[1][q] = 0.f;
      }
      if (!last) {
        tmem_st8(psi + c, y[0]);
        tmem_st8(psi + 64 + c, y[1]);
      }
      // slices: 16 columns of a row, slice and part are 32 bytes, staged so that a warp's global stores
      // take 16 whole rows each
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        uint32_t pk[4][NS];
#pragma unroll
        for (int q = 0; q < 4; ++q) split_pair<NS>(y[part][2 * q], y[part][2 * q + 1], pk[q]);
#pragma unroll
        for (int t = 0; t < NS; ++t)
          *reinterpret_cast<uint4*>(stage + (2 * t + part) * 1024 + lane * 32 +
                                    16 * (((c >> 3) & 1) ^ ((lane >> 2) & 1))) =
              make_uint4(pk[0][t], pk[1][t], pk[2][t], pk[3][t]);
      }
      if ((c & 8) == 0) continue;
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int r = 16 * k + (lane >> 1), u = lane & 1, j = row - lane + r;
        if (j < e.nc) {
          __nv_bfloat16* d = e.slice_out + (size_t)j * e.kp + col + (c - 8) + 8 * u;
#pragma unroll
          for (int t = 0; t < NS; ++t)
#pragma unroll
            for (int part = 0; part < 2; ++part)
              *reinterpret_cast<uint4*>(d + t * e.slice_stride + part * e.np) =
                  *reinterpret_cast<const uint4*>(stage + (2 * t + part) * 1024 + r * 32 + 16 * (u ^ ((r >> 2) & 1)));
        }
      }
      __syncwarp();
    }
    tmem_wait_st();
    if (last) {  // X to the masters
      const int ib = col + 4 * (lane & 7), cnt = min(4, e.n - ib);
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        float u[32];
        epi_transpose(reinterpret_cast<float*>(stage), lane, part ? ai : ar, u);
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          const int j = row - lane + 4 * g + (lane >> 3);
          const float v[4] = {u[4 * g], u[4 * g + 1], u[4 * g + 2], u[4 * g + 3]};
          if (j < e.nc) store4(part ? e.out_im : e.out_re, (size_t)j * e.ldm + ib, cnt, v);
        }
      }
    }
  }
};

// KEEP: every CTA owns one tile for the whole chain (grid = tiles), and its states and accumulator stay
// on the SM (KeptTile); only slices are exchanged.  A tile's epilogue otherwise reads 128 KB of FP32 masters
// and writes as much, between the last MMA of a product and the first of the next.  The second buffer
// of sums, which a CTA with one tile a product has no use for, makes room for the states.
// BF16X3 / X6 products, masters in memory / kept: N = 64 9.8 / 7.9 and 11.5 / 9.8 us, N = 256 12.9 / 11.9 and
// 17.5 / 16.8, N = 700 21.9 / 19.0 and 32.1 / 30.7, N = 1024 25.6 / 24.4 and 42.0 / 41.2.  What is left at N = 1000 is
// the MMAs (80 cycles each for 64 at the tensor rate: 8 KB of operands from shared memory), 16 of
// 24 us, then the epilogue (its arithmetic, 3 us), the release and the first stage's load.
template <int NS, int BN, int BKE, int EPI, bool HAS_A, bool KEEP>
__global__ void __launch_bounds__(PTHREADS, 1) k_split_chain(const __grid_constant__ ChainArgs args) {
  static_assert(EPI != EPI_DOT, "chains of forward or adjoint terms only");
  using Cfg = SplitCfg<NS, BN, BKE, HAS_A>;
  constexpr int STAGES = Cfg::STAGES;
  static_assert(!KEEP || ((Cfg::STACKED || Cfg::SLICED) && EPI == EPI_FWD), "kept tiles: 64-wide forward terms");
  constexpr uint32_t BUF_COLS = Cfg::ACC_COLS;
  constexpr uint32_t TMEM_COLS = 2 * BUF_COLS;  // two buffers of sums (KEEP: one, and the states)
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* gbase = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + STAGES * Cfg::STAGE_BYTES);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * STAGES + 5);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + STAGES);
  const uint32_t tfull0 = smem_u32(bars + 2 * STAGES), tempty0 = smem_u32(bars + 2 * STAGES + 2);
  const uint32_t done = smem_u32(bars + 2 * STAGES + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tiles = args.tiles_i * args.tiles_j;
  const int nunits = args.nprod * tiles;
  unsigned int* status = args.epi[0].t.status;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, EPI_WARPS);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  auto unit = [&](int u, int& p, int& tj, int& j0, int& i0) {
    p = u / tiles;
    const int t = u - p * tiles;
    tj = t / args.tiles_i;
    j0 = tj * BM;
    i0 = (t - tj * args.tiles_i) * BN;
  };

  if (warp == 0) {
    if (lane == 0) {  // ---------------- TMA producer: waits for each unit's left operand
      int g = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < nunits && ok; u += gridDim.x) {
        int p, tj, j0, i0;
        unit(u, p, tj, j0, i0);
        if (p > 0) {
          if (!(ok = wait_count(args.flags + (size_t)(p - 1) * args.tiles_j + tj, (unsigned)EPI_WARPS * args.tiles_i))) break;
          fence_proxy_async_global();  // the epilogues' generic stores, before this thread's TMA reads
        }
        const int np_ = args.epi[p].np;
        for (int kb = 0; kb < args.nk; ++kb) {
          const int s = g % STAGES;
          if (g >= STAGES && !(ok = mbar_wait(empty0 + 8 * s, ((g / STAGES) - 1) & 1))) break;
          if (*(volatile int*)abort_flag) {
            ok = false;
            break;
          }
          const uint32_t st = base + s * Cfg::STAGE_BYTES;
          const uint32_t bar = full0 + 8 * s;
          mbar_expect_tx(bar, Cfg::STAGE_BYTES);
          const int kx = kb * BKE;
          split_load_stage<NS, BN, BKE, HAS_A>(st, bar, args.left[p], args.rmaps.os, args.rmaps.oa, kx, np_, j0, i0);
          ++g;
        }
      }
      if (!ok) {
        atomicExch(abort_flag, 1);
        atomicOr(status, FQ_BIT_TIMEOUT);
      }
      for (int q = max(0, g - STAGES); q < g; ++q) mbar_wait(full0 + 8 * (q % STAGES), (q / STAGES) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ---------------- MMA issuer (as k_split_persist)
      int g = 0, i = 0;
      bool ok = true;
      for (int u = blockIdx.x; u < nunits && ok; u += gridDim.x, ++i) {
        const int b = KEEP ? 0 : i & 1;
        if (KEEP && i >= 1 && !(ok = mbar_wait(tempty0, (i - 1) & 1))) break;
        if (!KEEP && i >= 2 && !(ok = mbar_wait(tempty0 + 8 * b, ((i >> 1) - 1) & 1))) break;
        const uint32_t acc = tmem + (uint32_t)b * BUF_COLS;
        for (int kb = 0; kb < args.nk; ++kb, ++g) {
          const int s = g % STAGES;
          ok = mbar_wait(full0 + 8 * s, (g / STAGES) & 1);
          if (!ok || *(volatile int*)abort_flag) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t st = base + s * Cfg::STAGE_BYTES;
          split_issue_stage<NS, BN, BKE, HAS_A>(acc, st, kb == 0);
          mma_commit(empty0 + 8 * s);
        }
        if (!ok) break;
        mma_commit(tfull0 + 8 * b);
      }
      if (!ok) {
        atomicExch(abort_flag, 1);
        atomicOr(status, FQ_BIT_TIMEOUT);
      }
      mma_commit(done);
      mbar_wait(done, 0);
    }
  } else {  // ---------------- epilogue warps; then the unit's completion for its row block
    const int quarter = warp & 3;
    float* stage =
        reinterpret_cast<float*>(gbase + STAGES * Cfg::STAGE_BYTES + Cfg::TAIL + (warp - 2) * EPI_STAGE_BYTES);
    bool bad = false, ok = true;
    double dsr = 0.0, dsi = 0.0;
    int i = 0;
    KeptTile<NS, Cfg::STACKED> kept;
    const int half = (warp - 2) >> 2;
    if constexpr (KEEP) {
      int p, tj, j0, i0;
      unit(blockIdx.x, p, tj, j0, i0);
      kept.row = j0 + quarter * 32 + lane;
      kept.col = i0 + 32 * half;
      kept.trow = tmem + ((uint32_t)(quarter * 32) << 16);
      kept.stage = gbase + STAGES * Cfg::STAGE_BYTES + Cfg::TAIL + (warp - 2) * KEEP_STAGE_BYTES<NS>;
      kept.load(args.epi[0], half);
    }
    for (int u = blockIdx.x; u < nunits; u += gridDim.x, ++i) {
      int p, tj, j0, i0;
      unit(u, p, tj, j0, i0);
      const int b = KEEP ? 0 : i & 1;
      bool go = mbar_wait(tfull0 + 8 * b, KEEP ? i & 1 : (i >> 1) & 1);
      tc_fence_after();
      go = __all_sync(0xffffffffu, go && !*(volatile int*)abort_flag);
      if (!go) {
        ok = false;
        break;
      }
      const SplitEpi& e = args.epi[p];
      if constexpr (KEEP) {
        kept.term(e, p, half, lane, tempty0, bad);
      } else {
        // the previous product's outputs this epilogue reads (prev, acc) were released with its counter
        if (p > 0) ld_acquire_u32(args.flags + (size_t)(p - 1) * args.tiles_j + tj);
        const uint32_t trow = tmem + (uint32_t)b * BUF_COLS + ((uint32_t)(quarter * 32) << 16);
#pragma unroll 1
        for (int c0 = epi_begin<BN>(warp), c1 = c0 + BN * 4 / EPI_WARPS; c0 < c1; c0 += 32) {
          float yr[32], yi[32];
          split_load_y<NS, BN, BKE, HAS_A>(trow, c0, stage, lane, yr, yi);
          if (c0 + 32 >= c1) {  // this warp's sums are read: the buffer's next MMAs may start
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(tempty0 + 8 * b);
          }
          if (i0 + c0 < e.n) epi_block<NS, EPI, 4>(e, yr, yi, j0 + quarter * 32, i0 + c0, lane, bad, dsr, dsi);
        }
      }
      // this warp's stores of the unit made visible (to the async proxy too), then one release per
      // warp, which covers the lanes' stores through the barrier: a tile is done when its epilogue warps
      // have counted
      fence_proxy_async_global();
      __syncwarp();
      if (lane == 0) red_release_add(args.flags + (size_t)p * args.tiles_j + tj, 1u);
    }
    if (!ok) {
      atomicExch(abort_flag, 1);
      atomicOr(status, FQ_BIT_TIMEOUT);
    }
    if (bad) atomicOr(status, FQ_BIT_BOUND);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// Launches a chain cooperatively (all CTAs resident).  FQ_EUNSUPPORTED when that cannot be done
// (a capturing stream, or the device refuses the cooperative launch): the caller then runs the
// products one launch each.
template <int NS, int BN, int BKE, int EPI, bool HAS_A, bool KEEP = false>
fq_status launch_chain(const ChainArgs& args, cudaStream_t s) {
  using Cfg = SplitCfg<NS, BN, BKE, HAS_A>;
  constexpr size_t SMEM = KEEP ? Cfg::SMEM + EPI_WARPS * (KEEP_STAGE_BYTES<NS> - EPI_STAGE_BYTES) : Cfg::SMEM;
  static_assert(KEEP_STAGE_BYTES<NS> >= EPI_STAGE_BYTES && SMEM <= 232448, "shared memory of one CTA");
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) return FQ_EUNSUPPORTED;
  static std::atomic<unsigned> attr_set{0};
  if (fq_first_on_device(attr_set)) {
    cudaError_t e = cudaFuncSetAttribute(k_split_chain<NS, BN, BKE, EPI, HAS_A, KEEP>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM);
    if (e != cudaSuccess) return fq_cuda_fail(e, "chain kernel shared-memory attribute");
  }
  const int tiles = args.tiles_i * args.tiles_j;
  const int grid = std::min(tiles, fq_sm_count());
  void* kargs[] = {(void*)&args};
  cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_split_chain<NS, BN, BKE, EPI, HAS_A, KEEP>, dim3(grid),
                                              dim3(PTHREADS), kargs, SMEM, s);
  if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
    cudaGetLastError();
    return FQ_EUNSUPPORTED;
  }
  return e == cudaSuccess ? FQ_OK : fq_cuda_fail(e, "chain kernel launch");
}

// ------------------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

fq_status encode_fn() {
  std::call_once(g_encode_once, [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      g_encode = (PFN_cuTensorMapEncodeTiled_v12000)fn;
  });
  if (!g_encode) {
    fq_set_error("cuTensorMapEncodeTiled is not available from the driver");
    return FQ_ECUDA;
  }
  return FQ_OK;
}

// 2-D BF16 map over [rows][cols] (row-major, cols contiguous), box = box_cols x box_rows with the
// swizzle matching box_cols * 2 bytes (128, 64 or 32).
fq_status make_map(CUtensorMap* m, const void* ptr, int rows, int cols, int box_rows, int box_cols) {
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {(cuuint32_t)box_cols, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  const CUtensorMapSwizzle sw = box_cols == 64   ? CU_TENSOR_MAP_SWIZZLE_128B
                                : box_cols == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                 : CU_TENSOR_MAP_SWIZZLE_32B;
  CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    fq_set_error("cuTensorMapEncodeTiled failed (%d)", (int)r);
    return FQ_ECUDA;
  }
  return FQ_OK;
}

int grid_1d(size_t total) { return (int)std::min<size_t>(std::max<size_t>((total + 255) / 256, 1), 152 * 32); }

}  // namespace
