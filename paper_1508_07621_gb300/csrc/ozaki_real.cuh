// FP64 emulation of the products with a real right operand (the gradient's forward, adjoint and
// dot products: Omega~_m and E = H1 / Delta E are real symmetric there), with stacked rows.
//
// The real and imaginary parts of 64 states are stacked as the 128 rows of the MMA's left
// operand (rows 0-63: Re psi, rows 64-127: Im psi), so one MMA of N = 64 per slice pair makes both
// Y_r and Y_i of a 64 x 64 tile, and one accumulator group takes 64 tensor-memory columns.  The
// four groups of ozaki_core.cuh (three exact ones and the tail) then fill half of the tensor
// memory, and the chunks of K alternate between two halves: the drain warps fold chunk c while
// the MMAs of chunk c + 1 run.  With one MMA per pair and value of k, a group's sum over 256
// values of k is at most 3 pairs x 2^14 x 256 < 2^24 units: still exact.
//
// Warp 0 streams the stages (K = 16 each: the two 64-row halves of each left slice and the 64 rows of
// each right slice, two bulk copies), warp 1 issues the MMAs, warps 2-17 drain (four per lane quarter,
// 16 columns each) and finally run the FP64 epilogue.  Clusters split K where tiles are few, and the
// epilogue is kept short, as in ozaki_core.cuh.  Every wait is bounded as in the other tensor-core
// kernels.
#pragma once

#include "ozaki_core.cuh"

namespace {

constexpr int OZR_BM = 64;                        // states per tile (128 stacked rows)
constexpr int OZR_A_BYTES = 2 * OZR_BM * OZ_ROWB; // one left slice: Re and Im halves, 4 KB
constexpr int OZR_B_BYTES = OZ_BN * OZ_ROWB;      // one right slice, 2 KB
constexpr int OZR_STAGE_BYTES = OZ_S * (OZR_A_BYTES + OZR_B_BYTES);
constexpr int OZR_STAGES = 4;
constexpr int OZR_KB_PER_DRAIN = 16;              // 256 values of k per chunk
constexpr int OZR_BUF_COLS = 4 * OZ_BN;           // four groups of 64 columns
constexpr int OZR_XS_BYTES = 2 * OZ_XS_PLANE * 4;  // staged sums: hi, then lo
constexpr size_t OZR_SMEM = (size_t)OZR_STAGES * OZR_STAGE_BYTES + 1024 + 256;
static_assert((size_t)OZR_STAGES * OZR_STAGE_BYTES >= OZR_XS_BYTES + 16 * sizeof(double2), "epilogue staging");

template <int EPI>
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_real_term(const OzOperands op, int nk, int tiles_j, int tiles_i, int np, int csize, OzEpi e) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* gbase = smem_raw + (base - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + OZR_STAGES * OZR_STAGE_BYTES);
  // full[4], empty[4], tfull[2], tempty[2], done
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * OZR_STAGES + 5);
  int* abort_flag = reinterpret_cast<int*>(tmem_slot + 1);
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + OZR_STAGES);
  const uint32_t tfull0 = smem_u32(bars + 2 * OZR_STAGES), tempty0 = smem_u32(bars + 2 * OZR_STAGES + 2);
  const uint32_t done = smem_u32(bars + 2 * OZR_STAGES + 4);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x % csize;
  const int kb0 = nk * rank / csize, nkr = nk * (rank + 1) / csize - kb0;  // this CTA's K stages
  const int nchunks = (nkr + OZR_KB_PER_DRAIN - 1) / OZR_KB_PER_DRAIN;

  int tj, ti;
  {
    const int b = blockIdx.x / csize, per = RASTER_GROUP * tiles_i, g = b / per;
    const int gj = min(RASTER_GROUP, tiles_j - g * RASTER_GROUP), r = b - g * per;
    tj = g * RASTER_GROUP + r % gj;
    ti = r / gj;
  }
  const int j0 = tj * OZR_BM, i0 = ti * OZ_BN;

  if (threadIdx.x == 0) {
    for (int s = 0; s < OZR_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull0 + 8 * b, 1);
      mbar_init(tempty0 + 8 * b, OZ_EPI_WARPS);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(OZ_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {  // ---------------- TMA producer
      int issued = 0;
      bool ok = true;
      for (int kb = 0; kb < nkr && ok; ++kb) {
        const int s = kb % OZR_STAGES;
        if (kb >= OZR_STAGES && !(ok = mbar_wait(empty0 + 8 * s, ((kb / OZR_STAGES) - 1) & 1))) break;
        if (*(volatile int*)abort_flag) {
          ok = false;
          break;
        }
        const uint32_t st = base + s * OZR_STAGE_BYTES;
        const uint32_t bar = full0 + 8 * s;
        mbar_expect_tx(bar, OZR_STAGE_BYTES);
        const size_t kp = np / OZ_BKE, kx = kb0 + kb;  // K pieces of a block, and this one
        bulk_load(st, op.left + ((size_t)(j0 / OZR_BM) * kp + kx) * (OZ_S * OZR_A_BYTES / 2), OZ_S * OZR_A_BYTES, bar);
        bulk_load(st + OZ_S * OZR_A_BYTES, op.right + ((size_t)(i0 / OZ_BN) * kp + kx) * (OZ_S * OZR_B_BYTES / 2),
                  OZ_S * OZR_B_BYTES, bar);
        issued = kb + 1;
      }
      if (!ok) {
        atomicExch(abort_flag, 1);
        atomicOr(e.t.status, FQ_BIT_TIMEOUT);
      }
      for (int kb = max(0, issued - OZR_STAGES); kb < issued; ++kb)
        mbar_wait(full0 + 8 * (kb % OZR_STAGES), (kb / OZR_STAGES) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ---------------- MMA issuer
      constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(OZ_BN >> 3) << 17) |
                                 ((uint32_t)(128 >> 4) << 24);
      bool ok = true;
      int kb = 0;
      for (int c = 0; c < nchunks && ok; ++c) {
        const int b = c & 1;
        if (c >= 2 && !(ok = mbar_wait(tempty0 + 8 * b, ((c >> 1) - 1) & 1))) break;
        tc_fence_after();
        const uint32_t accb = tmem + (uint32_t)(b * OZR_BUF_COLS);
        for (int kq = 0; kq < OZR_KB_PER_DRAIN && kb < nkr; ++kq, ++kb) {
          const int s = kb % OZR_STAGES;
          ok = mbar_wait(full0 + 8 * s, (kb / OZR_STAGES) & 1);
          if (!ok || *(volatile int*)abort_flag) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint64_t d0 = oz_desc(base + s * OZR_STAGE_BYTES);
#pragma unroll
          for (int p = 0; p < OZ_PAIRS; ++p) {
            int a, bb;
            oz_pair(p, a, bb);
            const int g = a + bb < 3 ? a + bb : 3;
            const bool lead = p == 0 || p == 1 || p == 3 || p == 6;
            mma_bf16(accb + (uint32_t)(g * OZ_BN), d0 + (uint64_t)((a * OZR_A_BYTES) >> 4),
                     d0 + (uint64_t)((OZ_S * OZR_A_BYTES + bb * OZR_B_BYTES) >> 4), idesc,
                     (kq == 0 && lead) ? 0u : 1u);
          }
          mma_commit(empty0 + 8 * s);
        }
        if (!ok) break;
        mma_commit(tfull0 + 8 * b);
      }
      if (!ok) {
        atomicExch(abort_flag, 1);
        atomicOr(e.t.status, FQ_BIT_TIMEOUT);
      }
      mma_commit(done);
      mbar_wait(done, 0);
    }
  } else {  // ---------------- drain warps 2-17
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    const int row = quarter * 32 + lane;  // stacked row: Re of state row (< 64), Im of state row - 64
    float2 h[8], l[8];                    // double-float sums of columns (2p, 2p + 1)
#pragma unroll
    for (int q = 0; q < 8; ++q) h[q] = l[q] = make_float2(0.f, 0.f);
    bool ok = true;
    for (int c = 0; c < nchunks; ++c) {
      const int b = c & 1;
      bool go = mbar_wait(tfull0 + 8 * b, (c >> 1) & 1);
      tc_fence_after();
      go = __all_sync(0xffffffffu, go && !*(volatile int*)abort_flag);
      if (!go) {
        ok = false;
        break;
      }
      const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * OZR_BUF_COLS + part * 16);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        float v[16];
        tmem_ld16(trow + g * OZ_BN, v);
        tmem_wait_ld();
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const float2 w = make_float2(v[2 * q], v[2 * q + 1]);
          if (g < 3) dd_add2(h[q], l[q], w);
          else l[q] = __fadd2_rn(l[q], w);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8 * b);
    }
    if (!ok) {
      atomicExch(abort_flag, 1);
      atomicOr(e.t.status, FQ_BIT_TIMEOUT);
    }
    // stage the sums column-major (xs[col][row], hi then lo) in the idle stages: the last MMAs
    // have completed, and every stage's copies have landed
    if (ok) {
      float* xw = reinterpret_cast<float*>(gbase) + part * 16 * OZ_XS_LD + row;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        xw[q * OZ_XS_LD] = q & 1 ? h[q >> 1].y : h[q >> 1].x;
        xw[q * OZ_XS_LD + OZ_XS_PLANE] = q & 1 ? l[q >> 1].y : l[q >> 1].x;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (csize > 1) oz_cluster_sync();
  if (warp >= 2) {
    // ---------------- FP64 epilogue: this CTA's share of the columns, consecutive threads on
    // consecutive columns of a state
    const bool ok = !*(volatile int*)abort_flag;
    const float* xs = reinterpret_cast<const float*>(gbase);
    const int wd = OZ_BN / csize, t = threadIdx.x - 64;
    const int cc = rank * wd + t % wd, i = i0 + cc;
    double dsr = 0.0, dsi = 0.0;
    bool bad = false;
    if (ok && i < e.n) {
      const fq_term& tt = e.t;
      const int ei = e.et[i];
      const bool first = EPI == OZ_FWD && tt.first;
      const double* src_re = EPI == OZ_FWD && !first ? e.prev_re : e.cur_re;
      const double* src_im = EPI == OZ_FWD && !first ? e.prev_im : e.cur_im;
      const double* add_re = EPI == OZ_ADJ ? e.prev_re : e.acc_re;  // ADJ: b2 (may be absent); FWD: acc
      const double* add_im = EPI == OZ_ADJ ? e.prev_im : e.acc_im;
      const bool add = EPI != OZ_DOT && !first && add_re;
      const int step = 32 * OZ_EPI_WARPS / wd;
      for (int row0 = t / wd; row0 < OZR_BM && j0 + row0 < e.nc; row0 += OZ_EPI_ROWS * step) {
        double xr[OZ_EPI_ROWS], xi[OZ_EPI_ROWS], zr[OZ_EPI_ROWS], zi[OZ_EPI_ROWS];
        int ej[OZ_EPI_ROWS];
#pragma unroll
        for (int u = 0; u < OZ_EPI_ROWS; ++u) {
          const int srow = row0 + u * step, j = j0 + srow;
          const bool in = srow < OZR_BM && j < e.nc;
          const size_t idx = (size_t)j * e.n + i;
          xr[u] = in ? src_re[idx] : 0.0;
          xi[u] = in ? src_im[idx] : 0.0;
          zr[u] = in && add ? add_re[idx] : 0.0;
          zi[u] = in && add ? add_im[idx] : 0.0;
          ej[u] = in ? e.es[j] : 0;
        }
#pragma unroll
        for (int u = 0; u < OZ_EPI_ROWS; ++u) {
          const int srow = row0 + u * step, j = j0 + srow;
          if (srow >= OZR_BM || j >= e.nc) break;
          const int ex = ej[u] + ei, at = cc * OZ_XS_LD + srow;
          const size_t idx = (size_t)j * e.n + i;
          float h0, l0, h1, l1;
          oz_fold(xs, at, OZ_XS_PLANE, csize, h0, l0);
          oz_fold(xs, at + OZR_BM, OZ_XS_PLANE, csize, h1, l1);
          const double yr = oz_value(h0, l0, ex), yi = oz_value(h1, l1, ex);
          if (EPI == OZ_DOT) {  // conj(b) Y
            dsr = fma(xr[u], yr, fma(xi[u], yi, dsr));
            dsi = fma(xr[u], yi, fma(-xi[u], yr, dsi));
          } else if (EPI == OZ_ADJ) {  // out = cpa g + i cw Y + b2
            double orr = e.cpa_re * xr[u] - e.cpa_im * xi[u] - e.cw * yi;
            double oi = e.cpa_re * xi[u] + e.cpa_im * xr[u] + e.cw * yr;
            if (add) {
              orr += zr[u];
              oi += zi[u];
            }
            bad |= oz_outside(orr, oi, tt.bound2);
            e.out_re[idx] = orr;
            e.out_im[idx] = oi;
          } else {  // Chebyshev term (as in the plain FP64 path)
            double pr, pi, ar, ai;
            if (first) {
              pr = yi;
              pi = -yr;
              ar = fma(tt.coef, pr, tt.coef0 * xr[u]);
              ai = fma(tt.coef, pi, tt.coef0 * xi[u]);
            } else {
              pr = fma(2.0, yi, xr[u]);
              pi = fma(-2.0, yr, xi[u]);
              ar = fma(tt.coef, pr, zr[u]);
              ai = fma(tt.coef, pi, zi[u]);
            }
            bad |= oz_outside(pr, pi, tt.bound2);
            if (tt.last) {
              e.out_re[idx] = tt.ph_re * ar - tt.ph_im * ai;
              e.out_im[idx] = tt.ph_re * ai + tt.ph_im * ar;
            } else {
              e.out_re[idx] = pr;
              e.out_im[idx] = pi;
              e.acc_re[idx] = ar;
              e.acc_im[idx] = ai;
            }
          }
        }
      }
    }
    if (bad) atomicOr(e.t.status, FQ_BIT_BOUND);
    if (EPI == OZ_DOT) {  // per-CTA partial in a fixed order (bit-reproducible)
      double2* red = reinterpret_cast<double2*>(gbase + OZR_XS_BYTES);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        dsr += __shfl_xor_sync(0xffffffffu, dsr, o);
        dsi += __shfl_xor_sync(0xffffffffu, dsi, o);
      }
      if (lane == 0) red[warp - 2] = make_double2(dsr, dsi);
      asm volatile("bar.sync 1, %0;" ::"n"(32 * OZ_EPI_WARPS) : "memory");
      if (warp == 2 && lane == 0) {
        double sr = 0.0, si = 0.0;
        for (int q = 0; q < OZ_EPI_WARPS; ++q) {
          sr += red[q].x;
          si += red[q].y;
        }
        e.partial[tj * tiles_i + ti] = make_double2(sr, si);
      }
    }
  }
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS) : "memory");
  }
  if (csize > 1) oz_cluster_sync();  // no CTA leaves while a peer may still read its sums
}

}  // namespace
