// Tiled tridiagonal chain (FP64 or FP32): each CTA carries one segment of one state through all L
// products of a step on chip and writes it back, so HBM sees the state once per step instead of five
// times per product.  Where one CTA holds a whole state, one launch runs every step and the state
// stays on chip throughout; otherwise there is one launch per step.
//
// The step works in the real gauge frame of Omega~_m (gauge.cuh): X_m = D_m P(Omega'_m) D_m^+
// X_{m-1} with P(x) = e^{-i beta h} sum_k c_k T_k(x), c_k = (-i)^k a_k (Eqs. 10 and 12), applied by
// Clenshaw's backward recurrence.  A CTA holds (threads x EPT) consecutive rows: its segment of seg
// rows plus L halo rows on each side where the state goes on.  Every product can be wrong only one
// row further in from such an edge (the rows beyond it are taken as zero), so after the L products
// of a step the segment's rows are exact; only those are written.  An exact row takes the same
// operations on the same numbers in every segmentation, so the split never changes a result's bits.
// pick_tile chooses segments, threads and rows per thread for the state length and count.
//
// FQ_DF32 runs the same step in double-float arithmetic: every value is an unevaluated sum
// hi + lo of two FP32 numbers (Dekker's splitting, Knuth's two-sum, and two-product by FMA), so
// the products keep about 48 significant bits on the FP32 pipes, which GB300 runs at many times
// its FP64 rate.  States stay FP64 in HBM between steps.
//
// Layout: states as rows, planar re / im planes [nc][ld] (the streaming kernel's layout).
// Per step and row: (2 d, 2 e') and (cos theta, sin theta) of D_m, in the kernel's precision,
// computed once per call in FP64 by k_gauge_tile.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "dfl.cuh"
#include "gauge.cuh"
#include "internal.h"

namespace {

constexpr int TILE_NT = 256;  // most threads of a CTA
constexpr int TILE_SLOTS = TILE_NT / 32 + 1;  // rows exchanged between warps, and a zero at the end
constexpr int TILE_MAXL = 128;

// How the segments of a state lie: seg rows each, the tile of segment b from row b step - off on.
struct TileSpan {
  int seg, step, off;
};

// Rows base .. a CTA holds and the rows [first, last) of them it writes, for segment blockIdx.x.  LINEAR
// takes the base from the span (it may be negative: those rows are zero).  The other form starts no tile
// before row 0, as FP64 needs where the halos are as long as the state; the one-step FP32 kernel takes 8 % longer
// with it (800 x 9001), and the double-float one spills more.
template <bool LINEAR>
struct TileRows {
  int first, last, base;
  __device__ TileRows(TileSpan sp, int L, int n) {
    first = blockIdx.x * sp.seg;
    last = min(first + sp.seg, n);
    base = LINEAR ? (int)blockIdx.x * sp.step - sp.off : max(0, first - L);
  }
};

// FP64: rows of a CTA below which a product's time no longer falls, where the FP64 pipe's time for
// that many rows (2 multiply-adds a cycle and SM) equals the latency of a product.
constexpr int F64_FLOOR_ROWS = 128;

// Segments per state, threads per CTA and rows per thread.
struct TileShape {
  int segs, seg, nt, ept;
  // two segments have no halo on their outer sides, more have one on both
  TileSpan span(int L) const { return segs <= 2 ? TileSpan{seg, segs == 1 ? 0 : seg - L, 0} : TileSpan{seg, seg, L}; }
};

// The shape for states of n rows, nc of them.  The arithmetic of a step is the rows the CTAs hold, halo
// and padding included, so a CTA gets no more threads than its rows need, and as few segments as fit
// (one segment has no halo and runs all steps in one launch).  FP64 (floor_rows > 0) is bound by its
// pipe from 128 rows on, so there an SM's time is (CTAs on the fullest SM) x (rows of a CTA), and more
// segments are taken where few states would leave SMs idle; the FP32 pipes need two dozen warps before
// that pays.  Rows per thread: the smallest of `epts` that holds the rows with TILE_NT threads (many
// warps of few rows hide latency best).
// A step in us before (2048 rows a CTA in FP64 and FP32, 1024 in double-float, always) and now, states
// x rows: FP64 36 x 36 43 -> 7, 24 x 501 66 -> 14, 501 x 501 245 -> 62, 24 x 3001 116 -> 49, 160 x 10001
// 1317 -> 1141; double-float 36 x 36 16 -> 4.8, 501 x 501 48 -> 31, 1501 x 1501 253 -> 212; FP32 501 x 501
// 19 -> 6.5.
template <int NE>
TileShape pick_tile(int n, int nc, int L, const int (&epts)[NE], int floor_rows) {
  const int sms = fq_sm_count(), cap = TILE_NT * epts[NE - 1];
  TileShape best{};
  double cost = 0.0;
  for (int segs = 1; segs <= n; ++segs) {
    const int seg = (n + segs - 1) / segs;
    const int halo = segs == 1 ? 0 : (segs == 2 ? L : 2 * L);
    const int need = segs == 1 ? n : std::min(n, seg + halo);
    if (need > cap) continue;
    int ept = epts[NE - 1];
    if (segs == 1 || floor_rows > 0)
      for (int q = NE - 1; q >= 0; --q)
        if (need <= TILE_NT * epts[q]) ept = epts[q];
    const int nt = 32 * ((need + 32 * ept - 1) / (32 * ept));
    const int real = (n + seg - 1) / seg;  // segments that hold rows
    const double waves = std::ceil((double)nc * real / sms);
    const double c = std::max(waves * nt * ept, (double)floor_rows);
    if (best.segs == 0 || c < 0.999 * cost) {
      best = TileShape{real, seg, nt, ept};
      cost = c;
    }
    if (floor_rows == 0) break;
    if ((double)nc * real >= 4.0 * sms || seg <= 2 * L) break;  // more segments only add halo from here
  }
  return best;
}

template <typename T>
struct TileCoef {
  T c[TILE_MAXL + 1];  // |c_k|: c_k = c[k] for even k (real, sign included), i c[k] for odd k
};

template <typename T, int TILE_EPT>
struct Tile {
  using T2 = typename V2<T>::t;
  T2* slot_last;   // [2][TILE_SLOTS]: entry w + 1 the last row of warp w, entry 0 zero
  T2* slot_first;  // [2][TILE_SLOTS]: entry w the first row of warp w, the one after the last warp zero
  int lane, warp;

  __device__ __forceinline__ Tile(T2* slots) {
    slot_last = slots;
    slot_first = slots + 2 * TILE_SLOTS;
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
    if (threadIdx.x < 2) {  // visible from the first halo()'s barrier on
      slot_last[threadIdx.x * TILE_SLOTS] = T2{0, 0};
      slot_first[threadIdx.x * TILE_SLOTS + (blockDim.x >> 5)] = T2{0, 0};
    }
  }

  // rows i0 - 1 and i0 + EPT of x (neighbouring threads; zero beyond the tile)
  __device__ __forceinline__ void halo(const T2 (&x)[TILE_EPT], int par, T2& left, T2& right) {
    T lr = __shfl_up_sync(0xffffffffu, x[TILE_EPT - 1].x, 1);
    T li = __shfl_up_sync(0xffffffffu, x[TILE_EPT - 1].y, 1);
    T rr = __shfl_down_sync(0xffffffffu, x[0].x, 1);
    T ri = __shfl_down_sync(0xffffffffu, x[0].y, 1);
    if (lane == 31) slot_last[par * TILE_SLOTS + warp + 1] = x[TILE_EPT - 1];
    if (lane == 0) slot_first[par * TILE_SLOTS + warp] = x[0];
    __syncthreads();
    if (lane == 0) {
      const T2 w = slot_last[par * TILE_SLOTS + warp];
      lr = w.x;
      li = w.y;
    }
    if (lane == 31) {
      const T2 w = slot_first[par * TILE_SLOTS + warp + 1];
      rr = w.x;
      ri = w.y;
    }
    left = T2{lr, li};
    right = T2{rr, ri};
  }

  // out = c v + (2 Omega' x) - out (HALF: c v + Omega' x - out, the closing sum), c = cc (real) or
  // i cc (IM): four FMAs per component, five for the closing sum
  template <bool IM, bool HALF>
  __device__ __forceinline__ void apply(const T2 (&x)[TILE_EPT], T2 (&out)[TILE_EPT], const T2 (&v)[TILE_EPT],
                                        const T (&d)[TILE_EPT], const T (&e)[TILE_EPT], T el0, T cc, int par) {
    T2 left, right;
    halo(x, par, left, right);
#pragma unroll
    for (int q = 0; q < TILE_EPT; ++q) {
      const T2 xm = q == 0 ? left : x[q - 1];
      const T2 xp = q == TILE_EPT - 1 ? right : x[q + 1];
      const T el = q == 0 ? el0 : e[q - 1];
      T ar, ai;
      if (HALF) {
        ar = fma((T)0.5, fma(d[q], x[q].x, fma(el, xm.x, e[q] * xp.x)), -out[q].x);
        ai = fma((T)0.5, fma(d[q], x[q].y, fma(el, xm.y, e[q] * xp.y)), -out[q].y);
      } else {
        ar = fma(d[q], x[q].x, fma(el, xm.x, fma(e[q], xp.x, -out[q].x)));
        ai = fma(d[q], x[q].y, fma(el, xm.y, fma(e[q], xp.y, -out[q].y)));
      }
      if (IM) {
        out[q] = T2{fma(-cc, v[q].y, ar), fma(cc, v[q].x, ai)};
      } else {
        out[q] = T2{fma(cc, v[q].x, ar), fma(cc, v[q].y, ai)};
      }
    }
  }
};

// One step of the chain, or `steps` of them (MULTI: a single segment per state).
template <typename T, int TILE_EPT, bool MULTI>
__global__ void __launch_bounds__(TILE_NT)
k_tri_tile(const typename V2<T>::t* __restrict__ cf, const typename V2<T>::t* __restrict__ rot,
           const T* __restrict__ xr, const T* __restrict__ xi, T* __restrict__ yr, T* __restrict__ yi, int n, int ld,
           int L, TileSpan span, int steps, TileCoef<T> coef, T ph_re, T ph_im, T bound2, unsigned int* status) {
  using T2 = typename V2<T>::t;
  __shared__ T2 slots[4 * TILE_SLOTS];
  Tile<T, TILE_EPT> tl(slots);
  const size_t j = blockIdx.y;
  const TileRows<!MULTI> rows(span, L, n);
  const int i0 = rows.base + (int)threadIdx.x * TILE_EPT;
  T2 v[TILE_EPT], A[TILE_EPT], B[TILE_EPT];
  T d[TILE_EPT], e[TILE_EPT];
#pragma unroll
  for (int q = 0; q < TILE_EPT; ++q) {
    const int i = i0 + q;
    A[q] = (MULTI || i >= 0) && i < n ? T2{xr[j * ld + i], xi[j * ld + i]} : T2{0, 0};
  }
  bool bad = false;
  int par = 0;
  const T cL = coef.c[L];
  for (int m = 0; m < (MULTI ? steps : 1); ++m, cf += ld, rot += ld) {
#pragma unroll
    for (int q = 0; q < TILE_EPT; ++q) {
      const int i = i0 + q;
      const bool in = (MULTI || i >= 0) && i < n;
      const T2 r = in ? rot[i] : T2{0, 0}, c = in ? cf[i] : T2{0, 0};
      v[q] = T2{fma(r.x, A[q].x, r.y * A[q].y), fma(r.x, A[q].y, -(r.y * A[q].x))};  // D^+ x
      d[q] = c.x;
      e[q] = c.y;
    }
    // e' of the row before this thread's first row (constant over the step)
    T el0 = __shfl_up_sync(0xffffffffu, e[TILE_EPT - 1], 1);
    if (tl.lane == 0) el0 = i0 > 0 && i0 - 1 < n ? cf[i0 - 1].y : (T)0;
    // b_L = c_L v, b_{L+1} = 0
#pragma unroll
    for (int q = 0; q < TILE_EPT; ++q) {
      A[q] = (L & 1) ? T2{-cL * v[q].y, cL * v[q].x} : T2{cL * v[q].x, cL * v[q].y};
      B[q] = T2{0, 0};
    }
    int k = L - 1;
    // b_k = c_k v + 2 Omega' b_{k+1} - b_{k+2}; two per iteration so the array roles stay static
    while (k >= 2) {
      if (k & 1) tl.template apply<true, false>(A, B, v, d, e, el0, coef.c[k], par);
      else tl.template apply<false, false>(A, B, v, d, e, el0, coef.c[k], par);
      par ^= 1;
      --k;
      if (k & 1) tl.template apply<true, false>(B, A, v, d, e, el0, coef.c[k], par);
      else tl.template apply<false, false>(B, A, v, d, e, el0, coef.c[k], par);
      par ^= 1;
      --k;
    }
    if (k == 1) {  // b_1 into B, then sum = c_0 v + Omega' b_1 - b_2 into A
      tl.template apply<true, false>(A, B, v, d, e, el0, coef.c[1], par);
      par ^= 1;
      tl.template apply<false, true>(B, A, v, d, e, el0, coef.c[0], par);
    } else {  // b_1 in A, b_2 in B: sum into B, then moved to A
      tl.template apply<false, true>(A, B, v, d, e, el0, coef.c[0], par);
#pragma unroll
      for (int q = 0; q < TILE_EPT; ++q) A[q] = B[q];
    }
    par ^= 1;
    // X = D e^{-i beta h} sum on this CTA's own rows
#pragma unroll
    for (int q = 0; q < TILE_EPT; ++q) {
      const int i = i0 + q;
      if (i < rows.first || i >= rows.last) {
        A[q] = T2{0, 0};
        continue;
      }
      const T2 y = T2{fma(ph_re, A[q].x, -(ph_im * A[q].y)), fma(ph_re, A[q].y, ph_im * A[q].x)};
      const T2 r = rot[i];
      A[q] = T2{fma(r.x, y.x, -(r.y * y.y)), fma(r.x, y.y, r.y * y.x)};
      bad |= !(A[q].x * A[q].x + A[q].y * A[q].y <= bound2);
    }
  }
#pragma unroll
  for (int q = 0; q < TILE_EPT; ++q) {
    const int i = i0 + q;
    if (i >= rows.first && i < rows.last) {
      yr[j * ld + i] = A[q].x;
      yi[j * ld + i] = A[q].y;
    }
  }
  if (bad) atomicOr(status, FQ_BIT_BOUND);
}

// ---------------------------------------------------------------------------- double-float
// At most 4 rows a thread and an 80-register cap (a few spills) let three CTAs (24 warps) share an
// SM: the double-float FMA chains are long, and latency, not the FP32 pipe, limits fewer warps.
template <int DFL_EPT>
struct DflTile {
  dflc* slot_last;   // as Tile's
  dflc* slot_first;
  int lane, warp;

  __device__ __forceinline__ DflTile(dflc* slots) {
    const dflc z = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    slot_last = slots;
    slot_first = slots + 2 * TILE_SLOTS;
    lane = threadIdx.x & 31;
    warp = threadIdx.x >> 5;
    if (threadIdx.x < 2) {
      slot_last[threadIdx.x * TILE_SLOTS] = z;
      slot_first[threadIdx.x * TILE_SLOTS + (blockDim.x >> 5)] = z;
    }
  }

  __device__ __forceinline__ static dflc shfl(dflc a, bool up) {
    dflc r;
    if (up) {
      r.h.x = __shfl_up_sync(0xffffffffu, a.h.x, 1);
      r.h.y = __shfl_up_sync(0xffffffffu, a.h.y, 1);
      r.l.x = __shfl_up_sync(0xffffffffu, a.l.x, 1);
      r.l.y = __shfl_up_sync(0xffffffffu, a.l.y, 1);
    } else {
      r.h.x = __shfl_down_sync(0xffffffffu, a.h.x, 1);
      r.h.y = __shfl_down_sync(0xffffffffu, a.h.y, 1);
      r.l.x = __shfl_down_sync(0xffffffffu, a.l.x, 1);
      r.l.y = __shfl_down_sync(0xffffffffu, a.l.y, 1);
    }
    return r;
  }

  __device__ __forceinline__ void halo(const dflc (&x)[DFL_EPT], int par, dflc& left, dflc& right) {
    dflc l = shfl(x[DFL_EPT - 1], true);
    dflc r = shfl(x[0], false);
    if (lane == 31) slot_last[par * TILE_SLOTS + warp + 1] = x[DFL_EPT - 1];
    if (lane == 0) slot_first[par * TILE_SLOTS + warp] = x[0];
    __syncthreads();
    if (lane == 0) l = slot_last[par * TILE_SLOTS + warp];
    if (lane == 31) r = slot_first[par * TILE_SLOTS + warp + 1];
    left = l;
    right = r;
  }

  // out = c v + (2 Omega' x) - out, or with Omega' x (HALF); c = cc or i cc (IM); all double-float
  template <bool IM, bool HALF>
  __device__ __forceinline__ void apply(const dflc (&x)[DFL_EPT], dflc (&out)[DFL_EPT], const dflc (&v)[DFL_EPT],
                                        const dfl (&d)[DFL_EPT], const dfl (&e)[DFL_EPT], dfl el0, dfl cc, int par) {
    dflc left, right;
    halo(x, par, left, right);
#pragma unroll
    for (int q = 0; q < DFL_EPT; ++q) {
      const dflc xm = q == 0 ? left : x[q - 1];
      const dflc xp = q == DFL_EPT - 1 ? right : x[q + 1];
      dfl dq = d[q], el = q == 0 ? el0 : e[q - 1], eh = e[q];
      if (HALF) {  // the closing sum uses Omega' = (stored operator) / 2, halved exactly
        dq = {0.5f * dq.h, 0.5f * dq.l};
        el = {0.5f * el.h, 0.5f * el.l};
        eh = {0.5f * eh.h, 0.5f * eh.l};
      }
      const dflc acc = dflc_fma(dq, x[q], dflc_fma(el, xm, dflc_fma(eh, xp, dflc_neg(out[q]))));
      out[q] = IM ? dflc_ifma(cc, v[q], acc) : dflc_fma(cc, v[q], acc);
    }
  }
};

struct DflCoef {
  dfl c[TILE_MAXL + 1];  // as TileCoef: c_k = c[k] (even k) or i c[k] (odd k)
};

// One step of the double-float tiled chain, or `steps` of them (MULTI: a single segment per state);
// states FP64 planar in HBM, and FP64 between the steps of a launch.
template <int DFL_EPT, bool MULTI>
__global__ void __launch_bounds__(TILE_NT, 3)
k_tri_tile_dfl(const dfl2* __restrict__ cf, const dfl2* __restrict__ rot, const double* __restrict__ xr,
               const double* __restrict__ xi, double* __restrict__ yr, double* __restrict__ yi, int n, int ld, int L,
               TileSpan span, int steps, DflCoef coef, double ph_re, double ph_im, double bound2, unsigned int* status) {
  __shared__ dflc slots[4 * TILE_SLOTS];
  DflTile<DFL_EPT> tl(slots);
  const size_t j = blockIdx.y;
  const TileRows<!MULTI> rows(span, L, n);
  const int i0 = rows.base + (int)threadIdx.x * DFL_EPT;
  const dfl zero = {0.f, 0.f};
  const dflc zc = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  const dfl cL = coef.c[L];
  double o_r[DFL_EPT], o_i[DFL_EPT];  // MULTI: the state between steps
  if (MULTI) {
#pragma unroll
    for (int q = 0; q < DFL_EPT; ++q) {
      const int i = i0 + q;
      o_r[q] = i < n ? xr[j * ld + i] : 0.0;
      o_i[q] = i < n ? xi[j * ld + i] : 0.0;
    }
  }
  bool bad = false;
  int par = 0;
  for (int m = 0; m < (MULTI ? steps : 1); ++m, cf += ld, rot += ld) {
    dflc v[DFL_EPT], A[DFL_EPT], B[DFL_EPT];
    dfl d[DFL_EPT], e[DFL_EPT];
#pragma unroll
    for (int q = 0; q < DFL_EPT; ++q) {
      const int i = i0 + q;
      if ((MULTI || i >= 0) && i < n) {
        const dfl2 r = rot[i], c = cf[i];
        const double rc = dfl_value(r.x), rs = dfl_value(r.y);
        const double x_r = MULTI ? o_r[q] : xr[j * ld + i], x_i = MULTI ? o_i[q] : xi[j * ld + i];
        const dfl vr = dfl_of(fma(rc, x_r, rs * x_i)), vi = dfl_of(fma(rc, x_i, -(rs * x_r)));  // D^+ x
        v[q] = {make_float2(vr.h, vi.h), make_float2(vr.l, vi.l)};
        d[q] = c.x;
        e[q] = c.y;
      } else {
        v[q] = zc;
        d[q] = zero;
        e[q] = zero;
      }
    }
    dfl el0;
    el0.h = __shfl_up_sync(0xffffffffu, e[DFL_EPT - 1].h, 1);
    el0.l = __shfl_up_sync(0xffffffffu, e[DFL_EPT - 1].l, 1);
    if (tl.lane == 0) {
      el0 = zero;
      if (i0 > 0 && i0 - 1 < n) el0 = cf[i0 - 1].y;
    }
    // b_L = c_L v (L odd: i cL v)
#pragma unroll
    for (int q = 0; q < DFL_EPT; ++q) {
      A[q] = (L & 1) ? dflc_ifma(cL, v[q], zc) : dflc_fma(cL, v[q], zc);
      B[q] = zc;
    }
    int k = L - 1;
    while (k >= 2) {
      if (k & 1) tl.template apply<true, false>(A, B, v, d, e, el0, coef.c[k], par);
      else tl.template apply<false, false>(A, B, v, d, e, el0, coef.c[k], par);
      par ^= 1;
      --k;
      if (k & 1) tl.template apply<true, false>(B, A, v, d, e, el0, coef.c[k], par);
      else tl.template apply<false, false>(B, A, v, d, e, el0, coef.c[k], par);
      par ^= 1;
      --k;
    }
    if (k == 1) {
      tl.template apply<true, false>(A, B, v, d, e, el0, coef.c[1], par);
      par ^= 1;
      tl.template apply<false, true>(B, A, v, d, e, el0, coef.c[0], par);
    } else {
      tl.template apply<false, true>(A, B, v, d, e, el0, coef.c[0], par);
#pragma unroll
      for (int q = 0; q < DFL_EPT; ++q) A[q] = B[q];
    }
    par ^= 1;
#pragma unroll
    for (int q = 0; q < DFL_EPT; ++q) {
      const int i = i0 + q;
      if (MULTI) o_r[q] = o_i[q] = 0.0;
      if (i < rows.first || i >= rows.last) continue;  // FP64 arithmetic on this CTA's own rows only
      const double sr = (double)A[q].h.x + (double)A[q].l.x, si = (double)A[q].h.y + (double)A[q].l.y;
      const double y_r = fma(ph_re, sr, -(ph_im * si)), y_i = fma(ph_re, si, ph_im * sr);
      const dfl2 r = rot[i];
      const double rc = dfl_value(r.x), rs = dfl_value(r.y);
      o_r[q] = fma(rc, y_r, -(rs * y_i));
      o_i[q] = fma(rc, y_i, rs * y_r);
      bad |= !(o_r[q] * o_r[q] + o_i[q] * o_i[q] <= bound2);
      if (!MULTI || m == steps - 1) {
        yr[j * ld + i] = o_r[q];
        yi[j * ld + i] = o_i[q];
      }
    }
  }
  if (bad) atomicOr(status, FQ_BIT_BOUND);
}

template <typename T>
void gauge_tables(const fq_plan* p, fq_tables t, void* ws, cudaStream_t s) {
  using T2 = typename V2<T>::t;
  const int ld = (p->n + 3) & ~3;
  GaugeArgs ga{p->n, p->steps, p->d_h0, p->d_h0o, p->d_h1, p->d_k, p->d_scal, p->sbeta};
  k_gauge_tile<T><<<t.n, GAUGE_NT, 0, s>>>(ga, ld, t.m0, (T2*)ws, (T2*)ws + (size_t)t.n * ld);
}

fq_status dfl_chain(fq_plan* p, const double* x0, double* x, int nc, int m_begin, int m_end, int identity,
                    int transpose_out, void* ws, cudaStream_t s, const fq_tables* pre) {
  const int n = p->n, ld = (n + 3) & ~3, nsteps = m_end - m_begin, L = p->L;
  const fq_tables t = pre ? *pre : fq_tables{m_begin, nsteps};
  if (!pre) fq_tile_tables(p, t, ws, s);
  const dfl2* cf = (dfl2*)ws + (size_t)(m_begin - t.m0) * ld;
  const dfl2* rot = cf + (size_t)t.n * ld;
  double* bufs = (double*)((dfl2*)ws + 2 * (size_t)t.n * ld);
  const size_t plane = (size_t)nc * ld;
  fq_blk<double> b[2] = {{bufs, bufs + plane}, {bufs + 2 * plane, bufs + 3 * plane}};
  if (identity) fq_launch_identity_f64(b[0], nc, n, ld, s);
  else fq_launch_load_states(x0, b[0], nc, n, ld, s);
  DflCoef coef{};
  for (int k = 0; k <= L; ++k) {
    const double a = p->cheb[k];
    const double c = (k & 3) == 0 || (k & 3) == 3 ? a : -a;
    const float h = (float)c;
    coef.c[k] = {h, (float)(c - (double)h)};
  }
  const int epts[] = {1, 2, 4};
  TileShape sh = pick_tile(n, nc, L, epts, 0);
  // Four segments: where the CTAs are a few more than a whole number an SM, three segments as long as fit and
  // a short last one (its FP64 rotations are few) spare the SMs that extra CTA.  The lines were drawn on a sweep
  // of 28 lengths from 1051 to 7801 rows and 20 to 600 states: 120 x 3001 82 us a step against 90, 160 x 3001
  // 96 against 103, 230 x 3101 129 against 135; beside these lines, and at other numbers of segments, equal
  // ones take as long or up to 14 % less (320 x 1201).
  const int longest = 4 * TILE_NT - 2 * L;
  const double ctas = (double)nc * sh.segs / fq_sm_count();  // an SM
  if (sh.segs == 4 && n - 3 * longest <= longest / 3 && ctas > 3.0 && ctas < 7.0 && ctas - std::floor(ctas) < 0.27) {
    sh.seg = longest;
    sh.segs = (n + longest - 1) / longest;
    sh.nt = TILE_NT;
  }
  // At four rows a thread the form for one step spills less: it takes over where a launch is long beside its
  // gap, from twenty states an SM on.  Twelve steps in ms, all in one launch / one each, states x rows: 2000 x 516 1.45 /
  // 1.48, 2000 x 801 2.12 / 2.07, 4000 x 516 2.68 / 2.71, 4000 x 801 3.99 / 3.81, 10000 x 601 6.58 / 6.28.
  const bool one = sh.segs > 1 || (sh.ept == 4 && nc > 20 * fq_sm_count());
  const int per = one ? 1 : nsteps;  // steps a launch
  int cur = 0;
  for (int m = 0; m < nsteps; m += per) {
    for (int r0 = 0; r0 < nc; r0 += 65535) {  // gridDim.y limit
      const int rows = nc - r0 < 65535 ? nc - r0 : 65535;
      const size_t o = (size_t)r0 * ld;
      fq_ktimer_start(p, s, "k_tri_tile_dfl");
      const auto kern = one           ? k_tri_tile_dfl<4, false>
                        : sh.ept == 1 ? k_tri_tile_dfl<1, true>
                        : sh.ept == 2 ? k_tri_tile_dfl<2, true>
                                      : k_tri_tile_dfl<4, true>;
      kern<<<dim3(sh.segs, rows), sh.nt, 0, s>>>(cf + (size_t)m * ld, rot + (size_t)m * ld, b[cur].re + o,
                                                 b[cur].im + o, b[cur ^ 1].re + o, b[cur ^ 1].im + o, n, ld, L,
                                                 sh.span(L), per, coef, p->phase_re, p->phase_im, 1.0 + 1e-9, p->d_status);
      fq_ktimer_stop(p, s);
    }
    cur ^= 1;
  }
  if (transpose_out) fq_launch_store_transpose_f64(b[cur], x, n, ld, s);
  else fq_launch_store_states_f64(b[cur], x, nc, n, ld, s);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fq_cuda_fail(e, "double-float tiled chain");
  return FQ_OK;
}

// state load / store helpers of the streaming path, by precision
void load_block(const double* x0, fq_blk<double> b, int nc, int n, int ld, cudaStream_t s) {
  fq_launch_load_states(x0, b, nc, n, ld, s);
}
void load_block(const double* x0, fq_blk<float> b, int nc, int n, int ld, cudaStream_t s) {
  fq_launch_load_states_f32(x0, b, nc, n, ld, s);
}
void identity_block(fq_blk<double> b, int nc, int n, int ld, cudaStream_t s) { fq_launch_identity_f64(b, nc, n, ld, s); }
void identity_block(fq_blk<float> b, int nc, int n, int ld, cudaStream_t s) { fq_launch_identity_f32(b, nc, n, ld, s); }
void store_block(fq_blk<double> b, double* x, int nc, int n, int ld, bool transpose, cudaStream_t s) {
  if (transpose) fq_launch_store_transpose_f64(b, x, n, ld, s);
  else fq_launch_store_states_f64(b, x, nc, n, ld, s);
}
void store_block(fq_blk<float> b, double* x, int nc, int n, int ld, bool transpose, cudaStream_t s) {
  if (transpose) fq_launch_store_transpose_f32(b, x, n, ld, s);
  else fq_launch_store_states_f32(b, x, nc, n, ld, s);
}

template <typename T>
TileCoef<T> tile_coef(const fq_plan* p) {
  TileCoef<T> c{};
  for (int k = 0; k <= p->L; ++k) {
    // c_k = (-i)^k a_k: k % 4 = 0: a, 1: -i a, 2: -a, 3: i a; odd k are stored as the factor of i
    const double a = p->cheb[k];
    c.c[k] = (T)((k & 3) == 0 || (k & 3) == 3 ? a : -a);
  }
  return c;
}

template <typename T>
fq_status tile_chain(fq_plan* p, const double* x0, double* x, int nc, int m_begin, int m_end, int identity,
                     int transpose_out, void* ws, cudaStream_t s, const fq_tables* pre) {
  using T2 = typename V2<T>::t;
  const int n = p->n, ld = (n + 3) & ~3, nsteps = m_end - m_begin, L = p->L;
  const fq_tables t = pre ? *pre : fq_tables{m_begin, nsteps};
  if (!pre) fq_tile_tables(p, t, ws, s);
  const T2* cf = (T2*)ws + (size_t)(m_begin - t.m0) * ld;
  const T2* rot = cf + (size_t)t.n * ld;
  T* bufs = (T*)((T2*)ws + 2 * (size_t)t.n * ld);
  const size_t plane = (size_t)nc * ld;
  fq_blk<T> b[2] = {{bufs, bufs + plane}, {bufs + 2 * plane, bufs + 3 * plane}};
  if (identity) identity_block(b[0], nc, n, ld, s);
  else load_block(x0, b[0], nc, n, ld, s);
  const TileCoef<T> coef = tile_coef<T>(p);
  const T b2 = (T)(1.0 + (sizeof(T) == 8 ? 1e-9 : 2e-3));
  const int epts[] = {2, 4, 8};
  const TileShape sh = pick_tile(n, nc, L, epts, sizeof(T) == 8 ? F64_FLOOR_ROWS : 0);
  const int per = sh.segs == 1 ? nsteps : 1;  // steps a launch
  int cur = 0;
  for (int m = 0; m < nsteps; m += per) {
    for (int r0 = 0; r0 < nc; r0 += 65535) {  // gridDim.y limit
      const int rows = nc - r0 < 65535 ? nc - r0 : 65535;
      const size_t o = (size_t)r0 * ld;
      auto kern = sh.ept == 2 ? k_tri_tile<T, 2, true> : (sh.ept == 4 ? k_tri_tile<T, 4, true> : k_tri_tile<T, 8, true>);
      // FP32 in several segments (8 rows a thread): the form for one step needs 80 registers instead of 115, and
      // three CTAs share an SM instead of two.  Twelve steps of 4000 x 3001 3.07 ms against 3.91 on the form for
      // many steps, 800 x 9001 3.07 against 3.46, 300 x 20001 3.81 against 4.26.
      if constexpr (sizeof(T) == 4)
        if (sh.segs > 1) kern = k_tri_tile<T, 8, false>;
      kern<<<dim3(sh.segs, rows), sh.nt, 0, s>>>(cf + (size_t)m * ld, rot + (size_t)m * ld, b[cur].re + o,
                                                 b[cur].im + o, b[cur ^ 1].re + o, b[cur ^ 1].im + o, n, ld, L,
                                                 sh.span(L), per, coef, (T)p->phase_re, (T)p->phase_im, b2, p->d_status);
    }
    cur ^= 1;
  }
  store_block(b[cur], x, nc, n, ld, transpose_out != 0, s);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fq_cuda_fail(e, "tiled tridiagonal chain");
  return FQ_OK;
}

}  // namespace

int fq_tile_supported(int L) { return L >= 1 && L <= TILE_MAXL; }

size_t fq_tile_workspace(const fq_plan* p, int nc, int nsteps) {
  const size_t ld = (p->n + 3) & ~3;
  if (p->precision == FQ_DF32)  // double-float coefficients (16 B a pair), FP64 states
    return 2 * (size_t)nsteps * ld * sizeof(dfl2) + 4 * (size_t)nc * ld * sizeof(double);
  const size_t es = p->precision == FQ_FP64 ? sizeof(double) : sizeof(float);
  return 2 * (size_t)nsteps * ld * 2 * es + 4 * (size_t)nc * ld * es;
}

void fq_tile_tables(const fq_plan* p, fq_tables t, void* ws, cudaStream_t s) {
  if (p->precision == FQ_FP64) gauge_tables<double>(p, t, ws, s);
  else if (p->precision == FQ_DF32) gauge_tables<dfl>(p, t, ws, s);
  else gauge_tables<float>(p, t, ws, s);
}

fq_status fq_tile_propagate(fq_plan* p, const double* x0, double* x, int nc, int m_begin, int m_end, int identity,
                            int transpose_out, void* ws, cudaStream_t s, const fq_tables* pre) {
  if (p->precision == FQ_FP64)
    return tile_chain<double>(p, x0, x, nc, m_begin, m_end, identity, transpose_out, ws, s, pre);
  if (p->precision == FQ_DF32) return dfl_chain(p, x0, x, nc, m_begin, m_end, identity, transpose_out, ws, s, pre);
  return tile_chain<float>(p, x0, x, nc, m_begin, m_end, identity, transpose_out, ws, s, pre);
}
