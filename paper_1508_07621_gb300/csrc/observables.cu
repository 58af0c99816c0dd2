// Second propagation round (§3, last paragraph; §7): period averages of an observable along the
// chain (and, below, the overlap phase error of Eq. 20),  <A>_T = (1/T) int_0^T <psi(t)|A(t)|psi(t)> dt  (Eq. 17),
// for A(t) = a0 H0 + (a1 + s f(t)) H1 (A = H(t) for a0 = 1, a1 = 0, s = 1), evaluated at the
// step boundaries t_m = m h with composite Simpson weights (trapezoid for odd M).
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "internal.h"

namespace {

__device__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  return s;  // valid in thread 0
}

constexpr int EXPECT_STATES = 4;  // states per CTA (tridiagonal: one where they are few)
constexpr int EXPECT_BLOCK = 32;   // dense: rows of H per CTA
constexpr int EXPECT_WARPS = 8;    // tridiagonal: warps of a CTA
// tridiagonal: up to this many states an SM, a CTA a state (500 x 1001 0.41 ms against 0.37 with four, 400 0.34 either
// way, 300 0.32 against 0.35)
constexpr int EXPECT_SINGLE = 3;

// acc[r] += w <x_r| c0 H0 + c1 H1 |x_r>, tridiagonal H0 (diag, off), diagonal H1:
// sum_i d_i |x_i|^2 + 2 c0 o_i Re(conj(x_i) x_{i+1}), d = c0 diag + c1 H1, for S states a CTA.  Row i goes to lane
// i % 32 of warp (i / 32) % 8; the warps, then the lanes are added pairwise, whatever S is.  Bound by the FP64
// pipes (64 cycles a warp and instruction): 6 instructions an entry, and 4 for d and o, once for the S states.
// (One state per CTA and both neighbours of every entry took 14 instructions; a warp a state, H staged for four of
// them, left most FP64 pipes idle below a thousand states.)  Averages over ten FP32 steps in ms, a warp a state and
// now, states x rows: 30 x 10001 2.06 -> 1.03, 100 x 1001 0.38 -> 0.28, 600 x 1001 0.43 -> 0.37, 1500 x 1001 0.69 ->
// 0.70, 3000 x 301 0.43 -> 0.50 (more states than rows; two rounds of 256 rows for 301).
template <int S>
__global__ void __launch_bounds__(32 * EXPECT_WARPS)
    k_expect_tri(const double2* __restrict__ x, int nc, int n, const double* __restrict__ h0d,
                 const double* __restrict__ h0o, const double* __restrict__ h1d, double c0, double c1, double w,
                 double* acc) {
  __shared__ double part[S][EXPECT_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r0 = blockIdx.x * S;
  double sum[S];
#pragma unroll
  for (int q = 0; q < S; ++q) sum[q] = 0.0;
#pragma unroll(S > 1 ? 2 : 4)
  for (int i = threadIdx.x; i < n; i += 32 * EXPECT_WARPS) {
    const bool right = i + 1 < n;
    const double d = fma(c0, h0d[i], c1 * h1d[i]), o = right ? 2.0 * c0 * h0o[i] : 0.0;
#pragma unroll
    for (int q = 0; q < S; ++q) {
      const double2* row = x + (size_t)min(r0 + q, nc - 1) * n;
      const double2 a = row[i], b = right ? row[i + 1] : make_double2(0.0, 0.0);
      sum[q] = fma(d, fma(a.x, a.x, a.y * a.y), fma(o, fma(a.x, b.x, a.y * b.y), sum[q]));
    }
  }
#pragma unroll
  for (int q = 0; q < S; ++q) part[q][warp][lane] = sum[q];
  __syncthreads();
  if (warp >= S) return;
  double p[EXPECT_WARPS];
#pragma unroll
  for (int u = 0; u < EXPECT_WARPS; ++u) p[u] = part[warp][u][lane];
  double s = ((p[0] + p[1]) + (p[2] + p[3])) + ((p[4] + p[5]) + (p[6] + p[7]));
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0 && r0 + warp < nc) acc[r0 + warp] += w * s;
}

// A = c0 H0 + c1 H1
__global__ void k_expect_form(const double* __restrict__ h0, const double* __restrict__ h1, size_t nn, double c0,
                              double c1, double* __restrict__ a) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < nn; q += (size_t)gridDim.x * blockDim.x)
    a[q] = fma(c0, h0[q], c1 * h1[q]);
}

// acc[b][r] += w times the part of <x_r| A |x_r> (A dense real-symmetric) of the rows of block b: sum over
// its rows i of x_i^* (A_ii x_i + 2 sum_{k < i} A_ik x_k), blockwise, so that only the blocks on and left of
// the diagonal are visited.  Lane = row i, warp = state; the longest rows of blocks start first, and few
// states a CTA balance the rest.  Bound by the FP64 pipes: half of the 2 N^2 multiply-adds a state.  (One
// state per CTA, a thread per row of H walking it, formed A for every state on uncoalesced reads: 151 us
// at N = 256 and 256 states, now 53 us.)
// FORM: A's entries are formed here from H0 and H1 (16 more instructions for a warp's 64 a block), without
// k_expect_form's launch: up to N = 128, where every CTA has an SM to itself.  Averages over ten steps in ms, formed
// before / here: FP64 N = 40 0.41 / 0.38, 128 1.39 / 1.38, BF16X3 64 0.68 / 0.66, 200 1.14 / 1.14, 400 (40 states) 1.29 /
// 1.34, 1000 (16) 2.36 / 2.59: the CTA of the last rows forms all of them.
template <bool FORM>
__global__ void __launch_bounds__(32 * EXPECT_STATES)
    k_expect_dense(const double2* __restrict__ x, int nc, int n, const double* __restrict__ A,
                   const double* __restrict__ h1, double c0, double c1, double w, double* acc) {
  __shared__ double sa[EXPECT_BLOCK][EXPECT_BLOCK + 1];      // [k][i]
  __shared__ double2 sx[EXPECT_STATES][EXPECT_BLOCK];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = gridDim.y - 1 - blockIdx.y, i0 = b * EXPECT_BLOCK;
  const int r = blockIdx.x * EXPECT_STATES + warp;
  double yr = 0.0, yi = 0.0;
  for (int kb = 0; kb <= b; ++kb) {
    const int k0 = kb * EXPECT_BLOCK;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < EXPECT_BLOCK / EXPECT_STATES; ++q) {
      const int ii = warp + EXPECT_STATES * q;
      const size_t at = (size_t)(i0 + ii) * n + k0 + lane;
      double v = 0.0;
      if (i0 + ii < n && k0 + lane < n) v = FORM ? fma(c0, A[at], c1 * h1[at]) : A[at];
      sa[lane][ii] = v;
    }
    sx[warp][lane] = r < nc && k0 + lane < n ? x[(size_t)r * n + k0 + lane] : make_double2(0.0, 0.0);
    __syncthreads();
    if (kb == b) {
      yr += yr;
      yi += yi;
    }
#pragma unroll 8
    for (int kk = 0; kk < EXPECT_BLOCK; ++kk) {
      const double a = sa[kk][lane];
      const double2 v = sx[warp][kk];
      yr = fma(a, v.x, yr);
      yi = fma(a, v.y, yi);
    }
  }
  const double2 v = sx[warp][lane];  // the diagonal block's entries: rows i0 + lane
  double s = fma(v.x, yr, v.y * yi);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0 && r < nc) acc[(size_t)b * nc + r] += w * s;
}

// sigma[r] = |1 - e^{i eps_r T} <phi_r|moved_r>| (Eq. 20, reading R14), one CTA per state row.
__global__ void k_overlap_sigma(const double2* __restrict__ phi, const double2* __restrict__ moved, int n,
                                const double* __restrict__ eps, double period, double* __restrict__ sigma) {
  __shared__ double red[32];
  const double2* a = phi + (size_t)blockIdx.x * n;
  const double2* b = moved + (size_t)blockIdx.x * n;
  double sr = 0.0, si = 0.0;
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const double2 x = a[k], y = b[k];
    sr = fma(x.x, y.x, fma(x.y, y.y, sr));   // Re(conj(x) y)
    si = fma(x.x, y.y, fma(-x.y, y.x, si));  // Im(conj(x) y)
  }
  sr = block_sum(sr, red);
  __syncthreads();
  si = block_sum(si, red);
  if (threadIdx.x == 0) {
    double sn, cs;
    sincos(eps[blockIdx.x] * period, &sn, &cs);
    const double zr = 1.0 - (cs * sr - sn * si), zi = -(cs * si + sn * sr);
    sigma[blockIdx.x] = hypot(zr, zi);
  }
}

// out[r] = s * (sum of the nb blocks' parts)
__global__ void k_scale_out(const double* acc, int nc, int nb, double s, double* out) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nc; q += gridDim.x * blockDim.x) {
    double t = 0.0;
    for (int b = 0; b < nb; ++b) t += acc[(size_t)b * nc + q];
    out[q] = s * t;
  }
}

size_t up256(size_t v) { return (v + 255) & ~(size_t)255; }

// blocks of partial sums per state
int expect_blocks(const fq_plan* p) { return p->format == FQ_DENSE ? (p->n + EXPECT_BLOCK - 1) / EXPECT_BLOCK : 1; }

// the sums, and A of a dense plan
size_t expect_bytes(const fq_plan* p, int32_t ncols) {
  return up256((size_t)ncols * expect_blocks(p) * 8) + (p->format == FQ_DENSE ? up256((size_t)p->n * p->n * 8) : 0);
}

}  // namespace

extern "C" size_t floquet_observable_workspace_size(const fq_plan* p, int32_t ncols) {
  if (!p || ncols < 1) return 0;
  return up256((size_t)ncols * p->n * 16) + expect_bytes(p, ncols) + floquet_workspace_size(p, ncols);
}

static fq_status floquet_average_observable_body(fq_plan* p, const void* d_X0, int32_t ncols, double a0, double a1,
                                                 double s_drive, double* d_avg, void* d_ws, size_t ws_bytes,
                                                 void* stream) {
  if (!p || !d_X0 || !d_avg || ncols < 1) {
    fq_set_error("floquet_average_observable: bad arguments");
    return FQ_EINVAL;
  }
  if (p->drive_kind != FQ_DRIVE_COS) {
    fq_set_error("floquet_average_observable: needs a cosine drive plan");
    return FQ_EUNSUPPORTED;
  }
  if (p->format == FQ_DENSE && p->n > 8192) {
    fq_set_error("floquet_average_observable: dense N <= 8192");
    return FQ_EUNSUPPORTED;
  }
  const size_t need = floquet_observable_workspace_size(p, ncols);
  if (!d_ws || ws_bytes < need || ((uintptr_t)d_ws & 255)) {
    fq_set_error("floquet_average_observable: workspace must be >= %zu bytes, 256-byte aligned", need);
    return FQ_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const int n = p->n, M = p->steps;
  char* b = (char*)d_ws;
  double* X = (double*)b;
  double* acc = (double*)(b + up256((size_t)ncols * n * 16));
  void* inner = b + up256((size_t)ncols * n * 16) + expect_bytes(p, ncols);
  const size_t inner_bytes = ws_bytes - up256((size_t)ncols * n * 16) - expect_bytes(p, ncols);
  const int nb = expect_blocks(p);
  double* A = (double*)((char*)acc + up256((size_t)ncols * nb * 8));  // dense: c0 H0 + c1 H1
  cudaError_t e = cudaMemcpyAsync(X, d_X0, (size_t)ncols * n * 16, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(acc, 0, (size_t)ncols * nb * 8, s);
  if (e != cudaSuccess) return fq_cuda_fail(e, "observable setup");
  const double h = p->h;
  std::vector<double> w(M + 1, h);
  if (M % 2 == 0) {
    for (int m = 1; m < M; ++m) w[m] = (m & 1) ? 4.0 * h / 3.0 : 2.0 * h / 3.0;
    w[0] = w[M] = h / 3.0;
  } else {
    w[0] = w[M] = 0.5 * h;
  }
  auto observe = [&](int m) {
    const double t = m * h;
    const double f = fq_drive_f(0, p->f_dc, p->f_ac, p->omega, p->phi0, t);
    const double c0 = a0, c1 = a1 + s_drive * f;
    const int groups = (ncols + EXPECT_STATES - 1) / EXPECT_STATES;
    if (p->format == FQ_TRIDIAG) {
      const bool single = ncols <= EXPECT_SINGLE * fq_sm_count();
      const auto kern = single ? k_expect_tri<1> : k_expect_tri<EXPECT_STATES>;
      kern<<<single ? ncols : groups, 32 * EXPECT_WARPS, 0, s>>>((const double2*)X, ncols, n, p->d_h0, p->d_h0o, p->d_h1,
                                                                 c0, c1, w[m], acc);
    } else {
      const size_t nn = (size_t)n * n;
      const bool form = nb <= 4 && groups * nb <= fq_sm_count();
      if (!form)
        k_expect_form<<<(int)std::min<size_t>((nn + 255) / 256, 152 * 16), 256, 0, s>>>(p->d_h0, p->d_h1, nn, c0, c1, A);
      const auto kern = form ? k_expect_dense<true> : k_expect_dense<false>;
      kern<<<dim3(groups, nb), 32 * EXPECT_STATES, 0, s>>>((const double2*)X, ncols, n, form ? p->d_h0 : A, p->d_h1, c0, c1,
                                                           w[m], acc);
    }
  };
  // a tridiagonal plan's gauge tables for all steps at once: one CTA forms a step's, for tens of us
  const bool tables = fq_prepare_tables(p, ncols, inner, s);
  observe(0);
  for (int m = 0; m < M; ++m) {
    const fq_status st = tables ? fq_step_with_tables(p, X, X, ncols, m, inner, s)
                                : floquet_propagate(p, X, X, ncols, m, m + 1, inner, inner_bytes, stream);
    if (st != FQ_OK) return st;
    observe(m + 1);
  }
  k_scale_out<<<(ncols + 255) / 256, 256, 0, s>>>(acc, ncols, nb, 1.0 / p->period, d_avg);
  e = cudaGetLastError();
  return e == cudaSuccess ? FQ_OK : fq_cuda_fail(e, "observable kernels");
}

extern "C" fq_status floquet_average_observable(fq_plan* p, const void* d_X0, int32_t ncols, double a0, double a1,
                                                double s_drive, double* d_avg, void* d_ws, size_t ws_bytes,
                                                void* stream) {
  return fq_guard("floquet_average_observable", [&] {
    return floquet_average_observable_body(p, d_X0, ncols, a0, a1, s_drive, d_avg, d_ws, ws_bytes, stream);
  });
}

extern "C" size_t floquet_overlap_workspace_size(const fq_plan* p, int32_t ncols) {
  if (!p || ncols < 1) return 0;
  return up256((size_t)ncols * p->n * 16) + floquet_workspace_size(p, ncols);
}

static fq_status floquet_overlap_phase_error_body(fq_plan* p, const void* d_states, int32_t ncols,
                                                  const double* d_eps, double* d_sigma, void* d_ws, size_t ws_bytes,
                                                  void* stream) {
  if (!p || !d_states || !d_eps || !d_sigma || ncols < 1) {
    fq_set_error("floquet_overlap_phase_error: bad arguments");
    return FQ_EINVAL;
  }
  const size_t need = floquet_overlap_workspace_size(p, ncols);
  if (!d_ws || ws_bytes < need || ((uintptr_t)d_ws & 255)) {
    fq_set_error("floquet_overlap_phase_error: workspace must be >= %zu bytes, 256-byte aligned", need);
    return FQ_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const int n = p->n;
  char* b = (char*)d_ws;
  double* moved = (double*)b;
  const size_t head = up256((size_t)ncols * n * 16);
  // U_T phi~ for every state: the plan's whole chain (step h) on the given rows
  fq_status st = floquet_propagate(p, d_states, moved, ncols, 0, p->steps, b + head, ws_bytes - head, stream);
  if (st != FQ_OK) return st;
  k_overlap_sigma<<<ncols, 256, 0, s>>>((const double2*)d_states, (const double2*)moved, n, d_eps, p->period,
                                        d_sigma);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? FQ_OK : fq_cuda_fail(e, "overlap kernel");
}

extern "C" fq_status floquet_overlap_phase_error(fq_plan* p, const void* d_states, int32_t ncols, const double* d_eps,
                                                 double* d_sigma, void* d_ws, size_t ws_bytes, void* stream) {
  return fq_guard("floquet_overlap_phase_error", [&] {
    return floquet_overlap_phase_error_body(p, d_states, ncols, d_eps, d_sigma, d_ws, ws_bytes, stream);
  });
}
