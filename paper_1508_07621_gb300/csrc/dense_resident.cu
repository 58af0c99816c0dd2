// Resident dense chain for small N (FP64): a cluster of C = ceil(N/16) CTAs carries one state
// through every step of a chunk of the period, with the state on chip the whole time.
//
// The per-term dense path launches one tiled GEMM per Chebyshev term; at N = 64 each of those
// launches keeps only a handful of SMs busy and the chain is 1400 dependent launches long
// (M = 200, L = 7).  Here the independence of the columns of U_T (Algorithm 1 propagates each
// initial state on its own) is used instead: one cluster per state, each CTA owning 16 rows of
// Omega~_m, so 64 states fill the SMs and the whole chunk is one launch.
//
// Per step m (Eqs. 10-12): Phi_0 = X_{m-1}, Phi_1 = -i Omega~ Phi_0,
// Phi_{l+1} = -2i Omega~ Phi_l + Phi_{l-1}, X_m = e^{-i beta h} sum_{l<=L} a_l Phi_l.
//
// FP64 (k_dense_resident).  GB300 runs one FP64 multiply-add every second cycle in each quarter of an
// SM: an FP64 instruction of a warp takes 64 cycles of its quarter however many lanes it uses, so the
// kernel is bound by their number in the busiest warp.  A CTA owns 16 rows and has 4 warps (8 above
// N = 64) that share the values of k; lane (row, parity) holds up to 8 entries of its row of S_m and A_m
// (Omega~_m = S_m + i A_m) in registers, the next step's loaded while this one runs.  A product is at
// most 32 FP64 instructions a warp; the two parities of a row trade partial sums, one keeping Re y and
// one Im y (one addition), and the first warp adds the warps' partials and advances the recurrence of
// 16 complex rows on its 32 lanes (4 instructions at 4 warps).  The state vector Phi_l is kept whole in
// every CTA's shared memory, twice; the first warp writes its new entries into every CTA of the cluster
// (distributed shared memory), one cluster barrier per product publishes them, and the accumulator
// and the bound check follow while it is under way.  (Eight lanes a row with a shuffle reduction and the
// recurrence on every warp's leading lanes, 32 rows a CTA, took as many FP64 instructions again as the
// products themselves.)  A product of all states in us before and now: N = 16 3.3 -> 0.9, 32 3.8 -> 1.4, 48 4.2 -> 2.5,
// 64 4.2 -> 3.1, 100 23 -> 13, 128 31 -> 19.
//
// Omega~_m for the chunk's steps is formed beforehand in HBM (it is L2-resident: 64 steps x
// 2 x N^2 doubles = 4 MB at N = 64) by one batched launch (order 4) or one launch per step
// (order 6).
//
// FQ_DF32 runs the same chain in double-float arithmetic (dfl.cuh) on the FP32 pipes, which
// GB300 runs at many times its FP64 rate: Omega~ is converted once per step to FP32 pairs, the
// state lives in shared memory as packed complex pairs, and the states in HBM stay FP64.  There a
// thread pair (row i, k-group g) holds 8 entries of row i, and the KG threads of a row reduce their
// partial sums by shuffles.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "dfl.cuh"
#include "internal.h"

namespace {

constexpr int DR_ROWS = 16;   // rows of Omega~ per CTA
constexpr int DR_KPT = 8;     // entries of a row per thread
constexpr int DR_MAXW = 8;    // FP64: most warps per CTA
constexpr int DR_MAXN = 128;
constexpr int DR_CHUNK = 64;  // steps per launch
constexpr int DR_MAXL = 128;

struct DrCoef {
  double a[DR_MAXL + 1];
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// the two halves of cluster_sync_all
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

// stores x at the same shared-memory offset as `local` in cluster CTA `rank`
__device__ __forceinline__ void st_cluster_f64(const double* local, unsigned rank, double x) {
  const unsigned la = (unsigned)__cvta_generic_to_shared(local);
  unsigned ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(x) : "memory");
}

// S, A: [nsteps][n][n] (Omega~ of the chunk's steps); x: planar states [nc][n], updated in place.
// C CTAs of W warps per state, warp w on the columns 2 KPT w .. 2 KPT (w + 1).
template <int KPT>
__global__ void __launch_bounds__(32 * DR_MAXW)
    k_dense_resident(const double* __restrict__ S, const double* __restrict__ A, int n, int nsteps, int L, int C,
                     DrCoef cf, double ph_re, double ph_im, double bound2, double* xr, double* xi,
                     unsigned* status) {
  __shared__ double2 phi[2][DR_MAXN];
  __shared__ double part[DR_MAXW][32];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31, W = blockDim.x >> 5;
  const int row = lane & 15, kh = lane >> 4;
  const unsigned rank = C > 1 ? cluster_rank() : 0u;
  const int j = blockIdx.x / C;  // the state this cluster carries
  const int i = (int)rank * DR_ROWS + row;
  for (int q = t; q < 2 * DR_MAXN; q += 32 * W) {
    const int b = q / DR_MAXN, k = q % DR_MAXN;
    phi[b][k] = b == 0 && k < n ? make_double2(xr[(size_t)j * n + k], xi[(size_t)j * n + k]) : make_double2(0.0, 0.0);
  }
  __syncthreads();
  if (C > 1) cluster_sync_all();  // every CTA of the cluster is running before remote stores
  const size_t nn = (size_t)n * n;
  double s[KPT], a[KPT], sn[KPT], an[KPT];  // this step's entries and the next one's
  auto load = [&](int m, double (&ls)[KPT], double (&la)[KPT]) {
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      const int k = 2 * KPT * warp + 2 * q + kh;  // the parities interleave: no bank conflict on phi
      const bool ok = m < nsteps && i < n && k < n;
      ls[q] = ok ? S[m * nn + (size_t)i * n + k] : 0.0;
      la[q] = ok ? A[m * nn + (size_t)i * n + k] : 0.0;
    }
  };
  load(0, sn, an);
  // first warp: lanes with kh = 0 sum Re y and carry the imaginary component of row i, the others
  // the reverse (Phi_{l+1} = -2i y + Phi_{l-1})
  double acc = 0.0, pv = 0.0;
  int buf = 0;
  bool bad = false;
  for (int m = 0; m < nsteps; ++m) {
#pragma unroll
    for (int q = 0; q < KPT; ++q) {
      s[q] = sn[q];
      a[q] = an[q];
    }
    load(m + 1, sn, an);
    for (int l = 0; l < L; ++l) {
      const double2* v = phi[buf] + 2 * KPT * warp + kh;
      double yr = 0.0, yi = 0.0;
#pragma unroll
      for (int q = 0; q < KPT; ++q) {
        const double2 p = v[2 * q];
        yr = fma(s[q], p.x, fma(-a[q], p.y, yr));
        yi = fma(s[q], p.y, fma(a[q], p.x, yi));
      }
      const double other = __shfl_xor_sync(0xffffffffu, kh ? yr : yi, 16);
      double y = (kh ? yi : yr) + other;
      if (warp > 0) part[warp][lane] = y;
      __syncthreads();
      if (warp == 0) {
        // the warps' partials (W is 4 or 8), added pairwise
        const double y1 = part[2][lane] + part[3][lane];
        y += part[1][lane];
        if (W > 4) {
          y += part[4][lane] + part[5][lane];
          y += y1 + (part[6][lane] + part[7][lane]);
        } else {
          y += y1;
        }
        const double2 pc = phi[buf][i < n ? i : 0];
        const double cur = kh ? pc.x : pc.y;
        const double sy = kh ? y : -y;  // Phi_1 = -i y
        double nx = l == 0 ? sy : fma(2.0, sy, pv);
        const double psi = nx;
        auto accumulate = [&] { acc = fma(cf.a[l + 1], psi, l == 0 ? cf.a[0] * cur : acc); };
        if (l == L - 1) {  // X_m = e^{-i beta h} acc
          accumulate();
          const double ao = __shfl_xor_sync(0xffffffffu, acc, 16);
          nx = fma(ph_re, acc, (kh ? -ph_im : ph_im) * ao);
        }
        if (i < n) {
          double* dst = kh ? &phi[buf ^ 1][i].x : &phi[buf ^ 1][i].y;
          if (C > 1) {
            for (int c = 0; c < C; ++c) st_cluster_f64(dst, (unsigned)c, nx);
          } else {
            *dst = nx;
          }
        }
        __syncwarp();
        if (C > 1) cluster_arrive();
        // what the peers do not wait for
        pv = cur;
        if (l < L - 1) accumulate();
        // |T_l(Omega~) x| <= |x| inside the bounds; components below 2^-1/2 need no arithmetic
        if (__any_sync(0xffffffffu, (__double2hiint(psi) & 0x7FFFFFFF) >= 0x3FE6A09E)) {
          const double co = __shfl_xor_sync(0xffffffffu, psi, 16);
          bad |= i < n && !(psi * psi + co * co <= bound2);
        }
      } else if (C > 1) {
        cluster_arrive();
      }
      __syncwarp();
      if (C > 1) cluster_wait();
      else __syncthreads();
      buf ^= 1;
    }
  }
  if (warp == 0 && i < n) {
    if (kh) xr[(size_t)j * n + i] = phi[buf][i].x;
    else xi[(size_t)j * n + i] = phi[buf][i].y;
  }
  if (bad) atomicOr(status, FQ_BIT_BOUND);
  __syncwarp();
  if (C > 1) cluster_sync_all();  // no CTA leaves while a peer could still address its memory
}

__device__ __forceinline__ void st_cluster_f32x4(const void* local, unsigned rank, float4 v) {
  const unsigned la = (unsigned)__cvta_generic_to_shared(local);
  unsigned ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(la), "r"(rank));
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(ra), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}

__device__ __forceinline__ dflc dflc_shfl_xor(dflc a, int o) {
  return {make_float2(__shfl_xor_sync(0xffffffffu, a.h.x, o), __shfl_xor_sync(0xffffffffu, a.h.y, o)),
          make_float2(__shfl_xor_sync(0xffffffffu, a.l.x, o), __shfl_xor_sync(0xffffffffu, a.l.y, o))};
}

// The chain of k_dense_resident in double-float arithmetic: S, A as FP32 pairs [nsteps][n][n]
// (float2 = (hi, lo)), the state as packed complex pairs in shared memory.
template <int ROWS, int KG>
__global__ void __launch_bounds__(ROWS* KG)
    k_dense_resident_dfl(const float2* __restrict__ S, const float2* __restrict__ A, int n, int nsteps, int L, int C,
                         DrCoef cf, double ph_re, double ph_im, double bound2, double* xr, double* xi,
                         unsigned* status) {
  constexpr int NT = ROWS * KG;
  constexpr int NV = KG * DR_KPT;
  __shared__ dflc phi[2][NV];
  const int t = threadIdx.x, rl = t / KG, g = t % KG;
  const unsigned rank = C > 1 ? cluster_rank() : 0u;
  const int j = blockIdx.x / C;
  const int i = (int)rank * ROWS + rl;
  const bool own = g == 0 && i < n;
  const dflc zc = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  for (int q = t; q < 2 * NV; q += NT) {
    const int b = q / NV, k = q % NV;
    dflc v = zc;
    if (b == 0 && k < n) {
      const dfl r = dfl_of(xr[(size_t)j * n + k]), m = dfl_of(xi[(size_t)j * n + k]);
      v = {make_float2(r.h, m.h), make_float2(r.l, m.l)};
    }
    phi[b][k] = v;
  }
  __syncthreads();
  if (C > 1) cluster_sync_all();
  const size_t nn = (size_t)n * n;
  const dfl ph_c = dfl_of(ph_re), ph_s = dfl_of(ph_im);
  int buf = 0;
  bool bad = false;
  for (int m = 0; m < nsteps; ++m) {
    dfl s[DR_KPT], a[DR_KPT];
#pragma unroll
    for (int q = 0; q < DR_KPT; ++q) {
      const int k = g + KG * q;
      const bool ok = i < n && k < n;
      const float2 sv = ok ? S[m * nn + (size_t)i * n + k] : make_float2(0.f, 0.f);
      const float2 av = ok ? A[m * nn + (size_t)i * n + k] : make_float2(0.f, 0.f);
      s[q] = dfl{sv.x, sv.y};
      a[q] = dfl{av.x, av.y};
    }
    dflc acc = zc, pv = zc;
    for (int l = 0; l < L; ++l) {
      dflc ys = zc, ya = zc;  // S phi and i A phi, two independent chains
#pragma unroll
      for (int q = 0; q < DR_KPT; ++q) {
        const dflc v = phi[buf][g + KG * q];
        ys = dflc_fma(s[q], v, ys);
        ya = dflc_ifma2(a[q], v, ya);
      }
      dflc y = dflc_add(ys, ya);
#pragma unroll
      for (int o = KG / 2; o > 0; o >>= 1) y = dflc_add(y, dflc_shfl_xor(y, o));
      if (own) {
        const dflc cur = phi[buf][i];
        // -i y (first product) or -2i y + phi_{l-1}: (y_im, -y_re) scaled exactly
        const float sc = l == 0 ? 1.f : 2.f;
        const dflc my = {make_float2(sc * y.h.y, -sc * y.h.x), make_float2(sc * y.l.y, -sc * y.l.x)};
        const dflc nx = l == 0 ? my : dflc_add(my, pv);
        const dfl al = dfl_of(cf.a[l + 1]);
        acc = l == 0 ? dflc_fma(al, nx, dflc_fma(dfl_of(cf.a[0]), cur, zc)) : dflc_fma(al, nx, acc);
        pv = cur;
        const double nr = (double)nx.h.x + (double)nx.l.x, ni = (double)nx.h.y + (double)nx.l.y;
        bad |= !(nr * nr + ni * ni <= bound2);
        dflc out = nx;
        if (l == L - 1) out = dflc_ifma2(ph_s, acc, dflc_fma(ph_c, acc, zc));  // (ph_re + i ph_im) acc
        const float4 w = make_float4(out.h.x, out.h.y, out.l.x, out.l.y);
        if (C > 1) {
          for (int c = 0; c < C; ++c) st_cluster_f32x4(&phi[buf ^ 1][i], (unsigned)c, w);
        } else {
          phi[buf ^ 1][i] = out;
        }
      }
      if (C > 1) cluster_sync_all();
      else __syncthreads();
      buf ^= 1;
    }
  }
  if (own) {
    const dflc v = phi[buf][i];
    xr[(size_t)j * n + i] = (double)v.h.x + (double)v.l.x;
    xi[(size_t)j * n + i] = (double)v.h.y + (double)v.l.y;
  }
  if (bad) atomicOr(status, FQ_BIT_BOUND);
  if (C > 1) cluster_sync_all();
}

// S, A of a chunk as FP32 pairs
__global__ void k_to_dfl(const double* __restrict__ S, const double* __restrict__ A, size_t count, float2* Sd,
                         float2* Ad) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < count; q += (size_t)gridDim.x * blockDim.x) {
    const dfl s = dfl_of(S[q]), a = dfl_of(A[q]);
    Sd[q] = make_float2(s.h, s.l);
    Ad[q] = make_float2(a.h, a.l);
  }
}

// Omega~ of steps m0 .. m0+nsteps-1 (order 4, Eq. 11 on Omega_m/h): S = sa H0 + sb H1 - sbeta 1,
// A = sc [H0,H1], scalars from the plan's device copy (sa | sb | sc, M each).
__global__ void k_omega_dense_steps(const double* __restrict__ h0, const double* __restrict__ h1,
                                    const double* __restrict__ k, int n, const double* __restrict__ scal, int M,
                                    int m0, int nsteps, double sbeta, double* S, double* A) {
  const size_t nn = (size_t)n * n, total = nn * nsteps;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < total; q += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(q / nn);
    const size_t e = q % nn;
    const int i = (int)(e / n), jj = (int)(e % n);
    const double sa = scal[m0 + m], sb = scal[M + m0 + m], sc = scal[2 * M + m0 + m];
    S[q] = sa * h0[e] + sb * h1[e] - (i == jj ? sbeta : 0.0);
    A[q] = sc * k[e];
  }
}

// FP64: KG = 0 (the warps share the values of k); double-float: KG threads per row
template <int ROWS, int KG>
cudaError_t launch_resident(const fq_plan* p, const double* S, const double* A, const float2* Sd, const float2* Ad,
                            int nsteps, double* xr, double* xi, int nc, cudaStream_t s) {
  const int C = (p->n + ROWS - 1) / ROWS;
  DrCoef cf{};
  for (int l = 0; l <= p->L; ++l) cf.a[l] = p->cheb[l];
  const double bound2 = 1.0 + 1e-9;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(nc * C));
  const int W = p->n <= 64 ? 4 : DR_MAXW;  // FP64: warps
  cfg.blockDim = dim3(KG ? ROWS * KG : 32 * W);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  if (C > 1) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
  if constexpr (KG > 0)
    return cudaLaunchKernelEx(&cfg, k_dense_resident_dfl<ROWS, KG>, (const float2*)Sd, (const float2*)Ad, p->n, nsteps,
                              p->L, C, cf, p->phase_re, p->phase_im, bound2, xr, xi, p->d_status);
  const int need = (p->n + 2 * W - 1) / (2 * W);  // entries a lane
  static constexpr decltype(&k_dense_resident<1>) kerns[DR_KPT] = {
      k_dense_resident<1>, k_dense_resident<2>, k_dense_resident<3>, k_dense_resident<4>,
      k_dense_resident<5>, k_dense_resident<6>, k_dense_resident<7>, k_dense_resident<8>};
  const auto kern = kerns[need - 1];
  return cudaLaunchKernelEx(&cfg, kern, S, A, p->n, nsteps, p->L, C, cf, p->phase_re,
                            p->phase_im, bound2, xr, xi, p->d_status);
}

}  // namespace

bool fq_dense_resident_supported(int n, int L) { return n >= 1 && n <= DR_MAXN && L >= 1 && L <= DR_MAXL; }

size_t fq_dense_resident_omega_count(int n, int nsteps) {
  // FP64 S (or A) of a chunk, and room for its FP32-pair copy (FQ_DF32) after it
  return 2 * (size_t)std::min(nsteps, DR_CHUNK) * n * n;
}

fq_status fq_dense_resident_chain(const fq_plan* p, double* xr, double* xi, int nc, int m_begin, int m_end,
                                  double* S, double* A, cudaStream_t s) {
  const int n = p->n;
  const size_t nn = (size_t)n * n;
  for (int m0 = m_begin; m0 < m_end; m0 += DR_CHUNK) {
    const int cnt = std::min(DR_CHUNK, m_end - m0);
    if (p->order == 6) {
      const double inv = 1.0 / (p->h * p->delta_e);
      for (int m = 0; m < cnt; ++m) {
        double c[FQ_M6_TERMS];
        for (int q = 0; q < FQ_M6_TERMS; ++q) c[q] = p->coef6[(size_t)(m0 + m) * FQ_M6_TERMS + q] * inv;
        fq_launch_omega6_f64(p, c, S + m * nn, A + m * nn, s);
      }
    } else {
      const size_t total = nn * cnt;
      const int grid = (int)std::min<size_t>((total + 255) / 256, 152 * 16);
      k_omega_dense_steps<<<grid, 256, 0, s>>>(p->d_h0, p->d_h1, p->d_k, n, p->d_scal, p->steps, m0, cnt, p->sbeta,
                                               S, A);
    }
    // FQ_DF32: FP32-pair copies in the second half of each region
    const size_t cap = (size_t)std::min(m_end - m_begin, DR_CHUNK);  // chunk size the regions were sized for
    float2* Sd = reinterpret_cast<float2*>(S + cap * nn);
    float2* Ad = reinterpret_cast<float2*>(A + cap * nn);
    if (p->precision == FQ_DF32) {
      const size_t total = nn * cnt;
      k_to_dfl<<<(int)std::min<size_t>((total + 255) / 256, 152 * 16), 256, 0, s>>>(S, A, total, Sd, Ad);
    }
    // double-float: CTAs of 16 rows, a cluster of up to eight per state (the products are cheap
    // on the FP32 pipes; more SMs share each product)
    cudaError_t e;
    if (p->precision == FQ_DF32 && n <= 64) e = launch_resident<16, 8>(p, S, A, Sd, Ad, cnt, xr, xi, nc, s);
    else if (p->precision == FQ_DF32) e = launch_resident<16, 16>(p, S, A, Sd, Ad, cnt, xr, xi, nc, s);
    else e = launch_resident<DR_ROWS, 0>(p, S, A, Sd, Ad, cnt, xr, xi, nc, s);
    if (e != cudaSuccess) return fq_cuda_fail(e, "dense resident chain");
  }
  return FQ_OK;
}
