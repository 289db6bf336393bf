// pcg.cu -- multigrid-preconditioned conjugate gradients on one level (the
// paper names multigrid as the preconditioner of a CG solve, App. D.2).
//
// Flexible (Polak-Ribiere) CG, because a V-cycle that smooths red first in
// both legs is not exactly symmetric:
//   r0 = f - L phi0 (true residual, Dirichlet ghosts); z = M r; p = z (first)
//   loop: q = L0 p; alpha = (r, z) / (p, q); phi += alpha p; r' = r - alpha q;
//         stop on ||r'||; z' = M r'; beta = (z', r' - r) / (z, r); p = z' + beta p
// (r' - r = -alpha q, so the numerator is formed as -alpha (z', q) and the old
// residual is never stored)
// M = one V-cycle from zero with homogeneous coarse-fine values (the level's
// own V-cycle, reading its right-hand side array, which holds r during the
// iteration), or in mixed precision inner_cycles FP32 V-cycles on r / s scaled
// back by s, the power of two of ||r||'s binade (flexible CG tolerates the
// inexact FP32 solve);
// L0 = the operator with homogeneous coarse-fine values.  On a
// periodic level z is projected to zero mean (the operator's null space).
// Everything is FP64 and in the solver's pre-scaled units (d = -h^2 r / 6;
// the iteration is invariant to that scale); r lives in the level's
// right-hand side array, saved at set-up and restored at wrap-up.  Dot products are per-block
// partial sums reduced in a fixed order (deterministic), alpha and beta are
// formed on the device, and the iteration runs as the set-up / body /
// wrap-up segments of the level solve's CUDA graph (solve.cu): the residual
// norm goes to the same control block as the stationary iteration's.
#include <cmath>

#include "cmg_internal.cuh"
#include "oct_ops.cuh"

namespace cmg {
namespace {

constexpr int kPcgThreads = 256;

template <int THREADS>
__device__ __forceinline__ void block_partial(double v, double *part) {
  __shared__ double ws[THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double s = threadIdx.x < THREADS / 32 ? ws[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
  }
}

// The kernels below run per oct, per plane of an oct (two threads) or, on
// small levels, with four threads of two cells per oct; every block covers
// 256 octs and leaves one partial sum.
//
// GB300 issues an FP64 warp instruction about every 64 clocks per SM
// sub-partition, so their count is what these kernels are written for.  The
// direction and q = L0 p are two kernels: with the neighbours' p formed on the
// fly (z + beta p_old, twelve values a cell) an oct took 120 FP64
// instructions and 112 loads; now 8, then 16 with the neighbours summed in
// integers, for 192 bytes more traffic.
constexpr int kPlaneThreads = 2 * kPcgThreads, kCellThreads4 = 4 * kPcgThreads;

// r = g + nbsum(phi) / 6 - phi (phi's ghost octs hold the Dirichlet values),
// in place in the right-hand side array g (plane stride 4 n), which holds r
// for the rest of the iteration; partial sums of r^2
__global__ void __launch_bounds__(kPcgThreads) k_pcg_resid(const int32_t *__restrict__ nbr,
                                                          const double *__restrict__ phi, double *__restrict__ g,
                                                          int64_t n, int64_t n_alloc, double *__restrict__ part) {
  pdl_enter();
  double acc = 0.0;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) {
    double pv[2][4], qv[2][4], gv[4];
    dev::apply_oct<false>(i, nbr, phi, n, n_alloc, pv, qv);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      dev::load4<false>(g + (p * n + i) * 4, gv);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        gv[q] -= qv[p][q];
        acc = fma(gv[q], gv[q], acc);
      }
      dev::store4(g + (p * n + i) * 4, gv);
    }
  }
  block_partial<kPcgThreads>(acc, part);
}

// the oct and plane of a thread of a per-plane kernel
__device__ __forceinline__ int64_t plane_at(int64_t n, int &p) {
  p = threadIdx.x >= kPcgThreads;
  return blockIdx.x * (int64_t)kPcgThreads + (threadIdx.x & (kPcgThreads - 1));
}

// p = z + beta p on the real octs (p is zero on the ghost and zero octs)
__global__ void __launch_bounds__(kPlaneThreads) k_pcg_dir(const double *__restrict__ z, double *__restrict__ dir,
                                                          int64_t n, int64_t n_alloc, const double *__restrict__ sc) {
  pdl_enter();
  int p;
  const int64_t i = plane_at(n, p);
  if (i >= n) return;
  const int64_t k = (p * n_alloc + i) * 4;
  const double b = sc[3];
  double pv[4], zv[4];
  dev::load4<false>(dir + k, pv);
  dev::load4<false>(z + k, zv);
#pragma unroll
  for (int q = 0; q < 4; ++q) pv[q] = fma(b, pv[q], zv[q]);
  dev::store4(dir + k, pv);
}

// q = L0 p = p - nbsum(p) / 6; partial (p, q)
__global__ void __launch_bounds__(kPcgThreads) k_pcg_apply(const int32_t *__restrict__ nbr,
                                                          const double *__restrict__ dir, int64_t n, int64_t n_alloc,
                                                          double *__restrict__ q, double *__restrict__ part) {
  pdl_enter();
  double acc = 0.0;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) {
    double pv[2][4], qv[2][4];
    dev::apply_oct<false>(i, nbr, dir, n, n_alloc, pv, qv);
#pragma unroll
    for (int p = 0; p < 2; ++p) {
#pragma unroll
      for (int k = 0; k < 4; ++k) acc = fma(pv[p][k], qv[p][k], acc);
      dev::store4(q + (p * n_alloc + i) * 4, qv[p]);
    }
  }
  block_partial<kPcgThreads>(acc, part);
}
__global__ void __launch_bounds__(kCellThreads4) k_pcg_apply_cell(const int32_t *__restrict__ nbr,
                                                                 const double *__restrict__ dir, int64_t n,
                                                                 int64_t n_alloc, double *__restrict__ q,
                                                                 double *__restrict__ part) {
  pdl_enter();
  double acc = 0.0;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, i = t >> 2;
  if (i < n) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      double pv, qv;
      dev::apply_cell(i, plane_cell(p, (int)(t & 3)), nbr, dir, n, n_alloc, pv, qv);
      acc = fma(pv, qv, acc);
      q[(p * n_alloc + i) * 4 + (t & 3)] = qv;
    }
  }
  block_partial<kCellThreads4>(acc, part);
}

// x += alpha p; r -= alpha q (r in the right-hand side array); partial (r, r)
__global__ void __launch_bounds__(kPlaneThreads) k_pcg_step(double *__restrict__ x, const double *__restrict__ dir,
                                                           double *__restrict__ r, const double *__restrict__ q,
                                                           int64_t n, int64_t n_alloc, const double *__restrict__ sc,
                                                           double *__restrict__ part) {
  pdl_enter();
  double acc = 0.0;
  int p;
  const int64_t i = plane_at(n, p);
  if (i < n) {
    const double a = sc[5];
    const int64_t k = (p * n_alloc + i) * 4, gk = (p * n + i) * 4;
    double xv[4], pv[4], rv[4], qv[4];
    dev::load4<false>(x + k, xv);
    dev::load4<false>(dir + k, pv);
    dev::load4<false>(r + gk, rv);
    dev::load4<false>(q + k, qv);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      xv[j] = fma(a, pv[j], xv[j]);
      rv[j] = fma(-a, qv[j], rv[j]);
      acc = fma(rv[j], rv[j], acc);
    }
    dev::store4(x + k, xv);
    dev::store4(r + gk, rv);
  }
  block_partial<kPlaneThreads>(acc, part);
}

// partial (z, r) into part[b], (z, q) into part[nb + b]; q is the previous
// iteration's L0 p, so that r' - r = -alpha q
__global__ void __launch_bounds__(kPlaneThreads) k_pcg_dots(const double *__restrict__ z, const double *__restrict__ r,
                                                           const double *__restrict__ q, int64_t n, int64_t n_alloc,
                                                           double *__restrict__ part) {
  pdl_enter();
  double a = 0.0, b = 0.0;
  int p;
  const int64_t i = plane_at(n, p);
  if (i < n) {
    const int64_t k = (p * n_alloc + i) * 4;
    double zv[4], rv[4], qv[4];
    dev::load4<false>(z + k, zv);
    dev::load4<false>(r + (p * n + i) * 4, rv);
    dev::load4<false>(q + k, qv);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      a = fma(zv[j], rv[j], a);
      b = fma(zv[j], qv[j], b);
    }
  }
  block_partial<kPlaneThreads>(a, part);
  __syncthreads();
  block_partial<kPlaneThreads>(b, part + gridDim.x);
}

// sum of part[0..np) in a fixed order, on all threads of a one-block launch
__device__ double block_sum(const double *__restrict__ part, int np) {
  __shared__ double ws[32];
  __shared__ double total;
  double v = 0.0;
  for (int t = threadIdx.x; t < np; t += blockDim.x) v += part[t];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double s = threadIdx.x < (blockDim.x >> 5) ? ws[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) total = s;
  }
  __syncthreads();
  const double r = total;
  __syncthreads();
  return r;
}

// Scalars: sc[0] (z, r), sc[1] (z, q), sc[2] (z, r) of the last beta, sc[3]
// beta, sc[4] (p, q), sc[5] alpha, sc[6] (r, r), sc[7] first-iteration flag,
// sc[8] the FP32 right-hand side's scale.  The reductions finish into them:
enum { FIN_BETA, FIN_ALPHA, FIN_NORM, FIN_NORM_FIRST };

// beta = (z', r' - r) / (z, r) = -alpha (z', q) / (z, r) (Polak-Ribiere; 0 on
// the first iteration); alpha = (z, r) / (p, q); ||r||^2 to the solve control
// in source units (and, at set-up, the first-iteration flag)
template <int MODE>
__global__ void k_pcg_fin(const double *__restrict__ part, int np, double *sc, double d2f, double *scal2) {
  pdl_enter();
  const double a = block_sum(part, np);
  if (MODE == FIN_BETA) {
    const double b = block_sum(part + np, np);
    if (threadIdx.x == 0) {
      sc[0] = a;
      sc[1] = b;
      sc[3] = sc[7] != 0.0 ? 0.0 : -sc[5] * b / sc[2];
      sc[2] = a;
      sc[7] = 0.0;
    }
  } else if (threadIdx.x == 0) {
    if (MODE == FIN_ALPHA) {
      sc[4] = a;
      sc[5] = sc[2] / a;
    } else {
      sc[6] = a;
      sc[8] = dev::pow2_scale(sqrt(a));
      *scal2 = a * d2f;
      if (MODE == FIN_NORM_FIRST) sc[7] = 1.0;
    }
  }
}

// FP32 right-hand side of the mixed-precision preconditioner: r / s, s the
// power of two of ||r||'s binade (sc[8]), g layout [2][n][4]
__global__ void k_pcg_emit32(const double *__restrict__ r, int64_t n, const double *__restrict__ sc,
                             float *__restrict__ g32) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= 2 * n) return;
  const double inv = dev::inv_scale(sc[8]);
  double v[4];
  float w[4];
  dev::load4<false>(r + t * 4, v);
#pragma unroll
  for (int q = 0; q < 4; ++q) w[q] = dev::f32_scaled(v[q], inv);
  dev::store4(g32 + t * 4, w);
}

// z = s e in phi (real octs; FP64) from the FP32 correction e
__global__ void k_pcg_z64(const float *__restrict__ e, int64_t n, int64_t n_alloc, const double *__restrict__ sc,
                          double *__restrict__ z) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= 2 * n) return;
  const int p = t >= n ? 1 : 0;
  const int64_t k = (p * n_alloc + t - p * n) * 4;
  const double s = sc[8];
  float w[4];
  double v[4];
  dev::load4<false>(e + k, w);
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = s * dev::widen(w[q]);
  dev::store4(z + k, v);
}

struct PcgView {
  double *x, *p, *q, *gsave, *part, *sc;
  int64_t n, na, ps, nv;
  unsigned nb;
};

PcgView view(cmg_level *L) {
  MgLev &g = L->mg[0];
  PcgView v;
  v.n = g.n;
  v.na = g.n_alloc;
  v.ps = g.n_alloc * 4;
  v.nv = 8 * g.n_alloc;
  v.nb = blocks_for(g.n, kPcgThreads);
  v.x = L->pcg;
  v.p = v.x + v.nv;
  v.q = v.p + v.nv;
  v.gsave = v.q + v.nv;
  v.part = v.gsave + v.nv;
  v.sc = v.part + 2 * v.nb;
  return v;
}

double d2f_of(const cmg_level *L) {
  const double h = L->mg[0].h;
  return 36.0 / (h * h * h * h);  // squared pre-scaled norms -> source units
}

constexpr int kFinThreads = 1024;

}  // namespace

void pcg_prepare(cmg_level *L) {
  if (L->pcg) return;
  MgLev &g = L->mg[0];
  const int64_t nv = 8 * g.n_alloc;
  const unsigned nb = blocks_for(g.n, kPcgThreads);
  // x, direction, q, saved right-hand side; partials; scalars (zeroed, so
  // that q and the direction start finite)
  L->pcg = L->mem.alloc<double>(4 * nv + 2 * (int64_t)nb + 16, true, L->ctx->stream);
  CMG_CUDA(cudaStreamSynchronize(L->ctx->stream));
}

// Set-up (inside the solve graph): ghosts, ||f - L 0||^2 into scal[0], the
// true residual r0 in place of the right-hand side (the first right-hand side
// of the preconditioner) with ||r0||^2 into scal[2], x = phi, p = 0, ghost
// octs of phi cleared.
void pcg_pre(cmg_level *L) {
  MgLev &g = L->mg[0];
  cudaStream_t s = L->ctx->stream;
  const PcgView v = view(L);
  fill_ghosts(L);
  zero_phi_norm(L, L->scal + 0);
  CMG_CUDA(cudaMemcpyAsync(v.gsave, g.g, sizeof(double) * 8 * v.n, cudaMemcpyDeviceToDevice, s));
  CMG_CUDA(cudaMemcpyAsync(v.x, g.phi, sizeof(double) * v.nv, cudaMemcpyDeviceToDevice, s));
  CMG_CUDA(cudaMemsetAsync(v.p, 0, sizeof(double) * v.nv, s));
  {
    LaunchScope ls(L->ctx, K_RESID64, 8.0 * v.n * 24.0, 8.0 * v.n * 9.0);
    launch_k(k_pcg_resid, v.nb, kPcgThreads, s, g.nbr, g.phi, g.g, v.n, v.na, v.part);
  }
  {
    LaunchScope ls(L->ctx, K_REDUCE, 8.0 * v.nb, v.nb);
    launch_k(k_pcg_fin<FIN_NORM_FIRST>, 1, kFinThreads, s, v.part, (int)v.nb, v.sc, d2f_of(L), L->scal + 2);
  }
  // corrections see zero coarse-fine values: clear the ghost octs of phi
  if (g.n_alloc > v.n) {
    CMG_CUDA(cudaMemsetAsync(g.phi + 4 * v.n, 0, sizeof(double) * 4 * (g.n_alloc - v.n), s));
    CMG_CUDA(cudaMemsetAsync(g.phi + v.ps + 4 * v.n, 0, sizeof(double) * 4 * (g.n_alloc - v.n), s));
  }
  CMG_CUDA(cudaGetLastError());
}

// One CG iteration: z = M r (V-cycle), beta, p and q = L0 p, alpha, x and r
// updates; ||r||^2 into scal[2] for the control's check.
void pcg_body(cmg_level *L, const cmg_solve_params *p, int64_t *updates) {
  MgLev &g = L->mg[0];
  cudaStream_t s = L->ctx->stream;
  const PcgView v = view(L);
  int64_t upc = 0;
  if (p->precision == CMG_PREC_MIXED) {
    // z = s e, e = FP32 V-cycles on r / s (FP32 right-hand side)
    {
      LaunchScope ls(L->ctx, K_CONVERT, 8.0 * v.n * 12.0, 8.0 * v.n);
      launch_k(k_pcg_emit32, blocks_for(2 * v.n), kThreads, s, g.g, v.n, v.sc, g.g32);
    }
    vcycle32_from_zero(L, p, &upc);
    {
      LaunchScope ls(L->ctx, K_CONVERT, 8.0 * v.n * 12.0, 8.0 * v.n);
      launch_k(k_pcg_z64, blocks_for(2 * v.n), kThreads, s, g.phi32, v.n, v.na, v.sc, g.phi);
    }
  } else {
    vcycle64_from_zero(L, p, &upc);  // z = M r in phi
  }
  *updates += upc;
  if (L->periodic_full) subtract_mean(L);
  {
    LaunchScope ls(L->ctx, K_REDUCE, 8.0 * v.n * 24.0, 8.0 * v.n * 4.0);
    launch_k(k_pcg_dots, v.nb, kPlaneThreads, s, g.phi, g.g, v.q, v.n, v.na, v.part);
  }
  {
    LaunchScope ls(L->ctx, K_REDUCE, 16.0 * v.nb, 2.0 * v.nb);
    launch_k(k_pcg_fin<FIN_BETA>, 1, kFinThreads, s, v.part, (int)v.nb, v.sc, 0.0, (double *)nullptr);
  }
  {
    LaunchScope ls(L->ctx, K_CONVERT, 8.0 * v.n * 24.0, 8.0 * v.n * 2.0);
    launch_k(k_pcg_dir, v.nb, kPlaneThreads, s, g.phi, v.p, v.n, v.na, v.sc);
  }
  {
    LaunchScope ls(L->ctx, K_RESID64, 8.0 * v.n * 16.0 + 24.0 * v.n, 8.0 * v.n * 9.0);
    const bool cells = v.n <= kCellOcts;
    launch_k(cells ? k_pcg_apply_cell : k_pcg_apply, v.nb, cells ? kCellThreads4 : kPcgThreads, s, g.nbr, v.p, v.n, v.na,
             v.q, v.part);
  }
  {
    LaunchScope ls(L->ctx, K_REDUCE, 8.0 * v.nb, v.nb);
    launch_k(k_pcg_fin<FIN_ALPHA>, 1, kFinThreads, s, v.part, (int)v.nb, v.sc, 0.0, (double *)nullptr);
  }
  {
    LaunchScope ls(L->ctx, K_CONVERT, 8.0 * v.n * 48.0, 8.0 * v.n * 6.0);
    launch_k(k_pcg_step, v.nb, kPlaneThreads, s, v.x, v.p, g.g, v.q, v.n, v.na, v.sc, v.part);
  }
  {
    LaunchScope ls(L->ctx, K_REDUCE, 8.0 * v.nb, v.nb);
    launch_k(k_pcg_fin<FIN_NORM>, 1, kFinThreads, s, v.part, (int)v.nb, v.sc, d2f_of(L), L->scal + 2);
  }
  CMG_CUDA(cudaGetLastError());
}

// Wrap-up: phi = x, the source restored, the ghosts refilled.
void pcg_post(cmg_level *L) {
  MgLev &g = L->mg[0];
  cudaStream_t s = L->ctx->stream;
  const PcgView v = view(L);
  CMG_CUDA(cudaMemcpyAsync(g.phi, v.x, sizeof(double) * v.nv, cudaMemcpyDeviceToDevice, s));
  CMG_CUDA(cudaMemcpyAsync(g.g, v.gsave, sizeof(double) * 8 * v.n, cudaMemcpyDeviceToDevice, s));
}

}  // namespace cmg
