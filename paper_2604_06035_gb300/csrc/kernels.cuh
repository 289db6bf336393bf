// kernels.cuh -- one-operation-per-launch kernels of the multigrid V-cycle
// (thread per oct), built on the per-oct bodies of oct_ops.cuh:
//   red-black Gauss-Seidel colour pass      App. D.2 Eq. (gs_update)
//   residual (+ squared norm, + restriction) Sec. 5.1.1 item (iii); restriction = mean of 8 children
//   prolongation + correction               Sec. 5.1.1 (trilinear interpolation)
//   coarse-fine Dirichlet ghost values      interpolation of the parent's phi (morton_nbor_cell, App. B)
//   coarsest periodic 2^3 solve             exact (Walsh-Hadamard diagonalisation)
// Included by launch.cu only.
#pragma once

#include "oct_ops.cuh"

namespace cmg {
namespace {

// Deterministic block sum of one double per thread -> partials[blockIdx.x].
template <int THREADS = kThreads>
__device__ void block_sum_to(double v, double *partials) {
  __shared__ double ws[THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double w = threadIdx.x < (blockDim.x >> 5) ? ws[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
    if (threadIdx.x == 0) partials[blockIdx.x] = w;
  }
}

// FP32 kernels read their oct's index data (written only by the level build)
// before the grid-dependency wait, overlapping the preceding kernel's tail:
// measured on the two-level 128^3 workload, the mixed-precision solves got
// 2-3 % faster.  FP64 kernels, bound by GB300's FP64 issue rate, keep every
// load after the wait: with the early reads the refined level's FP64 solve
// got ~1-3 % slower.  FP32 colour passes preload only on levels of at most
// kPreloadSweepOcts octs: the HBM-bound pass over a 512^3 level got 3 %
// slower with it (the residual there got faster).
template <typename T>
constexpr bool kPreloadIdx = sizeof(T) == 4;
constexpr int64_t kPreloadSweepOcts = int64_t(1) << 20;

constexpr int kCellThreads = 128;

template <typename T, int P, bool ZERO, bool MASK, bool PRE>
__global__ void __launch_bounds__(kThreads) k_sweep(const int32_t *__restrict__ nbr, const T *__restrict__ src,
                                                   T *__restrict__ dst, const T *__restrict__ g,
                                                   const uint8_t *__restrict__ active, int64_t n) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if constexpr (PRE) {
    dev::SweepIdx x;
    if (i < n) x = dev::sweep_idx<ZERO, MASK>(i, nbr, active, n);
    pdl_enter();
    if (i >= n) return;
    dev::sweep_oct_idx<T, P, ZERO, MASK, false>(i, x, src, dst, g);
  } else {
    pdl_enter();
    if (i >= n) return;
    dev::sweep_oct<T, P, ZERO, MASK, false>(i, nbr, src, dst, g, active, n);
  }
}

// FP64 operations with one thread per cell (four per oct).
template <int P, bool ZERO, bool MASK>
__global__ void __launch_bounds__(kCellThreads) k_sweep_cell(const int32_t *__restrict__ nbr,
                                                            const double *__restrict__ src, double *__restrict__ dst,
                                                            const double *__restrict__ g,
                                                            const uint8_t *__restrict__ active, int64_t n) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_enter();
  if (t >= 4 * n) return;
  dev::sweep_cell<double, P, ZERO, MASK, false>(t >> 2, (int)(t & 3), nbr, src, dst, g, active, n);
}

// Restriction of the colour-0 residuals (the colour-1 ones are zero): the
// four lanes of an oct hand theirs to the first, which adds them in resid_oct's
// order.  Every thread of a warp runs it.
template <bool MASK>
__global__ void __launch_bounds__(kCellThreads)
    k_restrict_cell(const int32_t *__restrict__ nbr, const double *__restrict__ phi, const double *__restrict__ g,
                    const uint8_t *__restrict__ active, int64_t n, int64_t n_alloc,
                    const int32_t *__restrict__ father, double *__restrict__ cg, double *__restrict__ cphi, int64_t cn,
                    int64_t cn_alloc, int zero_cphi) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_enter();
  const int64_t i = t >> 2;
  const bool on = i < n;
  const double dv = on ? dev::resid_c0_cell<MASK>(i, (int)(t & 3), nbr, phi, g, active, n, n_alloc) : 0.0;
  const int base = (int)(threadIdx.x & 31) & ~3;
  double rsum = 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j) rsum += __shfl_sync(0xFFFFFFFFu, dv, base + j);
  if (!on || (t & 3)) return;
  const int32_t fa = __ldg(father + i);
  if (fa < 0) return;
  const int64_t pc = fa >> 3;
  const int cc = fa & 7;
  cg[((int64_t)cell_parity(cc) * cn + pc) * 4 + (cc >> 1)] = 0.5 * rsum;
  if (zero_cphi) cphi[((int64_t)cell_parity(cc) * cn_alloc + pc) * 4 + (cc >> 1)] = 0.0;
}

// Sum of the colour-0 residuals' squares, per block of 256 octs as in k_resid.
template <bool MASK>
__global__ void __launch_bounds__(4 * kThreads)
    k_norm_cell(const int32_t *__restrict__ nbr, const double *__restrict__ phi, const double *__restrict__ g,
                const uint8_t *__restrict__ active, int64_t n, int64_t n_alloc, double *__restrict__ partials) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_enter();
  const double dv = (t >> 2) < n ? dev::resid_c0_cell<MASK>(t >> 2, (int)(t & 3), nbr, phi, g, active, n, n_alloc) : 0.0;
  block_sum_to<4 * kThreads>(dv * dv, partials);
}

// Prolongation before a colour-0 pass: the colour-1 cells only.
template <bool MASK>
__global__ void __launch_bounds__(kCellThreads)
    k_prolong_cell(const uint64_t *__restrict__ keys, const int32_t *__restrict__ blk, int64_t n, int64_t n_alloc,
                   double *__restrict__ phi, const uint8_t *__restrict__ active, const double *__restrict__ cphi,
                   int64_t cn_alloc) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_enter();
  if (t >= 4 * n) return;
  dev::prolong_cell<double, MASK, false>(t >> 2, plane_cell(1, (int)(t & 3)), keys, blk, n, n_alloc, phi, active, cphi,
                                         cn_alloc);
}

template <typename T, bool NORM, bool RESTRICT, bool EMIT, bool ROUT, bool ZPHI, bool C1Z = false>
__global__ void __launch_bounds__(kThreads) k_resid(const int32_t *__restrict__ nbr, const T *__restrict__ phi,
                                                   const T *__restrict__ g, const uint8_t *__restrict__ active,
                                                   int64_t n, int64_t n_alloc, const int32_t *__restrict__ father,
                                                   T *__restrict__ cg, T *__restrict__ cphi, int64_t cn,
                                                   int64_t cn_alloc, int zero_cphi, double *__restrict__ partials,
                                                   float *__restrict__ g32, const double *__restrict__ emit_scale,
                                                   double *__restrict__ rout, double rscale) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double acc = 0.0;
  if constexpr (kPreloadIdx<T>) {
    dev::ResidIdx x;
    if (i < n) x = dev::resid_idx<RESTRICT>(i, nbr, active, n, father);
    pdl_enter();
    if (i < n) {
      const double inv_s = EMIT ? dev::inv_scale(*emit_scale) : 0.0;
      acc = dev::resid_oct_idx<T, NORM, RESTRICT, EMIT, ROUT, ZPHI, false, C1Z, C1Z>(i, x, phi, g, n, n_alloc, cg, cphi, cn,
                                                                           cn_alloc, zero_cphi, g32, inv_s, rout,
                                                                           rscale);
    }
  } else {
    pdl_enter();
    if (i < n) {
      const double inv_s = EMIT ? dev::inv_scale(*emit_scale) : 0.0;
      acc = dev::resid_oct<T, NORM, RESTRICT, EMIT, ROUT, ZPHI, false, C1Z, C1Z>(i, nbr, phi, g, active, n, n_alloc, father,
                                                                       cg, cphi, cn, cn_alloc, zero_cphi, g32, inv_s,
                                                                       rout, rscale);
    }
  }
  if (NORM) block_sum_to(acc, partials);
}

template <typename T, bool MASK, bool C0D>
__global__ void __launch_bounds__(kThreads) k_prolong(const uint64_t *__restrict__ keys, const int32_t *__restrict__ blk,
                                                     int64_t n, int64_t n_alloc, T *__restrict__ phi,
                                                     const uint8_t *__restrict__ active,
                                                     const T *__restrict__ cphi, int64_t cn_alloc) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if constexpr (kPreloadIdx<T>) {
    dev::ProlongIdx x;
    if (i < n) x = dev::prolong_idx<MASK>(i, keys, blk, n, active);
    pdl_enter();
    if (i >= n) return;
    dev::prolong_oct_idx<T, MASK, false, C0D>(i, x, n_alloc, phi, cphi, cn_alloc);
  } else {
    pdl_enter();
    if (i >= n) return;
    dev::prolong_oct<T, MASK, false, C0D>(i, keys, blk, n, n_alloc, phi, active, cphi, cn_alloc);
  }
}

__global__ void __launch_bounds__(kThreads) k_ghost_fill(const uint64_t *__restrict__ gkeys,
                                                        const int32_t *__restrict__ gblk,
                                                        const uint32_t *__restrict__ gmask, int64_t n_ghost,
                                                        int64_t n, int64_t n_alloc, double *__restrict__ phi,
                                                        const double *__restrict__ pphi, int64_t pn_alloc) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n_ghost) return;
  const int cc = (int)(gkeys[t] & 7);
  int32_t b[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) b[k] = __ldg(gblk + k * n_ghost + t);
  double val[8];
  dev::interp8<double, false>(pphi, pn_alloc, b, cc, val);
  const uint32_t m = gmask[t];
  const int64_t oct = n + t;
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = plane_cell(p, q);
      v[q] = ((m >> c) & 1) ? val[c] : 0.0;
    }
    dev::store4(phi + (p * n_alloc + oct) * 4, v);
  }
}

// Ghost values in the [n][6][4] API layout (NaN where the neighbour exists).
__global__ void k_get_ghosts(const int32_t *__restrict__ nbr, int64_t n, int64_t n_ghost, int64_t n_alloc,
                             const double *__restrict__ phi, double *__restrict__ out) {
  pdl_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int d = 0; d < 6; ++d) {
    const int64_t o = nbr[d * n + i];
    const bool ghost = o >= n && o < n + n_ghost;
    const int a = d >> 1, side = d & 1;
    int q = 0;
    for (int c = 0; c < 8; ++c) {
      if (((c >> a) & 1) != side) continue;
      const int c2 = c ^ (1 << a);
      out[(i * 6 + d) * 4 + q] = ghost ? phi[((int64_t)cell_parity(c2) * n_alloc + o) * 4 + (c2 >> 1)]
                                       : __longlong_as_double(0x7ff8000000000000ll);
      ++q;
    }
  }
}

template <typename T>
__global__ void k_wht(const T *__restrict__ g, T *__restrict__ phi, int64_t n_alloc, double h) {
  pdl_enter();
  if (threadIdx.x >= 32 || blockIdx.x != 0) return;
  dev::wht_solve_warp<T, T, false>(g, phi, n_alloc, h);
}

// The layout kernels below take one oct per thread: its 8 values in 16-byte
// accesses, which moves a 256^3 level's field at about twice the rate of one
// value per thread.  WIDE = false: the caller's array does not start on a
// 16-byte boundary and is accessed value by value.
template <bool WIDE, typename T>
__device__ __forceinline__ void load8(const T *p, T v[8]) {
  if (!WIDE) {
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = p[k];
    return;
  }
  T a[4], b[4];
  dev::load4<false>(p, a);
  dev::load4<false>(p + 4, b);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = a[k];
    v[k + 4] = b[k];
  }
}
template <bool WIDE, typename T>
__device__ __forceinline__ void store8(T *p, const T v[8]) {
  if (!WIDE) {
#pragma unroll
    for (int k = 0; k < 8; ++k) p[k] = v[k];
    return;
  }
  dev::store4(p, v);
  dev::store4(p + 4, v + 4);
}
// the plane's four values of an oct's eight (child order), and back
template <typename T>
__device__ __forceinline__ void to_plane(const T v[8], int p, T q4[4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q) q4[q] = p == 0 ? v[plane_cell(0, q)] : v[plane_cell(1, q)];
}

template <bool WIDE>
__global__ void __launch_bounds__(kThreads) k_set_density(const double *__restrict__ rho, int64_t n, double rho_bar,
                                                         double scale, double *__restrict__ g) {
  pdl_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  double v[8], w[4];
  load8<WIDE>(rho + i * 8, v);
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = scale * (v[c] - rho_bar);
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    to_plane(v, p, w);
    dev::store4(g + (p * n + i) * 4, w);
  }
}

// oct-major [n][8] <-> planar [2][stride][4], with a scale factor
template <bool WIDE, typename T>
__global__ void __launch_bounds__(kThreads) k_pack(const T *__restrict__ in, int64_t n, int64_t stride, double scale,
                                                  T *__restrict__ out) {
  pdl_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  T v[8], w[4];
  load8<WIDE>(in + i * 8, v);
  if (scale != 1.0) {
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = (T)(scale * (double)v[c]);
  }
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    to_plane(v, p, w);
    dev::store4(out + (p * stride + i) * 4, w);
  }
}

template <bool WIDE, typename T>
__global__ void __launch_bounds__(kThreads) k_unpack(const T *__restrict__ in, int64_t n, int64_t stride, double scale,
                                                    T *__restrict__ out) {
  pdl_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  T v[8];
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    T w[4];
    dev::load4<false>(in + (p * stride + i) * 4, w);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[plane_cell(p, q)] = w[q];
  }
  if (scale != 1.0) {
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = (T)(scale * (double)v[c]);
  }
  store8<WIDE>(out + i * 8, v);
}

// Sum of phi: a grid-stride loop, so that the block sums' FP64 additions
// (which issue once per ~64 clocks) are paid once per block and not per 256
// octs.
__global__ void __launch_bounds__(kThreads) k_sum_phi(const double *__restrict__ phi, int64_t n, int64_t n_alloc,
                                                     double *__restrict__ partials) {
  pdl_enter();
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += gridDim.x * (int64_t)blockDim.x) {
    double a[4], b[4];
    dev::load4<false>(phi + i * 4, a);
    dev::load4<false>(phi + (n_alloc + i) * 4, b);
    acc += ((a[0] + a[1]) + (a[2] + a[3])) + ((b[0] + b[1]) + (b[2] + b[3]));
  }
  block_sum_to(acc, partials);
}

__global__ void __launch_bounds__(kThreads) k_sub_scalar(double *__restrict__ phi, int64_t n, int64_t n_alloc,
                                                        const double *__restrict__ s) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= 2 * n) return;
  const int p = t >= n ? 1 : 0;
  double *at = phi + (p * n_alloc + (t - p * n)) * 4;
  const double x = *s;
  double v[4];
  dev::load4<false>(at, v);
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] -= x;
  dev::store4(at, v);
}

// phi64 += S * phi32 on the real octs (solution accumulation, FP64)
__global__ void k_accumulate(double *__restrict__ phi, const float *__restrict__ e, int64_t n, int64_t n_alloc,
                             const double *__restrict__ scale) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= 2 * n) return;
  const int p = t >= n ? 1 : 0;
  const int64_t i = t - p * n;
  const double S = *scale;
  double v[4];
  float w[4];
  dev::load4<false>(phi + (p * n_alloc + i) * 4, v);
  dev::load4<false>(e + (p * n_alloc + i) * 4, w);
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = fma(S, dev::widen(w[q]), v[q]);
  dev::store4(phi + (p * n_alloc + i) * 4, v);
}

// Sum partials in a fixed order; out[0] = scale * sum (and its sqrt to out[1]).
__global__ void k_finalize(const double *__restrict__ partials, int np, double scale, double *__restrict__ out,
                           int with_sqrt) {
  pdl_enter();
  __shared__ double ws[32];
  double v = 0.0;
  for (int t = threadIdx.x; t < np; t += blockDim.x) v += partials[t];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    double w = threadIdx.x < (blockDim.x >> 5) ? ws[threadIdx.x] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xffffffffu, w, o);
    if (threadIdx.x == 0) {
      out[0] = scale * w;
      if (with_sqrt) out[1] = sqrt(scale * w);
    }
  }
}

__global__ void k_copy_convert_f2d(const float *__restrict__ a, double *__restrict__ b, int64_t m) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < m) b[t] = (double)a[t];
}
__global__ void k_copy_convert_d2f(const double *__restrict__ a, float *__restrict__ b, int64_t m) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t < m) b[t] = (float)a[t];
}

template <typename T>
T *phi_of(MgLev &g);
template <>
double *phi_of<double>(MgLev &g) { return g.phi; }
template <>
float *phi_of<float>(MgLev &g) { return g.phi32; }
template <typename T>
T *g_of(MgLev &g);
template <>
double *g_of<double>(MgLev &g) { return g.g; }
template <>
float *g_of<float>(MgLev &g) { return g.g32; }

}  // namespace
}  // namespace cmg
