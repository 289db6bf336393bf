// oct_ops.cuh -- per-oct bodies of the multigrid operators, shared by the
// one-kernel-per-operation path (launch.cu, kernels.cuh) and the tail kernels
// (tail.cu).  Layout: see cmg_internal.cuh.  CG = true routes every load of
// data that another thread block of the same launch may have written through
// L2 (ld.global.cg), as the grid tail's blocks exchange data via global
// memory between grid barriers.
#pragma once

#include "cmg_internal.cuh"

namespace cmg {
namespace dev {

template <bool CG>
__device__ __forceinline__ double2 ldv(const double2 *p) {
  if constexpr (CG) return __ldcg(p); else return *p;
}
template <bool CG>
__device__ __forceinline__ float4 ldv(const float4 *p) {
  if constexpr (CG) return __ldcg(p); else return *p;
}
template <bool CG, typename T>
__device__ __forceinline__ T ld1(const T *p) {
  if constexpr (CG) return __ldcg(p); else return *p;
}

// The four values of one plane of an oct in one access (16 bytes FP32, 32
// bytes FP64; oct arrays start on 32-byte boundaries).
__device__ __forceinline__ void load_oct(const double *p, double v[4]) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void load_oct(const float *p, float v[4]) {
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
               : "l"(p)
               : "memory");
}

template <bool CG>
__device__ __forceinline__ void load4(const double *p, double v[4]) {
  const double2 a = ldv<CG>(reinterpret_cast<const double2 *>(p));
  const double2 b = ldv<CG>(reinterpret_cast<const double2 *>(p + 2));
  v[0] = a.x;
  v[1] = a.y;
  v[2] = b.x;
  v[3] = b.y;
}
template <bool CG>
__device__ __forceinline__ void load4(const float *p, float v[4]) {
  const float4 a = ldv<CG>(reinterpret_cast<const float4 *>(p));
  v[0] = a.x;
  v[1] = a.y;
  v[2] = a.z;
  v[3] = a.w;
}
__device__ __forceinline__ void store4(double *p, const double v[4]) {
  *reinterpret_cast<double2 *>(p) = make_double2(v[0], v[1]);
  *reinterpret_cast<double2 *>(p + 2) = make_double2(v[2], v[3]);
}
__device__ __forceinline__ void store4(float *p, const float v[4]) {
  *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], v[3]);
}

// ---------------------------------------------------------------------------
// The six-neighbour sum of the 7-point stencil.
//
// GB300 issues FP64 at about 2 lanes per SM per clock, 1/64 of its FP32 rate,
// while its integer pipes sit idle in these kernels.  An FP64 sum can instead
// be formed exactly in integers: with E the largest biased exponent of the
// operands, each operand's 53-bit significand is shifted to the common scale
// 2^(E - 1082) (operands more than 7 binades below the largest lose the bits
// under that scale: at most 2^-59 of the largest operand each), the signed
// 64-bit integers are added (|sum| < 6 * 2^60, no overflow), and the integer
// sum is rounded once to the nearest FP64 value, ties to even.  The result is
// within half an ulp of the exact sum plus those truncations, more accurate
// than five sequential FP64 additions, and does not depend on the order of
// the operands.  Zero and subnormal operands contribute nothing (a subnormal
// is below 2^-1022, far under the scale).  The rounding is written out in
// integer operations too: the int64 -> FP64 conversion issues on the FP64
// pipe.  The alignment costs ~15 integer instructions per operand.
// x >> s with PTX semantics: a shift of 64 or more gives 0.
__device__ __forceinline__ unsigned long long shr_clamped(unsigned long long x, unsigned s) {
  unsigned long long r;
  asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));
  return r;
}

// S 2^(E - 1082) rounded to the nearest FP64 value, ties to even; Ex = E << 20
// with 64 <= E < 0x7FC, |S| < 2^63.
__device__ __forceinline__ double fixed_round(long long S, int Ex) {
  const int sg = (int)(S >> 63);  // 0 or -1
  // |S|, or |S| - 1 for a negative S: the 1 is added with the rounding bias
  // below.  Where it would change the leading bit or the last kept bit, the
  // bits rounded off are all zero and the same value comes out.
  const uint32_t alo = (uint32_t)S ^ (uint32_t)sg, ahi = (uint32_t)((unsigned long long)S >> 32) ^ (uint32_t)sg;
  if (ahi >= (1u << 21)) {  // leading bit at p = 63 - c > 52: r = p - 52 bits are rounded off
    const int c = __clz((int)ahi), r = 11 - c;
    // round half to even by one biased truncation: adding 2^(r-1) - 1 plus
    // the last kept bit carries into the kept bits exactly when the dropped
    // part is above half, or equal to it with the kept part odd
    const uint32_t bias = ((1u << (r - 1)) - 1u) + (__funnelshift_r(alo, ahi, r) & 1u) - (uint32_t)sg;
    const unsigned long long b = (((unsigned long long)ahi << 32) | alo) + bias;
    const uint32_t bhi = (uint32_t)(b >> 32);
    // the kept part carries its leading bit at 2^52 (2^53 after a rounding
    // carry), which adds the last 1 (or 2) to the exponent field E + p - 59
    const uint32_t hi = (bhi >> r) + (uint32_t)(Ex + ((3 - c) << 20));
    return __hiloint2double((int)(hi | ((uint32_t)sg & 0x80000000u)), (int)__funnelshift_r((uint32_t)b, bhi, r));
  }
  if (S == 0) return 0.0;
  const unsigned long long a = S < 0 ? 0ull - (unsigned long long)S : (unsigned long long)S;
  const int p = 63 - __clzll((long long)a), eb = (Ex >> 20) + p - 59;
  if (eb <= 0) return ldexp((double)S, (Ex >> 20) - 1082);  // subnormal sum (never in practice)
  if (p > 52)  // |S| = 2^53 alone, above the test on |S| - 1
    return __longlong_as_double((long long)(((unsigned long long)eb << 52) + ((S < 0 ? 1ull : 0ull) << 63)));
  return __longlong_as_double(
      (long long)(((unsigned long long)(eb - 1) << 52) + (a << (52 - p)) + ((S < 0 ? 1ull : 0ull) << 63)));
}

template <int N>
__device__ __forceinline__ double fixed_sum(const double *v) {
  uint32_t hi[N], lo[N];
  int e[N];
  int E = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    hi[k] = (uint32_t)__double2hiint(v[k]);
    lo[k] = (uint32_t)__double2loint(v[k]);
    e[k] = (int)((hi[k] >> 20) & 0x7FFu);
    E = max(E, e[k]);
  }
  // an infinity or NaN, an operand of 2^1021 or more (whose sum could
  // overflow the exponent field below), or every operand below 2^-960 (zeros
  // included): FP64 additions
  if (E >= 0x7FC || E < 64) {
    if (E == 0) {
      // all operands +-0 (a solve's first passes and residuals see whole
      // neighbourhoods of zeros): the FP64 additions' result without them,
      // -0 only when every operand is -0
      uint32_t nz = 0, neg = 0xFFFFFFFFu;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        nz |= (hi[k] & 0x7FFFFFFFu) | lo[k];
        neg &= hi[k];
      }
      if (nz == 0) return __longlong_as_double((long long)((unsigned long long)(neg & 0x80000000u) << 32));
    }
    double s = v[0];
#pragma unroll
    for (int k = 1; k < N; ++k) s += v[k];
    return s;
  }
  // each significand with its leading bit at bit 63 (one funnel shift and
  // the bit), then one right shift by E - e + 4 to the scale 2^(E - 1082);
  // zero and subnormal operands (e = 0) shift by E + 4 >= 68 and vanish.
  // Negative operands enter as ones' complements; the count of them, added
  // once, completes the two's complements.
  long long S = 0;
  int negs = 0;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const uint32_t top = __funnelshift_l(lo[k], hi[k], 11) | 0x80000000u;
    const unsigned long long m = ((unsigned long long)top << 32) | (lo[k] << 11);
    const unsigned long long a = shr_clamped(m, (unsigned)(E - e[k] + 4));
    const long long sg = (long long)((int)hi[k] >> 31);  // 0 or -1
    S += (long long)a ^ sg;
    negs -= (int)sg;
  }
  S += negs;
  return fixed_round(S, E << 20);
}

// Neighbour sum in the order (-x, +x, -y, +y, -z, +z).  FP32: sequential
// additions.  FP64: the first five in the integer sum, the last by one FP64
// addition (the FP64 and integer pipes share the work).  Every kernel forms
// every neighbour sum with these bits, so a residual formed right after a
// colour pass repeats that pass's sums bit for bit.
__device__ __forceinline__ float nbsum6(const float v[6]) {
  return ((((v[0] + v[1]) + v[2]) + v[3]) + v[4]) + v[5];
}
__device__ __forceinline__ double nbsum6(const double v[6]) { return fixed_sum<5>(v) + v[5]; }

// The neighbour sum of a colour-0 residual cell: FP64 takes all six in the
// integer sum.  No colour-0 residual has to repeat a colour pass's sum (only
// the colour-1 residuals after a colour-1 pass do, and they keep nbsum6), and
// the residual spends twice the sweep's FP64 instructions per cell (the
// subtraction of phi and the norm or restriction sum), so its best split
// differs: measured on GB300 (256^3 + 3-level FP64 chain, one box), the
// residual family 11.6 -> 10.9 ms per step with all six in integers.
__device__ __forceinline__ float nbsum6_r0(const float v[6]) { return nbsum6(v); }
__device__ __forceinline__ double nbsum6_r0(const double v[6]) { return fixed_sum<6>(v); }

template <typename T>
__device__ __forceinline__ T fma_t(T a, T b, T c);
template <>
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }
template <>
__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }

// One colour pass of red-black Gauss-Seidel (App. D.2 Eq. (gs_update)) on
// oct i: plane P from the other plane of the oct and of its six face
// neighbours.  ZERO: the other plane is known to be zero, so phi = g.
//
// The *_idx loaders read an oct's index data (neighbours, active mask,
// father, interpolation block, octant), which only the level build writes;
// a one-launch-per-operation kernel reads it before its grid-dependency wait,
// overlapping the preceding kernel, and passes it to the *_oct_idx body.
struct SweepIdx {
  int32_t nb[6];
  unsigned m;
};
template <bool ZERO, bool MASK>
__device__ __forceinline__ SweepIdx sweep_idx(int64_t i, const int32_t *__restrict__ nbr,
                                              const uint8_t *__restrict__ active, int64_t n) {
  SweepIdx x;
#pragma unroll
  for (int d = 0; d < 6; ++d) x.nb[d] = ZERO ? 0 : __ldg(nbr + d * n + i);
  x.m = MASK ? __ldg(active + i) : 0xFFu;
  return x;
}

// The values a pass reads for an oct, apart from the arithmetic on them, so
// that a loop over octs can have the next oct's in flight.
template <typename T>
struct SweepVals {
  T g[4], own[4], nb[6][4];
};
template <typename T, bool ZERO, bool CG>
__device__ __forceinline__ void sweep_load(int64_t i, const SweepIdx &x, const T *src, const T *g, SweepVals<T> &v) {
  load4<CG>(g + i * 4, v.g);
  if (ZERO) return;
  load4<CG>(src + i * 4, v.own);
  // whole neighbour octs, two of their values used each: fewer, wider loads
  // than one per value (256^3 + 3-level chains: FP32 passes 16.95 -> 16.35
  // ms per step, FP64 ones 26.96 -> 26.52)
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    if (CG) load4<CG>(src + (int64_t)x.nb[d] * 4, v.nb[d]);
    else load_oct(src + (int64_t)x.nb[d] * 4, v.nb[d]);
  }
}
template <typename T, int P, bool ZERO, bool MASK>
__device__ __forceinline__ void sweep_finish(int64_t i, const SweepIdx &x, const SweepVals<T> &w, T *dst) {
  T out[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = plane_cell(P, q);
    out[q] = w.g[q];
    if (!ZERO) {
      T v[6];
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        const int a = d >> 1, side = d & 1, c2 = c ^ (1 << a);
        v[d] = ((c >> a) & 1) != side ? w.own[c2 >> 1] : w.nb[d][c2 >> 1];
      }
      out[q] = fma_t(nbsum6(v), T(1) / T(6), out[q]);
    }
    if (MASK && !((x.m >> c) & 1)) out[q] = T(0);
  }
  store4(dst + i * 4, out);
}

template <typename T, int P, bool ZERO, bool MASK, bool CG>
__device__ __forceinline__ void sweep_oct_idx(int64_t i, const SweepIdx &x, const T *src, T *dst, const T *g) {
  SweepVals<T> v;
  sweep_load<T, ZERO, CG>(i, x, src, g, v);
  sweep_finish<T, P, ZERO, MASK>(i, x, v, dst);
}

template <typename T, int P, bool ZERO, bool MASK, bool CG>
__device__ __forceinline__ void sweep_oct(int64_t i, const int32_t *__restrict__ nbr, const T *src, T *dst,
                                          const T *g, const uint8_t *__restrict__ active, int64_t n) {
  sweep_oct_idx<T, P, ZERO, MASK, CG>(i, sweep_idx<ZERO, MASK>(i, nbr, active, n), src, dst, g);
}

// sweep_oct for one cell (cell plane_cell(P, q) of oct i), one thread per
// cell: the same loads, sums in the same order and the same FMA, so the
// result is bit-identical to sweep_oct's.
template <typename T, int P, bool ZERO, bool MASK, bool CG>
__device__ __forceinline__ void sweep_cell(int64_t i, int q, const int32_t *__restrict__ nbr, const T *src, T *dst,
                                           const T *g, const uint8_t *__restrict__ active, int64_t n) {
  T out = ld1<CG>(g + i * 4 + q);
  if (!ZERO) {
    const int c = plane_cell(P, q);
    const T inv6 = T(1) / T(6);
    T v[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const int a = d >> 1, side = d & 1, c2 = c ^ (1 << a);
      const int64_t o = (((c >> a) & 1) != side) ? i : (int64_t)__ldg(nbr + d * n + i);
      v[d] = ld1<CG>(src + o * 4 + (c2 >> 1));
    }
    out = fma_t(nbsum6(v), inv6, out);
  }
  if (MASK && !((__ldg(active + i) >> plane_cell(P, q)) & 1)) out = T(0);
  dst[i * 4 + q] = out;
}

// sweep_cell with what a run of passes over a level reads again each time
// (index data, right-hand sides) kept in registers: slot q of both planes of
// oct i.  The two cells differ in their x bit alone, so they share their y and
// z neighbours.
struct CellRun {
  int32_t xn[2], yn, zn;  // neighbour octs the two cells look out to
  unsigned m;             // their activity, by plane
  double g[2];
};
template <bool MASK>
__device__ __forceinline__ CellRun cell_run(int64_t i, int q, const int32_t *__restrict__ nbr, const double *g,
                                            const uint8_t *__restrict__ active, int64_t n) {
  CellRun r;
  r.yn = __ldg(nbr + (2 + (q & 1)) * n + i);
  r.zn = __ldg(nbr + (4 + (q >> 1)) * n + i);
  const unsigned m = MASK ? __ldg(active + i) : 0xFFu;
  r.m = 0;
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const int c = plane_cell(p, q);
    r.xn[p] = __ldg(nbr + (c & 1) * n + i);
    r.m |= ((m >> c) & 1u) << p;
    r.g[p] = g[(p * n + i) * 4 + q];
  }
  return r;
}
template <int P, bool ZERO, bool MASK>
__device__ __forceinline__ void sweep_cell_run(int64_t i, int q, const CellRun &r, const double *src, double *dst) {
  double out = r.g[P];
  if (!ZERO) {
    // the cell's slots one step along x, y, z are q, q ^ 1, q ^ 2
    const double *own = src + i * 4;
    const double ze = src[(int64_t)r.zn * 4 + (q ^ 2)], zi = own[q ^ 2];
    const bool up = (q & 2) != 0;  // the outer z neighbour is the one above
    const double v[6] = {own[q], src[(int64_t)r.xn[P] * 4 + q], own[q ^ 1], src[(int64_t)r.yn * 4 + (q ^ 1)],
                         up ? zi : ze, up ? ze : zi};
    out = fma(nbsum6(v), 1.0 / 6.0, out);
  }
  if (MASK && !((r.m >> P) & 1u)) out = 0.0;
  dst[i * 4 + q] = out;
}

// The FP32 right-hand side of a mixed-precision solve's correction problem,
// (float)(x * s) with s a power of two: the scaling and the rounding to FP32
// (to nearest, ties to even) formed in integer operations, since GB300
// issues FP64 multiplications and conversions at its low FP64 rate (the
// residual kernel that emits it went 11 % faster).  Zero, a scale that is
// not a normal power of two, and results outside FP32's normal range take
// the FP64 operations instead (same results).
__device__ __forceinline__ float f32_scaled(double x, double s) {
  const unsigned long long sb = (unsigned long long)__double_as_longlong(s);
  const unsigned long long xb = (unsigned long long)__double_as_longlong(x);
  const int es = (int)((sb >> 52) & 0x7FF), ex = (int)((xb >> 52) & 0x7FF);
  const int fe = ex + es - 2046 + 127;  // FP32 biased exponent of x * s
  if ((sb & 0x800FFFFFFFFFFFFFull) != 0 || es == 0 || es == 0x7FF || ex == 0 || fe <= 0 || fe >= 255)
    return (float)(x * s);
  const unsigned long long mant = xb & 0x000FFFFFFFFFFFFFull;
  // round the 52-bit fraction to 23 bits: a carry runs into the exponent
  // field (and from the largest binade to infinity, as the conversion does)
  const uint32_t m = (uint32_t)((mant + 0x0FFFFFFFull + ((mant >> 29) & 1ull)) >> 29);
  return __uint_as_float((((uint32_t)fe << 23) + m) | ((uint32_t)(xb >> 32) & 0x80000000u));
}
// (double)x in integer operations (the conversion issues on the FP64 pipe).
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x), m = b & 0x7FFFFFFFu;
  if (m - 0x00800000u >= 0x7F000000u && m != 0) return (double)x;  // subnormal, infinite, NaN
  return __hiloint2double((int)((b & 0x80000000u) | (m ? (m >> 3) + 0x38000000u : 0u)), (int)(b << 29));
}
// The FP32 right-hand sides' scale for a norm: the power of two of its binade
// (products with it are exact), itself if infinite, else 1.
__device__ __forceinline__ double pow2_scale(double v) {
  if (!(v > 0.0)) return 1.0;
  if (v == INFINITY) return v;
  int e;
  (void)frexp(v, &e);
  return ldexp(1.0, e - 1);
}
// 1 / s: exact and without the FP64 pipe's ten-odd instructions for a normal
// power of two.
__device__ __forceinline__ double inv_scale(double s) {
  const int hi = __double2hiint(s);
  if ((hi & 0x800FFFFF) == 0 && __double2loint(s) == 0 && hi >= 0x00100000 && hi <= 0x7FD00000)
    return __hiloint2double(0x7FE00000 - hi, 0);
  return 1.0 / s;
}
struct ResidIdx {
  int32_t nb[6];
  unsigned m;
  int32_t fa;
};
template <bool RESTRICT>
__device__ __forceinline__ ResidIdx resid_idx(int64_t i, const int32_t *__restrict__ nbr,
                                              const uint8_t *__restrict__ active, int64_t n,
                                              const int32_t *__restrict__ father) {
  ResidIdx x;
#pragma unroll
  for (int d = 0; d < 6; ++d) x.nb[d] = __ldg(nbr + d * n + i);
  x.m = active ? __ldg(active + i) : 0xFFu;
  x.fa = RESTRICT ? __ldg(father + i) : -1;
  return x;
}

// Residual of oct i: d = fma(s, 1/6, g) - phi per cell, r = (-6 / h^2) d.
// Returns the sum of d^2 over the oct (NORM; accumulated in FP64 for FP64
// data, in FP32 within the oct for FP32 data, whose FP64 conversions would
// otherwise bind the kernel to GB300's FP64 pipe).  RESTRICT: a fully active oct
// writes its father cell g_c = 0.5 * sum_8 d (= -h_c^2/6 * mean_8 r) and, if
// zero_cphi, zeroes the father's phi.  EMIT: g32 = (float)(d * inv_s).
// ROUT: r oct-major.  ZPHI: phi taken as zero on real octs.
//
// C1Z: the last operation on this level was a colour-1 pass over every oct
// with the colour-0 values, g and ghost values the residual now reads.  That
// pass wrote fma(s, 1/6, g) at each active colour-1 cell, and this function
// forms the same s from the same values in the same order, so each
// colour-1 residual is exactly +0 (inactive cells are +0 anyway): their
// stencils are skipped.  Skipping changes no result bit: the norm gains
// +0 terms (acc >= +0 throughout), the restriction sum would gain +0 four
// times, which leaves it unchanged (it is never -0), and EMIT / ROUT write
// what dv = +0 gives.
//
// WIDE: the neighbours' planes in one access each (as in sweep_load) instead
// of value by value.  For the colour-0 residuals alone it is faster (batch of
// 512 patches: restriction 570 -> 447 us, norm 631 -> 519 us), for both
// colours' its registers cost the one-launch kernels occupancy (256^3 mixed
// chain 23.9 -> 24.3 ms).
template <typename T, bool NORM, bool RESTRICT, bool EMIT, bool ROUT, bool ZPHI, bool CG, bool C1Z = false,
          bool WIDE = false>
__device__ __forceinline__ double resid_oct_idx(int64_t i, const ResidIdx &x, const T *phi, const T *g, int64_t n,
                                                int64_t n_alloc, T *cg, T *cphi, int64_t cn, int64_t cn_alloc,
                                                int zero_cphi, float *g32, double inv_s, double *rout,
                                                double rscale) {
  T pl[2][4], gv[2][4];
  if (ZPHI) {
#pragma unroll
    for (int q = 0; q < 4; ++q) pl[0][q] = pl[1][q] = T(0);
  } else {
    load4<CG>(phi + i * 4, pl[0]);
    load4<CG>(phi + (n_alloc + i) * 4, pl[1]);
  }
  load4<CG>(g + i * 4, gv[0]);
  if (!C1Z) load4<CG>(g + (n + i) * 4, gv[1]);
  const int32_t *nb = x.nb;
  const T inv6 = T(1) / T(6);
  const unsigned m = x.m;
  T rsum = T(0);
  double acc = 0.0;
  if constexpr (ZPHI && NORM && !RESTRICT && !EMIT && !ROUT) {
    // phi taken as zero: away from the Dirichlet ghosts every sum is zero and
    // fma(0, 1/6, g) = g (256^3 level, cold cache: 118 -> 59 us)
    if (max(max(max(nb[0], nb[1]), max(nb[2], nb[3])), max(nb[4], nb[5])) < n && m == 0xFFu) {
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc = fma((double)gv[p][q], (double)gv[p][q], acc);
      return acc;
    }
  }
  T tacc = T(0);  // FP32 data: the oct's squares summed in FP32, one conversion
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    if (C1Z && p == 1) {
      // rsum needs no + 0 for the four zeros: it starts at +0 and a sum that
      // cancels rounds to +0, so it is never -0
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (EMIT) g32[(p * n + i) * 4 + q] = f32_scaled((double)T(0), inv_s);
        if (ROUT) rout[i * 8 + plane_cell(p, q)] = rscale * 0.0;
      }
      continue;
    }
    // the neighbours' other planes, whole (as in sweep_load)
    T nv[6][4];
    if (WIDE && !ZPHI) {
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        const T *at = phi + ((1 - p) * n_alloc + (int64_t)nb[d]) * 4;
        if (CG) load4<CG>(at, nv[d]);
        else load_oct(at, nv[d]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = plane_cell(p, q);
      T v[6];
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        const int a = d >> 1, side = d & 1, c2 = c ^ (1 << a);
        if (((c >> a) & 1) != side) {
          v[d] = pl[1 - p][c2 >> 1];
        } else if (WIDE && !ZPHI) {
          v[d] = nv[d][c2 >> 1];
        } else {
          const int64_t o = nb[d];
          v[d] = (ZPHI && o < n) ? T(0) : ld1<CG>(phi + ((1 - p) * n_alloc + o) * 4 + (c2 >> 1));
        }
      }
      T dv = fma_t(p == 0 ? nbsum6_r0(v) : nbsum6(v), inv6, gv[p][q]) - pl[p][q];
      if (!((m >> c) & 1)) dv = T(0);
      if (NORM) {
        if constexpr (sizeof(T) == 8)
          acc = fma((double)dv, (double)dv, acc);
        else
          tacc = fma_t(dv, dv, tacc);
      }
      if (RESTRICT) rsum += dv;
      if (EMIT) g32[(p * n + i) * 4 + q] = f32_scaled((double)dv, inv_s);
      if (ROUT) rout[i * 8 + c] = rscale * (double)dv;
    }
  }
  if (NORM && sizeof(T) == 4) acc = (double)tacc;
  if (RESTRICT) {
    const int32_t fa = x.fa;
    if (fa >= 0) {
      const int64_t pc = fa >> 3;
      const int cc = fa & 7;
      cg[((int64_t)cell_parity(cc) * cn + pc) * 4 + (cc >> 1)] = T(0.5) * rsum;
      if (zero_cphi) cphi[((int64_t)cell_parity(cc) * cn_alloc + pc) * 4 + (cc >> 1)] = T(0);
    }
  }
  return acc;
}

template <typename T, bool NORM, bool RESTRICT, bool EMIT, bool ROUT, bool ZPHI, bool CG, bool C1Z = false,
          bool WIDE = false>
__device__ __forceinline__ double resid_oct(int64_t i, const int32_t *__restrict__ nbr, const T *phi, const T *g,
                                            const uint8_t *__restrict__ active, int64_t n, int64_t n_alloc,
                                            const int32_t *__restrict__ father, T *cg, T *cphi, int64_t cn,
                                            int64_t cn_alloc, int zero_cphi, float *g32, double inv_s,
                                            double *rout, double rscale) {
  return resid_oct_idx<T, NORM, RESTRICT, EMIT, ROUT, ZPHI, CG, C1Z, WIDE>(i, resid_idx<RESTRICT>(i, nbr, active, n, father),
                                                                phi, g, n, n_alloc, cg, cphi, cn, cn_alloc,
                                                                zero_cphi, g32, inv_s, rout, rscale);
}

// p - (sum of the six neighbours of p) / 6 on an oct: pv the oct's own values,
// qv the result, by planes; missing neighbours are ghost octs or the zero oct
// of p ([2][n_alloc][4]).  Whole planes and the integer sum, as above.
template <bool CG>
__device__ __forceinline__ void apply_oct(int64_t i, const int32_t *__restrict__ nbr, const double *p, int64_t n,
                                          int64_t n_alloc, double pv[2][4], double qv[2][4]) {
  int32_t nb[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) nb[d] = __ldg(nbr + d * n + i);
  load4<CG>(p + i * 4, pv[0]);
  load4<CG>(p + (n_alloc + i) * 4, pv[1]);
#pragma unroll
  for (int pl = 0; pl < 2; ++pl) {
    double nv[6][4];
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const double *at = p + ((1 - pl) * n_alloc + (int64_t)nb[d]) * 4;
      if (CG) load4<CG>(at, nv[d]);
      else load_oct(at, nv[d]);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = plane_cell(pl, q);
      double v[6];
#pragma unroll
      for (int d = 0; d < 6; ++d) {
        const int a = d >> 1, side = d & 1, c2 = c ^ (1 << a);
        v[d] = ((c >> a) & 1) != side ? pv[1 - pl][c2 >> 1] : nv[d][c2 >> 1];
      }
      qv[pl][q] = fma(fixed_sum<6>(v), -1.0 / 6.0, pv[pl][q]);
    }
  }
}
// The same for cell c of oct i.
__device__ __forceinline__ void apply_cell(int64_t i, int c, const int32_t *__restrict__ nbr, const double *p, int64_t n,
                                           int64_t n_alloc, double &pv, double &qv) {
  const int pl = cell_parity(c);
  double v[6];
  pv = p[(pl * n_alloc + i) * 4 + (c >> 1)];
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const int a = d >> 1, side = d & 1, c2 = c ^ (1 << a);
    const int64_t o = (((c >> a) & 1) != side) ? i : (int64_t)__ldg(nbr + d * n + i);
    v[d] = p[((1 - pl) * n_alloc + o) * 4 + (c2 >> 1)];
  }
  qv = fma(fixed_sum<6>(v), -1.0 / 6.0, pv);
}

// resid_oct<NORM = false, RESTRICT = true> with one thread per cell: lane k
// of an aligned group of 8 lanes takes cell plane_cell(k >> 2, k & 3) of oct
// i (plane k >> 2, slot k & 3).  Every lane of the warp calls it (the father
// value is summed across the group by shuffles, in resid_oct's order);
// `valid` is false for a group past the end of the range.
template <typename T, bool CG>
__device__ __forceinline__ void resid_restrict_cell(bool valid, int64_t i, const int32_t *__restrict__ nbr, const T *phi,
                                                    const T *g, const uint8_t *__restrict__ active, int64_t n,
                                                    int64_t n_alloc, const int32_t *__restrict__ father, T *cg, T *cphi,
                                                    int64_t cn, int64_t cn_alloc, int zero_cphi) {
  const int k = (int)(threadIdx.x & 7), p = k >> 2, q = k & 3, c = plane_cell(p, q);
  T dv = T(0);
  if (valid) {
    const T pv = ld1<CG>(phi + (p * n_alloc + i) * 4 + q);
    const T gv = ld1<CG>(g + (p * n + i) * 4 + q);
    const T inv6 = T(1) / T(6);
    T v[6];
#pragma unroll
    for (int d = 0; d < 6; ++d) {
      const int a = d >> 1, side = d & 1, c2 = c ^ (1 << a);
      const int64_t o = (((c >> a) & 1) != side) ? i : (int64_t)__ldg(nbr + d * n + i);
      v[d] = ld1<CG>(phi + ((1 - p) * n_alloc + o) * 4 + (c2 >> 1));
    }
    if (p == 0)
      dv = fma_t(nbsum6_r0(v), inv6, gv) - pv;
    else
      dv = fma_t(nbsum6(v), inv6, gv) - pv;
    const unsigned m = active ? __ldg(active + i) : 0xFFu;
    if (!((m >> c) & 1)) dv = T(0);
  }
  const int base = (int)(threadIdx.x & 31) & ~7;
  T rsum = T(0);
#pragma unroll
  for (int j = 0; j < 8; ++j) rsum += __shfl_sync(0xFFFFFFFFu, dv, base + j);
  if (valid && k == 0) {
    const int32_t fa = __ldg(father + i);
    if (fa >= 0) {
      const int64_t pc = fa >> 3;
      const int cc = fa & 7;
      cg[((int64_t)cell_parity(cc) * cn + pc) * 4 + (cc >> 1)] = T(0.5) * rsum;
      if (zero_cphi) cphi[((int64_t)cell_parity(cc) * cn_alloc + pc) * 4 + (cc >> 1)] = T(0);
    }
  }
}

// resid_oct<..., C1Z = true> with four threads per oct: the residual of colour
// 0 cell q of oct i (d-units), the same sum and operations.
template <bool MASK>
__device__ __forceinline__ double resid_c0_cell(int64_t i, int q, const int32_t *__restrict__ nbr, const double *phi,
                                                const double *g, const uint8_t *__restrict__ active, int64_t n,
                                                int64_t n_alloc) {
  const int c = plane_cell(0, q);
  const double pv = phi[i * 4 + q], gv = g[i * 4 + q];
  double v[6];
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    const int a = d >> 1, side = d & 1, c2 = c ^ (1 << a);
    const int64_t o = (((c >> a) & 1) != side) ? i : (int64_t)__ldg(nbr + d * n + i);
    v[d] = phi[(n_alloc + o) * 4 + (c2 >> 1)];
  }
  const double dv = fma(nbsum6_r0(v), 1.0 / 6.0, gv) - pv;
  return MASK && !((__ldg(active + i) >> c) & 1) ? 0.0 : dv;
}

// Trilinear cell-centred interpolation of a coarse field onto the 8 children
// of a coarse cell: per axis weight 3/4 for the father, 1/4 for its neighbour
// toward the child (Sec. 5.1.1).
//
// The father is child cc of the block's oct 0; block oct t is displaced along
// the axes in t toward the father's octant.  On an axis the neighbour toward
// a child lies in the displaced oct where the child's bit equals the father's,
// else it is the father's sibling; in both cases its child bit there is the
// father's flipped.  So with r = c ^ cc ^ 7 (the axes on which child c looks
// out of the oct), the value child c combines for the axes in t is child
// cc ^ t of block oct t & r, with weight 3^(3 - |t|) / 64.
//
// 64 x the value is formed as one weighted sum.  FP32: separably, 3 a + b in
// one FMA along x, y and z.  FP64: in integers, as the neighbour sums are
// (GB300's FP64 pipe ran the separable form's 26 FMAs per oct at 81 % busy
// while the others idled): significands at the common scale 2^(E - 1078), E
// the largest biased exponent of the eight (bits under that scale are
// truncated), times the weights, added as 64-bit integers
// (|sum| < 64 * 2^56) and rounded once, ties to even: half an ulp plus at
// most 63/512 ulp of 64 x the largest value, below the three nested roundings
// of the separable form.  The 64 is divided out exactly (a power of two) in
// the FMA that adds the correction to phi, or by a multiplication for a
// plain value.
// Measured on GB300 (256^3 + 3-level chain, per step): FP64 prolongations
// 6.73 ms (separable) -> 4.30 ms; FP32 ones 3.51 -> 2.48 ms, from finding the
// eight values by t & r instead of by selects among 27 places.
// 3 a + b with one rounding
template <typename T>
__device__ __forceinline__ T tri3(T father, T side) {
  return fma_t(T(3), father, side);
}
// v[t]: the value for the axes in t
template <typename T>
__device__ __forceinline__ T interp64_sep(const T v[8]) {
  return tri3(tri3(tri3(v[0], v[1]), tri3(v[2], v[3])), tri3(tri3(v[4], v[5]), tri3(v[6], v[7])));
}
__device__ __forceinline__ float interp64(const float v[8]) { return interp64_sep(v); }
__device__ __forceinline__ double interp64(const double v[8]) {
  uint32_t hi[8], lo[8];
  int e[8], E = 0;
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    hi[t] = (uint32_t)__double2hiint(v[t]);
    lo[t] = (uint32_t)__double2loint(v[t]);
    e[t] = (int)((hi[t] >> 20) & 0x7FFu);
    E = max(E, e[t]);
  }
  // infinities, NaN and values whose sum could overflow, or all below 2^-960:
  // FP64 operations; all zero: 0
  if (E >= 0x7F0 || E < 64) {
    if (E == 0) {
      uint32_t nz = 0;
#pragma unroll
      for (int t = 0; t < 8; ++t) nz |= (hi[t] & 0x7FFFFFFFu) | lo[t];
      if (nz == 0) return 0.0;
    }
    return interp64_sep(v);
  }
  // each significand with its leading bit at bit 63, shifted right by
  // E - e + 8 (zero and subnormal values vanish); the sign goes with the
  // weight for the high word, and as a ones' complement for the low one:
  // -w a = w (~a) - w (2^32 - 1)
  unsigned long long L = 0;
  int H = 0, C = 0;
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const int w = t == 0 ? 27 : t == 7 ? 1 : (t == 3 || t == 5 || t == 6) ? 3 : 9;
    const uint32_t top = __funnelshift_l(lo[t], hi[t], 11) | 0x80000000u;
    const unsigned long long a =
        shr_clamped(((unsigned long long)top << 32) | (lo[t] << 11), (unsigned)(E - e[t] + 8));
    const int sg = (int)hi[t] >> 31;  // 0 or -1
    H += (int)(a >> 32) * (w * (sg | 1));
    L += (unsigned long long)((uint32_t)a ^ (uint32_t)sg) * (unsigned)w;
    C += sg * w;
  }
  const long long S = (long long)L + ((long long)(H + C) << 32) - C;
  return fixed_round(S, (E + 4) << 20);
}
constexpr double kInv64 = 0.015625;

// Where a block's coarse values lie: p[t] + 4 oct is the value of child
// cc ^ t of an oct.
template <typename T>
struct CoarseView {
  const T *p[8];
};
template <typename T>
__device__ __forceinline__ CoarseView<T> coarse_view(const T *cphi, int64_t cn_alloc, int cc) {
  CoarseView<T> w;
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const int ch = cc ^ t;
    w.p[t] = cphi + (cell_parity(ch) ? cn_alloc * 4 : (int64_t)0) + (ch >> 1);
  }
  return w;
}

// 64 x the values of all 8 children (X64) or the values, out[c].
template <typename T, bool CG, bool X64 = false>
__device__ __forceinline__ void interp8(const T *cphi, int64_t cn_alloc, const int32_t b[8], int cc, T out[8]) {
  const CoarseView<T> w = coarse_view(cphi, cn_alloc, cc);
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    T v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) v[t] = ld1<CG>(w.p[t] + (int64_t)b[t & r] * 4);
    const T z = interp64(v);
    out[r] = X64 ? z : z * T(kInv64);
  }
  // out[r] is child r ^ (cc ^ 7): put them in child order
#pragma unroll
  for (int bit = 1; bit < 8; bit <<= 1) {
    const bool flip = ((cc ^ 7) & bit) != 0;
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (!(c & bit)) {
        const T x = out[c], y = out[c | bit];
        out[c] = flip ? y : x;
        out[c | bit] = flip ? x : y;
      }
  }
}

// 64 x the values of the colour-1 children, out[q] for slot q.
template <typename T, bool CG>
__device__ __forceinline__ void interp4_c1(const T *cphi, int64_t cn_alloc, const int32_t b[8], int cc, T out[4]) {
  const CoarseView<T> w = coarse_view(cphi, cn_alloc, cc);
  // r = c ^ cc ^ 7 of an odd-parity c has cc's parity: r = R_j, or R_j ^ 7,
  // with R_j = 0, 3, 5, 6; the slot c >> 1 is then j ^ k
  const bool odd = cell_parity(cc) != 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int R = plane_cell(0, j);
    T v[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const int32_t o = (t & R) == (t & ~R) ? b[0] : odd ? b[t & ~R] : b[t & R];
      v[t] = ld1<CG>(w.p[t] + (int64_t)o * 4);
    }
    out[j] = interp64(v);
  }
  const int k = ((odd ? cc : cc ^ 7) >> 1) & 3;
#pragma unroll
  for (int bit = 1; bit < 4; bit <<= 1) {
    const bool flip = (k & bit) != 0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (!(q & bit)) {
        const T x = out[q], y = out[q | bit];
        out[q] = flip ? y : x;
        out[q | bit] = flip ? x : y;
      }
  }
}

// phi + the child's correction, given as 64 x its value
template <typename T>
__device__ __forceinline__ T add_corr(T phi, T corr) {
  return fma_t(corr, T(kInv64), phi);
}

// phi[i] += trilinear interpolation of the coarse correction (active cells).
struct ProlongIdx {
  int32_t b[8];
  int cc;
  unsigned m;
};
template <bool MASK>
__device__ __forceinline__ ProlongIdx prolong_idx(int64_t i, const uint64_t *__restrict__ keys,
                                                  const int32_t *__restrict__ blk, int64_t n,
                                                  const uint8_t *__restrict__ active) {
  ProlongIdx x;
  x.cc = (int)(__ldg(keys + i) & 7);
#pragma unroll
  for (int t = 0; t < 8; ++t) x.b[t] = __ldg(blk + t * n + i);
  x.m = MASK ? __ldg(active + i) : 0xFFu;
  return x;
}

// C0D: a colour-0 pass over every oct comes next; it overwrites each
// colour-0 value without reading it (the update uses only the colour-1
// neighbours and g), so the colour-0 corrections are dead and only colour-1
// cells are corrected (the unused interpolation terms and loads drop out).
template <typename T, bool MASK, bool CG, bool C0D = false>
__device__ __forceinline__ void prolong_oct_idx(int64_t i, const ProlongIdx &x, int64_t n_alloc, T *phi,
                                                const T *cphi, int64_t cn_alloc) {
  const unsigned m = x.m;
  T corr[8];
  if (C0D) {
    T c1[4];
    interp4_c1<T, CG>(cphi, cn_alloc, x.b, x.cc, c1);
#pragma unroll
    for (int q = 0; q < 4; ++q) corr[plane_cell(1, q)] = c1[q];
  } else {
    interp8<T, CG, true>(cphi, cn_alloc, x.b, x.cc, corr);
  }
#pragma unroll
  for (int p = C0D ? 1 : 0; p < 2; ++p) {
    T v[4];
    load4<CG>(phi + (p * n_alloc + i) * 4, v);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = plane_cell(p, q);
      if ((m >> c) & 1) v[q] = add_corr(v[q], corr[c]);
    }
    store4(phi + (p * n_alloc + i) * 4, v);
  }
}

template <typename T, bool MASK, bool CG, bool C0D = false>
__device__ __forceinline__ void prolong_oct(int64_t i, const uint64_t *__restrict__ keys,
                                            const int32_t *__restrict__ blk, int64_t n, int64_t n_alloc, T *phi,
                                            const uint8_t *__restrict__ active, const T *cphi, int64_t cn_alloc) {
  prolong_oct_idx<T, MASK, CG, C0D>(i, prolong_idx<MASK>(i, keys, blk, n, active), n_alloc, phi, cphi, cn_alloc);
}

// prolong_oct for one cell c of oct i, one thread per cell: the 8 coarse
// values interp8 combines for this cell, in its order and with its weights
// (bit-identical); inactive cells are left untouched.
template <typename T, bool MASK, bool CG>
__device__ __forceinline__ void prolong_cell(int64_t i, int c, const uint64_t *__restrict__ keys,
                                             const int32_t *__restrict__ blk, int64_t n, int64_t n_alloc, T *phi,
                                             const uint8_t *__restrict__ active, const T *cphi, int64_t cn_alloc) {
  if (MASK && !((__ldg(active + i) >> c) & 1)) return;
  const int cc = (int)(__ldg(keys + i) & 7);
  const CoarseView<T> w = coarse_view(cphi, cn_alloc, cc);
  const int r = c ^ cc ^ 7;
  T v[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) v[t] = ld1<CG>(w.p[t] + (int64_t)__ldg(blk + (int64_t)(t & r) * n + i) * 4);
  const T acc = interp64(v);
  T *dst = phi + ((int64_t)cell_parity(c) * n_alloc + i) * 4 + (c >> 1);
  *dst = add_corr(ld1<CG>(dst), acc);
}

// Exact solve of the periodic 2^3 oct by one warp (all 32 lanes call it;
// lanes 0..7 own cell c = lane): eigenvectors (-1)^{k.b}, eigenvalues
// -4 |k|_1 / h^2, mean mode dropped; FP64 inside.  Each lane forms one
// transform coefficient and one output from the others' values (shuffles),
// in the same order of operations as a serial evaluation.
template <typename S, typename T, bool CG>
__device__ void wht_solve_warp(const S *g, T *phi, int64_t n_alloc, double h) {
  const unsigned all = 0xFFFFFFFFu;
  const int c = (int)(threadIdx.x & 7);
  const double f = (double)ld1<CG>(g + cell_parity(c) * 4 + (c >> 1)) * (-6.0 / (h * h));
  double s = 0.0;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const double fb = __shfl_sync(all, f, b);
    s += cell_parity(c & b) ? -fb : fb;
  }
  const double fh = s * 0.125;
  const int odd = (c & 1) + ((c >> 1) & 1) + ((c >> 2) & 1);
  const double x = c ? fh / (-4.0 * odd / (h * h)) : 0.0;
  double t = 0.0;
#pragma unroll
  for (int k = 1; k < 8; ++k) {
    const double xk = __shfl_sync(all, x, k);
    t += cell_parity(k & c) ? -xk : xk;
  }
  if ((threadIdx.x & 31) < 8) phi[(int64_t)cell_parity(c) * n_alloc * 4 + (c >> 1)] = (T)t;
}

}  // namespace dev
}  // namespace cmg
