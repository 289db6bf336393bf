// unet.cu -- the learned warm start: a 3-level 3-D U-Net (16/32/64 channels)
// mapping (rho, phi_prev) on a periodic D^3 block to the change of phi, with
// hand-written BF16 x BF16 -> FP32 tensor-core training and inference kernels.
// (No counterpart in the paper; the layer graph is listed in include/cmg.h.)
//
// Layout: activations are channels-last bf16 [B][D^3][C] (voxel v = (z D + y)
// D + x); conv weights are bf16 [Cout][27][Cin] for the forward pass and
// [Cin][27][Cout] for the input gradient, tap t = 9 (dz+1) + 3 (dy+1) + (dx+1);
// master parameters, gradients and Adam moments are FP32.
//
// Convolutions and input gradients on grids of a multiple of 16 run on the
// tcgen05 kernels of conv_tc.cuh.  Below that (or on request) they are implicit
// GEMMs on mma.sync m16n8k16 (bf16 in, fp32 accumulate): a block owns a 4x4x4
// voxel brick, per 16-channel slice it stages the brick's 6x6x6 periodic halo
// (216 rows of 32 B) and the 27 taps of the weight slice in shared memory, and
// every tap's A fragment is an ldmatrix of halo rows shifted by the tap offset
// -- each input value is read from global memory once per slice instead of 27
// times.  The weight gradient (k_conv_wgrad) stages the same bricks, in another
// layout, and sums over runs of them.
#include <cuda_bf16.h>

#include <cmath>
#include <cstring>

#include "cmg_internal.cuh"
#include "conv_tc.cuh"

namespace cmg {
namespace {

using bf16 = __nv_bfloat16;

constexpr int kConvThreads = 128;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void ldsm_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(addr));
}

__device__ __forceinline__ void mma16816(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ int wrap(int a, int D) { return a < 0 ? a + D : (a >= D ? a - D : a); }

// Global voxel row of halo cell (hz, hy, hx) (0..5) around brick (bz, by, bx).
__device__ __forceinline__ int64_t halo_row(int64_t sbase, int D, int bz, int by, int bx, int hz, int hy, int hx) {
  const int z = wrap(bz * 4 + hz - 1, D), y = wrap(by * 4 + hy - 1, D), x = wrap(bx * 4 + hx - 1, D);
  return sbase + ((int64_t)z * D + y) * D + x;
}

// out[v][n] = sum_t sum_k in[v + SIGN d_t][k] * W[n][t][k] (+ bias, ReLU).
// SIGN = +1: forward conv (W = [Cout][27][Cin]); SIGN = -1: input gradient
// (in = output gradient, W = [Cin][27][Cout]).  N = 8 NT output channels.
template <int NT, int SIGN, bool BIAS_RELU>
__global__ void __launch_bounds__(kConvThreads) k_conv(const bf16 *__restrict__ in, int K, const bf16 *__restrict__ W,
                                                      const float *__restrict__ bias, const bf16 *__restrict__ mask,
                                                      bf16 *__restrict__ out, int D) {
  extern __shared__ __align__(16) uint8_t smem[];
  constexpr int N = NT * 8;
  bf16 *halo = reinterpret_cast<bf16 *>(smem);  // [216][16]
  bf16 *wt = halo + 216 * 16;                   // [N][27][16]
  const int D4 = D >> 2;
  const int brick = blockIdx.x;
  const int bx = brick % D4, by = (brick / D4) % D4, bz = brick / (D4 * D4);
  const int64_t sbase = (int64_t)blockIdx.y * D * D * D;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float acc[NT][4];
#pragma unroll
  for (int j = 0; j < NT; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.f;
  // A-fragment row of this lane: voxel m of the warp's 16 (z = warp)
  const int am = (lane & 7) + ((lane >> 3) & 1) * 8, akofs = (lane >> 4) * 8;
  const int ay = am >> 2, ax = am & 3;
  const int bn = (lane & 7) + ((lane >> 4) & 1) * 8, bkofs = ((lane >> 3) & 1) * 8;
  for (int kc = 0; kc < K / 16; ++kc) {
    for (int p = threadIdx.x; p < 432; p += kConvThreads) {
      const int row = p >> 1, half = p & 1;
      const int hz = row / 36, hy = (row / 6) % 6, hx = row % 6;
      const int64_t g = halo_row(sbase, D, bz, by, bx, hz, hy, hx);
      *reinterpret_cast<uint4 *>(halo + row * 16 + half * 8) =
          *reinterpret_cast<const uint4 *>(in + g * K + kc * 16 + half * 8);
    }
    for (int p = threadIdx.x; p < N * 27 * 2; p += kConvThreads) {
      const int r = p >> 1, half = p & 1;
      *reinterpret_cast<uint4 *>(wt + r * 16 + half * 8) =
          *reinterpret_cast<const uint4 *>(W + (int64_t)r * K + kc * 16 + half * 8);
    }
    __syncthreads();
#pragma unroll 1
    for (int t = 0; t < 27; ++t) {
      const int dz = SIGN * (t / 9 - 1), dy = SIGN * ((t / 3) % 3 - 1), dx = SIGN * (t % 3 - 1);
      const int hrow = ((warp + dz + 1) * 6 + (ay + dy + 1)) * 6 + (ax + dx + 1);
      uint32_t a0, a1, a2, a3;
      ldsm_x4(smem_u32(halo + hrow * 16 + akofs), a0, a1, a2, a3);
#pragma unroll
      for (int np = 0; np < NT / 2; ++np) {
        uint32_t b0, b1, b2, b3;
        ldsm_x4(smem_u32(wt + ((np * 16 + bn) * 27 + t) * 16 + bkofs), b0, b1, b2, b3);
        mma16816(acc[2 * np], a0, a1, a2, a3, b0, b1);
        mma16816(acc[2 * np + 1], a0, a1, a2, a3, b2, b3);
      }
    }
    __syncthreads();
  }
  const int g = lane >> 2, q = lane & 3;
#pragma unroll
  for (int j = 0; j < NT; ++j) {
    const int c0 = j * 8 + q * 2;
    float bv0 = 0.f, bv1 = 0.f;
    if (BIAS_RELU) {
      bv0 = bias[c0];
      bv1 = bias[c0 + 1];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m = g + h * 8;
      const int64_t v = sbase + ((int64_t)(bz * 4 + warp) * D + by * 4 + (m >> 2)) * D + bx * 4 + (m & 3);
      float x0 = acc[j][2 * h] + bv0, x1 = acc[j][2 * h + 1] + bv1;
      if (BIAS_RELU) {
        x0 = fmaxf(x0, 0.f);
        x1 = fmaxf(x1, 0.f);
      } else if (mask != nullptr) {  // ReLU derivative from the stored activations
        const __nv_bfloat162 act = *reinterpret_cast<const __nv_bfloat162 *>(mask + v * N + c0);
        if (!(__low2float(act) > 0.f)) x0 = 0.f;
        if (!(__high2float(act) > 0.f)) x1 = 0.f;
      }
      *reinterpret_cast<__nv_bfloat162 *>(out + v * N + c0) = __floats2bfloat162_rn(x0, x1);
    }
  }
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// Weight and bias gradients of one layer:
//   dW[co][t][ci] += sum_v dout[v][co] in[v + d_t][ci],  db[co] += sum_v dout[v][co].
// `in` is a tensor of CIN channels, or (up) the channel concatenation of the
// nearest-upsampled `in` (Ca channels on the D/2 grid) and `skip` (Cb), read
// in place.
//
// The order of the sums is part of the result: the tensor cores truncate as
// they accumulate, an error that grows with the length of a run of MMAs (up to
// 4e-6 of a layer's gradient between runs of different lengths), and Adam's
// first steps and the weights' rounding to bf16 turn such a difference into
// one of 1e-4 of the next gradients.  So a layer's bricks of 4x4x4 voxels are
// dealt out in runs of `per_run` consecutive ones, every weight is one
// accumulator over each run (a brick's four z slices one after the other, the
// 16 voxels of a slice in one MMA), and the runs' sums meet in FP32 additions:
// a training step repeats the steps of earlier versions up to the order of
// those additions (3e-7).
//
// What bounds it: with 16 output channels every B fragment (16 voxels x 16
// input channels, one ldmatrix.x4) feeds only two MMAs, so the ldmatrix reads
// of shared memory (4 clocks each) weigh as much as the MMAs.  Hence the
// split: a block takes one run, one slice of 16 input channels, NM tiles of
// 16 output channels (2 where the layer has them) and all 27 taps, so that a
// brick's halo is staged once for all of them; a warp takes the 9 taps of one
// dz, so that its A fragments (dout^T) are read once for 9 taps and its B
// fragments serve NM tiles.  Halo rows hold their 6 voxels' lower channels and then the upper
// ones (12 x 16 bytes), dout planes of 8 channels: the 8 addresses of an
// ldmatrix phase (two halo rows of 4 voxels, 8 voxels of dout) lie in
// different banks, and a tap's offset is an immediate.  Several blocks per SM
// walk their bricks through a cp.async ring with one barrier per brick, so
// that their staging and MMA phases overlap.  The bias gradient is one more
// MMA per A fragment, against ones, whose 16-voxel sums are added in FP32.
// Measured on GB300: all layers of a training step on 8 blocks of 64^3 take
// 1.08 ms (245 TFLOP/s; the mma.sync rate, about 1024 multiply-adds per SM and
// clock, would give 0.42 ms); with a brick's halo staged once per group of taps
// and dout fragments read once per tap, the same sums took 3.61 ms.  Bricks of
// 8x8x4 voxels with another order of the sums: 1.03 ms.
// A block's output channels: 16 NM.
template <int NM>
struct WgradGeom {
  static constexpr int kThreads = 96, kCo = 16 * NM;
  static constexpr int kBlocks = 4;  // per SM: what the accumulators leave registers for
  static constexpr int kStages = 3;
  static constexpr int kHalo = 216 * 32;
  // plane stride: 8 lanes of a copy (8 / planes voxels x planes) hit distinct banks
  static constexpr int kDoutPlane = 64 * 16 + 1024 / kCo;
  static constexpr int kStage = kHalo + (kCo / 8) * kDoutPlane;
  static constexpr int kSmem = kStages * kStage;
  static constexpr int kHaloPieces = (432 + kThreads - 1) / kThreads;  // 16-byte pieces per thread
  static constexpr int kDoutPieces = (64 * (kCo / 8) + kThreads - 1) / kThreads;
};

template <int NM>
__global__ void __launch_bounds__(WgradGeom<NM>::kThreads, WgradGeom<NM>::kBlocks)
    k_conv_wgrad(const bf16 *__restrict__ dout, int COUT, const bf16 *__restrict__ in, int CIN,
                 const bf16 *__restrict__ skip, int Cb, float *__restrict__ dW, float *__restrict__ db, int D,
                 int nbricks, int per_run) {
  using G = WgradGeom<NM>;
  constexpr int C8 = G::kCo / 8, kUnroll = NM == 1 ? 4 : 1;  // one tile leaves registers to unroll
  extern __shared__ __align__(16) uint8_t smem[];
  const int lane = threadIdx.x & 31, dz = threadIdx.x >> 5, co_first = blockIdx.z * G::kCo;
  const int first = blockIdx.x * per_run, last = min(first + per_run, nbricks);
  const int nb = D >> 2;
  // this block's slice of 16 input channels
  const int Ca = CIN - Cb, c_first = blockIdx.y * 16;
  const bool two = skip != nullptr, up = two && c_first < Ca;
  const int cstride = up ? Ca : (two ? Cb : CIN), cbase = (two && !up) ? c_first - Ca : c_first;
  const bf16 *src = ((two && !up) ? skip : in) + cbase;
  const int Dg = up ? D >> 1 : D, sh = up ? 1 : 0;
  const uint32_t base = smem_u32(smem);

  // the brick staged next
  int bx = first % nb, by = (first / nb) % nb, bz = (first / (nb * nb)) % nb, smp = first / (nb * nb * nb);
  auto stage = [&](int buf) {
    const uint32_t halo = base + buf * G::kStage, dt = halo + G::kHalo;
    const bf16 *ss = src + (int64_t)smp * Dg * Dg * Dg * cstride;
    const int x0 = bx * 4, y0 = by * 4, z0 = bz * 4;
    // 16-byte pieces in the order of the rows in shared memory: voxel (hz, hy,
    // hx) and channel half
#pragma unroll
    for (int k = 0; k < G::kHaloPieces; ++k) {
      const int p = threadIdx.x + k * G::kThreads;
      const int hz = p / 72, hy = (p / 12) % 6, half = (p / 6) & 1, hx = p % 6;
      const int z = wrap(z0 + hz - 1, D) >> sh, y = wrap(y0 + hy - 1, D) >> sh, x = wrap(x0 + hx - 1, D) >> sh;
      if (p < 432) cp_async16(halo + p * 16, ss + ((int64_t)(z * Dg + y) * Dg + x) * cstride + half * 8);
    }
    const bf16 *ds = dout + ((((int64_t)smp * D + z0) * D + y0) * D + x0) * COUT + co_first;
#pragma unroll
    for (int k = 0; k < G::kDoutPieces; ++k) {
      const int p = threadIdx.x + k * G::kThreads, v = p / C8, c8 = p % C8;
      if (p < 64 * C8)
        cp_async16(dt + c8 * G::kDoutPlane + v * 16, ds + (((v >> 4) * D + ((v >> 2) & 3)) * D + (v & 3)) * COUT + c8 * 8);
    }
    if (++bx == nb) {
      bx = 0;
      if (++by == nb) {
        by = 0;
        if (++bz == nb) {
          bz = 0;
          ++smp;
        }
      }
    }
  };

  float acc[9][NM][2][4], sum[NM][2];
#pragma unroll
  for (int m = 0; m < NM; ++m) {
#pragma unroll
    for (int t = 0; t < 9; ++t)
#pragma unroll
      for (int h = 0; h < 2; ++h) acc[t][m][h][0] = acc[t][m][h][1] = acc[t][m][h][2] = acc[t][m][h][3] = 0.f;
    sum[m][0] = sum[m][1] = 0.f;
  }
  const bool bias = blockIdx.y == 0 && dz == 0;
  const int bk = (lane & 7) + ((lane >> 3) & 1) * 8, bhalf = (lane >> 4) & 1;  // B rows: voxel bk, channel half
  const int ak = (lane & 7) + ((lane >> 4) & 1) * 8, ahalf = (lane >> 3) & 1;  // A rows
  const uint32_t lane_a = G::kHalo + ahalf * G::kDoutPlane + ak * 16;
  const uint32_t lane_b = ((dz * 6 + (bk >> 2)) * 12 + bhalf * 6 + (bk & 3)) * 16;
  int buf = 0;
#pragma unroll
  for (int k = 0; k < G::kStages - 1; ++k) {
    if (first + k < last) stage(k);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int bi = first; bi < last; ++bi, buf = buf + 1 == G::kStages ? 0 : buf + 1) {
    asm volatile("cp.async.wait_group %0;" ::"n"(G::kStages - 2) : "memory");
    __syncthreads();  // this brick has landed, and the buffer filled next was read a brick ago
    if (bi + G::kStages - 1 < last) stage(buf == 0 ? G::kStages - 1 : buf - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const uint32_t at = base + buf * G::kStage;
#pragma unroll(kUnroll)
    for (int i = 0; i < 4; ++i) {  // the brick's z slices
      uint32_t a[NM][4];
#pragma unroll
      for (int m = 0; m < NM; ++m)
        ldsm_x4_t(at + lane_a + 2 * m * G::kDoutPlane + i * 256, a[m][0], a[m][1], a[m][2], a[m][3]);
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        uint32_t b0, b1, b2, b3;
        ldsm_x4_t(at + lane_b + ((i * 6 + t / 3) * 12 + t % 3) * 16, b0, b1, b2, b3);
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          mma16816(acc[t][m][0], a[m][0], a[m][1], a[m][2], a[m][3], b0, b1);
          mma16816(acc[t][m][1], a[m][0], a[m][1], a[m][2], a[m][3], b2, b3);
        }
      }
      if (bias) {
        constexpr uint32_t kOnes = 0x3F803F80u;  // bf16 1, 1
#pragma unroll
        for (int m = 0; m < NM; ++m) {
          float c[4] = {0.f, 0.f, 0.f, 0.f};
          mma16816(c, a[m][0], a[m][1], a[m][2], a[m][3], kOnes, kOnes);
          sum[m][0] += c[0];
          sum[m][1] += c[2];
        }
      }
    }
  }
  // one red.v2 per pair of ci
  const int g = lane >> 2, q = lane & 3;
#pragma unroll
  for (int m = 0; m < NM; ++m)
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int co = co_first + m * 16 + g + 8 * hh;
      float *dst = dW + ((int64_t)co * 27 + dz * 9) * CIN + c_first + 2 * q;
#pragma unroll
      for (int t = 0; t < 9; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(dst + t * CIN + 8 * h),
                       "f"(acc[t][m][h][2 * hh]), "f"(acc[t][m][h][2 * hh + 1])
                       : "memory");
      if (bias && q == 0) atomicAdd(db + co, sum[m][hh]);
    }
}

// ---- per-sample input statistics and the network input
// stats[b] = {sum rho, sum rho^2, sum phi^2}: per-thread FP32 partial sums,
// combined in FP64 (GB300's FP64 rate is a small fraction of FP32's)
__global__ void k_stats(const float *__restrict__ rho, const float *__restrict__ phi, int64_t V,
                        double *__restrict__ stats) {
  const int b = blockIdx.y;
  float f0 = 0.f, f1 = 0.f, f2 = 0.f;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    const float r = rho[b * V + v], p = phi[b * V + v];
    f0 += r;
    f1 = fmaf(r, r, f1);
    f2 = fmaf(p, p, f2);
  }
  double s0 = f0, s1 = f1, s2 = f2;
  for (int o = 16; o > 0; o >>= 1) {
    s0 += __shfl_down_sync(0xffffffffu, s0, o);
    s1 += __shfl_down_sync(0xffffffffu, s1, o);
    s2 += __shfl_down_sync(0xffffffffu, s2, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(stats + 3 * b, s0);
    atomicAdd(stats + 3 * b + 1, s1);
    atomicAdd(stats + 3 * b + 2, s2);
  }
}

// norm[b] = {mean, 1/std, out_scale * rms}, plus 1/rms at norm_in[b] (one thread per sample)
__global__ void k_norm(const double *__restrict__ stats, int64_t V, int B, float out_scale, float *__restrict__ norm,
                       float *__restrict__ inv_rms) {
  const int b = threadIdx.x;
  if (b >= B) return;
  const double n = (double)V;
  const double mean = stats[3 * b] / n;
  const double var = fmax(stats[3 * b + 1] / n - mean * mean, 1e-300);
  const double rms = sqrt(stats[3 * b + 2] / n);
  norm[3 * b] = (float)mean;
  norm[3 * b + 1] = (float)(1.0 / sqrt(var));
  norm[3 * b + 2] = (float)(out_scale * rms);
  inv_rms[b] = (float)(1.0 / rms);
}

// x[b][v][0] = (rho - mean) / std, x[..][1] = phi / rms, channels 2..15 = 0
__global__ void k_input(const float *__restrict__ rho, const float *__restrict__ phi, int64_t V,
                        const float *__restrict__ norm, const float *__restrict__ inv_rms, bf16 *__restrict__ x) {
  const int b = blockIdx.y;
  const float mean = norm[3 * b], inv_std = norm[3 * b + 1], ir = inv_rms[b];
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < V; v += (int64_t)gridDim.x * blockDim.x) {
    __align__(16) __nv_bfloat162 row[8];
    row[0] = __floats2bfloat162_rn((rho[b * V + v] - mean) * inv_std, phi[b * V + v] * ir);
#pragma unroll
    for (int c = 1; c < 8; ++c) row[c] = __floats2bfloat162_rn(0.f, 0.f);
    uint4 *dst = reinterpret_cast<uint4 *>(x + (b * V + v) * 16);
    dst[0] = reinterpret_cast<const uint4 *>(row)[0];
    dst[1] = reinterpret_cast<const uint4 *>(row)[1];
  }
}

// 2x2x2 mean pooling: in [B][D^3][C] -> out [B][(D/2)^3][C]
__global__ void k_pool(const bf16 *__restrict__ in, int D, int C, int B, bf16 *__restrict__ out) {
  const int Dh = D / 2;
  const int64_t total = (int64_t)B * Dh * Dh * Dh * C;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % C);
    const int64_t u = e / C;
    const int64_t b = u / ((int64_t)Dh * Dh * Dh);
    const int64_t r = u % ((int64_t)Dh * Dh * Dh);
    const int z = (int)(r / (Dh * Dh)), y = (int)((r / Dh) % Dh), x = (int)(r % Dh);
    float s = 0.f;
    for (int k = 0; k < 8; ++k) {
      const int64_t v = b * D * D * D + ((int64_t)(2 * z + (k >> 2)) * D + 2 * y + ((k >> 1) & 1)) * D + 2 * x + (k & 1);
      s += __bfloat162float(in[v * C + c]);
    }
    out[e] = __float2bfloat16_rn(s * 0.125f);
  }
}

// out [B][D^3][Ca+Cb] = [nearest-upsampled a (D/2 grid, Ca), b (D grid, Cb)],
// 8 channels (16 bytes) per thread
__global__ void k_up_concat(const bf16 *__restrict__ a, int Ca, const bf16 *__restrict__ b, int Cb, int D, int B,
                            bf16 *__restrict__ out) {
  const int C8 = (Ca + Cb) / 8, Ca8 = Ca / 8, Dh = D / 2;
  const int64_t total = (int64_t)B * D * D * D * C8;
  const uint4 *av = reinterpret_cast<const uint4 *>(a), *bv = reinterpret_cast<const uint4 *>(b);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = e / C8;
    const int c = (int)(e - v * C8);
    uint4 x;
    if (c < Ca8) {
      const int xx = (int)(v % D), y = (int)((v / D) % D);
      const int64_t sz = v / ((int64_t)D * D);  // sample * D + z, D even
      x = av[(((sz >> 1) * Dh + (y >> 1)) * Dh + (xx >> 1)) * Ca8 + c];
    } else {
      x = bv[v * (Cb / 8) + (c - Ca8)];
    }
    reinterpret_cast<uint4 *>(out)[e] = x;
  }
}

// head: delta[v] = sum_c d0[v][c] w[c] + b; phi_pred = phi_prev + rms delta
__global__ void k_head(const bf16 *__restrict__ d0, const float *__restrict__ hw, const float *__restrict__ hb,
                       const float *__restrict__ phi_prev, const float *__restrict__ norm, int64_t V, int B,
                       float *__restrict__ delta, float *__restrict__ phi_pred) {
  const int64_t total = (int64_t)B * V;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    float s = hb[0];
#pragma unroll
    for (int c = 0; c < 16; ++c) s = fmaf(__bfloat162float(d0[e * 16 + c]), hw[c], s);
    if (delta) delta[e] = s;
    if (phi_pred) phi_pred[e] = phi_prev[e] + norm[3 * (e / V) + 2] * s;
  }
}

// loss = mean (delta - target)^2, target = (phi_next - phi_prev) / rms;
// ddelta = 2 (delta - target) / (B V); dact = bf16(ddelta w) where d0 > 0,
// else 0 (the ReLU derivative); head grads.  One voxel (32 bytes of d0 and
// dact) per thread and step.  The grid is part of the head gradients' rounding
// (see k_conv_wgrad): up to 4096 blocks, whose FP32 sums are added up.
__global__ void __launch_bounds__(256) k_head_grad(const bf16 *__restrict__ d0, const float *__restrict__ hw,
                                                  const float *__restrict__ delta, const float *__restrict__ phi_prev,
                                                  const float *__restrict__ phi_next, const float *__restrict__ norm,
                                                  int64_t V, int B, bf16 *__restrict__ dact, float *__restrict__ ghw,
                                                  float *__restrict__ ghb, double *__restrict__ loss) {
  __shared__ float sh[17][8];
  const int64_t total = (int64_t)B * V;
  const float inv_n = 1.f / (float)total;
  float acc[17], w[16];
#pragma unroll
  for (int c = 0; c < 17; ++c) acc[c] = 0.f;
#pragma unroll
  for (int c = 0; c < 16; ++c) w[c] = hw[c];
  double l = 0.0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    __align__(16) __nv_bfloat162 d[8], o[8];
    reinterpret_cast<uint4 *>(d)[0] = __ldg(reinterpret_cast<const uint4 *>(d0 + e * 16));
    reinterpret_cast<uint4 *>(d)[1] = __ldg(reinterpret_cast<const uint4 *>(d0 + e * 16) + 1);
    const float target = (phi_next[e] - phi_prev[e]) / norm[3 * (e / V) + 2];
    const float diff = delta[e] - target;
    l += (double)diff * diff;
    const float dd = 2.f * diff * inv_n;
    acc[16] += dd;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float x0 = __low2float(d[q]), x1 = __high2float(d[q]);
      acc[2 * q] = fmaf(x0, dd, acc[2 * q]);
      acc[2 * q + 1] = fmaf(x1, dd, acc[2 * q + 1]);
      o[q] = __floats2bfloat162_rn(x0 > 0.f ? dd * w[2 * q] : 0.f, x1 > 0.f ? dd * w[2 * q + 1] : 0.f);
    }
    uint4 *dst = reinterpret_cast<uint4 *>(dact + e * 16);
    dst[0] = reinterpret_cast<const uint4 *>(o)[0];
    dst[1] = reinterpret_cast<const uint4 *>(o)[1];
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 17; ++c) {
    float v = acc[c];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) sh[c][warp] = v;
  }
  for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
  if (lane == 0) atomicAdd(loss, l);
  __syncthreads();
  if (threadIdx.x < 17) {
    float v = 0.f;
    for (int w2 = 0; w2 < (int)(blockDim.x >> 5); ++w2) v += sh[threadIdx.x][w2];
    if (threadIdx.x < 16) atomicAdd(ghw + threadIdx.x, v); else atomicAdd(ghb, v);
  }
}

// bf16 x 8 with entries zeroed where act is not above 0 (the ReLU derivative)
__device__ __forceinline__ uint4 pack_masked(const float v[8], const bf16 *act) {
  __align__(16) __nv_bfloat162 o[4], a[4];
  *reinterpret_cast<uint4 *>(a) = __ldg(reinterpret_cast<const uint4 *>(act));
#pragma unroll
  for (int q = 0; q < 4; ++q)
    o[q] = __floats2bfloat162_rn(__low2float(a[q]) > 0.f ? v[2 * q] : 0.f, __high2float(a[q]) > 0.f ? v[2 * q + 1] : 0.f);
  return *reinterpret_cast<const uint4 *>(o);
}
__device__ __forceinline__ void unpack8(const bf16 *p, float v[8]) {
  __align__(16) __nv_bfloat162 a[4];
  *reinterpret_cast<uint4 *>(a) = __ldg(reinterpret_cast<const uint4 *>(p));
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    v[2 * q] = __low2float(a[q]);
    v[2 * q + 1] = __high2float(a[q]);
  }
}

// gradient split of a concat [up(a) (Ca), b (Cb)] on the D grid, 8 channels
// (16 bytes) per thread:
//   da[u][c] = bf16(sum over the 8 children of dcat[..][c]), c < Ca (D/2
//   grid), 0 where the activation a is
__global__ void k_up_grad(const bf16 *__restrict__ dcat, int Ca, int Cb, const bf16 *__restrict__ act, int D, int B,
                          bf16 *__restrict__ da) {
  const int C = Ca + Cb, Ca8 = Ca / 8, Dh = D / 2;
  const int64_t total = (int64_t)B * Dh * Dh * Dh * Ca8;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = e / Ca8;
    const int c = (int)(e - u * Ca8) * 8;
    const int x = (int)(u % Dh), y = (int)((u / Dh) % Dh);
    const int64_t sz = u / ((int64_t)Dh * Dh);  // sample * Dh + z
    const bf16 *p = dcat + ((2 * sz * D + 2 * y) * D + 2 * x) * C + c;
    float acc[8] = {};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      float v[8];
      unpack8(p + (((int64_t)(k >> 2) * D + ((k >> 1) & 1)) * D + (k & 1)) * C, v);
#pragma unroll
      for (int q = 0; q < 8; ++q) acc[q] += v[q];
    }
    *reinterpret_cast<uint4 *>(da + e * 8) = pack_masked(acc, act + e * 8);
  }
}

// skip gradient: ds[v][c] = bf16(dcat[v][Ca + c] + dpool[parent(v)][c] / 8),
// 0 where the skip's activation is; 8 channels per thread
__global__ void k_skip_grad(const bf16 *__restrict__ dcat, int Ca, int Cb, const bf16 *__restrict__ dpool,
                            const bf16 *__restrict__ act, int D, int B, bf16 *__restrict__ ds) {
  const int C = Ca + Cb, Cb8 = Cb / 8, Dh = D / 2;
  const int64_t total = (int64_t)B * D * D * D * Cb8;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = e / Cb8;
    const int c = (int)(e - v * Cb8) * 8;
    const int x = (int)(v % D), y = (int)((v / D) % D);
    const int64_t sz = v / ((int64_t)D * D);  // sample * D + z, D even
    float a[8], b[8];
    unpack8(dcat + v * C + Ca + c, a);
    unpack8(dpool + (((sz >> 1) * Dh + (y >> 1)) * Dh + (x >> 1)) * Cb + c, b);
#pragma unroll
    for (int q = 0; q < 8; ++q) a[q] = a[q] + b[q] * 0.125f;
    *reinterpret_cast<uint4 *>(ds + e * 8) = pack_masked(a, act + e * 8);
  }
}

// Sum of squares of the gradient into clip[0] (block sums, one atomic each).
__global__ void k_grad_sq(const float *__restrict__ g, int64_t n, double *__restrict__ clip) {
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    acc += (double)g[i] * (double)g[i];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
  __shared__ double ws[32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += ws[w];
    atomicAdd(clip, t);
  }
}

// The clipping scale of this step: the gradient's 2-norm is capped at k times
// the running mean of the earlier steps' (capped) norms, once 20 steps have
// formed that mean; the mean then takes the capped norm.  Resets the sum.
__global__ void k_clip_scale(double *clip, float k) {
  const double norm = sqrt(clip[0]);
  const double mean = clip[1], seen = clip[2];
  double scale = 1.0, kept = norm;
  if (seen >= 20.0 && norm > k * mean && norm > 0.0) {
    scale = k * mean / norm;
    kept = k * mean;
    clip[4] += 1.0;
  }
  clip[1] = seen == 0.0 ? kept : 0.95 * mean + 0.05 * kept;
  clip[2] = seen + 1.0;
  clip[3] = scale;
  clip[5] = norm;
  clip[0] = 0.0;
}

// Adam on the FP32 master parameters; with clip, the gradient is scaled by
// clip[3] first.
__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, int64_t n, float lr, float b1, float b2, float eps, float c1, float c2,
                       const double *__restrict__ clip) {
  const float gs = clip ? (float)clip[3] : 1.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i] * gs;
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// bf16 weight copies of every layer (blockIdx.y) from the master vector: W
// [co][t][ci], WT [ci][t][co], and both arranged for the tcgen05 kernels.
struct WeightPlan {
  struct Layer {
    const float *w;
    int co, ci;
    bf16 *W, *WT, *WI, *WTI;
  } l[10];
};
__global__ void k_prepare_weights(const __grid_constant__ WeightPlan P) {
  const WeightPlan::Layer &L = P.l[blockIdx.y];
  const int n = L.co * 27 * L.ci;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int ci = e % L.ci, t = (e / L.ci) % 27, co = e / (27 * L.ci);
    const bf16 x = __float2bfloat16_rn(L.w[e]);
    L.W[e] = x;
    L.WT[(ci * 27 + t) * L.co + co] = x;
    L.WI[tc::image_index(L.co, 1, co, t, ci)] = x;
    L.WTI[tc::image_index(L.ci, -1, ci, t, co)] = x;
  }
}

// dense [B][D^3] (z, y, x) <-> oct-major [n][8] of a full periodic level whose
// octs are listed x fastest (child c = bx + 2 by + 4 bz)
__global__ void k_dense_octs(const double *__restrict__ src, int D, int64_t n, double *__restrict__ dst, int to_octs) {
  const int Do = D / 2;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < 8 * n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = e >> 3;
    const int c = (int)(e & 7);
    const int ox = (int)(o % Do), oy = (int)((o / Do) % Do), oz = (int)(o / ((int64_t)Do * Do));
    const int64_t v = ((int64_t)(2 * oz + ((c >> 2) & 1)) * D + 2 * oy + ((c >> 1) & 1)) * D + 2 * ox + (c & 1);
    if (to_octs) dst[e] = src[v]; else dst[v] = src[e];
  }
}

unsigned gsz(int64_t n) { return (unsigned)std::min<int64_t>((n + 255) / 256, 4096); }

}  // namespace
}  // namespace cmg

// ----------------------------------------------------------------- network

namespace {

struct LayerSpec {
  const char *name;
  int cin, cout, lvl;
};
constexpr LayerSpec kLayers[10] = {{"enc0a", 16, 16, 0}, {"enc0b", 16, 16, 0}, {"enc1a", 16, 32, 1},
                                   {"enc1b", 32, 32, 1}, {"bota", 32, 64, 2},  {"botb", 64, 64, 2},
                                   {"dec1a", 96, 32, 1}, {"dec1b", 32, 32, 1}, {"dec0a", 48, 16, 0},
                                   {"dec0b", 16, 16, 0}};

int64_t layer_offset(int l) {
  int64_t o = 0;
  for (int k = 0; k < l; ++k) o += (int64_t)kLayers[k].cout * 27 * kLayers[k].cin + kLayers[k].cout;
  return o;
}
int64_t total_params() { return layer_offset(10) + 17; }

}  // namespace

struct cmg_unet {
  cmg_ctx *ctx = nullptr;
  int D = 0, max_batch = 0;
  int64_t np = 0;
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
  __nv_bfloat16 *W[10] = {}, *WT[10] = {};
  // the same weights arranged for the tcgen05 kernels (conv_tc.cuh)
  __nv_bfloat16 *WI[10] = {}, *WTI[10] = {};
  int *d_err = nullptr;  // device status word of the bounded waits
  bool use_tc = true;    // tcgen05 convolutions where the grid allows
  // activations (bf16) and their gradients, per batch sample
  __nv_bfloat16 *x = nullptr, *a[10] = {}, *p0 = nullptr, *p1 = nullptr, *c1 = nullptr, *c0 = nullptr;
  __nv_bfloat16 *g0 = nullptr, *g1 = nullptr, *gc = nullptr, *gx = nullptr, *gs0 = nullptr, *gs1 = nullptr;
  __nv_bfloat16 *gp = nullptr, *gu = nullptr;
  float *delta = nullptr, *norm = nullptr;
  double *stats = nullptr, *loss = nullptr;
  // inputs: rho, field (its rms scales the output), base (the output is
  // base + rms(field) delta), target (training); out = the prediction
  float *in_rho = nullptr, *in_phi = nullptr, *in_base = nullptr, *in_next = nullptr, *out_phi = nullptr;
  // the prediction is base + out_scale * rms(field) * delta
  float out_scale = 1.f;
  int adam_t = 0;
  // gradient-norm clipping (cmg_unet_set_grad_clip): clip_k = 0 off; clip on
  // the device: [0] sum of squares of the step's gradient, [1] running mean
  // of the (clipped) norm, [2] steps seen, [3] scale applied, [4] steps
  // clipped, [5] last norm
  float clip_k = 0.f;
  double *clip = nullptr;
  bool weights_ready = false;
  cmg::DeviceBuffers mem;
};

namespace cmg {
namespace {

using bf16 = __nv_bfloat16;

template <int N, int ZB, bool FWD>
void conv_tc_launch(cmg_unet *U, const bf16 *in, int K, const bf16 *skip, int Cb, const bf16 *WI, const float *bias,
                    bf16 *out, int D, int B, const tc::ConvEpi &ep) {
  using G = tc::ConvGeom<N, ZB>;
  static int attr_dev = -1;
  if (attr_dev != U->ctx->device) {
    CMG_CUDA(cudaFuncSetAttribute(tc::k_conv_tc<N, ZB, FWD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  227 * 1024));
    attr_dev = U->ctx->device;
  }
  const int total = (D / 8) * (D / 16) * (D / ZB) * B;
  const int grid = std::min(total, U->ctx->num_sms);
  LaunchScope ls(U->ctx, FWD ? K_CONV_FWD : K_CONV_DGRAD, 0.0, 2.0 * 27 * K * N * (double)D * D * D * B);
  tc::k_conv_tc<N, ZB, FWD><<<grid, tc::kConvThreads, G::smem_bytes(K), U->ctx->stream>>>(in, K, skip, Cb, WI, bias, out,
                                                                                     D, total, U->d_err, ep);
  CMG_CUDA(cudaGetLastError());
}

template <int NT, int SIGN, bool BR>
void conv_launch(cmg_unet *U, const bf16 *in, int K, const bf16 *W, const float *bias, const bf16 *mask, bf16 *out,
                 int D, int B) {
  const size_t smem = (216 * 16 + (size_t)NT * 8 * 27 * 16) * sizeof(bf16);
  static bool attr = false;
  if (!attr) {
    CMG_CUDA(cudaFuncSetAttribute(k_conv<NT, SIGN, BR>, cudaFuncAttributeMaxDynamicSharedMemorySize, 160 * 1024));
    attr = true;
  }
  const int nb = (D / 4) * (D / 4) * (D / 4);
  LaunchScope ls(U->ctx, SIGN > 0 ? K_CONV_FWD : K_CONV_DGRAD, 0.0, 2.0 * 27 * K * NT * 8 * (double)D * D * D * B);
  k_conv<NT, SIGN, BR><<<dim3(nb, B), kConvThreads, smem, U->ctx->stream>>>(in, K, W, bias, mask, out, D);
  CMG_CUDA(cudaGetLastError());
}

// The tcgen05 path needs bricks of 8 x 16 x ZB voxels: D a multiple of 16.
bool tc_eligible(const cmg_unet *U, int N, int D) {
  return U->use_tc && D >= 16 && D % 16 == 0 && (N == 16 || N == 32 || N == 48 || N == 64 || N == 96);
}

// Deep bricks (ZB = 8 for N = 16, 4 for N = 32, 2 above) when they still
// give every SM a brick, else one-slice bricks.  The epilogue extras need
// N <= 32 (head: N = 16), and the pooling also needs the deep (even) ZB:
// returns whether ep.pool was done (else the caller pools separately).
bool conv_tc(cmg_unet *U, const bf16 *in, int K, const bf16 *skip, int Cb, const bf16 *WI, const float *bias,
             bf16 *out, int N, int D, int B, bool fwd, tc::ConvEpi ep = tc::ConvEpi()) {
  const int zb = N == 16 ? 8 : N == 32 ? 4 : 2;
  const bool deep = (D / 8) * (D / 16) * (D / zb) * B >= U->ctx->num_sms;
  const bool pooled = ep.pool != nullptr && deep && N <= 32;
  tc::ConvEpi e = ep;
  if (!pooled) e.pool = nullptr;
#define CMG_CONV_TC(NN, ZB)                                                                           \
  case NN:                                                                                            \
    if (deep) {                                                                                       \
      if (fwd) conv_tc_launch<NN, ZB, true>(U, in, K, skip, Cb, WI, bias, out, D, B, e);              \
      else conv_tc_launch<NN, ZB, false>(U, in, K, nullptr, 0, WI, nullptr, out, D, B, e);            \
    } else {                                                                                          \
      if (fwd) conv_tc_launch<NN, 1, true>(U, in, K, skip, Cb, WI, bias, out, D, B, e);               \
      else conv_tc_launch<NN, 1, false>(U, in, K, nullptr, 0, WI, nullptr, out, D, B, e);             \
    }                                                                                                 \
    break;
  switch (N) {
    CMG_CONV_TC(16, 8)
    CMG_CONV_TC(32, 4)
    CMG_CONV_TC(48, 2)
    CMG_CONV_TC(64, 2)
    CMG_CONV_TC(96, 2)
    default: throw Error(CMG_ERR_INVALID_ARG, "unsupported channel count");
  }
#undef CMG_CONV_TC
  return pooled;
}

// Convolution of layer l: forward (in = activations, N = cout) or input
// gradient (in = output gradient, N = cin; mask: the activations whose ReLU
// derivative multiplies it, or nullptr).
void conv(cmg_unet *U, int l, const bf16 *in, int K, const float *bias, const bf16 *mask, bf16 *out, int N, int D,
          int B, bool fwd) {
  if (tc_eligible(U, N, D)) {
    tc::ConvEpi ep;
    ep.mask = mask;
    conv_tc(U, in, K, nullptr, 0, fwd ? U->WI[l] : U->WTI[l], bias, out, N, D, B, fwd, ep);
    return;
  }
  const bf16 *W = fwd ? U->W[l] : U->WT[l];
#define CMG_CONV(NT)                                                             \
  case NT:                                                                       \
    if (fwd) conv_launch<NT, 1, true>(U, in, K, W, bias, nullptr, out, D, B);    \
    else conv_launch<NT, -1, false>(U, in, K, W, nullptr, mask, out, D, B);      \
    break;
  switch (N / 8) {
    CMG_CONV(2)
    CMG_CONV(4)
    CMG_CONV(6)
    CMG_CONV(8)
    CMG_CONV(12)
    default: throw Error(CMG_ERR_INVALID_ARG, "unsupported channel count");
  }
#undef CMG_CONV
}

template <int NM>
void wgrad_launch(cmg_ctx *ctx, const bf16 *dout, int Cout, const bf16 *in, int Cin, const bf16 *skip, int Cb, float *dW,
                  float *db, int D, int B) {
  using G = WgradGeom<NM>;
  static_assert(G::kSmem <= 48 * 1024, "more needs an attribute");
  // Runs of bricks (k_conv_wgrad): about 4 per SM, a third or a ninth as many
  // where the layer has more than 3 or 8 tiles of 16 x 16 channels.
  const int nbricks = B * (D / 4) * (D / 4) * (D / 4), slices = Cin / 16, tiles = slices * (Cout / 16);
  const int most = std::max(1, std::min(nbricks, 4 * ctx->num_sms / (tiles <= 3 ? 1 : tiles <= 8 ? 3 : 9)));
  const int per_run = (nbricks + most - 1) / most, runs = (nbricks + per_run - 1) / per_run;
  LaunchScope ls(ctx, K_CONV_WGRAD, 0.0, 2.0 * 27 * Cout * Cin * (double)D * D * D * B);
  k_conv_wgrad<NM><<<dim3(runs, slices, Cout / G::kCo), G::kThreads, G::kSmem, ctx->stream>>>(
      dout, Cout, in, Cin, skip, Cb, dW, db, D, nbricks, per_run);
  CMG_CUDA(cudaGetLastError());
}

// Weight and bias gradients; skip: see k_conv_wgrad.
void wgrad(cmg_ctx *ctx, const bf16 *dout, int Cout, const bf16 *in, int Cin, const bf16 *skip, int Cb, float *dW,
           float *db, int D, int B) {
  if (Cin % 16 || (Cout != 16 && Cout % 32)) throw Error(CMG_ERR_INVALID_ARG, "unsupported channel count");
  if (Cout == 16) wgrad_launch<1>(ctx, dout, Cout, in, Cin, skip, Cb, dW, db, D, B);
  else wgrad_launch<2>(ctx, dout, Cout, in, Cin, skip, Cb, dW, db, D, B);
}

// After a synchronisation: a bounded wait that expired in a tcgen05
// convolution is reported (and the status word cleared).
void check_status(cmg_unet *U) {
  int e = 0;
  CMG_CUDA(cudaMemcpy(&e, U->d_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (e != 0) {
    CMG_CUDA(cudaMemset(U->d_err, 0, sizeof(int)));
    throw Error(e, "U-Net convolution: a bounded wait expired (tensor-core pipeline stalled)");
  }
}

int dim_of(const cmg_unet *U, int lvl) { return U->D >> lvl; }
int64_t vox(const cmg_unet *U, int lvl) {
  const int64_t d = dim_of(U, lvl);
  return d * d * d;
}

void prepare_weights(cmg_unet *U) {
  if (U->weights_ready) return;
  cudaStream_t s = U->ctx->stream;
  WeightPlan P;
  for (int l = 0; l < 10; ++l)
    P.l[l] = {U->params + layer_offset(l), kLayers[l].cout, kLayers[l].cin, U->W[l], U->WT[l], U->WI[l], U->WTI[l]};
  k_prepare_weights<<<dim3(32, 10), 256, 0, s>>>(P);
  CMG_CUDA(cudaGetLastError());
  U->weights_ready = true;
}

const float *bias_of(cmg_unet *U, int l) {
  return U->params + layer_offset(l) + (int64_t)kLayers[l].cout * 27 * kLayers[l].cin;
}

// Device arrays of one call: inputs (base may be the field, next only in
// training) and outputs (pred, delta or nullptr).  Device-memory arguments are
// read and written in place, host-memory ones through the network's buffers.
struct Fields {
  const float *rho, *phi, *base, *next;
  float *pred, *delta;
};

// Forward pass on F.rho / F.phi (B samples); leaves activations,
// delta and (if phi_pred) phi_prev + rms * delta.
void forward(cmg_unet *U, int B, const Fields &F, bool training) {
  cudaStream_t s = U->ctx->stream;
  prepare_weights(U);
  const int64_t V0 = vox(U, 0);
  CMG_CUDA(cudaMemsetAsync(U->stats, 0, sizeof(double) * 3 * B, s));
  k_stats<<<dim3(64, B), 256, 0, s>>>(F.rho, F.phi, V0, U->stats);
  k_norm<<<1, (B + 31) / 32 * 32, 0, s>>>(U->stats, V0, B, U->out_scale, U->norm, U->norm + 3 * U->max_batch);
  k_input<<<dim3(gsz(V0), B), 256, 0, s>>>(F.rho, F.phi, V0, U->norm, U->norm + 3 * U->max_batch, U->x);
  CMG_CUDA(cudaGetLastError());
  const int D0 = dim_of(U, 0), D1 = dim_of(U, 1);
  auto layer = [&](int l, const bf16 *in, bf16 *out) {
    const LayerSpec &L = kLayers[l];
    conv(U, l, in, L.cin, bias_of(U, l), nullptr, out, L.cout, dim_of(U, L.lvl), B, true);
  };
  // encoder convolution + 2x2x2 pooling (fused into the tcgen05 epilogue
  // where the bricks allow it)
  auto layer_pool = [&](int l, const bf16 *in, bf16 *out, bf16 *pooled) {
    const LayerSpec &L = kLayers[l];
    const int D = dim_of(U, L.lvl);
    bool done = false;
    if (tc_eligible(U, L.cout, D)) {
      tc::ConvEpi ep;
      ep.pool = pooled;
      done = conv_tc(U, in, L.cin, nullptr, 0, U->WI[l], bias_of(U, l), out, L.cout, D, B, true, ep);
    } else {
      layer(l, in, out);
    }
    if (!done) k_pool<<<gsz(B * (int64_t)(D / 2) * (D / 2) * (D / 2) * L.cout), 256, 0, s>>>(out, D, L.cout, B, pooled);
  };
  layer(0, U->x, U->a[0]);
  layer_pool(1, U->a[0], U->a[1], U->p0);  // s0
  layer(2, U->p0, U->a[2]);
  layer_pool(3, U->a[2], U->a[3], U->p1);  // s1
  layer(4, U->p1, U->a[4]);
  layer(5, U->a[4], U->a[5]);
  // decoder convolutions: the tcgen05 kernels read the upsampled coarse map
  // and the skip map directly (so does the weight gradient); the warp-level
  // kernels read the concatenation
  auto up_layer = [&](int l, const bf16 *coarse, int Ca, const bf16 *skipm, int Cb, bf16 *cat, bf16 *out) {
    const LayerSpec &L = kLayers[l];
    const int D = dim_of(U, L.lvl);
    if (tc_eligible(U, L.cout, D)) {
      conv_tc(U, coarse, Ca + Cb, skipm, Cb, U->WI[l], bias_of(U, l), out, L.cout, D, B, true);
      return;
    }
    k_up_concat<<<gsz(B * (int64_t)D * D * D * (Ca + Cb)), 256, 0, s>>>(coarse, Ca, skipm, Cb, D, B, cat);
    layer(l, cat, out);
  };
  up_layer(6, U->a[5], 64, U->a[3], 32, U->c1, U->a[6]);
  layer(7, U->a[6], U->a[7]);
  up_layer(8, U->a[7], 32, U->a[1], 16, U->c0, U->a[8]);
  const float *hw = U->params + layer_offset(10);
  if (!training && tc_eligible(U, 16, D0)) {
    // last convolution + head in one kernel; its activations are not kept
    tc::ConvEpi ep;
    ep.hw = hw;
    ep.base = F.base;
    ep.norm = U->norm;
    ep.delta = F.delta;
    ep.pred = F.pred;
    ep.store_out = 0;
    conv_tc(U, U->a[8], 16, nullptr, 0, U->WI[9], bias_of(U, 9), U->a[9], 16, D0, B, true, ep);
  } else {
    layer(9, U->a[8], U->a[9]);
    k_head<<<gsz(B * V0), 256, 0, s>>>(U->a[9], hw, hw + 16, F.base, U->norm, V0, B, F.delta, F.pred);
  }
  CMG_CUDA(cudaGetLastError());
}

// Backward pass after forward(): gradients (summed over the batch's voxels,
// loss = mean over all voxels) into U->grads; loss into U->loss.
void backward(cmg_unet *U, int B, const Fields &F) {
  cudaStream_t s = U->ctx->stream;
  const int64_t V0 = vox(U, 0), V1 = vox(U, 1), V2 = vox(U, 2);
  const int D0 = dim_of(U, 0), D1 = dim_of(U, 1);
  CMG_CUDA(cudaMemsetAsync(U->grads, 0, sizeof(float) * U->np, s));
  CMG_CUDA(cudaMemsetAsync(U->loss, 0, sizeof(double), s));
  float *ghw = U->grads + layer_offset(10);
  k_head_grad<<<gsz(B * V0), 256, 0, s>>>(
      U->a[9], U->params + layer_offset(10), F.delta, F.base, F.next, U->norm, V0, B, U->g0, ghw, ghw + 16,
      U->loss);
  CMG_CUDA(cudaGetLastError());
  // back through layer l: g (gradient of its pre-activation, bf16) -> its
  // weights' and biases' gradients and the gradient gin of its input, times
  // the ReLU derivative of the layer that made the input (below) if that
  // layer alone did
  auto back = [&](int l, const bf16 *g, const bf16 *in, const bf16 *skip, int Cb, bf16 *gin, const bf16 *below) {
    const LayerSpec &L = kLayers[l];
    const int D = dim_of(U, L.lvl);
    float *gw = U->grads + layer_offset(l);
    wgrad(U->ctx, g, L.cout, in, L.cin, skip, Cb, gw, gw + (int64_t)L.cout * 27 * L.cin, D, B);
    if (gin) conv(U, l, g, L.cout, nullptr, below, gin, L.cin, D, B, false);
  };
  // decoder level 0
  back(9, U->g0, U->a[8], nullptr, 0, U->g1, U->a[8]);           // g1 = grad a8 (16 ch, V0)
  back(8, U->g1, U->a[7], U->a[1], 16, U->gc, nullptr);          // gc = grad [up a7, a1] (48 ch, V0)
  k_up_grad<<<gsz(B * V1 * 4), 256, 0, s>>>(U->gc, 32, 16, U->a[7], D0, B, U->gu);  // grad a7 (32 ch, V1)
  // decoder level 1
  back(7, U->gu, U->a[6], nullptr, 0, U->gx, U->a[6]);           // gx = grad a6 (32 ch, V1)
  back(6, U->gx, U->a[5], U->a[3], 32, U->g0, nullptr);          // g0 reused: grad [up a5, a3] (96 ch, V1)
  k_up_grad<<<gsz(B * V2 * 8), 256, 0, s>>>(U->g0, 64, 32, U->a[5], D1, B, U->gu);  // grad a5 (64 ch, V2)
  // bottleneck
  back(5, U->gu, U->a[4], nullptr, 0, U->gx, U->a[4]);           // grad a4 (64, V2)
  back(4, U->gx, U->p1, nullptr, 0, U->gp, nullptr);             // grad p1 (32, V2)
  k_skip_grad<<<gsz(B * V1 * 4), 256, 0, s>>>(U->g0, 64, 32, U->gp, U->a[3], D1, B, U->gs1);  // grad s1 = a3
  // encoder level 1
  back(3, U->gs1, U->a[2], nullptr, 0, U->gx, U->a[2]);          // grad a2 (32, V1)
  back(2, U->gx, U->p0, nullptr, 0, U->gp, nullptr);             // grad p0 (16, V1)
  k_skip_grad<<<gsz(B * V0 * 2), 256, 0, s>>>(U->gc, 32, 16, U->gp, U->a[1], D0, B, U->gs0);  // grad s0 = a1
  // encoder level 0
  back(1, U->gs0, U->a[0], nullptr, 0, U->g1, U->a[0]);          // grad a0 (16, V0)
  back(0, U->g1, U->x, nullptr, 0, nullptr, nullptr);
  CMG_CUDA(cudaGetLastError());
}

// The kind is left to the runtime: one memory flag stands for all arrays of a
// call, and an array of the other kind is copied all the same.
void copy_async(cmg_unet *U, void *dst, const void *src, int64_t bytes) {
  CMG_CUDA(cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDefault, U->ctx->stream));
}

// The fields of a device-memory call are read and written in place where that
// gives what copies of the inputs at the start and of the outputs at the end
// give; else they go through the network's buffers.
struct FieldArgs {
  cmg_unet *U;
  int64_t n;          // values per field
  bool host;          // a host-memory call
  bool wait = false;  // host memory is copied: the call waits for it

  static cudaPointerAttributes where(const void *p) {
    cudaPointerAttributes a = {};
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
      cudaGetLastError();
      a.type = cudaMemoryTypeUnregistered;
    }
    return a;
  }
  // memory that the kernels can take as it is: the context's GPU's own (host
  // memory in a call marked as device memory is not, nor another GPU's)
  bool resident(const void *p) const {
    if (host) return false;
    const cudaPointerAttributes a = where(p);
    return a.type == cudaMemoryTypeDevice && a.device == U->ctx->device;
  }
  void copy(float *dst, const float *src, const void *callers) {
    copy_async(U, dst, src, sizeof(float) * n);
    const cudaMemoryType t = where(callers).type;
    wait = wait || t == cudaMemoryTypeUnregistered || t == cudaMemoryTypeHost;
  }
  const float *in(float *buf, const float *src) {
    if (resident(src)) return src;
    copy(buf, src, src);
    return buf;
  }
  bool overlap(const float *a, const float *b) const { return a && b && a < b + n && b < a + n; }
  // Where the kernels write an output.  The last one reads the base field and
  // writes both outputs, voxel by voxel, so none of the three may overlap.
  float *out(float *buf, float *dst, const float *base, const float *other) const {
    if (!dst) return nullptr;
    return resident(dst) && !overlap(dst, base) && !overlap(dst, other) ? dst : buf;
  }
  void deliver(float *dst, const float *from) {
    if (dst && dst != from) copy(dst, from, dst);
  }
};

}  // namespace
}  // namespace cmg

// ------------------------------------------------------------------ C ABI

namespace {
template <class F>
int unet_guard(F &&f) {
  try {
    cmg::record_error("");
    return f();
  } catch (const cmg::Error &e) {
    cmg::record_error(e.what());
    return e.code;
  } catch (const std::exception &e) {
    cmg::record_error(e.what());
    return CMG_ERR_CUDA;
  }
}
}  // namespace

extern "C" {

int cmg_unet_create(cmg_ctx *ctx, int grid_dim, int max_batch, cmg_unet **out) {
  return unet_guard([&] {
    if (!out || !ctx || grid_dim < 16 || grid_dim % 16 || max_batch < 1) return (int)CMG_ERR_INVALID_ARG;
    *out = nullptr;
    cudaSetDevice(ctx->device);
    auto *U = new cmg_unet();
    try {
      U->ctx = ctx;
      U->D = grid_dim;
      U->max_batch = max_batch;
      U->np = total_params();
      cudaStream_t s = ctx->stream;
      auto &M = U->mem;
      U->params = M.alloc<float>(U->np, true, s);
      U->grads = M.alloc<float>(U->np, true, s);
      U->m = M.alloc<float>(U->np, true, s);
      U->v = M.alloc<float>(U->np, true, s);
      U->clip = M.alloc<double>(8, true, s);
      for (int l = 0; l < 10; ++l) {
        const int64_t n = (int64_t)kLayers[l].cout * 27 * kLayers[l].cin;
        U->W[l] = reinterpret_cast<__nv_bfloat16 *>(M.alloc<uint16_t>(n));
        U->WT[l] = reinterpret_cast<__nv_bfloat16 *>(M.alloc<uint16_t>(n));
        U->WI[l] = reinterpret_cast<__nv_bfloat16 *>(M.alloc<uint16_t>(n));
        U->WTI[l] = reinterpret_cast<__nv_bfloat16 *>(M.alloc<uint16_t>(n));
      }
      const int64_t B = max_batch;
      const int64_t V0 = (int64_t)grid_dim * grid_dim * grid_dim, V1 = V0 / 8, V2 = V0 / 64;
      auto act = [&](int64_t n) { return reinterpret_cast<__nv_bfloat16 *>(M.alloc<uint16_t>(n)); };
      U->x = act(B * V0 * 16);
      const int64_t vox_of[3] = {V0, V1, V2};
      for (int l = 0; l < 10; ++l) U->a[l] = act(B * vox_of[kLayers[l].lvl] * kLayers[l].cout);
      U->p0 = act(B * V1 * 16);
      U->p1 = act(B * V2 * 32);
      U->c1 = act(B * V1 * 96);
      U->c0 = act(B * V0 * 48);
      const int64_t big = B * std::max(V0 * 48, V1 * 96);
      U->g0 = act(big);
      U->g1 = act(B * V0 * 16);
      U->gc = act(B * V0 * 48);
      U->gx = act(B * std::max(V1 * 32, V2 * 64));
      U->gs0 = act(B * V0 * 16);
      U->gs1 = act(B * V1 * 32);
      U->gp = act(B * std::max(V1 * 16, V2 * 32));
      U->gu = act(B * std::max(V1 * 32, V2 * 64));
      U->delta = M.alloc<float>(B * V0);
      U->norm = M.alloc<float>(4 * B);  // {mean, 1/std, c rms} per sample, then 1/rms per sample
      U->stats = M.alloc<double>(3 * B);
      U->loss = M.alloc<double>(1);
      U->d_err = M.alloc<int32_t>(1, true, s);
      U->in_rho = M.alloc<float>(B * V0);
      U->in_phi = M.alloc<float>(B * V0);
      U->in_base = M.alloc<float>(B * V0);
      U->in_next = M.alloc<float>(B * V0);
      U->out_phi = M.alloc<float>(B * V0);
      CMG_CUDA(cudaStreamSynchronize(s));
    } catch (...) {
      U->mem.release();
      delete U;
      throw;
    }
    *out = U;
    return (int)CMG_OK;
  });
}

int cmg_unet_destroy(cmg_unet *U) {
  if (!U) return CMG_OK;
  cudaSetDevice(U->ctx->device);
  cudaStreamSynchronize(U->ctx->stream);
  U->mem.release();
  delete U;
  return CMG_OK;
}

int cmg_unet_n_params(const cmg_unet *U, int64_t *n) {
  if (!U || !n) return CMG_ERR_INVALID_ARG;
  *n = U->np;
  return CMG_OK;
}

int cmg_unet_set_params(cmg_unet *U, const float *params, cmg_mem mem) {
  return unet_guard([&] {
    if (!U || !params) return (int)CMG_ERR_INVALID_ARG;
    cudaSetDevice(U->ctx->device);
    cudaStream_t s = U->ctx->stream;
    CMG_CUDA(cudaMemcpyAsync(U->params, params, sizeof(float) * U->np,
                             mem == CMG_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, s));
    CMG_CUDA(cudaMemsetAsync(U->m, 0, sizeof(float) * U->np, s));
    CMG_CUDA(cudaMemsetAsync(U->v, 0, sizeof(float) * U->np, s));
    CMG_CUDA(cudaMemsetAsync(U->clip, 0, sizeof(double) * 8, s));
    U->adam_t = 0;
    U->weights_ready = false;
    CMG_CUDA(cudaStreamSynchronize(s));
    return (int)CMG_OK;
  });
}

int cmg_unet_set_kernels(cmg_unet *U, int tensor_path) {
  if (!U || (tensor_path != 0 && tensor_path != 1)) return CMG_ERR_INVALID_ARG;
  U->use_tc = tensor_path == 1;
  return CMG_OK;
}

int cmg_unet_set_output_scale(cmg_unet *U, float scale) {
  if (!U || !(scale > 0.f) || !std::isfinite(scale)) return CMG_ERR_INVALID_ARG;
  U->out_scale = scale;
  return CMG_OK;
}

int cmg_unet_get_output_scale(const cmg_unet *U, float *scale) {
  if (!U || !scale) return CMG_ERR_INVALID_ARG;
  *scale = U->out_scale;
  return CMG_OK;
}

int cmg_unet_get_params(cmg_unet *U, float *out, cmg_mem mem) {
  return unet_guard([&] {
    if (!U || !out) return (int)CMG_ERR_INVALID_ARG;
    cudaSetDevice(U->ctx->device);
    CMG_CUDA(cudaMemcpyAsync(out, U->params, sizeof(float) * U->np,
                             mem == CMG_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice,
                             U->ctx->stream));
    CMG_CUDA(cudaStreamSynchronize(U->ctx->stream));
    return (int)CMG_OK;
  });
}

int cmg_unet_forward(cmg_unet *U, const float *rho, const float *field, const float *base, int batch,
                     float *phi_pred, float *delta, cmg_mem mem) {
  return unet_guard([&] {
    if (!U || !rho || !field || batch < 1 || batch > U->max_batch) return (int)CMG_ERR_INVALID_ARG;
    cudaSetDevice(U->ctx->device);
    const int64_t n = (int64_t)batch * U->D * U->D * U->D;
    cudaStream_t s = U->ctx->stream;
    cmg::FieldArgs A = {U, n, mem == CMG_MEM_HOST};
    cmg::Fields F = {};
    F.rho = A.in(U->in_rho, rho);
    F.phi = A.in(U->in_phi, field);
    F.base = base ? A.in(U->in_base, base) : F.phi;
    F.pred = A.out(U->out_phi, phi_pred, F.base, delta);
    F.delta = A.out(U->delta, delta, F.base, phi_pred);
    cmg::forward(U, batch, F, false);
    A.deliver(phi_pred, F.pred);
    A.deliver(delta, F.delta);
    if (A.host || A.wait) CMG_CUDA(cudaStreamSynchronize(s));
    if (A.host) cmg::check_status(U);
    return (int)CMG_OK;
  });
}

int cmg_unet_gradients(cmg_unet *U, const float *rho, const float *field, const float *base, const float *target,
                       int batch, float *grads, double *loss, cmg_mem mem) {
  return unet_guard([&] {
    if (!U || !rho || !field || !target || batch < 1 || batch > U->max_batch) return (int)CMG_ERR_INVALID_ARG;
    cudaSetDevice(U->ctx->device);
    const int64_t n = (int64_t)batch * U->D * U->D * U->D;
    cudaStream_t s = U->ctx->stream;
    cmg::FieldArgs A = {U, n, mem == CMG_MEM_HOST};
    cmg::Fields F = {};
    F.rho = A.in(U->in_rho, rho);
    F.phi = A.in(U->in_phi, field);
    F.base = base ? A.in(U->in_base, base) : F.phi;
    F.next = A.in(U->in_next, target);
    F.delta = U->delta;
    cmg::forward(U, batch, F, true);
    cmg::backward(U, batch, F);
    const cudaMemcpyKind k = mem == CMG_MEM_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice;
    if (grads) CMG_CUDA(cudaMemcpyAsync(grads, U->grads, sizeof(float) * U->np, k, s));
    if (loss) {
      CMG_CUDA(cudaMemcpyAsync(loss, U->loss, sizeof(double), k, s));
    }
    if (A.wait && !A.host && !loss) CMG_CUDA(cudaStreamSynchronize(s));
    if (A.host || loss) {
      CMG_CUDA(cudaStreamSynchronize(s));
      cmg::check_status(U);
    }
    if (loss && mem == CMG_MEM_HOST) *loss /= (double)n;
    return (int)CMG_OK;
  });
}

int cmg_unet_adam_step(cmg_unet *U, float lr, float beta1, float beta2, float eps) {
  return unet_guard([&] {
    if (!U || !(lr >= 0.f)) return (int)CMG_ERR_INVALID_ARG;
    cudaSetDevice(U->ctx->device);
    U->adam_t += 1;
    const float c1 = 1.f - std::pow(beta1, (float)U->adam_t), c2 = 1.f - std::pow(beta2, (float)U->adam_t);
    const bool clip = U->clip_k > 0.f;
    if (clip) {
      cmg::k_grad_sq<<<cmg::gsz(U->np), 256, 0, U->ctx->stream>>>(U->grads, U->np, U->clip);
      cmg::k_clip_scale<<<1, 1, 0, U->ctx->stream>>>(U->clip, U->clip_k);
    }
    cmg::k_adam<<<cmg::gsz(U->np), 256, 0, U->ctx->stream>>>(U->params, U->grads, U->m, U->v, U->np, lr, beta1,
                                                              beta2, eps, c1, c2, clip ? U->clip : nullptr);
    CMG_CUDA(cudaGetLastError());
    U->weights_ready = false;
    return (int)CMG_OK;
  });
}

int cmg_unet_set_grad_clip(cmg_unet *U, float k) {
  return unet_guard([&] {
    if (!U || !(k == 0.f || k >= 1.f)) return (int)CMG_ERR_INVALID_ARG;
    U->clip_k = k;
    return (int)CMG_OK;
  });
}

int cmg_unet_grad_clip_stats(cmg_unet *U, double *last_norm, double *mean_norm, int64_t *steps, int64_t *clipped) {
  return unet_guard([&] {
    if (!U) return (int)CMG_ERR_INVALID_ARG;
    cudaSetDevice(U->ctx->device);
    double h[8];
    CMG_CUDA(cudaMemcpyAsync(h, U->clip, sizeof(h), cudaMemcpyDeviceToHost, U->ctx->stream));
    CMG_CUDA(cudaStreamSynchronize(U->ctx->stream));
    if (last_norm) *last_norm = h[5];
    if (mean_norm) *mean_norm = h[1];
    if (steps) *steps = (int64_t)h[2];
    if (clipped) *clipped = (int64_t)h[4];
    return (int)CMG_OK;
  });
}

int cmg_debug_conv_wgrad(cmg_ctx *ctx, const uint16_t *dout, int cout, const uint16_t *in, int cin,
                         const uint16_t *skip, int skip_channels, int grid_dim, int batch, float *dw, float *db) {
  return unet_guard([&] {
    if (!ctx || !dout || !in || !dw || !db || grid_dim < 4 || grid_dim % 4 || batch < 1) return (int)CMG_ERR_INVALID_ARG;
    if ((cout != 16 && cout != 32 && cout != 64) || cin < 16 || cin > 96 || cin % 16) return (int)CMG_ERR_INVALID_ARG;
    if (skip ? skip_channels < 16 || skip_channels % 16 || skip_channels >= cin : skip_channels != 0)
      return (int)CMG_ERR_INVALID_ARG;
    cudaSetDevice(ctx->device);
    CMG_CUDA(cudaMemsetAsync(dw, 0, sizeof(float) * cout * 27 * cin, ctx->stream));
    CMG_CUDA(cudaMemsetAsync(db, 0, sizeof(float) * cout, ctx->stream));
    auto b16 = [](const uint16_t *p) { return reinterpret_cast<const __nv_bfloat16 *>(p); };
    cmg::wgrad(ctx, b16(dout), cout, b16(in), cin, b16(skip), skip_channels, dw, db, grid_dim, batch);
    return (int)CMG_OK;
  });
}

int cmg_dense_octs(cmg_ctx *ctx, const double *src, int grid_dim, double *dst, int to_octs) {
  return unet_guard([&] {
    if (!ctx || !src || !dst || grid_dim < 2 || grid_dim % 2) return (int)CMG_ERR_INVALID_ARG;
    cudaSetDevice(ctx->device);
    const int64_t n = (int64_t)(grid_dim / 2) * (grid_dim / 2) * (grid_dim / 2);
    cmg::k_dense_octs<<<cmg::gsz(8 * n), 256, 0, ctx->stream>>>(src, grid_dim, n, dst, to_octs);
    CMG_CUDA(cudaGetLastError());
    return (int)CMG_OK;
  });
}

}  // extern "C"
