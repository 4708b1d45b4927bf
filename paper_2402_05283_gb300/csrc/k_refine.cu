// k_refine.cu - Step D tomographic refinement on the assembled spectrum.
//
// The paper's Step D is conventional 3D CXDI run on the gridded spectrum E(q):
// alternating projections between the support-positivity set of a 3D
// support S3 and the spectra equal to the gridded E(q) on the cells the
// slices reach (the measured mask M, the same for every kz).  Volumes are
// [z][y][x], N^3, in the centred frame of the Step D volume (the frame of
// the 2D supports); V is the spectrum of that volume.  One iteration is four
// passes over the half spectrum of rho (refine_kernels.cuh):
//   y lines   forward FFT_y
//   z lines   forward FFT_z -> error, X <- V where M -> IFFT_z
//   y lines   inverse FFT_y
//   x rows    inverse FFT_x -> rho = Re -> P_{S3+} rho -> forward FFT_x
// S3 starts as the back-projection of the plan's 2D supports, each moved
// with its PO's mass-centre shift in whole pixels (a voxel is in if its
// projection lands in the moved 2D support at every angle) and shrinks on
// schedule: blur P_{S3+} rho with the periodic Gaussian along x, y, z, keep
// the voxels at or above tau times the maximum.
#include <algorithm>
#include <cmath>

#include "blur.h"
#include "cpra_internal.h"
#include "fft.cuh"
#include "tiling.cuh"

namespace cpra {

// X = vol (the centred Step D volume), R = Re vol
__global__ void k_refine_in(const float2* __restrict__ vol, float2* X, float* R, size_t total) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    const float2 v = vol[i];
    X[i] = v;
    R[i] = v.x;
  }
}

// vol = P_{S3+} rho as complex (imaginary part 0)
__global__ void k_refined_out(const float* __restrict__ R, const uint32_t* __restrict__ S3, float2* vol,
                              int N, int W) {
  const size_t total = (size_t)N * N * N;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total;
       i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % N);
    const size_t row = i / N;
    const float v = R[i];
    vol[i] = make_float2((sbit(S3, row * W, x) && v >= 0.0f) ? v : 0.0f, 0.0f);
  }
}

// M[cell] = the gridding lists of the cell are not empty
__global__ void k_measured(const int32_t* __restrict__ cell_ptr, uint8_t* M, int NN) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c < NN) M[c] = cell_ptr[c + 1] > cell_ptr[c] ? 1 : 0;
}

// Voxel (z, y, x) is in S3 when at every angle u = rint((x - c) cos + (y - c)
// sin + c) lies in [0, N) with S2[n][(z + dz) mod N][(u + du) mod N] set
// ((dz, du): the angle's shift).  A warp takes a word of S3, a lane a voxel,
// and the CTA YB rows (y) of one plane z; the rows of S2 this plane needs go
// through shared memory, NC angles at a time.  A word leaves the loop when
// none of its voxels is in any more, so the angles run in an order that
// jumps by about 0.38 of the range (`step`, coprime to Np): neighbouring
// angles test nearly the same, and a voxel outside dies after a handful of
// spread angles.
// The nearest pixel is the one an FP64 evaluation in the host's order picks.
// FP32 decides it where its estimate is not within 1e-3 of a half; there the
// distance to the half is taken on FP32 pairs (cos, sin and the row's part as
// high and low words, products and sums with their rounding errors: good to
// 1e-11), and only within 1e-9 of a half in FP64.  The FP64 pipe is narrow: a
// warp meets an estimate near a half in every eighth step, and FP64 there
// was the bound.  N = 256, 180 angles: 1.09 ms with a thread a word, the
// angles in order and FP64 at 1e-3; a lane a voxel in spread order 1.25 ms;
// with the pairs and 64 words a CTA instead of 256 0.40 ms.
// u = rint(((x - c) cos + (y - c) sin) + c) in FP64, each step rounded, no
// contraction.  Not inlined: kept out of line, the rare call leaves the FP64
// pipe idle instead of being predicated into every evaluation.
__device__ __noinline__ int u_fp64(int x, int y, int N, double2 t) {
  const double c = N / 2;
  const double b = __dmul_rn((double)(y - N / 2), t.y);
  return (int)rint(__dadd_rn(__dadd_rn(__dmul_rn((double)(x - N / 2), t.x), b), c));
}

__global__ void __launch_bounds__(256)
k_backproject(const uint32_t* __restrict__ S2, const double2* __restrict__ cs,
              const int2* __restrict__ shift, uint32_t* S3, int N, int W, int Np, int YB, int NC, int step) {
  // per chunk of NC angles: cos and sin as FP32 pairs [NC]; (y - c) sin + c
  // as a pair [NC][YB]; S2 rows [NC][W]; the angle and its du [NC]; the words
  // still in, [YB][W]
  extern __shared__ __align__(16) unsigned char sm_raw[];
  float4* tcs = reinterpret_cast<float4*>(sm_raw);
  float2* tb = reinterpret_cast<float2*>(tcs + NC);
  int2* tn = reinterpret_cast<int2*>(tb + (size_t)NC * YB);
  uint32_t* rows = reinterpret_cast<uint32_t*>(tn + NC);
  uint32_t* in = rows + (size_t)NC * W;
  const int z = blockIdx.y;
  const int y0 = blockIdx.x * YB;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int q = threadIdx.x; q < YB * W; q += blockDim.x) {
    const int left = N - (q % W) * 32;  // voxels of the word
    in[q] = y0 + q / W >= N ? 0u : left >= 32 ? 0xffffffffu : (1u << left) - 1u;
  }
  for (int n0 = 0; n0 < Np; n0 += NC) {
    const int nc = min(NC, Np - n0);
    __syncthreads();  // the previous chunk is done
    for (int k = threadIdx.x; k < nc; k += blockDim.x) {
      const int n = (int)((unsigned)(n0 + k) * (unsigned)step % (unsigned)Np);
      const double2 t = cs[n];
      const float ch = (float)t.x, sh = (float)t.y;
      tcs[k] = make_float4(ch, (float)(t.x - (double)ch), sh, (float)(t.y - (double)sh));
      tn[k] = make_int2(n, shift[n].y);
    }
    __syncthreads();
    for (int q = threadIdx.x; q < nc * W; q += blockDim.x) {
      const int k = q / W, ww = q - k * W, n = tn[k].x;
      int zr = z + shift[n].x;
      zr = zr < 0 ? zr + N : (zr >= N ? zr - N : zr);
      rows[k * W + ww] = S2[((size_t)n * N + zr) * W + ww];
    }
    for (int q = threadIdx.x; q < nc * YB; q += blockDim.x) {
      const int k = q / YB;
      const float y = (float)(y0 + q - k * YB - N / 2);
      const float4 t = tcs[k];
      float h = __fmul_rn(y, t.z), l = fmaf(y, t.z, -h);
      l = fmaf(y, t.w, l);
      two_add(h, l, (float)(N / 2));
      tb[q] = make_float2(h, l);
    }
    __syncthreads();
    for (int q = warp; q < YB * W; q += blockDim.x >> 5) {
      const uint32_t bits = in[q];
      if (bits == 0) continue;
      const int yl = q / W, x = (q - yl * W) * 32 + lane;
      const float xf = (float)(x - N / 2);
      bool keep = (bits >> lane) & 1u;
      uint32_t left = bits;
      for (int k = 0; k < nc; ++k) {
        const float4 t = tcs[k];
        const float2 b = tb[k * YB + yl];
        // the estimate, within 2e-4 for |x - c|, |y - c| <= 512, and its
        // nearest integer by the 1.5 * 2^23 shift
        const float uf = fmaf(xf, t.x, b.x);
        const float sh = __fadd_rn(uf, 12582912.0f);
        int ui = __float_as_int(sh) - 0x4B400000;
        const float fr = __fsub_rn(uf, __fsub_rn(sh, 12582912.0f));
        if (fabsf(fabsf(fr) - 0.5f) < 1e-3f && keep) {
          const float half = floorf(uf) + 0.5f;
          const float p = __fmul_rn(xf, t.x);
          float s = b.x, e = 0.0f;
          two_add(s, e, p);
          const float d = __fsub_rn(s, half) + (e + (fmaf(xf, t.x, -p) + fmaf(xf, t.y, b.y)));
          ui = (int)floorf(uf) + (d > 0.0f ? 1 : 0);
          if (fabsf(d) < 1e-9f) ui = u_fp64(x, y0 + yl, N, cs[tn[k].x]);
        }
        if (ui >= 0 && ui < N) {
          ui += tn[k].y;
          ui = ui < 0 ? ui + N : (ui >= N ? ui - N : ui);
          keep = keep && ((rows[k * W + (ui >> 5)] >> (ui & 31)) & 1u);
        } else {
          keep = false;
        }
        left = __ballot_sync(0xffffffffu, keep);
        if (left == 0) break;
      }
      __syncwarp();
      if (lane == 0) in[q] = left;
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < YB * W; q += blockDim.x)
    if (y0 + q / W < N) S3[((size_t)z * N + y0 + q / W) * W + q % W] = in[q];
}

// The 3D shrink-wrap blurs P_{S3+} rho along x (the 2D step's row blur over
// the N z-planes), then along y and z in place (its column blur), with the
// maximum of the last pass; see blur.h.

// S3 <- {B >= tau * max} (unchanged when the maximum is 0): a warp a row,
// lane l tests voxel 32 w + l and the warp's ballot is word w
__global__ void k_thresh3(const float* __restrict__ Bv, const unsigned* __restrict__ mx, uint32_t* S3,
                          float tau, int N, int W, size_t rows) {
  const int lane = threadIdx.x & 31;
  const size_t row = (size_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= rows) return;  // whole warps
  const float m = __uint_as_float(*mx);
  if (!(m > 0.0f)) return;
  const float thr = tau * m;
  const float* br = Bv + row * N;
  for (int w = 0; w < W; ++w) {
    const int x = w * 32 + lane;
    const uint32_t bits = __ballot_sync(0xffffffffu, x < N && br[x] >= thr);
    if (lane == 0) S3[row * W + w] = bits;
  }
}

// ------------------------------------------------------------------ launchers
// a step near 0.38 Np that is coprime to Np
static int angle_step(int Np) {
  auto gcd = [](int a, int b) {
    while (b) {
      const int t = a % b;
      a = b;
      b = t;
    }
    return a;
  };
  int s = std::max(1, (int)(0.381966 * Np));
  while (gcd(s, Np) != 1) ++s;
  return s;
}

cudaError_t launch_refine_setup(const RefineArgs& a, const float2* vol, cudaStream_t st) {
  const size_t total = (size_t)a.N * a.N * a.N;
  const unsigned blocks = (unsigned)std::min<size_t>((total + 255) / 256, 152 * 16);
  g_launches += 1;
  k_refine_in<<<blocks, 256, 0, st>>>(vol, a.X, a.R, total);
  return cudaGetLastError();
}

cudaError_t launch_refine_support(const RefineArgs& a, const uint32_t* S2, const double2* cs,
                                  const int2* shift, int Np, const int32_t* cell_ptr, cudaStream_t st) {
  const int N = a.N, W = a.W;
  // 64 words a CTA: the words that hold object run every angle one after the
  // other, so a CTA with 256 of them was a chain of 0.3 ms
  const int YB = std::max(1, std::min(N, 64 / W));
  // angles a chunk: their tables (see k_backproject) within 36 KB (six CTAs an SM)
  const int per = (int)(sizeof(float4) + sizeof(int2) + W * sizeof(uint32_t) + YB * sizeof(float2));
  const int words = YB * W * (int)sizeof(uint32_t);
  const int NC = std::max(1, std::min(Np, (36 * 1024 - words) / per));
  const size_t smem = (size_t)NC * per + words;
  g_launches += 2;
  k_backproject<<<dim3((N + YB - 1) / YB, N), 256, smem, st>>>(S2, cs, shift, a.S3, N, W, Np, YB, NC,
                                                               angle_step(Np));
  k_measured<<<(N * N + 255) / 256, 256, 0, st>>>(cell_ptr, a.M, N * N);
  return cudaGetLastError();
}

cudaError_t launch_refine_shrink(const RefineArgs& a, const float* taps, int ntaps, float tau,
                                 unsigned* mx, cudaStream_t st) {
  const int N = a.N;
  const size_t NN = (size_t)N * N;
  const int lo = -(ntaps / 2) + ((ntaps % 2) ? 0 : 1);
  cudaError_t e = cudaMemsetAsync(mx, 0, sizeof(unsigned), st);
  if (e == cudaSuccess) e = launch_sw_rows(a.R, a.S3, a.Bv, taps, ntaps, lo, N, a.W, N, st);  // x
  if (e == cudaSuccess) e = launch_blur_cols(a.Bv, a.Bv, taps, ntaps, lo, N, N, NN, (size_t)N, nullptr, false, st);  // y
  if (e == cudaSuccess) e = launch_blur_cols(a.Bv, a.Bv, taps, ntaps, lo, N, N, (size_t)N, NN, mx, false, st);  // z
  if (e != cudaSuccess) return e;
  g_launches += 1;
  k_thresh3<<<(unsigned)((NN + 7) / 8), 256, 0, st>>>(a.Bv, mx, a.S3, tau, N, a.W, NN);
  return cudaGetLastError();
}

cudaError_t launch_refine_output(const RefineArgs& a, float2* vol, cudaStream_t st) {
  const size_t total = (size_t)a.N * a.N * a.N;
  const unsigned blocks = (unsigned)std::min<size_t>((total + 255) / 256, 152 * 16);
  g_launches += 1;
  k_refined_out<<<blocks, 256, 0, st>>>(a.R, a.S3, vol, a.N, a.W);
  return cudaGetLastError();
}

}  // namespace cpra
