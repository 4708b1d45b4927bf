// twopass.cuh - steps of the block-wide passes (k_twopass.cu) that the sweep
// kernel (k_sweep.cu) shares, so that both round the same way.
#pragma once
#include "cpra_internal.h"
#include "fft.cuh"

namespace cpra {

template <int N>
__device__ __forceinline__ void load_twiddles(float2* tw_s, const float2* tw) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw_s[i] = tw[i];
}

// G' = a G / |G|; err += w (|G| - a)^2 in FP32 (a thread's few dozen
// terms; FP64 across threads and blocks)
__device__ __forceinline__ float2 project(float2 G, float a, float& err, float w) {
  if (a < 0.0f) return G;  // an unmeasured pair (mask): free, no error term
  const float m = sqrtf(G.x * G.x + G.y * G.y);
  const float d = m - a;
  err = fmaf(w * d, d, err);
  if (m > 0.0f) {
    const float s = a / m;
    return make_float2(G.x * s, G.y * s);
  }
  return make_float2(a, 0.0f);
}

template <int NT>
__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int i = 0; i < NT / 32; ++i) s += red[i];
  return s;
}

// Projection of the packed column 0 (buf[ky * B], the block's column 0 of
// pitch B): a0(ky) = A_sym at kx = 0, an(ky) = A_sym at kx = N/2.
template <int N, int B, int NT, class A0, class AN>
__device__ __forceinline__ void project_column0(float2* buf, A0&& a0, AN&& an, float& err) {
  constexpr int H = N / 2;
  // packed column: Z = G(.,0) + i G(.,N/2), both Hermitian along ky
  for (int ky = threadIdx.x; ky <= H; ky += NT) {
    const int km = (N - ky) % N;
    const float2 z = buf[ky * B], zm = buf[km * B];
    const float2 g0 = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
    const float2 gn = make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
    const float w = (ky == 0 || ky == H) ? 1.0f : 2.0f;
    const float2 p0 = project(g0, a0(ky), err, w);
    const float2 pn = project(gn, an(ky), err, w);
    buf[ky * B] = make_float2(p0.x - pn.y, p0.y + pn.x);
    if (km != ky) buf[km * B] = make_float2(p0.x + pn.y, pn.x - p0.y);
  }
}

}  // namespace cpra
