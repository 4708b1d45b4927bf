// k_refine_w.cu - dispatch of the line passes over volumes
// (refine_kernels.cuh), and the data of the half spectrum.
#include "refine_kernels.cuh"

namespace cpra {

#define CPRA_CASE(NN) CPRA_REFINE_INSTANCES(NN, extern)
CPRA_FOR_EACH_N(CPRA_CASE)
#undef CPRA_CASE

// W and the constant sums from V = FFT3 of the data volume (full), a block a
// row ky of every gridDim.y-th plane kz: konst[0] += sum K_k, konst[1] +=
// sum_M |V|^2
__global__ void k_rdata(const float2* __restrict__ V, const uint8_t* __restrict__ M, float2* W, double* konst,
                        int N, int HP) {
  const int H = N / 2, ky = blockIdx.x, my = (N - ky) % N;
  double sk = 0.0, sd = 0.0;
  for (int c = threadIdx.x; c <= H; c += blockDim.x) {
    const int mc = (N - c) % N;
    const bool m1 = M[ky * N + c], m2 = M[my * N + mc];
    if (!m1 && !m2) continue;
    const float wt = (c == 0 || c == H) ? 0.5f : 1.0f;  // the partner is in the same column
    float k = 0.0f, ke = 0.0f, d = 0.0f, de = 0.0f;  // N/16 planes
#pragma unroll 4
    for (int kz = blockIdx.y; kz < N; kz += gridDim.y) {
      const int mz = (N - kz) % N;
      const float2 v1 = V[((size_t)kz * N + ky) * N + c];
      const float2 p = V[((size_t)mz * N + my) * N + mc];
      const float2 v2 = make_float2(p.x, -p.y);
      float2 w = make_float2(0.0f, 0.0f);
      if (m1) w = v1;
      if (m2) w = make_float2(w.x + v2.x, w.y + v2.y);
      W[((size_t)kz * N + ky) * HP + c] = make_float2(0.5f * w.x, 0.5f * w.y);
      if (m1) two_add(d, de, wt * fmaf(v1.x, v1.x, v1.y * v1.y));
      if (m2) two_add(d, de, wt * fmaf(v2.x, v2.x, v2.y * v2.y));
      if (m1 && m2) {
        const float dx = v1.x - v2.x, dy = v1.y - v2.y;
        two_add(k, ke, 0.5f * wt * fmaf(dx, dx, dy * dy));
      }
    }
    sk += pair_value(k, ke);
    sd += pair_value(d, de);
  }
  sk = warp_sum(sk);
  sd = warp_sum(sd);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(konst + 0, sk);
    atomicAdd(konst + 1, sd);
  }
}

cudaError_t launch_refine_w_data(const RefineArgs& a, int HP, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(a.konst, 0, 2 * sizeof(double), st);
  if (e != cudaSuccess) return e;
  g_launches += 1;
  k_rdata<<<dim3(a.N, 16), 128, 0, st>>>(a.X, a.M, a.Wd, a.konst, a.N, HP);
  return cudaGetLastError();
}

cudaError_t launch_volume_ylines(int N, float2* vol, float2* out, const float2* xtw, cudaStream_t st) {
  switch (N) {
#define CPRA_CASE(NN) \
  case NN: return volume_ylines_n<NN>(vol, out, xtw, st);
    CPRA_FOR_EACH_N(CPRA_CASE)
#undef CPRA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_refine_data(const RefineArgs& a, cudaStream_t st) {
  switch (a.N) {
#define CPRA_CASE(NN) \
  case NN: return data_w<NN>(a, st);
    CPRA_FOR_EACH_N(CPRA_CASE)
#undef CPRA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_refine_iter(const RefineArgs& a, double* err2, bool first, bool last, cudaStream_t st) {
  switch (a.N) {
#define CPRA_CASE(NN) \
  case NN: return iter_w<NN>(a, err2, first, last, st);
    CPRA_FOR_EACH_N(CPRA_CASE)
#undef CPRA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace cpra
