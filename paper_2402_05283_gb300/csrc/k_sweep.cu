// k_sweep.cu - Gauss-Seidel sweeps at the block-wide engine's sizes, one
// launch an episode.
//
// A sweep is a chain: angle n starts from the image of angle n - 1.  One
// launch per angle and pass (k_prime, k_colpass, k_rowpass) leaves a few
// dozen CTAs of three warps on the device for 25 to 57 us each (N = 160,
// 16 guesses: 163 us an angle), so the chain is bound by the latency of the
// passes and their launches, not by bytes.  Here one cluster of C CTAs runs
// the whole chain of one guess: it keeps the angle's packed half spectrum in
// distributed shared memory (CTA r holds columns [CW r, CW (r + 1)) of all
// rows, and works on image rows [2 CW r, 2 CW (r + 1))), with a thread for
// every butterfly, and the iterate of the angle in registers: pixel idx of
// the CTA's rows belongs to the same thread from the coupling to the last
// update.  Rows never leave their CTA, so the taps on earlier angles read
// what this CTA wrote.  Per angle: the taps are read, the amplitudes and
// support bits once an iteration, and the iterate is written once.
// The transforms, the projection and the update are those of k_twopass.cu,
// term by term, so the iterates are the same bits; the error sums are taken
// in another order.
// The chains of a wave of clusters take as long as one; with enough guesses the
// passes, which fill the device as guesses are added, are the faster form
// (sweep_choice).
#include <cooperative_groups.h>

#include "cluster.cuh"
#include "cpra_internal.h"
#include "fft.cuh"
#include "taps.cuh"
#include "tiling.cuh"
#include "twopass.cuh"

namespace cg = cooperative_groups;

namespace cpra {

namespace {

// Threads: one a radix-4 butterfly of the CTA's lines, one a radix-8 butterfly
// where that would be more than 640.
template <int N, int C_> struct SweepCfg {
  static constexpr int H = N / 2, C = C_, CW = H / C;
  static constexpr int P = CW;            // row pairs of a CTA
  static constexpr int PI = P | 1;        // odd pitch of the row buffer
  static constexpr int NT = warps32(clampi(CW * N / 4 <= 640 ? CW * N / 4 : CW * N / 8, 64, 1024));
  static constexpr int KG = (P * N + NT - 1) / NT;   // row-pair pixels a thread
  static constexpr int KA = (N * CW + NT - 1) / NT;  // spectrum values a thread
  static constexpr int KH = (P * H + NT - 1) / NT;   // row-pair frequencies a thread
  static constexpr size_t SMEM = sizeof(float2) * (N * CW + N * PI + N);
  static_assert(H % C == 0 && 2 * KG <= 32 && H + 1 <= NT && NT >= 64, "sweep tiles");
};

// the thread index, opaque: keeps the compiler from holding the index
// arithmetic of every loop in registers across the loop over angles
__device__ __forceinline__ int opaque_tid() {
  int t = threadIdx.x;
  asm volatile("" : "+r"(t));
  return t;
}

// adds the warp's error terms to hist[at] (at < 0: nowhere) in FP64
__device__ __forceinline__ void add_error(float e, double* hist, long long at) {
  const double s = warp_sum(e, 0.0f);
  if ((threadIdx.x & 31) == 0 && at >= 0) atomicAdd(hist + at, s);
}

template <int N, int C>
__global__ void __launch_bounds__(SweepCfg<N, C>::NT, 1)
k_sweep(const JobStatic* __restrict__ js, const JobStep* __restrict__ st,
        const int2* __restrict__ tiles) {
  using F = SweepCfg<N, C>;
  constexpr int H = F::H, CW = F::CW, P = F::P, PI = F::PI, NT = F::NT;
  extern __shared__ float2 smem[];
  float2* slab = smem;           // [row][CW]
  float2* buf = slab + N * CW;   // row pairs, [x][PI]
  float2* tw_s = buf + N * PI;
  __shared__ TapTab taps[2];  // of this angle and the next
  const int job = tiles[blockIdx.y].x;
  const JobStatic* J = js + job;
  const JobStep* Z = st + job;
  if (!Z->active) return;  // the same for every CTA of the cluster
  const int rank = (int)cg::this_cluster().block_rank();
  const int Np = J->Np, W = J->W, n_iters = Z->n_iters, hio_left = Z->hio_left;
  const float beta = J->beta, c2 = 1.0f - 2.0f * beta, inv = 1.0f / N;
  const CoupleArgs& ca = Z->ca;
  float* g = Z->g;
  const int y0 = rank * 2 * P, c0 = rank * CW;
  const uint32_t sb = smem_u32(slab);
  load_twiddles<N>(tw_s, J->tw);

  // packed spectra of this CTA's rows (buf) -> the slabs that own the columns
  auto scatter = [&] {
    for (int idx = opaque_tid(); idx < P * H; idx += NT) {
      const int p = idx / H, k = idx - p * H;
      float2 h0, h1;
      if (k == 0) {
        const float2 z0 = buf[p], zn = buf[H * PI + p];
        h0 = make_float2(z0.x, zn.x);
        h1 = make_float2(z0.y, zn.y);
      } else {
        const float2 z = buf[k * PI + p], zm = buf[(N - k) * PI + p];
        h0 = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
        h1 = make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
      }
      const uint32_t a = dsm_map(sb + 8u * (uint32_t)((y0 + 2 * p) * CW + k % CW), (uint32_t)(k / CW));
      dsm_st(a, h0);
      dsm_st(a + 8u * CW, h1);
    }
  };
  // A_sym of this thread's spectrum values of angle n (and its frequency of
  // the packed column 0)
  auto load_a = [&](int n, float (&av)[F::KA], float& a0, float& an) {
    const float* An = J->A_main + ((size_t)n * H + c0) * N;
    const int tid = opaque_tid();
#pragma unroll
    for (int q = 0; q < F::KA; ++q) {
      const int idx = tid + q * NT;
      if (idx < N * CW) av[q] = __ldg(An + (size_t)(idx % CW) * N + idx / CW);
    }
    if (c0 == 0 && tid <= H) {
      a0 = __ldg(An + tid);
      an = __ldg(J->A_nyq + (size_t)n * N + tid);
    }
  };

  float old0[F::KG], old1[F::KG];  // the iterate at this thread's pixels
  float av[F::KA], a0 = 0.0f, an = 0.0f;
  if (rank == 0 && Z->err_slot >= 0)  // the error terms add up in the history itself
    for (int i = threadIdx.x; i < n_iters * Np; i += NT) J->err_hist[(size_t)Z->err_slot * Np + i] = 0.0;
  fill_taps<N>(taps[0], ca, Z->g_src, Z->g_dst, J->S, 0, Np, W, J->present);
  __syncthreads();
  for (int n = 0; n < Np; ++n) {
    const TapTab& tt = taps[n & 1];
    // what the next angle will read first, on its way to L2
    if (n + 1 < Np) {
      const float* gn = Z->g_src + (size_t)(n + 2 < Np ? n + 2 : n + 1) * N * N + (size_t)y0 * N;
      for (int q = threadIdx.x; q < 2 * P * N / 32; q += NT)
        asm volatile("prefetch.global.L2 [%0];\n" ::"l"(gn + q * 32));
      const float* An = J->A_main + ((size_t)(n + 1) * H + c0) * N;
      for (int q = threadIdx.x; q < CW * N / 32; q += NT)
        asm volatile("prefetch.global.L2 [%0];\n" ::"l"(An + q * 32));
    }
    // Eq. 4, then R2C rows
    // (the loads of three taps are all in flight together)
    uint32_t bits = 0;
    const int tid = opaque_tid();
#pragma unroll
    for (int q = 0; q < F::KG; ++q) {
      old0[q] = old1[q] = 0.0f;
      const int idx = tid + q * NT;
      if (idx < P * N) {
        const int p = idx / N, x = idx - p * N;
        const size_t row = ((size_t)n * N + y0 + 2 * p) * W;
        bits |= ((uint32_t)sbit(J->S, row, x) | (uint32_t)sbit(J->S, row + W, x) << 1) << (2 * q);
      }
    }
    for (int k0 = 0; k0 < ca.n_taps; k0 += 3) {
      float v0[3][F::KG], v1[3][F::KG];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int k = k0 + u;
        if (k >= ca.n_taps || tt.w[k] == 0.0f) continue;  // (a tap on an absent angle)
        const float* src = tt.src[k] + (size_t)y0 * N;
        const int mir = tt.mir[k];
#pragma unroll
        for (int q = 0; q < F::KG; ++q) {
          const int idx = tid + q * NT;
          if (idx >= P * N) continue;
          const int p = idx / N, x = idx - p * N;
          const int xs = mir ? (N - x) % N : x;
          v0[u][q] = src[2 * p * N + xs];
          v1[u][q] = src[(2 * p + 1) * N + xs];
          if (ca.object) {
            const size_t row = (size_t)(y0 + 2 * p) * W;
            v0[u][q] = (sbit(tt.s[k], row, xs) && v0[u][q] >= 0.0f) ? v0[u][q] : 0.0f;
            v1[u][q] = (sbit(tt.s[k], row + W, xs) && v1[u][q] >= 0.0f) ? v1[u][q] : 0.0f;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int k = k0 + u;
        if (k >= ca.n_taps || tt.w[k] == 0.0f) continue;
        const float w = tt.w[k];
#pragma unroll
        for (int q = 0; q < F::KG; ++q) {
          old0[q] = (ca.n_taps == 1) ? v0[u][q] : fmaf(w, v0[u][q], old0[q]);
          old1[q] = (ca.n_taps == 1) ? v1[u][q] : fmaf(w, v1[u][q], old1[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < F::KG; ++q) {
      const int idx = tid + q * NT;
      if (idx < P * N) buf[(idx % N) * PI + idx / N] = make_float2(old0[q], old1[q]);
    }
    if (n + 1 < Np) fill_taps<N>(taps[(n + 1) & 1], ca, Z->g_src, Z->g_dst, J->S, n + 1, Np, W, J->present);
    __syncthreads();
    fft_lines<N, -1, P, PI, NT, true>(buf, tw_s);
    scatter();
    cluster_arrive();
    load_a(n, av, a0, an);  // in flight across the barrier
    cluster_wait();
    for (int it = 0; it < n_iters; ++it) {
      fft_lines<N, -1, CW, CW, NT, true>(slab, tw_s);
      float err = 0.0f;
      const int ta = opaque_tid();
#pragma unroll
      for (int q = 0; q < F::KA; ++q) {
        const int idx = ta + q * NT;
        if (idx < N * CW && c0 + idx % CW != 0) slab[idx] = project(slab[idx], av[q], err, 2.0f);
      }
      if (c0 == 0)
        project_column0<N, CW, NT>(slab, [&](int) { return a0; }, [&](int) { return an; }, err);
      __syncthreads();
      fft_lines<N, +1, CW, CW, NT, true>(slab, tw_s);
      add_error(err, J->err_hist, Z->err_slot < 0 ? -1 : (Z->err_slot + it) * Np + n);
      cluster_sync_all();
      // rows of the spectrum -> buf, C2R, update, R2C
      const int tg = opaque_tid();
      float2 s0[F::KH], s1[F::KH];
#pragma unroll
      for (int q = 0; q < F::KH; ++q) {  // every remote load in flight first
        const int idx = tg + q * NT;
        if (idx >= P * H) continue;
        const int p = idx / H, k = idx - p * H;
        const uint32_t a = dsm_map(sb + 8u * (uint32_t)((y0 + 2 * p) * CW + k % CW), (uint32_t)(k / CW));
        s0[q] = dsm_ld(a);
        s1[q] = dsm_ld(a + 8u * CW);
      }
#pragma unroll
      for (int q = 0; q < F::KH; ++q) {
        const int idx = tg + q * NT;
        if (idx >= P * H) continue;
        const int p = idx / H, k = idx - p * H;
        const float2 h0 = cscale(s0[q], inv), h1 = cscale(s1[q], inv);
        if (k == 0) {
          buf[p] = make_float2(h0.x, h1.x);
          buf[H * PI + p] = make_float2(h0.y, h1.y);
        } else {
          buf[k * PI + p] = make_float2(h0.x - h1.y, h0.y + h1.x);
          buf[(N - k) * PI + p] = make_float2(h0.x + h1.y, h1.x - h0.y);
        }
      }
      __syncthreads();
      fft_lines<N, +1, P, PI, NT, true>(buf, tw_s);
      const int rule = it < hio_left ? Z->algo : kER;
      const bool last = it + 1 == n_iters;
      const int tu = opaque_tid();
#pragma unroll
      for (int q = 0; q < F::KG; ++q) {
        const int idx = tu + q * NT;
        if (idx >= P * N) break;
        const int p = idx / N, x = idx - p * N;
        const float2 z = buf[x * PI + p];
        old0[q] = update_pixel(old0[q], z.x * inv, (bits >> (2 * q)) & 1u, rule, beta, c2);
        old1[q] = update_pixel(old1[q], z.y * inv, (bits >> (2 * q + 1)) & 1u, rule, beta, c2);
        buf[x * PI + p] = make_float2(old0[q], old1[q]);
        if (last) {
          float* d = g + ((size_t)n * N + y0 + 2 * p) * N + x;
          d[0] = old0[q];
          d[N] = old1[q];
        }
      }
      __syncthreads();  // buf, and (last) the rows the next angle's taps read
      if (!last) {
        fft_lines<N, -1, P, PI, NT, true>(buf, tw_s);
        scatter();
        cluster_sync_all();
      }
    }
  }
  cluster_sync_all();  // no CTA leaves while another reads its shared memory
  if (rank == 0 && Z->err_slot >= 0)  // the raw sums -> Fourier errors
    for (int i = threadIdx.x; i < n_iters * Np; i += NT) {
      double* e = J->err_hist + (size_t)Z->err_slot * Np + i;
      *e = publish_error(__ldcg(e), J->Cn[i % Np], J->sumA2[i % Np], J->status, i % Np);
    }
}

template <int N, int C>
cudaLaunchConfig_t sweep_config(int members, cudaLaunchAttribute* at, cudaStream_t st) {
  using F = SweepCfg<N, C>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(F::C, members);
  cfg.blockDim = dim3(F::NT);
  cfg.dynamicSmemBytes = F::SMEM;
  cfg.stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = F::C;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// clusters of this shape that the current device holds at a time (0: none)
template <int N, int C>
int sweep_resident() {
  static PerDevice<int> resident;
  int clusters = 0;
  const cudaError_t e = on_device(resident, clusters, [](int& n) {
    const cudaError_t r = smem_attr(k_sweep<N, C>, SweepCfg<N, C>::SMEM);
    cudaLaunchAttribute at;
    const cudaLaunchConfig_t cfg = sweep_config<N, C>(1, &at, nullptr);
    return r == cudaSuccess ? cudaOccupancyMaxActiveClusters(&n, k_sweep<N, C>, &cfg) : r;
  });
  if (e == cudaSuccess) return clusters;
  cudaGetLastError();
  return 0;
}

// How a group of guesses is swept: a cluster of FEW CTAs a guess has the
// shortest chain, of MANY CTAs (0: no such form) a longer one with more
// clusters resident; per_few and per_many are the times of an angle (2
// iterations) with the device full, a wave of guesses at a time.  The passes of
// k_twopass.cu take max(pass0 + pass1 G, pass2 G) for G guesses.  Measured, us an
// angle, few / many / passes:
//   N = 96:  1 guess 18.1 / 22.0 / 120, 24: 36.4 / 22.7 / 134, 256: 241 / 189 / 172
//   N = 160: 1 guess 27.2 / 32.1 / 138, 16: 58.4 / 34.0 / 166, 256: 533 / 336 / 356
//   N = 320: 1 guess 71.4 / 116 / 165, 16: 155 / 137 / 205, 32: 236 / 273 / 233,
//            48: 319 / 295 / 306, 64: 404 / 427 / 485
//   N = 32:  1 guess 8.9 / 13.2 / 52.7, 96: 20.2 / 13.6 / 60.4
// At N = 16 and 48 one form is the fastest throughout (N = 16: 2 CTAs 8.7 for 1
// guess and 10.7 for 256, 8 CTAs 8.6 and 39.1; N = 48: 4 CTAs 13.3 and 61.1, 8
// CTAs 14.9 and 71.3; passes 33.8 and 47.3, 48.6 and 78.1).
template <int N> struct SweepForms;
#define CPRA_SWEEP_FORMS(N, FEW_, MANY_, T_FEW, T_MANY, P0, P1, P2)                      \
  template <> struct SweepForms<N> {                                                     \
    static constexpr int FEW = FEW_, MANY = MANY_;                                       \
    static constexpr float per_few = T_FEW, per_many = T_MANY, pass0 = P0, pass1 = P1, pass2 = P2; \
  };
CPRA_SWEEP_FORMS(16, 2, 0, 9.5f, 0.0f, 34.0f, 0.052f, 0.1f)
CPRA_SWEEP_FORMS(32, 8, 2, 10.3f, 14.5f, 53.0f, 0.1f, 0.1f)
CPRA_SWEEP_FORMS(48, 4, 0, 14.9f, 0.0f, 49.0f, 0.12f, 0.1f)
CPRA_SWEEP_FORMS(96, 6, 4, 19.0f, 23.5f, 120.0f, 0.2f, 0.5f)
CPRA_SWEEP_FORMS(160, 8, 5, 29.7f, 34.4f, 145.0f, 0.5f, 1.4f)
CPRA_SWEEP_FORMS(320, 8, 5, 79.0f, 148.0f, 165.0f, 2.0f, 6.3f)
#undef CPRA_SWEEP_FORMS

enum SweepChoice { kSweepPasses, kSweepFew, kSweepMany };

template <int N>
SweepChoice sweep_choice(int members) {
  using S = SweepForms<N>;
  const float g = (float)members;
  float best = S::pass0 + S::pass1 * g > S::pass2 * g ? S::pass0 + S::pass1 * g : S::pass2 * g;
  SweepChoice choice = kSweepPasses;
  auto offer = [&](SweepChoice c, int resident, float us) {
    if (resident < 1) return;
    const float t = (float)((members + resident - 1) / resident) * us;
    if (t < best) {
      best = t;
      choice = c;
    }
  };
  offer(kSweepFew, sweep_resident<N, S::FEW>(), S::per_few);
  if constexpr (S::MANY > 0) offer(kSweepMany, sweep_resident<N, S::MANY>(), S::per_many);
  return choice;
}

template <int N, int C>
cudaError_t sweep_go(const Launch& L) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = sweep_config<N, C>(L.ntiles, &at, L.stream);
  g_launches += 1;
  return cudaLaunchKernelEx(&cfg, k_sweep<N, C>, L.js, L.st, L.tiles);
}

template <int N>
cudaError_t sweep_launch(const Launch& L) {
  using S = SweepForms<N>;
  const SweepChoice c = sweep_choice<N>(L.ntiles);
  if constexpr (S::MANY > 0)
    if (c == kSweepMany) return sweep_go<N, S::MANY>(L);
  return c == kSweepFew ? sweep_go<N, S::FEW>(L) : cudaErrorInvalidValue;
}

}  // namespace

// sizes whose slab and row buffer fit the shared memory of eight CTAs
#define CPRA_FOR_EACH_SWEEP_N(X) X(16) X(32) X(48) X(96) X(160) X(320)

bool sweep_supported(int N, int engine, int members) {
  if (engine == CPRA_ENGINE_FUSED) return fused_sweep_supported(N);
  if (engine != CPRA_ENGINE_TWO_PASS) return false;
  switch (N) {
#define CPRA_CASE(NN) \
  case NN: return sweep_choice<NN>(members) != kSweepPasses;
    CPRA_FOR_EACH_SWEEP_N(CPRA_CASE)
#undef CPRA_CASE
    default:
      return false;
  }
}

cudaError_t launch_sweep(const Launch& L) {
  if (L.engine == CPRA_ENGINE_FUSED) return launch_fused_sweep(L);
  switch (L.N) {
#define CPRA_CASE(NN) \
  case NN: return sweep_launch<NN>(L);
    CPRA_FOR_EACH_SWEEP_N(CPRA_CASE)
#undef CPRA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace cpra
