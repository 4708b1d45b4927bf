// k_fused.cu - cluster-resident fused iteration, N in {64, 128, 256, 512}.
//
// One thread-block cluster of C CTAs owns one angle for a whole launch: the
// prime (Eq. 4 coupling, or a plain read of g, then the row R2C) and
// n_iters iterations of
//   column FFT -> modulus projection onto A_sym (FP64 Fourier error) ->
//   column IFFT -> row C2R -> HIO / RAAR / ER update -> row R2C,
// with the packed half spectrum (N x N/2 complex, column 0 holding
// (Re H(y,0), Re H(y,N/2)) as in the two-pass engine) never leaving the
// cluster's distributed shared memory.  CTA r keeps packed columns
// [CW r, CW (r + 1)) of all N rows (its slab; CW = 32, or 16 at N = 512)
// and does the row work of image rows [2 CW r, 2 CW (r + 1)):
//   column phase  local to the CTA: its CW columns, one or two tasks a warp;
//   row phase     each row pair gathered from the C slabs over DSMEM,
//                 inverted, updated against g in global memory, transformed
//                 again and scattered back to the same slab places.
// Two cluster barriers per iteration separate the phases; loads that do not
// depend on other CTAs (A_sym, the old iterate) are issued between the
// arrive and the wait.  Global memory per angle-iteration: g read (HIO and
// RAAR need the old iterate) and written, A_sym read; within one launch these
// stay in L2, and the support bits are read once per launch into registers.
// Up to N = 256 the line transforms are the warp-resident FFTs of fftw.cuh
// with the same task-to-lane maps as the two-pass warp engine (bit-identical
// iterates); N = 512 uses the one-line FFT of fftw_pair.cuh.
#include <cooperative_groups.h>

#include "cluster.cuh"
#include "fast_kernels.cuh"

namespace cg = cooperative_groups;

namespace cpra {

// Line transforms of the fused kernel: the L-line plans of fftw.cuh, or the
// one-line 512-point plan of fftw_pair.cuh (half the registers, so 16 warps
// fit beside the slab).
template <int N> struct FusedLines { using type = typename WLines<N, kPrecFP32>::type; };

// Packed columns per CTA: 32, or 16 at N = 512, where a cluster of 16 CTAs
// of 108 KB each puts two CTAs of different angles on an SM, so that one
// CTA's barrier and DSMEM waits overlap the other's arithmetic.
// Q tasks a warp and phase: 2, which leaves the registers and shared memory
// for more clusters an SM, or 1 for launches whose clusters would leave the
// SMs with a few warps each (fused_launch has the rule).
template <int N, int Q> struct FusedCfg {
  using FL = typename FusedLines<N>::type;
  static constexpr int H = N / 2;
  static constexpr int CW = N == 512 ? 16 : 32;  // packed columns per CTA
  static constexpr int C = H / CW;               // CTAs per cluster
  static constexpr int ROWS = N / C;             // image rows of a CTA's row phase
  static constexpr int TASKS = CW / FL::L;       // tasks per phase per CTA
  static constexpr int NW = TASKS / Q;           // warps
  static constexpr int NT = NW * 32;
  static constexpr int SP = CW + 1;              // slab pitch in float2: odd, so column reads are conflict-free
  static constexpr int SLAB = N * SP;
  static constexpr int MINB = (N >= 256 ? 2 : 4) * Q / 2;
  static constexpr int MASKW = (2 * FL::TA * FL::E1 + 31) / 32;  // support-bit words of a row task
  static constexpr size_t SMEM = sizeof(float2) * (SLAB + NW * FL::TSIZE + N) + sizeof(double) * NW;
  static_assert(ROWS == 2 * CW, "row pairs of a CTA = its packed columns");
  static_assert(C >= 1 && C <= 16, "cluster size");
  static_assert(TASKS == Q * NW, "tasks a warp");
};

// ---------------------------------------------------------------- DSMEM (cluster.cuh)
// slab address of (row y, packed column c): CTA c / 32, local column c % 32
template <int N>
__device__ __forceinline__ uint32_t slab_at(uint32_t sb, int y, int c) {
  using F = FusedCfg<N, 2>;  // (the slabs do not depend on Q)
  return dsm_map(sb + 8u * (uint32_t)(y * F::SP + (c & (F::CW - 1))), (uint32_t)(c / F::CW));
}

// Z = H(row 2p) + i H(row 2p+1) of this warp's row pairs, B layout, from the
// packed spectra in the cluster's slabs.  Frequencies k and N - k need the same
// packed value in different lanes, so the rows come into the warp's tile
// first, each value once over the cluster's network, all loads in flight
// (ten iterations of 180 angles at N = 256: 704 us with a remote load a use,
// 651 so).  A cluster of one CTA (N = 64) reads its own slab directly.
template <int N, class FL>
__device__ __forceinline__ void gather_pairs(float2 (&b)[FL::TB][FL::E2], float2* T, const float2* slab,
                                             uint32_t sb, int pair0, int lane) {
  using F = FusedCfg<N, 2>;
  constexpr int H = N / 2, RV = 2 * FL::L * H / 32;  // values a lane
  static_assert(H % 32 == 0, "row spectra");
  constexpr bool local = F::C == 1;
  constexpr int R1 = local ? F::SP : H;  // from a pair's first row to its second
  if constexpr (!local) {
    float2 v[RV];
#pragma unroll
    for (int q = 0; q < RV; ++q)
      v[q] = dsm_ld(slab_at<N>(sb, 2 * pair0 + q / (H / 32), lane + 32 * (q % (H / 32))));
#pragma unroll
    for (int q = 0; q < RV; ++q) T[lane + 32 * q] = v[q];
    __syncwarp();
  }
  static_for<0, FL::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const float2* r0 = local ? slab + 2 * (pair0 + FL::b_line(t)) * F::SP : T + FL::b_line(t) * N;
    const float2* r1 = r0 + R1;
    static_for<0, FL::E2>([&](auto KK) {
      constexpr int j = decltype(KK)::value;
      const int k = FL::b_k(t, j);
      const bool up = k > H;
      const int c = up ? N - k : (k == H ? 0 : k);
      const float s = up ? -1.0f : 1.0f;
      const float2 h0 = r0[c], h1 = r1[c];
      float2 z = make_float2(fmaf(-s, h1.y, h0.x), fmaf(s, h0.y, h1.x));
      if (c == 0) z = k == 0 ? make_float2(h0.x, h1.x) : make_float2(h0.y, h1.y);
      b[i][j] = z;
    });
  });
  __syncwarp();  // the tile is the transforms' scratch from here on
}

// Z (B layout) of this warp's row pairs -> packed half spectra of both rows
// of each pair, written to the slabs (T pairs index k with N - k)
template <int N, class FL>
__device__ __forceinline__ void scatter_pairs(float2 (&b)[FL::TB][FL::E2], float2* T, float2* slab,
                                              uint32_t sb, int pair0, int lane) {
  using F = FusedCfg<N, 2>;
  constexpr int H = N / 2;
  static_for<0, FL::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const int line = FL::b_line(t);
    static_for<0, FL::E2>([&](auto KK) {
      constexpr int j = decltype(KK)::value;
      T[line * N + FL::b_k(t, j)] = b[i][j];
    });
  });
  __syncwarp();
#pragma unroll
  for (int line = 0; line < FL::L; ++line) {
    const float2* Zl = T + line * N;
    const int y0 = 2 * (pair0 + line);
#pragma unroll
    for (int k = lane; k < H; k += 32) {
      float2 h0, h1;
      if (k == 0) {
        const float2 z0 = Zl[0], zn = Zl[H];
        h0 = make_float2(z0.x, zn.x);
        h1 = make_float2(z0.y, zn.y);
      } else {
        const float2 z = Zl[k], zm = Zl[N - k];
        h0 = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
        h1 = make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
      }
      if constexpr (F::C == 1) {
        slab[y0 * F::SP + k] = h0;
        slab[(y0 + 1) * F::SP + k] = h1;
      } else {
        const uint32_t a0 = slab_at<N>(sb, y0, k);
        dsm_st(a0, h0);
        dsm_st(a0 + 8u * F::SP, h1);
      }
    }
  }
  __syncwarp();
}

// support bits of this lane's pixels of one row task (A layout), bit
// (i * E1 + m) * 2 + r for row 2 (pair0 + line) + r
template <int N, class FL>
__device__ __forceinline__ void support_mask(uint32_t (&mk)[FusedCfg<N, 2>::MASKW], const uint32_t* Sn,
                                             int W, int pair0, int lane) {
  static_for<0, FusedCfg<N, 2>::MASKW>([&](auto WW) { mk[decltype(WW)::value] = 0u; });
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const uint32_t* s0 = Sn + (size_t)(2 * (pair0 + FL::a_line(t))) * W;
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      constexpr int bit = (i * FL::E1 + m) * 2;
      const int x = FL::a_x(t, m);
      const uint32_t b0 = (__ldg(s0 + (x >> 5)) >> (x & 31)) & 1u;
      const uint32_t b1 = (__ldg(s0 + W + (x >> 5)) >> (x & 31)) & 1u;
      mk[bit >> 5] |= (b0 << (bit & 31)) | (b1 << ((bit + 1) & 31));
    });
  });
}

// Few angles at N = 64 stay as they were, two tasks a warp and the error
// published in every iteration (90 us for ten iterations of eight angles, 65
// in the other form): a test of the serving loop submits 2000 iterations of
// eight angles and needs them to outlast 20 ms.
constexpr int kFewTiles64 = 8;
template <int N, int Q>
__device__ __forceinline__ bool publish_at_once() { return N == 64 && Q == 2 && gridDim.y <= kFewTiles64; }

// SWEEP: a Gauss-Seidel episode, the angles of the member one after the other
// inside the launch (a launch per angle left its one to four CTAs a guess alone
// on the device; 90 angles, 16 guesses, 2 iterations: N = 64 25 us an angle,
// 128 42, 256 54; in one launch 16, 28 and 40).
// An angle's rows stay with their warp, so the taps on earlier angles read
// what the warp wrote itself.
template <int N, bool MASKED, int Q, bool SWEEP = false>
__global__ void __launch_bounds__(FusedCfg<N, Q>::NT, FusedCfg<N, Q>::MINB)
k_fused(const JobStatic* __restrict__ js, const JobStep* __restrict__ st,
        const int2* __restrict__ tiles) {
  using F = FusedCfg<N, Q>;
  using FL = typename F::FL;
  constexpr int H = N / 2;
  extern __shared__ __align__(16) float2 smem[];
  float2* slab = smem;
  float2* xs = smem + F::SLAB + F::NW * FL::TSIZE;
  double* red = reinterpret_cast<double*>(xs + N);
  __shared__ TapTab tt;
  const int2 tl = tiles[blockIdx.y];
  const JobStatic* J = js + tl.x;
  const JobStep* Z = st + tl.x;
  if (!Z->active) return;  // the same for every CTA of the cluster
  const int rank = (int)cg::this_cluster().block_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* T = smem + F::SLAB + warp * FL::TSIZE;
  const uint32_t sb = smem_u32(slab);
  const int Np = J->Np, W = J->W;
  const float beta = J->beta;
  const float c2 = 1.0f - 2.0f * beta;
  const float* __restrict__ A_T = J->A_main;
  float* g = Z->g;
  const CoupleArgs& ca = Z->ca;
  const int n_iters = Z->n_iters, hio_left = Z->hio_left;
  const long long err_slot = Z->err_slot;

  load_xtw<N>(xs, J->xtw, F::NT);
  const int n_end = SWEEP ? Np : tl.y + 1;
#pragma unroll 1
  for (int n = SWEEP ? 0 : tl.y; n < n_end; ++n) {
    fill_taps<N>(tt, ca, Z->g_src, Z->g_dst, J->S, n, Np, W, J->present);
    // the support is fixed during a launch: each lane keeps its pixels' bits
    uint32_t mask[Q][F::MASKW];
    static_for<0, Q>([&](auto QQ) {
      constexpr int q = decltype(QQ)::value;
      support_mask<N, FL>(mask[q], J->S + (size_t)n * N * W, W,
                          rank * F::CW + (warp + q * F::NW) * FL::L, lane);
    });
    cluster_sync_all();  // every CTA runs before any DSMEM access; xs and taps visible

    // ---- prime: (coupled) rows -> R2C -> slabs
#pragma unroll 1
    for (int q = 0; q < Q; ++q) {
      const int pair0 = rank * F::CW + (warp + q * F::NW) * FL::L;
      float2 a[FL::TA][FL::E1];
      blend_rows<N, FL, !SWEEP>(a, tt, ca, W, pair0, lane);
      if (ca.store_g) store_rows<N, FL>(a, Z->g_dst + (size_t)n * N * N, pair0, lane);
      float2 b[FL::TB][FL::E2];
      FL::fwd(a, b, T, xs, lane);
      scatter_pairs<N, FL>(b, T, slab, sb, pair0, lane);
    }
    cluster_sync_all();

    const float inv = 1.0f / N;
    // A_sym of column task q (B layout), read through L1
    auto load_av = [&](int q, float (&av)[FL::TB][FL::E2]) {
      const int cg0 = rank * F::CW + (warp + q * F::NW) * FL::L;
      static_for<0, FL::TB>([&](auto II) {
        constexpr int i = decltype(II)::value;
        const int t = lane + 32 * i;
        const float* Ac = A_T + ((size_t)n * H + cg0 + FL::b_line(t)) * N;
        static_for<0, FL::E2>([&](auto KK) {
          constexpr int j = decltype(KK)::value;
          av[i][j] = __ldg(Ac + FL::b_k(t, j));
        });
      });
    };
    // the old iterate of row task q (A layout), read by the HIO and RAAR rules
    auto load_old = [&](int q, float2 (&old)[FL::TA][FL::E1]) {
      const int pair0 = rank * F::CW + (warp + q * F::NW) * FL::L;
      static_for<0, FL::TA>([&](auto II) {
        constexpr int i = decltype(II)::value;
        const int t = lane + 32 * i;
        const float* g0 = g + ((size_t)n * N + 2 * (pair0 + FL::a_line(t))) * N;
        static_for<0, FL::E1>([&](auto MM) {
          constexpr int m = decltype(MM)::value;
          const int x = FL::a_x(t, m);
          old[i][m] = make_float2(g0[x], g0[N + x]);
        });
      });
    };
    // column task q: FFT_y, projection onto A_sym (error terms of weight 2
    // into err2, of weight 1 into err1), IFFT_y
    auto col_task = [&](int q, const float (&av)[FL::TB][FL::E2], float& err2, float& err1) {
      const int cl0 = (warp + q * F::NW) * FL::L;  // first local column of the task
      const int cg0 = rank * F::CW + cl0;           // its packed column index
      float2 a[FL::TA][FL::E1];
      static_for<0, FL::TA>([&](auto II) {
        constexpr int i = decltype(II)::value;
        const int t = lane + 32 * i;
        const int line = FL::a_line(t);
        static_for<0, FL::E1>([&](auto MM) {
          constexpr int m = decltype(MM)::value;
          a[i][m] = slab[FL::a_x(t, m) * F::SP + cl0 + line];
        });
      });
      float2 b[FL::TB][FL::E2];
      FL::fwd(a, b, T, xs, lane);
      static_for<0, FL::TB>([&](auto II) {
        constexpr int i = decltype(II)::value;
        const int t = lane + 32 * i;
        if (cg0 + FL::b_line(t) != 0) {
          static_for<0, FL::E2>([&](auto KK) {
            constexpr int j = decltype(KK)::value;
            b[i][j] = project_w<MASKED>(b[i][j], av[i][j], err2);
          });
        }
      });
      if (cg0 == 0) {
        // column 0 packs G(., 0) + i G(., N/2); both are Hermitian along ky
        static_for<0, FL::TB>([&](auto II) {
          constexpr int i = decltype(II)::value;
          const int t = lane + 32 * i;
          if (FL::b_line(t) == 0) {
            static_for<0, FL::E2>([&](auto KK) {
              constexpr int j = decltype(KK)::value;
              T[FL::b_k(t, j)] = b[i][j];
            });
          }
        });
        __syncwarp();
        const float* An = J->A_nyq + (size_t)n * N;
        static_for<0, FL::TB>([&](auto II) {
          constexpr int i = decltype(II)::value;
          const int t = lane + 32 * i;
          if (FL::b_line(t) == 0) {
            static_for<0, FL::E2>([&](auto KK) {
              constexpr int j = decltype(KK)::value;
              const int ky = FL::b_k(t, j);
              const float2 z = T[ky], zm = T[(N - ky) % N];
              const float2 g0 = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
              const float2 gn = make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
              const float2 p0 = project_w<MASKED>(g0, av[i][j], err1);
              const float2 pn = project_w<MASKED>(gn, __ldg(An + ky), err1);
              b[i][j] = make_float2(p0.x - pn.y, p0.y + pn.x);
            });
          }
        });
        __syncwarp();
      }
      FL::inv(b, a, T, xs, lane);
      static_for<0, FL::TA>([&](auto II) {
        constexpr int i = decltype(II)::value;
        const int t = lane + 32 * i;
        const int line = FL::a_line(t);
        static_for<0, FL::E1>([&](auto MM) {
          constexpr int m = decltype(MM)::value;
          slab[FL::a_x(t, m) * F::SP + cl0 + line] = cscale(a[i][m], inv);
        });
      });
    };
    // HIO / RAAR / ER update of row task q from g' = a / N; a <- the new iterate
    auto update = [&](int q, float2 (&a)[FL::TA][FL::E1], const float2 (&old)[FL::TA][FL::E1],
                      int rule) {
      const int pair0 = rank * F::CW + (warp + q * F::NW) * FL::L;
      uint32_t mq[F::MASKW];
      static_for<0, F::MASKW>([&](auto WW) {
        constexpr int w = decltype(WW)::value;
        mq[w] = q ? mask[Q - 1][w] : mask[0][w];
      });
      static_for<0, FL::TA>([&](auto II) {
        constexpr int i = decltype(II)::value;
        const int t = lane + 32 * i;
        float* g0 = g + ((size_t)n * N + 2 * (pair0 + FL::a_line(t))) * N;
        static_for<0, FL::E1>([&](auto MM) {
          constexpr int m = decltype(MM)::value;
          constexpr int bit = (i * FL::E1 + m) * 2;
          const int x = FL::a_x(t, m);
          const float2 z = a[i][m];
          const float gp0 = z.x * inv, gp1 = z.y * inv;
          const bool s0 = (mq[bit >> 5] >> (bit & 31)) & 1u;
          const bool s1 = (mq[bit >> 5] >> ((bit + 1) & 31)) & 1u;
          const float n0 = update_pixel(old[i][m].x, gp0, s0, rule, beta, c2);
          const float n1 = update_pixel(old[i][m].y, gp1, s1, rule, beta, c2);
          g0[x] = n0;
          g0[N + x] = n1;
          a[i][m] = make_float2(n0, n1);
        });
      });
    };

    float av[FL::TB][FL::E2];
    float2 old[FL::TA][FL::E1];
    load_av(0, av);
    for (int it = 0; it < n_iters; ++it) {
      const int rule = it < hio_left ? Z->algo : kER;  // HIO or RAAR, then ER
      const bool fwd = it + 1 < n_iters;
      float es = 0.0f, ee = 0.0f;  // error terms as an FP32 pair
#pragma unroll 1
      for (int q = 0; q < Q; ++q) {
        if (q) load_av(q, av);
        float err2 = 0.0f, err1 = 0.0f;
        col_task(q, av, err2, err1);
        two_add(es, ee, eighths2(err2));
        two_add(es, ee, eighths1(err1));
      }
      const double errd = warp_sum(es, ee);
      if (lane == 0) red[warp] = errd;
      cluster_arrive();
      if (rule != kER) load_old(0, old);  // in flight across the barrier
      cluster_wait();
#pragma unroll 1
      for (int q = 0; q < Q; ++q) {
        const int pq = rank * F::CW + (warp + q * F::NW) * FL::L;
        if (rule != kER && q) load_old(q, old);
        float2 b[FL::TB][FL::E2];
        float2 a[FL::TA][FL::E1];
        gather_pairs<N, FL>(b, T, slab, sb, pq, lane);
        FL::inv(b, a, T, xs, lane);
        update(q, a, old, rule);
        if (fwd) {
          FL::fwd(a, b, T, xs, lane);
          scatter_pairs<N, FL>(b, T, slab, sb, pq, lane);
        }
      }
      if (rank == 0 && warp == 0 && err_slot >= 0) {
        // Fourier error of the iterate entering this iteration, summed in a
        // fixed order over the cluster's warps (the partials stay put until
        // every CTA has passed the barrier below)
        double s = 0.0;
        for (int q = lane; q < F::C * F::NW; q += 32)
          s += dsm_ld_f64(dsm_map(smem_u32(red + q % F::NW), (uint32_t)(q / F::NW)));
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        // the raw sum in eighths; the square root and division wait until the last
        // iteration (see publish_at_once for the exception)
        if (lane == 0)
          J->err_hist[(size_t)(err_slot + it) * Np + n] =
              publish_at_once<N, Q>() ? publish_error(kEighths * s, J->Cn[n], J->sumA2[n], J->status, n) : s;
      }
      cluster_arrive();
      if (fwd) load_av(0, av);  // in flight across the barrier
      cluster_wait();
    }
    if (!publish_at_once<N, Q>() && rank == 0 && warp == 0 && err_slot >= 0) {
      __syncwarp();
      for (int it = lane; it < n_iters; it += 32) {
        double* e = J->err_hist + (size_t)(err_slot + it) * Np + n;
        *e = publish_error(kEighths * __ldcg(e), J->Cn[n], J->sumA2[n], J->status, n);
      }
    }
  }
}

// ---------------------------------------------------------------- host side
template <int N, int Q>
static cudaLaunchConfig_t fused_config(int ntiles, cudaLaunchAttribute* at, cudaStream_t st) {
  using F = FusedCfg<N, Q>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(F::C, ntiles);
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

// attributes of both instances; *clusters: resident clusters of this shape
template <int N, int Q, bool SWEEP = false>
static cudaError_t fused_attrs(int* clusters) {
  using F = FusedCfg<N, Q>;
  cudaError_t e = cudaSuccess;
  for (auto kernel : {k_fused<N, false, Q, SWEEP>, k_fused<N, true, Q, SWEEP>}) {
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)F::SMEM);
    if (e == cudaSuccess && F::C > 8)
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute at;
  cudaLaunchConfig_t cfg = fused_config<N, Q>(1, &at, nullptr);
  e = cudaOccupancyMaxActiveClusters(clusters, k_fused<N, false, Q, SWEEP>, &cfg);
  return e == cudaSuccess && *clusters < 1 ? cudaErrorNotSupported : e;
}

// N = 512 has one instance: its two tasks a warp fill the SM with 16 warps
template <int N> constexpr bool kFusedWide = N <= 256;

// a cluster of C CTAs with this much shared memory must fit on the current
// device; *wide: clusters of the one-task form that are resident at a time
template <int N>
static cudaError_t fused_prepare(int* wide) {
  static PerDevice<int> resident;
  int one = 0;
  const cudaError_t e = on_device(resident, one, [](int& n) {
    int c = 0;
    const cudaError_t r = fused_attrs<N, 2>(&c);
    if constexpr (kFusedWide<N>)
      if (r == cudaSuccess && fused_attrs<N, 1>(&n) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
      }
    return r;
  });
  if (wide) *wide = one;
  return e;
}

// One task a warp where all of the launch's clusters are resident at a time in
// that form: the SMs then hold twice the warps and each runs half the chain.
// Ten iterations, two tasks / one: N = 64, 32 angles 90 / 66 us, 200 angles
// 101 / 79; N = 128, 90 angles 182 / 158, 150 angles 186 / 165; N = 256, 30
// angles 200 / 190.  Beyond that the two-task form holds more clusters an SM.
template <int N>
static cudaError_t fused_launch(const Launch& L) {
  int wide = 0;
  cudaError_t e = fused_prepare<N>(&wide);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute at;
  g_launches += 1;
  if constexpr (kFusedWide<N>)
    if (L.ntiles <= wide && !(N == 64 && L.ntiles <= kFewTiles64)) {
      const cudaLaunchConfig_t cfg = fused_config<N, 1>(L.ntiles, &at, L.stream);
      if (L.masked) return cudaLaunchKernelEx(&cfg, k_fused<N, true, 1>, L.js, L.st, L.tiles);
      return cudaLaunchKernelEx(&cfg, k_fused<N, false, 1>, L.js, L.st, L.tiles);
    }
  const cudaLaunchConfig_t cfg = fused_config<N, 2>(L.ntiles, &at, L.stream);
  if (L.masked) return cudaLaunchKernelEx(&cfg, k_fused<N, true, 2>, L.js, L.st, L.tiles);
  return cudaLaunchKernelEx(&cfg, k_fused<N, false, 2>, L.js, L.st, L.tiles);
}

// The sweep form: one task a warp while the members fit that way (a chain is
// as long as its angle), else two.
template <int N>
static int sweep_wide() {  // members that fit with one task a warp, 0: no sweep form here
  static PerDevice<int> resident;
  int one = 0;
  const cudaError_t e = on_device(resident, one, [](int& n) {
    int two = 0;
    const cudaError_t r = fused_attrs<N, 2, true>(&two);
    return r == cudaSuccess ? fused_attrs<N, 1, true>(&n) : r;
  });
  if (e == cudaSuccess) return one;
  cudaGetLastError();
  return 0;
}

template <int N, int Q>
static cudaError_t fused_sweep_go(const Launch& L) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t cfg = fused_config<N, Q>(L.ntiles, &at, L.stream);
  g_launches += 1;
  if (L.masked) return cudaLaunchKernelEx(&cfg, k_fused<N, true, Q, true>, L.js, L.st, L.tiles);
  return cudaLaunchKernelEx(&cfg, k_fused<N, false, Q, true>, L.js, L.st, L.tiles);
}

// However many the members: a launch an angle runs the same clusters in the same
// waves (256 guesses, us an angle, one launch / a launch an angle: N = 64 22 /
// 34, 128 56 / 69, 256 217 / 252).
bool fused_sweep_supported(int N) {
  switch (N) {
    case 64: return sweep_wide<64>() > 0;
    case 128: return sweep_wide<128>() > 0;
    case 256: return sweep_wide<256>() > 0;
    default: return false;
  }
}

cudaError_t launch_fused_sweep(const Launch& L) {
#define CPRA_CASE(NN) \
  case NN: return L.ntiles <= sweep_wide<NN>() ? fused_sweep_go<NN, 1>(L) : fused_sweep_go<NN, 2>(L);
  switch (L.N) {
    CPRA_CASE(64)
    CPRA_CASE(128)
    CPRA_CASE(256)
    default: return cudaErrorInvalidValue;
  }
#undef CPRA_CASE
}

#define CPRA_FOR_EACH_FUSED_N(X) X(64) X(128) X(256) X(512)

bool fused_supported(int N) {
  switch (N) {
#define CPRA_CASE(NN) case NN:
    CPRA_FOR_EACH_FUSED_N(CPRA_CASE)
#undef CPRA_CASE
    return true;
    default:
      return false;
  }
}

cudaError_t prepare_kernels_fused(int N) {
  switch (N) {
#define CPRA_CASE(NN) \
  case NN: return fused_prepare<NN>(nullptr);
    CPRA_FOR_EACH_FUSED_N(CPRA_CASE)
#undef CPRA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t launch_fused(const Launch& L) {
  if (L.prec != kPrecFP32) return cudaErrorInvalidValue;
  switch (L.N) {
#define CPRA_CASE(NN) \
  case NN: return fused_launch<NN>(L);
    CPRA_FOR_EACH_FUSED_N(CPRA_CASE)
#undef CPRA_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace cpra
