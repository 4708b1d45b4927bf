// assemble_kernels.cuh - the per-size kernels of the assembly and the merge
// (k_assemble.cu describes the steps) and their launchers.
#pragma once
#include "cpra_internal.h"
#include "fast_kernels.cuh"
#include "tiling.cuh"

namespace cpra {

// ramps of one angle: [0, N) along z (FFT order, signed k), then [0, N/2]
// along u, the last one for ku = -N/2
__host__ __device__ constexpr int ramp_len(int N) { return N + N / 2 + 1; }

// Q = sum over a cell's samples of ku < 0 of weight * corr
cudaError_t launch_grid_corr(cpra_plan_s* p);
cudaError_t launch_prtf(const unsigned long long* rings, const unsigned* counts, float* prtf, int H, int total,
                        cudaStream_t st);

// ---------------------------------------------------------------- columns
// Staging of CB adjacent packed columns (rows H apart) of the column kernels,
// thread to (row, column) as in the column pass.
template <int N> struct SpecCols {
  using C = ColW<N, kPrecFP32>;
  static constexpr int H = N / 2, RS = C::NT / C::CB, SR = (N + RS - 1) / RS;
  int y0, cc;
  __device__ SpecCols() {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    y0 = 32 % C::CB == 0 ? warp + C::WARPS * (lane / C::CB) : threadIdx.x / C::CB;
    cc = 32 % C::CB == 0 ? lane % C::CB : threadIdx.x % C::CB;
  }
  template <class F>
  __device__ __forceinline__ void each(F&& f) const {  // f(row)
#pragma unroll
    for (int k = 0; k < SR; ++k)
      if (N % RS == 0 || y0 + k * RS < N) f(y0 + k * RS);
  }
  // columns c0 .. c0 + CB of Hn -> registers (A layout); buf is free after
  template <class FL>
  __device__ __forceinline__ void load(const float2* Hn, int c0, float2* buf,
                                       float2 (&a)[FL::TA][FL::E1]) const {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    each([&](int y) { cp_async8(buf + y * C::SP + cc, Hn + (size_t)y * H + c0 + cc); });
    cp_async_commit();
    cp_async_wait_all();
    __syncthreads();
    static_for<0, FL::TA>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int t = lane + 32 * i;
      if (!FL::a_on(t)) return;
      const int col = warp * FL::L + FL::a_line(t);
      static_for<0, FL::E1>([&](auto MM) {
        constexpr int m = decltype(MM)::value;
        a[i][m] = buf[FL::a_x(t, m) * C::SP + col];
      });
    });
    __syncthreads();
  }
};

// f(i, j, t) over the B-layout values that exist
template <class FL, class F>
__device__ __forceinline__ void each_b(int lane, F&& f) {
  static_for<0, FL::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::b_on(t)) return;
    static_for<0, FL::E2>([&](auto JJ) { f(II, JJ, t); });
  });
}

// F[z / 8][n][ku][z % 8]: a chunk of eight planes of all samples is
// contiguous, so the grid kernel streams it once through L2
__device__ __forceinline__ size_t f_at(int z, int n, int c, int Np, int HC) {
  return (((size_t)(z >> 3) * Np + n) * HC + c) * 8 + (z & 7);
}

// inverse-transformed lines a (A layout) of columns cl0 + line -> F, 1/N;
// only(line) selects lines
template <int N, class FL, class Only>
__device__ __forceinline__ void store_f(const float2 (&a)[FL::TA][FL::E1], float2* F, int n, int Np,
                                        int c, int lane, Only&& only) {
  constexpr int H = N / 2;
  constexpr Const<FL::ACC> inv(1.0 / N);
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const int line = FL::a_line(t);
    if (!FL::a_on(t) || !only(line)) return;
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      const int z = FL::a_x(t, m);
      F[f_at(z < H ? z + H : z - H, n, c + line, Np, H + 1)] = inv.mul(a[i][m]);
    });
  });
}

template <int N>
constexpr size_t spec_smem() { return sizeof(float2) * (SpecLines<N>::XN + 2 * N + ColW<N, kPrecFP32>::BUF); }

// What the spectra kernel makes of a block of columns: F (one guess, all
// angles: blockIdx.y = angle), REF or DIST (one angle n0 of guess blockIdx.y)
template <int N, int MODE>
__global__ void __launch_bounds__(ColW<N, kPrecFP32>::NT, ColW<N, kPrecFP32>::MINB)
k_spectra(const float2* __restrict__ Hp, const float2* __restrict__ ramps, float2* F, float2* corr,
          const float2* __restrict__ xtw, const MergeArgs ma) {
  using C = ColW<N, kPrecFP32>;
  using FL = SpecLines<N>;
  constexpr int H = N / 2;
  extern __shared__ float2 smem[];
  float2* xs = smem;
  float2* rz = xs + FL::XN;
  float2* z0 = rz + N;  // the packed column 0 after its forward transform
  float2* buf = z0 + N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* T = buf + warp * FL::TSIZE;
  const int n = MODE == kSpecF ? blockIdx.y : ma.n0;
  const int Np = gridDim.y;
  const int c0 = blockIdx.x * C::CB;
  if constexpr (MODE != kSpecF) {
    Hp = ma.guess[blockIdx.y].Hp;
    ramps = ma.guess[blockIdx.y].ramps;
  }
  const float2* rn = ramps + (size_t)n * ramp_len(N);
  const float2* ru = rn + N;
  for (int i = threadIdx.x; i < N; i += C::NT) {
    xs[i] = xtw[i];
    if constexpr (FL::XN > N) xs[N + i] = xtw[N + i];
    rz[i] = rn[i];
  }
  float2 a[FL::TA][FL::E1], b[FL::TB][FL::E2];
  const SpecCols<N> cols;
  cols.template load<FL>(Hp + (size_t)n * N * H, c0, buf, a);
  FL::fwd(a, b, T, xs, lane);
  const int cl = warp * FL::L;  // first column of the warp in the block
  const bool packed = c0 == 0 && warp == 0;
  if (packed) {  // column 0 packs G(., 0) + i G(., N/2), both Hermitian along kz
    each_b<FL>(lane, [&](auto II, auto JJ, int t) {
      if (FL::b_line(t) == 0) z0[FL::b_k(t, decltype(JJ)::value)] = b[decltype(II)::value][decltype(JJ)::value];
    });
    __syncwarp();
  }
  auto g_zero = [&](int k) {
    const float2 z = z0[k], zm = z0[(N - k) % N];
    return make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
  };
  auto g_nyq = [&](int k) {
    const float2 z = z0[k], zm = z0[(N - k) % N];
    return make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
  };
  if constexpr (MODE == kSpecF) {
    const float inv = 1.0f / N;
    each_b<FL>(lane, [&](auto II, auto JJ, int t) {
      constexpr int i = decltype(II)::value, j = decltype(JJ)::value;
      const int k = FL::b_k(t, j), c = c0 + cl + FL::b_line(t);
      const float2 w = __ldg(ru + c);
      const float2 G = c == 0 ? g_zero(k) : b[i][j];
      const float2 E = cmul(cmul(G, rz[k]), w);
      if (k == H && c > 0) {  // E(-N/2, -c) - conj E(-N/2, c)
        const float2 M = cmul(cmul(cconj(G), rz[H]), cconj(w));
        corr[(size_t)n * (H + 1) + c] = make_float2(inv * (M.x - E.x), inv * (M.y + E.y));
      }
      b[i][j] = E;
    });
    __syncwarp();
    FL::inv(b, a, T, xs, lane);
    store_f<N, FL>(a, F, n, Np, c0 + cl, lane, [](int) { return true; });
    if (packed) {  // the column ku = -N/2
      __syncwarp();
      const float2 w = __ldg(ru + H);
      each_b<FL>(lane, [&](auto II, auto JJ, int t) {
        const int k = FL::b_k(t, decltype(JJ)::value);
        b[decltype(II)::value][decltype(JJ)::value] = cmul(cmul(g_nyq(k), rz[k]), w);
      });
      FL::inv(b, a, T, xs, lane);
      store_f<N, FL>(a, F, n, Np, H, lane, [](int line) { return line == 0; });
    }
  } else {
    // |ref - E|^2 - |ref - conj E|^2 = -4 Im ref Im E: one FP64 product a value
    // decides (a merge of four guesses, N = 256, 144 angles: 0.775 ms with both
    // distances in FP64, 0.737 so)
    double dot = 0.0;
    auto take = [&](int kz, int ku, float2 v) {
      if constexpr (MODE == kSpecRef) {
        ma.ref[(size_t)kz * N + ku] = v;
      } else {
        const float2 r = ma.ref[(size_t)kz * N + ku];
        dot += (double)r.y * (double)v.y;
      }
    };
    each_b<FL>(lane, [&](auto II, auto JJ, int t) {
      const int k = FL::b_k(t, decltype(JJ)::value), c = c0 + cl + FL::b_line(t);
      const float2 G = b[decltype(II)::value][decltype(JJ)::value];
      if (c == 0) {
        take(k, 0, cmul(g_zero(k), rz[k]));
        take(k, H, cmul(cmul(g_nyq(k), rz[k]), __ldg(ru + H)));
      } else {
        const int km = (N - k) % N;
        const float2 w = __ldg(ru + c);
        take(k, c, cmul(cmul(G, rz[k]), w));
        take(km, N - c, cmul(cmul(cconj(G), rz[km]), cconj(w)));
      }
    });
    if constexpr (MODE == kSpecDist) {
      dot = warp_sum(dot);
      if (lane == 0) atomicAdd(ma.dist + blockIdx.y, dot);
    }
  }
}

// The PRTF's ring sums are whole numbers of 2^-50, so they are exact in any
// order: a ring holds fewer than 2^12 values of at most 1.  Bit 63 (out of the
// sums' reach) says that one was not a number.  (FP64 sums in shared memory
// depend on the order in their last bits, and their atomics are loops: N = 256,
// 144 angles, four guesses 0.783 ms a merge; with FP32 sums 0.722, so 0.734.)
constexpr double kRingUnit = 8.8817841970012523e-16;  // 2^-50
constexpr unsigned long long kRingNaN = 1ull << 63;
// |v| / m (0 where m is 0): the FP32 quotient and its remainder over m
__device__ __forceinline__ unsigned long long prtf_ratio(float2 v, float m) {
  if (!(m > 0.0f)) return 0;
  const float a = sqrtf(fmaf(v.x, v.x, v.y * v.y)), q = a / m;
  if (!(q <= 2.0f)) return kRingNaN;
  const float rest = fmaf(-q, m, a) / m;  // (m infinite: not a number, and q is 0)
  const long long lo = fabsf(rest) < q ? __float2ll_rn(rest * 0x1p50f) : 0;
  return (unsigned long long)(__float2ll_rn(q * 0x1p50f) + lo);
}
__device__ __forceinline__ void add_ring(unsigned long long* ring, unsigned long long f) {
  if (f < kRingNaN) atomicAdd(ring, f);
  else atomicOr(ring, kRingNaN);
}

// One block of columns of angle blockIdx.y through every kept guess: the mean
// of the corrected spectra (full plane, into acc), the ring sums of
// |sum E'| / sum |E'| and F of the mean.  E(-k) = conj E(k) but for the row
// kz = -N/2, whose partner sum is kept beside the block.  Bound by HBM: every
// guess's packed spectrum is read once, the mean and F are written once
// (one pass over the full-plane sums a guess, then separate PRTF and IDFT_z
// passes, took 1.88 ms for four guesses at N = 256, 144 angles; one pass 0.25
// ms at one CTA an SM and 0.16 at two).
template <int N>
__global__ void __launch_bounds__(ColW<N, kPrecFP32>::NT, ColW<N, kPrecFP32>::NT <= 256 && N <= 512 ? 2 : 1)
k_merge(const MergeArgs ma, int n_l, float2* acc, unsigned long long* rings, unsigned* counts, float2* F,
        float2* corr, const float2* __restrict__ xtw) {
  using C = ColW<N, kPrecFP32>;
  using FL = SpecLines<N>;
  constexpr int H = N / 2;
  extern __shared__ float2 smem[];
  float2* xs = smem;
  float2* rz = xs + FL::XN;
  float2* z0 = rz + N;
  float2* buf = z0 + N;
  __shared__ float2 sh[C::CB];  // mean of the partner row kz = -N/2 of the block's columns
  __shared__ unsigned long long ring[H];
  __shared__ unsigned cnt[H];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* T = buf + warp * FL::TSIZE;
  const int n = blockIdx.y, Np = gridDim.y;
  const int c0 = blockIdx.x * C::CB, cl = warp * FL::L;
  const SpecCols<N> cols;
  const float scale = 1.0f / (float)n_l;
  const bool packed = c0 == 0 && warp == 0;
  for (int i = threadIdx.x; i < FL::XN; i += C::NT) xs[i] = xtw[i];
  for (int i = threadIdx.x; i < H; i += C::NT) {
    ring[i] = 0;
    cnt[i] = 0u;
  }
  // pass 0: columns c0 .. (column 0 of the packed pair); pass 1, first block
  // only: the column ku = -N/2
  for (int pass = 0; pass < (c0 == 0 ? 2 : 1); ++pass) {
    float2 a[FL::TA][FL::E1], b[FL::TB][FL::E2];
    float2 s[FL::TB][FL::E2];
    float mg[FL::TB][FL::E2];
    float2 sm[FL::TB];  // partner sum of the row kz = -N/2 (the task that holds it)
    float mh[FL::TB];
    static_for<0, FL::TB>([&](auto II) {
      constexpr int i = decltype(II)::value;
      sm[i] = make_float2(0.f, 0.f);
      mh[i] = 0.0f;
      static_for<0, FL::E2>([&](auto JJ) {
        s[i][decltype(JJ)::value] = make_float2(0.f, 0.f);
        mg[i][decltype(JJ)::value] = 0.0f;
      });
    });
    for (int q = 0; q < n_l; ++q) {
      const MergeGuess mq = ma.guess[q];
      const float2* rn = mq.ramps + (size_t)n * ramp_len(N);
      const float2* ru = rn + N;
      __syncthreads();  // the previous guess is done with rz, buf and z0
      for (int i = threadIdx.x; i < N; i += C::NT) rz[i] = rn[i];
      cols.template load<FL>(mq.Hp + (size_t)n * N * H, c0, buf, a);
      FL::fwd(a, b, T, xs, lane);
      if (packed) {
        each_b<FL>(lane, [&](auto II, auto JJ, int t) {
          if (FL::b_line(t) == 0) z0[FL::b_k(t, decltype(JJ)::value)] = b[decltype(II)::value][decltype(JJ)::value];
        });
        __syncwarp();
      }
      each_b<FL>(lane, [&](auto II, auto JJ, int t) {
        constexpr int i = decltype(II)::value, j = decltype(JJ)::value;
        const int k = FL::b_k(t, j), c = c0 + cl + FL::b_line(t);
        float2 G = b[i][j];
        if (c == 0) {
          const float2 z = z0[k], zm = z0[(N - k) % N];
          G = pass == 0 ? make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y))
                        : make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
        }
        const float2 w = __ldg(ru + (c == 0 && pass ? H : c));
        const float2 E = cmul(cmul(G, rz[k]), w);
        s[i][j] = make_float2(s[i][j].x + E.x, s[i][j].y + (mq.inv ? -E.y : E.y));
        if (rings) mg[i][j] += sqrtf(fmaf(E.x, E.x, E.y * E.y));
        if (k == H && c > 0) {
          const float2 M = cmul(cmul(cconj(G), rz[H]), cconj(w));
          sm[i] = make_float2(sm[i].x + M.x, sm[i].y + (mq.inv ? -M.y : M.y));
          if (rings) mh[i] += sqrtf(fmaf(M.x, M.x, M.y * M.y));
        }
      });
    }
    // ring sums, the mean, its correction for the columns ku < 0
    __syncthreads();
    each_b<FL>(lane, [&](auto II, auto JJ, int t) {
      constexpr int i = decltype(II)::value, j = decltype(JJ)::value;
      const int k = FL::b_k(t, j), line = FL::b_line(t), c = c0 + cl + line;
      if (pass && c > 0) return;
      const float2 v = s[i][j];
      if (rings) {
        const int kz = k < H ? k : k - N, ku = c == 0 && pass ? H : c;
        const int r = (int)rintf(sqrtf((float)(kz * kz + ku * ku)));  // exact: no square is near (m + 1/2)^2
        if (r < H) {
          const unsigned long long f = prtf_ratio(v, mg[i][j]);
          const bool two = c > 0;  // and its partner (-kz, -ku)
          if (two && k == H) add_ring(ring + r, prtf_ratio(sm[i], mh[i]));
          add_ring(ring + r, two && k != H && f < kRingNaN ? 2 * f : f);
          if (n == 0) atomicAdd(cnt + r, two ? 2u : 1u);
        }
      }
      const float2 m = cscale(v, scale);
      b[i][j] = m;
      buf[k * C::SP + cl + line] = m;
      if (k == H && c > 0) {
        const float2 p = cscale(sm[i], scale);
        sh[cl + line] = p;
        const float inv = 1.0f / N;
        corr[(size_t)n * (H + 1) + c] = make_float2(inv * (p.x - m.x), inv * (p.y + m.y));
      }
    });
    __syncthreads();
    // the mean's rows: CB columns of ku >= 0, their partners of ku < 0
    float2* an = acc + (size_t)n * N * N;
    if (pass == 0) {
      const int c = c0 + cols.cc;
      cols.each([&](int kz) { an[(size_t)kz * N + c] = buf[kz * C::SP + cols.cc]; });
      if (c > 0)
        cols.each([&](int kz) {
          an[(size_t)((N - kz) % N) * N + N - c] = kz == H ? sh[cols.cc] : cconj(buf[kz * C::SP + cols.cc]);
        });
    } else {
      for (int kz = threadIdx.x; kz < N; kz += C::NT) an[(size_t)kz * N + H] = buf[kz * C::SP];
    }
    __syncthreads();  // buf becomes the warps' tiles again
    FL::inv(b, a, T, xs, lane);
    if (pass == 0) store_f<N, FL>(a, F, n, Np, c0 + cl, lane, [](int) { return true; });
    else if (packed) store_f<N, FL>(a, F, n, Np, H, lane, [](int line) { return line == 0; });
  }
  if (rings) {
    __syncthreads();
    for (int i = threadIdx.x; i < H; i += C::NT) {
      if (ring[i]) {
        add_ring(rings + (size_t)n * H + i, ring[i] & ~kRingNaN);
        if (ring[i] >= kRingNaN) add_ring(rings + (size_t)n * H + i, kRingNaN);
      }
      if (n == 0 && cnt[i]) atomicAdd(counts + i, cnt[i]);
    }
  }
}

// ---------------------------------------------------------------- grid
// A block takes row ky of L chunks of eight planes (L: lines a warp of the
// plan, so that its eight warps have one transform each).  Four lanes hold a
// cell's eight planes of a chunk (16 bytes each), so a sample's 64 bytes are
// one access and 64 cells are in work at a time.  The cells near the origin
// collect thousands of samples (all angles meet there): a cell of more than
// kHeavy is summed by the whole block, its samples spread over the 64 quads
// (one thread a cell walked the list alone: 80 us of 83 at N = 128, 90
// angles).  Sums run in a fixed order.  Bound by L2: four reads a sample and
// plane.  N = 512, 360 angles, with the transform along kx: 0.91 ms; gather
// 1.04 and rows 0.63 as separate passes over V.
constexpr int kHeavy = 32;
template <int N> struct GridCfg {
  using FL = VolLines<N>;
  static constexpr int L = FL::L, H = N / 2, HC = H + 1;
  static constexpr int NZC = (N + 7) / 8;  // chunks of eight planes
  static constexpr int STAGED = 2560;  // samples of a row held in shared memory (else read from L2)
  // pitch of a line: at least N, room for the warp's tile, 2 mod 8 (the four
  // plane pairs of a quad then start four banks apart)
  static constexpr int P0 = (FL::TSIZE + L - 1) / L > N ? (FL::TSIZE + L - 1) / L : N;
  static constexpr int LP = (P0 + 5) / 8 * 8 + 2;
  static constexpr size_t SMEM = sizeof(float2) * (FL::XN + 8 * L * LP + STAGED) + sizeof(int) * (N + 4);
  static_assert(LP >= P0 && LP % 8 == 2, "line pitch");
};

// s (planes 2q and 2q + 1) += the samples e0, e0 + step, ... < e1, four lines
// of F in flight; a sample of ku < 0 reads the conjugate
template <class E>
__device__ __forceinline__ void grid_sum(float4& s, E ents, int e0, int e1, int step,
                                         const float4* __restrict__ Fc) {
  for (int e = e0; e < e1; e += 4 * step) {
    GridEnt g[4];
    float4 f[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (e + i * step < e1) {
        g[i] = ents[e + i * step];
        f[i] = __ldg(Fc + (size_t)(g[i].at & 0x7fffffffu) * 4);
      }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (e + i * step < e1) {
        const float wy = __uint_as_float(__float_as_uint(g[i].w) ^ (g[i].at & 0x80000000u));
        s.x = fmaf(g[i].w, f[i].x, s.x);
        s.y = fmaf(wy, f[i].y, s.y);
        s.z = fmaf(g[i].w, f[i].z, s.z);
        s.w = fmaf(wy, f[i].w, s.w);
      }
  }
}

template <int N>
__global__ void __launch_bounds__(256, 3)
k_grid(const float2* __restrict__ F, const float2* __restrict__ Q, const int32_t* __restrict__ cell_ptr,
       const GridEnt* __restrict__ ents, float2* V, const float2* __restrict__ xtw, int Np) {
  using G = GridCfg<N>;
  using FL = typename G::FL;
  constexpr int L = G::L, LP = G::LP;
  extern __shared__ __align__(16) float2 smem[];
  float2* xs = smem;
  float2* lines = smem + FL::XN;  // [8 L][LP]
  GridEnt* es = reinterpret_cast<GridEnt*>(lines + 8 * L * LP);
  int* ptr = reinterpret_cast<int*>(es + G::STAGED);  // [N + 1]
  __shared__ unsigned short heavy[N];
  __shared__ int n_heavy;
  __shared__ float part[8][4][4];
  const int ky = blockIdx.x, ch0 = blockIdx.y * L;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int quad = threadIdx.x >> 2, q = threadIdx.x & 3;
  if (threadIdx.x == 0) n_heavy = 0;
  const int first = __ldg(cell_ptr + ky * N), count = __ldg(cell_ptr + ky * N + N) - first;
  const bool staged = count <= G::STAGED;
  for (int i = threadIdx.x; i <= N; i += 256) ptr[i] = __ldg(cell_ptr + ky * N + i) - first;
  if (staged)
    for (int i = threadIdx.x; i < count; i += 256) cp_async8(es + i, ents + first + i);
  cp_async_commit();
  for (int i = threadIdx.x; i < FL::XN; i += 256) xs[i] = xtw[i];
  cp_async_wait_all();
  __syncthreads();
  auto put = [&](int x, int ch, const float4& s) {
    const float sg = ((x + ky) & 1) ? -1.0f : 1.0f;
    const float2 c = __ldg(Q + ky * N + x);  // what the conjugates leave out, (-1)^z
    float2* d = lines + (ch * 8 + 2 * q) * LP + x;
    d[0] = make_float2(sg * (s.x + c.x), sg * (s.y + c.y));
    d[LP] = make_float2(sg * (s.z - c.x), sg * (s.w - c.y));
  };
  const size_t chunk4 = (size_t)Np * G::HC * 4;  // float4s a chunk
  auto chunk = [&](int ch) { return reinterpret_cast<const float4*>(F) + (size_t)(ch0 + ch) * chunk4 + q; };
  auto sum_cell = [&](float4& s, int e0, int e1, int step, int ch) {
    if (staged) grid_sum(s, (const GridEnt*)es, e0, e1, step, chunk(ch));
    else grid_sum(s, ents + first, e0, e1, step, chunk(ch));
  };
#pragma unroll 2
  for (int u = quad; u < N * L; u += 64) {
    const int x = u % N, ch = u / N;
    if (ch0 + ch >= G::NZC) break;
    const int e0 = ptr[x], e1 = ptr[x + 1];
    if (e1 - e0 > kHeavy) {
      if (ch == 0 && q == 0) heavy[atomicAdd(&n_heavy, 1)] = (unsigned short)x;
      continue;
    }
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    sum_cell(s, e0, e1, 1, ch);
    put(x, ch, s);
  }
  __syncthreads();
  const int nh = n_heavy;
  for (int h = 0; h < nh; ++h) {
    const int x = heavy[h];
    const int e0 = ptr[x], e1 = ptr[x + 1];
    for (int ch = 0; ch < L; ++ch) {
      if (ch0 + ch >= G::NZC) break;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
      sum_cell(s, e0 + quad, e1, 64, ch);
      float r[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) r[i] += __shfl_xor_sync(0xffffffffu, r[i], o);
        if (lane < 4) part[warp][lane][i] = r[i];
      }
      __syncthreads();
      if (threadIdx.x < 4) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          r[i] = 0.0f;
          for (int w = 0; w < 8; ++w) r[i] += part[w][threadIdx.x][i];
        }
        put(x, ch, make_float4(r[0], r[1], r[2], r[3]));
      }
      __syncthreads();
    }
  }
  // the warp's L lines of kx, inverse, into the row of their planes
  float2* T = lines + warp * L * LP;
  float2 a[FL::TA][FL::E1], b[FL::TB][FL::E2];
  static_for<0, FL::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::b_on(t)) return;
    static_for<0, FL::E2>([&](auto JJ) {
      constexpr int j = decltype(JJ)::value;
      b[i][j] = T[FL::b_line(t) * LP + FL::b_k(t, j)];
    });
  });
  __syncwarp();
  FL::inv(b, a, T, xs, lane);
  constexpr Const<FL::ACC> inv(1.0 / N);
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const int z = ch0 * 8 + warp * L + FL::a_line(t);
    if (!FL::a_on(t) || z >= N) return;
    float2* row = V + ((size_t)z * N + ky) * N;
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      row[FL::a_x(t, m)] = inv.mul(a[i][m]);
    });
  });
}

// ------------------------------------------------------------------ launchers
template <int N, int MODE>
static cudaError_t spectra_n(const float2* Hp, const float2* ramps, float2* F, float2* corr, const float2* xtw,
                             const MergeArgs& ma, int count, cudaStream_t st) {
  using C = ColW<N, kPrecFP32>;
  static PerDevice<bool> attr;
  cudaError_t e = smem_once(k_spectra<N, MODE>, spec_smem<N>(), attr);
  if (e != cudaSuccess) return e;
  g_launches += 1;
  k_spectra<N, MODE><<<dim3((N / 2) / C::CB, count), C::NT, spec_smem<N>(), st>>>(Hp, ramps, F, corr, xtw, ma);
  return cudaGetLastError();
}

// gather into rows of the grid with their inverse FFT, then the y lines
template <int N>
static cudaError_t grid_n(cpra_plan_s* p, float2* out) {
  using G = GridCfg<N>;
  Assembly& a = p->asmb;
  static PerDevice<bool> attr;
  cudaError_t e = smem_once(k_grid<N>, G::SMEM, attr);
  if (e == cudaSuccess) e = launch_grid_corr(p);
  if (e != cudaSuccess) return e;
  g_launches += 1;
  k_grid<N><<<dim3(N, (G::NZC + G::L - 1) / G::L), 256, G::SMEM, p->stream>>>(
      a.F, a.Q, a.cell_ptr, a.ents, a.vol, p->xtw, p->Np);
  e = cudaGetLastError();
  return e == cudaSuccess ? launch_volume_ylines(N, a.vol, out, p->xtw, p->stream) : e;
}

template <int N>
cudaError_t assemble_n(cpra_plan_s* p, float2* out) {
  Assembly& a = p->asmb;
  cudaError_t e =
      spectra_n<N, kSpecF>(p->Hp, a.ramps, a.F, a.corr, p->xtw, MergeArgs{}, p->Np, p->stream);
  return e == cudaSuccess ? grid_n<N>(p, out) : e;
}

template <int N>
cudaError_t merge_twins_n(cpra_plan_s* d, const MergeArgs& ma, int n_l) {
  cudaStream_t st = d->stream;
  cudaError_t e = spectra_n<N, kSpecRef>(nullptr, nullptr, nullptr, nullptr, d->xtw, ma, 1, st);
  if (e != cudaSuccess || n_l < 2) return e;
  e = cudaMemsetAsync(ma.dist, 0, sizeof(double) * n_l, st);
  return e == cudaSuccess
             ? spectra_n<N, kSpecDist>(nullptr, nullptr, nullptr, nullptr, d->xtw, ma, n_l, st)
             : e;
}

template <int N>
cudaError_t merge_n(cpra_plan_s* d, const MergeArgs& ma, int n_l, float2* acc, unsigned long long* rings,
                           float* prtf) {
  using C = ColW<N, kPrecFP32>;
  cudaStream_t st = d->stream;
  static PerDevice<bool> attr;
  cudaError_t e = smem_once(k_merge<N>, spec_smem<N>(), attr);
  const size_t total = (size_t)d->Np * (N / 2);
  unsigned* counts = reinterpret_cast<unsigned*>(rings + total);
  if (e == cudaSuccess && rings)
    e = cudaMemsetAsync(rings, 0, sizeof(unsigned long long) * total + sizeof(unsigned) * (N / 2), st);
  if (e != cudaSuccess) return e;
  g_launches += 1;
  k_merge<N><<<dim3((N / 2) / C::CB, d->Np), C::NT, spec_smem<N>(), st>>>(
      ma, n_l, acc, rings, counts, d->asmb.F, d->asmb.corr, d->xtw);
  e = cudaGetLastError();
  if (e == cudaSuccess && rings) e = launch_prtf(rings, counts, prtf, N / 2, (int)total, st);
  return e == cudaSuccess ? grid_n<N>(d, nullptr) : e;
}


// The instances of one N, compiled in the translation unit that names them
// (k_assemble_*.cu) and only declared elsewhere.
#define CPRA_ASSEMBLE_INSTANCES(NN, EXTERN)                                                   \
  EXTERN template cudaError_t assemble_n<NN>(cpra_plan_s*, float2*);                          \
  EXTERN template cudaError_t merge_twins_n<NN>(cpra_plan_s*, const MergeArgs&, int);         \
  EXTERN template cudaError_t merge_n<NN>(cpra_plan_s*, const MergeArgs&, int, float2*, unsigned long long*, float*);

}  // namespace cpra
