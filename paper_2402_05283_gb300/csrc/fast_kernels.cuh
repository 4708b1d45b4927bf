// fast_kernels.cuh - two-pass iteration with warp-resident FFTs, every supported N.
//
// Same dataflow and the same packed half spectrum Hp as k_twopass.cu, but
// every line transform is the two-level register FFT of fftw.cuh: one
// warp-local transpose per transform instead of one block-wide shared-memory
// round trip per radix pass, and no block barriers inside a transform.
//   k_rowpass_w  Hp rows -> C2R -> HIO/RAAR/ER update of g -> R2C -> Hp rows
//   k_prime_w    Eq. 4 coupling of g (optional) -> R2C -> Hp rows
//   k_colpass_w  Hp column block -> FFT_y -> modulus projection onto A_sym
//                with the FP64 Fourier error -> IFFT_y -> Hp column block
// A_sym is read column-major (A_T[n][kx][ky]) so a warp's B-layout reads
// are coalesced.  PREC selects the arithmetic of the DFT stages: FP32
// register FFTs, or BF16 / FP16 tensor-core DFT GEMMs (fftw_tc.cuh).
#pragma once
#include "cpra_internal.h"
#include "fft.cuh"
#include "fftw.cuh"
#include "fftw_pair.cuh"
#include "taps.cuh"

namespace cpra {

// Line transforms of the warp engine: the L-line plans of fftw.cuh, or, at
// N = 512 in FP32, the one-line plan of fftw_pair.cuh (half the registers a
// thread, so twice the warps an SM).  The tensor-core forms keep the L-line
// plans.
template <int N, int PREC> struct WLines { using type = WarpLines<N>; };
template <> struct WLines<512, kPrecFP32> { using type = PairLines512; };
// lines of the assembly and the merge: the spectra's, and the volume's.
// Unless N is a power of two (there the plain ones are as near to 64 bits as
// the full-plane passes were) with accurate constants.  Error and time, plain /
// accurate: N = 192, 90 angles 3.8e-7 in 0.153 ms / 3.6e-7 in 0.154; N = 700, 20
// angles 2.9e-7 in 3.87 ms / 2.8e-7 in 4.28
template <int N>
using SpecLines = std::conditional_t<WP<N>::POW2, typename WLines<N, kPrecFP32>::type,
                                     typename WLines<N, kPrecFP32>::type::Acc>;
template <int N>
using VolLines = std::conditional_t<WP<N>::POW2, typename WLines<N, kPrecFP32>::type,
                                    typename WLines<N, kPrecFP32>::type::AccConst>;
// the one-line plan holds 16 values a lane: small enough for 24 warps an SM
template <class FL> constexpr bool kSlimLines = FL::L == 1 && FL::E1 <= 16 && FL::E2 <= 16;

template <int N, int PREC, class FL>
__device__ __forceinline__ void lines_fwd(float2 (&a)[FL::TA][FL::E1], float2 (&b)[FL::TB][FL::E2],
                                          float2* T, const float2* xs, int lane, const TcCtx* tc) {
  if constexpr (PREC == kPrecFP32) FL::fwd(a, b, T, xs, lane);
  else warp_fft_fwd<N, PREC>(a, b, T, xs, lane, tc);
}
template <int N, int PREC, class FL>
__device__ __forceinline__ void lines_inv(float2 (&b)[FL::TB][FL::E2], float2 (&a)[FL::TA][FL::E1],
                                          float2* T, const float2* xs, int lane, const TcCtx* tc) {
  if constexpr (PREC == kPrecFP32) FL::inv(b, a, T, xs, lane);
  else warp_fft_inv<N, PREC>(b, a, T, xs, lane, tc);
}

// v = row `lane` of a 32 x 32 bit matrix (bit c = column c); returns column
// `lane`: five butterfly rounds that swap the off-diagonal blocks of size
// 16, 8, 4, 2, 1 between lane pairs.
__device__ __forceinline__ uint32_t warp_bit_transpose(uint32_t v, int lane) {
  static_for<0, 5>([&](auto KK) {
    constexpr int j = 16 >> decltype(KK)::value;
    constexpr uint32_t m = j == 16 ? 0x0000FFFFu : j == 8 ? 0x00FF00FFu : j == 4 ? 0x0F0F0F0Fu
                         : j == 2 ? 0x33333333u : 0x55555555u;
    const uint32_t o = __shfl_xor_sync(0xffffffffu, v, j);
    v = (lane & j) ? ((v & ~m) | ((o >> j) & m)) : ((v & m) | ((o & m) << j));
  });
  return v;
}

// The one-line 512-point plan holds pixels x = lane + 32 m (m < 16) of two
// rows, so its support bits are the 32 words of those rows (16 each) read
// one a lane and transposed: bit 16 r + m of the result is the bit of pixel
// lane + 32 m in row r.
template <int N, class FL>
constexpr bool kRowMaskInRegs = kSlimLines<FL> && FL::L == 1 && N == 512;

// per-warp shared memory of the row kernels: transpose tile + the warp's g
// rows; 4 warps a block with the L-line plans (the largest number up to 5
// that divides the angle's warp tasks where 4 does not), 8 with the one-line
// plan
__host__ __device__ constexpr int row_warps(int tasks) {
  return tasks % 4 == 0 ? 4 : tasks % 5 == 0 ? 5 : tasks % 3 == 0 ? 3 : tasks % 2 == 0 ? 2 : 1;
}
// GS: the rows have shared memory of their own; else the old rows are copied
// into the transpose tile once the inverse transform has left it, which takes
// half the shared memory and so lets four CTAs of the L-line plans share an SM
// (row pass, us an angle, own rows / tile: N = 1024 3.28 / 2.58, 700 2.01 /
// 1.79, 384 0.50 / 0.39; prime, which has no old rows, 1024 3.12 / 2.56)
template <int N, class FL_, bool GS_ = true> struct RowCfg {
  using FL = FL_;
  static constexpr bool GS = GS_;
  static_assert((N / 2) % FL::L == 0, "row pairs fill whole warps");
  static constexpr int WARPS = kSlimLines<FL> ? 8 : row_warps((N / 2) / FL::L);
  static constexpr int GROWS = 2 * FL::L;                  // image rows per warp
  static constexpr int GFLOATS = GROWS * N;
  static constexpr int WARP_F2 = FL::TSIZE + (GS ? GFLOATS / 2 : 0);  // float2 per warp
  static constexpr int MINB = GS || WARPS > 4 ? 3 : 4;
  static constexpr size_t SMEM = sizeof(float2) * (N + WARPS * WARP_F2);
};
template <int N, int PREC>
using RowW = RowCfg<N, typename WLines<N, PREC>::type, PREC != kPrecFP32 || kSlimLines<typename WLines<N, PREC>::type>>;
// the prime keeps the L-line plans: its three taps a pixel are loaded in
// registers, where the extra warps of the one-line plan do not pay
template <int N, int PREC> using PrimeW = RowCfg<N, WarpLines<N>, PREC != kPrecFP32>;

// extra shared memory of the tensor-core path (TcLayout of fftw_tc.cuh): the
// block DFT matrices, the CTA's A tile, the unscale factors, the mbarrier
template <int N, int PREC> struct TcSmem {
  using P = WP<N>;
  template <int W>
  static constexpr size_t bytes() {
    if constexpr (PREC == kPrecFP32) return 0;
    else return TcLayout<P::E1, P::E2, W>::BYTES;
  }
};
template <int N, int PREC>
constexpr size_t row_smem() {
  return RowW<N, PREC>::SMEM + TcSmem<N, PREC>::template bytes<RowW<N, PREC>::WARPS>();
}
template <int N, int PREC, bool MOM = false>
constexpr size_t prime_smem() {
  if (MOM && !WP<N>::POW2) return PrimeW<N, PREC>::SMEM + sizeof(float2) * N;
  return PrimeW<N, PREC>::SMEM + TcSmem<N, PREC>::template bytes<PrimeW<N, PREC>::WARPS>();
}

// The CTA's tensor-core state (every thread calls it; tc_end releases it):
// base = the kernel's tensor-core region, gW = the plan's matrices.
template <int N, int PREC, int W>
__device__ __forceinline__ TcCtx tc_setup(char* base, const uint16_t* gW, DevStatus* status,
                                          uint32_t* phase) {
  if constexpr (PREC != kPrecFP32) return tc_begin<WP<N>::E1, WP<N>::E2, W>(base, gW, status, phase);
  else return TcCtx{};
}
template <int PREC>
__device__ __forceinline__ void tc_finish(const TcCtx& c) {
  if constexpr (PREC != kPrecFP32) tc_end(c);
}

template <int N>
__device__ __forceinline__ void load_xtw(float2* xs, const float2* xtw, int) {
  for (int i = threadIdx.x; i < N; i += blockDim.x) xs[i] = xtw[i];
}

// Z (B layout) of the row pairs of this warp -> packed half spectra of both
// rows of every pair, stored to Hp.  Z goes through the warp tile so each
// output index k can meet its partner N - k.
template <int N, class FL>
__device__ __forceinline__ void store_pairs_w(float2 (&b)[FL::TB][FL::E2], float2* T, float2* Hn,
                                              int pair0, int lane) {
  constexpr int H = N / 2;
  static_for<0, FL::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const int line = FL::b_line(t);
    if (FL::b_on(t))
      static_for<0, FL::E2>([&](auto KK) {
        constexpr int j = decltype(KK)::value;
        T[line * N + FL::b_k(t, j)] = b[i][j];
      });
  });
  __syncwarp();
#pragma unroll
  for (int line = 0; line < FL::L; ++line) {
    const float2* Z = T + line * N;
    float2* r0 = Hn + (size_t)(2 * (pair0 + line)) * H;
    float2* r1 = r0 + H;
#pragma unroll
    for (int kk = 0; kk < (H + 31) / 32; ++kk) {
      const int k = lane + 32 * kk;
      if (H % 32 != 0 && k >= H) break;
      float2 h0, h1;
      if (kk == 0 && lane == 0) {
        const float2 z0 = Z[0], zn = Z[H];
        h0 = make_float2(z0.x, zn.x);
        h1 = make_float2(z0.y, zn.y);
      } else {
        const float2 z = Z[k], zm = Z[N - k];
        h0 = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
        h1 = make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
      }
      r0[k] = h0;
      r1[k] = h1;
    }
  }
  __syncwarp();
}

// ---------------------------------------------------------------- row pass
// One CTA of the row pass: row pairs [bx * WARPS * L, (bx + 1) * WARPS * L)
// of tile tl = (job, angle).
template <int N, int PREC>
__device__ __forceinline__ void rowpass_tile(const JobStatic* __restrict__ js,
                                             const JobStep* __restrict__ st, const int2 tl,
                                             const int bx) {
  using RW = RowW<N, PREC>;
  using FL = typename RW::FL;
  constexpr int H = N / 2;
  extern __shared__ float2 smem[];
  const JobStatic* J = js + tl.x;
  const JobStep* Z = st + tl.x;
  if (!Z->active) return;
  float* g = Z->g;
  float2* Hp = J->Hp;
  const uint32_t* __restrict__ S = J->S;
  double* err_acc = J->err_acc;
  const double* __restrict__ Cn = J->Cn;
  const double* __restrict__ sumA2 = J->sumA2;
  double* err_hist = J->err_hist;
  const long long err_slot = Z->err_slot;
  const float2* __restrict__ xtw = J->xtw;
  const int Np = J->Np, W = J->W;
  const float beta = J->beta;
  const float c2 = 1.0f - 2.0f * beta;
  const int algo = Z->algo, forward = Z->forward;
  float2* xs = smem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* T = smem + N + warp * RW::WARP_F2;
  float* Gs = reinterpret_cast<float*>(T + (RW::GS ? FL::TSIZE : 0));  // this warp's 2L rows of g
  uint32_t tc_phase = 0;
  const TcCtx tc = tc_setup<N, PREC, RW::WARPS>(reinterpret_cast<char*>(smem + N + RW::WARPS * RW::WARP_F2),
                                                J->tcw, J->status, &tc_phase);
  const int n = tl.y;
  const int pair0 = (bx * RW::WARPS + warp) * FL::L;
  float* grow = g + ((size_t)n * N + 2 * pair0) * N;  // 2L contiguous rows
  float2* Hn = Hp + (size_t)n * N * H;
  // the warp's 2L packed spectrum rows (contiguous) into its tile, then the
  // old iterate, which is needed only after the inverse FFT
  {
    constexpr int HC = FL::L * N / 2;  // 16-byte pieces
    const float2* hrow = Hn + (size_t)(2 * pair0) * H + 2 * lane;
#pragma unroll
    for (int k = 0; k < (HC + 31) / 32; ++k)
      if (HC % 32 == 0 || lane + 32 * k < HC) cp_async16(T + 2 * (lane + 32 * k), hrow + 64 * k);
    cp_async_commit();
  }
  constexpr int GC = RW::GFLOATS / 4;  // 16-byte pieces
  auto load_old = [&] {  // ER does not look at the old iterate: 4 of 16 N^2 bytes less
    if (algo != kER) {
#pragma unroll
      for (int k = 0; k < (GC + 31) / 32; ++k)
        if (GC % 32 == 0 || lane + 32 * k < GC) cp_async16(Gs + 4 * (lane + 32 * k), grow + 4 * lane + 128 * k);
    }
    cp_async_commit();
  };
  if constexpr (RW::GS) load_old();
  if (bx == 0 && threadIdx.x == 0) {
    if (err_slot >= 0) {
      const double den = sumA2[n];
      // err_acc from L2: a persistent launch's column tasks on other SMs sum into it
      err_hist[(size_t)err_slot * Np + n] = publish_error(__ldcg(err_acc + n), Cn[n], den, J->status, n);
    }
    err_acc[n] = 0.0;
  }
  uint32_t smask = 0;  // the one-line plan's support bits (kRowMaskInRegs)
  if constexpr (kRowMaskInRegs<N, FL>)
    smask = __ldg(S + ((size_t)n * N + 2 * pair0 + (lane >> 4)) * W + (lane & 15));
  load_xtw<N>(xs, xtw, RW::WARPS * 32);
  cp_async_wait_group<RW::GS ? 1 : 0>();  // this lane's spectrum copies have landed
  __syncthreads();           // xs, and every lane's copies
  // packed row spectra -> Z = H(row 2p) + i H(row 2p+1), B layout, without
  // branches: k < H reads column k, k > H column N - k (sign s = -1)
  float2 b[FL::TB][FL::E2];
  if constexpr (std::is_same_v<FL, PairLines512>) {
    // lane (kl, h) holds k = kl + 16 j + H h: column c = kl + 16 j (h = 0)
    // or N - k = H - kl - 16 j (h = 1), one base and one stride a lane;
    // only j = 0 of lanes 0 and 1 meets column 0 (k = 0 and k = H)
    const int h = lane & 1, kl = lane >> 1;
    const int bo = h ? H - kl : kl, sj = h ? -16 : 16;
    const float s = h ? -1.0f : 1.0f;
    static_for<0, FL::E2>([&](auto KK) {
      constexpr int j = decltype(KK)::value;
      const int c = (bo + sj * j) & (H - 1);
      const float2 h0 = T[c], h1 = T[H + c];
      float2 z = make_float2(fmaf(-s, h1.y, h0.x), fmaf(s, h0.y, h1.x));
      if constexpr (j == 0)
        if (c == 0) z = h ? make_float2(h0.y, h1.y) : make_float2(h0.x, h1.x);
      b[0][j] = z;
    });
  } else {
    static_for<0, FL::TB>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int t = lane + 32 * i;
      if (!FL::b_on(t)) return;
      const float2* r0 = T + FL::b_line(t) * N;
      const float2* r1 = r0 + H;
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
  }
  __syncwarp();  // the tile is the transforms' scratch from here on
  float2 a[FL::TA][FL::E1];
  if constexpr (RW::GS) lines_inv<N, PREC, FL>(b, a, T, xs, lane, &tc);
  else FL::inv(b, a, T, xs, lane, load_old);
  if constexpr (kRowMaskInRegs<N, FL>) smask = warp_bit_transpose(smask, lane);
  cp_async_wait_all();
  __syncwarp();
  const float inv = 1.0f / N;
  // the real-space rule is uniform over the launch: one specialised loop each
  auto update_rows = [&](auto AA) {
    constexpr int ALGO = decltype(AA)::value;
    static_for<0, FL::TA>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int t = lane + 32 * i;
      if (!FL::a_on(t)) return;
      const int line = FL::a_line(t);
      const int y0 = 2 * (pair0 + line);
      float* g0 = g + ((size_t)n * N + y0) * N;
      float* g1 = g0 + N;
      const float* o0s = Gs + (2 * line) * N;
      const float* o1s = o0s + N;
      const uint32_t* s0 = S + ((size_t)n * N + y0) * W;
      const uint32_t* s1 = s0 + W;
      static_for<0, FL::E1>([&](auto MM) {
        constexpr int m = decltype(MM)::value;
        const int x = FL::a_x(t, m);
        const float2 z = a[i][m];
        const float gp0 = z.x * inv, gp1 = z.y * inv;
        bool in0, in1;
        if constexpr (kRowMaskInRegs<N, FL>) {
          in0 = (smask >> m) & 1u;
          in1 = (smask >> (16 + m)) & 1u;
        } else {
          in0 = (__ldg(s0 + (x >> 5)) >> (x & 31)) & 1u;
          in1 = (__ldg(s1 + (x >> 5)) >> (x & 31)) & 1u;
        }
        const float n0 = update_pixel_t<ALGO>(ALGO == kER ? 0.0f : o0s[x], gp0, in0, beta, c2);
        const float n1 = update_pixel_t<ALGO>(ALGO == kER ? 0.0f : o1s[x], gp1, in1, beta, c2);
        g0[x] = n0;
        g1[x] = n1;
        a[i][m] = make_float2(n0, n1);
      });
    });
  };
  if (algo == kHIO) update_rows(std::integral_constant<int, kHIO>{});
  else if (algo == kER) update_rows(std::integral_constant<int, kER>{});
  else update_rows(std::integral_constant<int, kRAAR>{});
  if (forward) {
    if constexpr (!RW::GS) __syncwarp();  // the old rows leave the tile
    lines_fwd<N, PREC, FL>(a, b, T, xs, lane, &tc);
    store_pairs_w<N, FL>(b, T, Hn, pair0, lane);
  }
  tc_finish<PREC>(tc);
}

template <int N, int PREC>
__global__ void __launch_bounds__(RowW<N, PREC>::WARPS * 32, RowW<N, PREC>::MINB)
k_rowpass_w(const JobStatic* __restrict__ js, const JobStep* __restrict__ st,
            const int2* __restrict__ tiles) {
  rowpass_tile<N, PREC>(js, st, tiles[blockIdx.y], blockIdx.x);
}

// ---------------------------------------------------------------- Eq. 4 taps
// a (A layout) of this warp's row pairs = sum_k alpha_k tap_k (Eq. 4), or
// the image itself for a single tap.  Taps outermost: every load of one tap
// is independent, so a warp keeps 2 * TA * E1 loads in flight per tap.  The
// mirror and object choices are uniform over a tap, so each (mirrored,
// object) combination runs its own loop: pixel x reads column x, or N - x
// mirrored (0 for x = 0, which only m = 0 can hold), at a per-lane base plus
// a constant offset.
// NC: the images are not written during the launch (read-only loads).
template <int N, class FL, bool MIR, bool OBJ, bool NC>
__device__ __forceinline__ void blend_tap(float2 (&a)[FL::TA][FL::E1], const float* src,
                                          const uint32_t* sk, float alpha, int W, int pair0,
                                          int lane) {
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::a_on(t)) return;
    const int y0 = 2 * (pair0 + FL::a_line(t));
    const float* r0 = src + (size_t)y0 * N;
    const uint32_t* m0 = sk + (size_t)y0 * W;
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      const int x = FL::a_x(t, m);
      const int xs_ = MIR ? (m == 0 && x == 0 ? 0 : N - x) : x;
      float v0 = NC ? __ldg(r0 + xs_) : r0[xs_];
      float v1 = NC ? __ldg(r0 + N + xs_) : r0[N + xs_];
      if constexpr (OBJ) {
        const bool in0 = (__ldg(m0 + (xs_ >> 5)) >> (xs_ & 31)) & 1u;
        const bool in1 = (__ldg(m0 + W + (xs_ >> 5)) >> (xs_ & 31)) & 1u;
        v0 = (in0 && v0 >= 0.0f) ? v0 : 0.0f;
        v1 = (in1 && v1 >= 0.0f) ? v1 : 0.0f;
      }
      a[i][m].x = fmaf(alpha, v0, a[i][m].x);
      a[i][m].y = fmaf(alpha, v1, a[i][m].y);
    });
  });
}

template <int N, class FL = WarpLines<N>, bool NC = true>
__device__ __forceinline__ void blend_rows(float2 (&a)[FL::TA][FL::E1], const TapTab& tt,
                                           const CoupleArgs& ca, int W, int pair0, int lane) {
  const int ntaps = ca.n_taps;
  static_for<0, FL::TA>([&](auto II) {
    static_for<0, FL::E1>([&](auto MM) { a[decltype(II)::value][decltype(MM)::value] = make_float2(0.f, 0.f); });
  });
  const bool obj = ca.object != 0;
  for (int k = 0; k < ntaps; ++k) {
    const float alpha = tt.w[k];
    if (alpha == 0.0f) continue;  // a tap on an absent angle
    const float* src = tt.src[k];
    const uint32_t* sk = tt.s[k];
    if (tt.mir[k]) {
      if (obj) blend_tap<N, FL, true, true, NC>(a, src, sk, alpha, W, pair0, lane);
      else blend_tap<N, FL, true, false, NC>(a, src, sk, alpha, W, pair0, lane);
    } else {
      if (obj) blend_tap<N, FL, false, true, NC>(a, src, sk, alpha, W, pair0, lane);
      else blend_tap<N, FL, false, false, NC>(a, src, sk, alpha, W, pair0, lane);
    }
  }
}

// a (A layout) of this warp's row pairs -> rows of one image
template <int N, class FL = WarpLines<N>>
__device__ __forceinline__ void store_rows(const float2 (&a)[FL::TA][FL::E1], float* img, int pair0,
                                           int lane) {
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::a_on(t)) return;
    float* d0 = img + (size_t)(2 * (pair0 + FL::a_line(t))) * N;
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      const int x = FL::a_x(t, m);
      d0[x] = a[i][m].x;
      d0[N + x] = a[i][m].y;
    });
  });
}

// ---------------------------------------------------------------- moments
// A lane's sum rho, sum rho z, sum rho u of its rows (p: a row's sum, pu: its
// sum of rho x) as FP32 pairs, with the exact products by z.
struct Moments {
  float s0 = 0.0f, e0 = 0.0f, sz = 0.0f, ez = 0.0f, su = 0.0f, eu = 0.0f;
  __device__ __forceinline__ void add(float p, float pu, float y) {
    two_add(s0, e0, p);
    two_add(su, eu, pu);
    const float pz = __fmul_rn(p, y);
    two_add(sz, ez, pz);
    ez = __fadd_rn(ez, fmaf(p, y, -pz));
  }
  // no lane of the warp has left FP32's range (a moment is up to N times the
  // sum of rho): else the rows are added again in FP64
  __device__ __forceinline__ bool in_range() const {
    return __all_sync(0xffffffffu, isfinite(s0) && isfinite(sz) && isfinite(su));
  }
  __device__ __forceinline__ void total(double (&m)[3]) const {
    m[0] = warp_sum(s0, e0);
    m[1] = warp_sum(sz, ez);
    m[2] = warp_sum(su, eu);
  }
};
__device__ __forceinline__ void add_moments(double (&d)[3], float p, float pu, float y) {
  d[0] += (double)p;
  d[1] += (double)p * (double)y;
  d[2] += (double)pu;
}

// ---------------------------------------------------------------- prime
// MOM (rows of rho for the assembly, a single plain tap): also the FP64
// moments sum rho, sum rho z, sum rho u of the angle, so that rho is not read
// a second time for them.  Each lane sums its pixels of a row in FP32 and its
// rows as FP32 pairs (48 bits), with the exact products by z; FP64 across
// warps and CTAs.  N = 512, 360 angles: rows 210 us and moments 128 us
// apart, 230 us together.
template <int N, int PREC, bool MOM = false>
__global__ void __launch_bounds__(PrimeW<N, PREC>::WARPS * 32, 3)
k_prime_w(const JobStatic* __restrict__ js, const JobStep* __restrict__ st,
          const int2* __restrict__ tiles, double* moments) {
  using RW = PrimeW<N, PREC>;
  // (rows of rho: the lines of the assembly, with the tiles of the prime)
  using FL = std::conditional_t<MOM && !WP<N>::POW2, typename RW::FL::Acc, typename RW::FL>;
  constexpr int H = N / 2;
  extern __shared__ float2 smem[];
  const int2 tl = tiles[blockIdx.y];
  const JobStatic* J = js + tl.x;
  const JobStep* Z = st + tl.x;
  if (!Z->prime) return;
  const float* __restrict__ g_src = Z->g_src;
  float* __restrict__ g_dst = Z->ca.store_g ? Z->g_dst : nullptr;
  float2* Hp = J->Hp;
  const uint32_t* __restrict__ S = J->S;
  const float2* __restrict__ xtw = J->xtw;
  const int Np = J->Np, W = J->W;
  const CoupleArgs& ca = Z->ca;
  float2* xs = smem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* T = smem + FL::XN + warp * RW::WARP_F2;
  uint32_t tc_phase = 0;
  const TcCtx tc = tc_setup<N, PREC, RW::WARPS>(reinterpret_cast<char*>(smem + FL::XN + RW::WARPS * RW::WARP_F2),
                                                J->tcw, J->status, &tc_phase);
  const int n = tl.y;
  const int pair0 = (blockIdx.x * RW::WARPS + warp) * FL::L;
  __shared__ TapTab tt;
  load_xtw<FL::XN>(xs, xtw, RW::WARPS * 32);
  fill_taps<N>(tt, ca, g_src, Z->g_dst, S, n, Np, W, J->present);
  __syncthreads();
  float2 a[FL::TA][FL::E1];
  blend_rows<N, FL>(a, tt, ca, W, pair0, lane);
  if (ca.store_g) store_rows<N, FL>(a, g_dst + (size_t)n * N * N, pair0, lane);
  __shared__ double red[MOM ? 3 : 1][RW::WARPS];
  if constexpr (MOM) {
    // f(sum, sum of x values, y) of the lane's rows
    auto rows = [&](auto&& f) {
      static_for<0, FL::TA>([&](auto II) {
        constexpr int i = decltype(II)::value;
        const int t = lane + 32 * i;
        if (!FL::a_on(t)) return;
        float p[2] = {0.0f, 0.0f}, pu[2] = {0.0f, 0.0f};
        static_for<0, FL::E1>([&](auto MM) {
          constexpr int m = decltype(MM)::value;
          const float x = (float)FL::a_x(t, m);
          p[0] += a[i][m].x;
          p[1] += a[i][m].y;
          pu[0] = fmaf(a[i][m].x, x, pu[0]);
          pu[1] = fmaf(a[i][m].y, x, pu[1]);
        });
#pragma unroll
        for (int r = 0; r < 2; ++r) f(p[r], pu[r], (float)(2 * (pair0 + FL::a_line(t)) + r));
      });
    };
    Moments mom;
    rows([&](float p, float pu, float y) { mom.add(p, pu, y); });
    double m[3];
    if (mom.in_range()) {
      mom.total(m);
    } else {
      double d[3] = {0.0, 0.0, 0.0};
      rows([&](float p, float pu, float y) { add_moments(d, p, pu, y); });
#pragma unroll
      for (int q = 0; q < 3; ++q) m[q] = warp_sum(d[q]);
    }
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < 3; ++q) red[MOM ? q : 0][warp] = m[q];
  }
  float2 b[FL::TB][FL::E2];
  lines_fwd<N, PREC, FL>(a, b, T, xs, lane, &tc);
  store_pairs_w<N, FL>(b, T, Hp + (size_t)n * N * H, pair0, lane);
  tc_finish<PREC>(tc);
  if constexpr (MOM) {
    __syncthreads();
    if (threadIdx.x < 3) {
      double s = 0.0;
      for (int w = 0; w < RW::WARPS; ++w) s += red[threadIdx.x][w];
      atomicAdd(moments + 3 * n + threadIdx.x, s);
    }
  }
}

// ---------------------------------------------------------------- column pass
// packed columns per CTA: 16 (128 B of each row) with the L-line plans; 8
// with the one-line plan (8 warps, three CTAs an SM), for the one-line sizes
// whose 8 columns leave room for two CTAs an SM (640, 768), and for the
// 16-bit path at N >= 512, where the tensor-core region (block DFT matrices,
// A tile) beside 16 columns would leave room for one CTA an SM; where N/2 is
// not a multiple of 16, a divisor of it (all 24 columns at N = 48, 10 of the
// 350 at N = 700: 80 B of each row)
template <int N, int PREC> struct ColW {
  using FL = typename WLines<N, PREC>::type;
  static constexpr int CB = N == 700 ? 10 : N == 48 ? 24 : N == 16 ? 8
                            : ((PREC != kPrecFP32 && N >= 512) || kSlimLines<FL> || N == 640 || N == 768) ? 8 : 16;
  static_assert((N / 2) % CB == 0 && CB % FL::L == 0, "column blocks");
  static constexpr int WARPS = CB / FL::L;
  static constexpr int NT = WARPS * 32;
  static constexpr int MINB = kSlimLines<FL> ? 3 : NT <= 128 ? 4 : (NT <= 256 || N == 700 ? 2 : 1);
  static constexpr int SP = CB + 1;  // staging pitch
  static constexpr int N2 = N / 2;
  static constexpr int STAGE = N * SP;
  static constexpr int TILES = WARPS * FL::TSIZE;
  static constexpr int BUF = STAGE > TILES ? STAGE : TILES;
  // A_sym of the block in shared memory, column c at c * AP, frequency ky at
  // a_pos(ky): the upper half moved on by 16 floats, so lanes reading ky and
  // ky + N/2 (the one-line plan's lane pairs) or the same ky of neighbouring
  // columns (the L-line plans) fall in different banks; no shift where a
  // 16-byte piece would straddle the halves (N = 700, one line a warp)
  static constexpr int AS = (N / 2) % 4 == 0 ? 16 : 0;
  static constexpr int AP = N + 16;
  static __device__ __forceinline__ int a_pos(int ky) { return ky + (ky >= N / 2 ? AS : 0); }
  static constexpr size_t SMEM = sizeof(float2) * (N + BUF) + sizeof(float) * CB * AP;
};
// a_pos of the B-layout frequency b_k(t, j) of a column-pass task: the half
// is fixed by t in the one-line plan and by j in the L-line plans, so the
// offset over j stays a compile-time constant
template <class C, int j>
__device__ __forceinline__ int col_a_pos(int t) {
  using FL = typename C::FL;
  if constexpr (std::is_same_v<FL, PairLines512>)
    return FL::b_k(t, 0) + ((t & 1) ? 16 : 0) + 16 * j;
  else
    return FL::b_k(t, 0) + FL::E1 * j + (FL::E1 * j >= C::N2 ? C::AS : 0);
}
template <int N, int PREC>
constexpr size_t col_smem() {
  return ColW<N, PREC>::SMEM + TcSmem<N, PREC>::template bytes<ColW<N, PREC>::WARPS>();
}

// G' = a G / |G| (a where G = 0); e += (|G| - a)^2, unweighted (the caller
// keeps one sum per weight).  In plans with a missing-data mask (MASKED),
// a < 0 marks a pixel left free.  Branch-free: G = 0 takes rsqrt(1) and the
// direction (1, 0), and |G| - a = 0 * 1 - a.  The per-thread partial sum
// stays in FP32 (at most a few hundred terms); across a warp's threads it is an
// FP32 pair, across warps, blocks and columns FP64.
template <bool MASKED>
__device__ __forceinline__ float2 project_w(float2 G, float a, float& e) {
  if constexpr (MASKED)
    if (a < 0.0f) return G;  // an unmeasured pair (mask): free, no error term
  const float r2 = fmaf(G.x, G.x, G.y * G.y);
  const bool zero = !(r2 > 0.0f);
  const float inv = rsqrtf(zero ? 1.0f : r2);
  const float d = fmaf(r2, inv, -a);
  e = fmaf(d, d, e);
  const float s = a * inv;
  // __fmul_rn: a product the compiler may not contract into the caller's
  // next add, so every instance of the kernels rounds the same way
  return make_float2(__fmul_rn(zero ? 1.0f : G.x, s), zero ? 0.0f : __fmul_rn(G.y, s));
}

// One CTA of the column pass: packed columns [bx * CB, (bx + 1) * CB) of
// tile tl = (job, angle).
//
// L2_ONLY: stage the spectrum with L2-only loads instead of the 8-byte
// cp.async (which allocates in L1): inside a persistent kernel other SMs
// rewrite the spectrum between two reads of the same lines by this SM.
template <int N, int PREC, bool MASKED, bool L2_ONLY = false>
__device__ __forceinline__ void colpass_tile(const JobStatic* __restrict__ js,
                                             const JobStep* __restrict__ st, const int2 tl,
                                             const int bx) {
  using C = ColW<N, PREC>;
  using FL = typename C::FL;
  constexpr int H = N / 2;
  extern __shared__ float2 smem[];
  const JobStatic* J = js + tl.x;
  if (!st[tl.x].active) return;
  float2* Hp = J->Hp;
  const float* __restrict__ A_T = J->A_main;
  const float* __restrict__ A_nyq = J->A_nyq;
  double* err_acc = J->err_acc;
  const float2* __restrict__ xtw = J->xtw;
  float2* xs = smem;
  float2* buf = smem + N;  // staging, then the warps' transpose tiles
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* As = reinterpret_cast<float*>(buf + C::BUF);  // A_sym of the block, [c][ky]
  uint32_t tc_phase = 0;
  const TcCtx tc = tc_setup<N, PREC, C::WARPS>(reinterpret_cast<char*>(As + C::CB * C::AP), J->tcw, J->status,
                                               &tc_phase);
  float2* T = buf + warp * FL::TSIZE;
  const int n = tl.y;
  const int c0 = bx * C::CB;
  float2* Hn = Hp + (size_t)n * N * H;
  // thread (row y0 + k RS, column cc) of the block: constant strides, so
  // the unrolled copies differ only in immediate offsets.  A warp's 32 / CB
  // rows are WARPS apart: with 8 columns (pitch 9) rows 8 apart start 16
  // banks apart, so a warp's 256 bytes take the minimum two wavefronts
  // (blocks whose columns do not divide a warp take plain thread order)
  constexpr int RS = C::NT / C::CB, SR = (N + RS - 1) / RS;
  constexpr int AC = C::CB * N / 4, AR = (AC + C::NT - 1) / C::NT;
  static_assert(C::NT % C::CB == 0, "column staging");
  const int y0 = 32 % C::CB == 0 ? warp + C::WARPS * (lane / C::CB) : threadIdx.x / C::CB;
  const int cc = 32 % C::CB == 0 ? lane % C::CB : threadIdx.x % C::CB;
  {
    const float2* src = Hn + (size_t)y0 * H + c0 + cc;
    float2* dst = buf + y0 * C::SP + cc;
    if constexpr (L2_ONLY) {
#pragma unroll
      for (int k = 0; k < SR; ++k)
        if (N % RS == 0 || y0 + k * RS < N) dst[k * RS * C::SP] = ld_cg(src + (size_t)k * RS * H);
    } else {
#pragma unroll
      for (int k = 0; k < SR; ++k)
        if (N % RS == 0 || y0 + k * RS < N) cp_async8(dst + k * RS * C::SP, src + (size_t)k * RS * H);
    }
    const float* Ablk = A_T + ((size_t)n * H + c0) * N;  // CB contiguous columns
#pragma unroll
    for (int k = 0; k < AR; ++k) {
      const int f = 4 * (threadIdx.x + k * C::NT);  // 4 floats, never across a column (4 | N) or a shifted half
      if (AC % C::NT == 0 || f < 4 * AC) cp_async16(As + (f / N) * C::AP + C::a_pos(f % N), Ablk + f);
    }
  }
  cp_async_commit();
  load_xtw<N>(xs, xtw, C::NT);
  cp_async_wait_all();
  __syncthreads();
  float2 a[FL::TA][FL::E1];
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
  float2 b[FL::TB][FL::E2];
  lines_fwd<N, PREC, FL>(a, b, T, xs, lane, &tc);
  float err2 = 0.0f, err1 = 0.0f;  // error terms of weight 2 and 1
  const bool warp_packed = (c0 == 0 && warp == 0);  // line 0 of warp 0 holds column 0
  static_for<0, FL::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const int col = warp * FL::L + FL::b_line(t);
    if (FL::b_on(t) && c0 + col != 0) {
      const float* Ac = As + col * C::AP;
      static_for<0, FL::E2>([&](auto KK) {
        constexpr int j = decltype(KK)::value;
        b[i][j] = project_w<MASKED>(b[i][j], Ac[col_a_pos<C, j>(t)], err2);
      });
    }
  });
  if (warp_packed) {
    // column 0 packs G(., 0) + i G(., N/2); both are Hermitian along ky
    static_for<0, FL::TB>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int t = lane + 32 * i;
      if (FL::b_on(t) && FL::b_line(t) == 0) {
        static_for<0, FL::E2>([&](auto KK) {
          constexpr int j = decltype(KK)::value;
          T[FL::b_k(t, j)] = b[i][j];
        });
      }
    });
    __syncwarp();
    static_for<0, FL::TB>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int t = lane + 32 * i;
      if (FL::b_on(t) && FL::b_line(t) == 0) {
        const float* A0 = As;  // column 0 of the block
        const float* An = A_nyq + (size_t)n * N;
        static_for<0, FL::E2>([&](auto KK) {
          constexpr int j = decltype(KK)::value;
          const int ky = FL::b_k(t, j);
          const float2 z = T[ky], zm = T[(N - ky) % N];
          const float2 g0 = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
          const float2 gn = make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
          const float2 p0 = project_w<MASKED>(g0, A0[col_a_pos<C, j>(t)], err1);
          const float2 pn = project_w<MASKED>(gn, __ldg(An + ky), err1);
          b[i][j] = make_float2(p0.x - pn.y, p0.y + pn.x);
        });
      }
    });
    __syncwarp();
  }
  lines_inv<N, PREC, FL>(b, a, T, xs, lane, &tc);
  __syncthreads();
  const float inv = 1.0f / N;
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::a_on(t)) return;
    const int col = warp * FL::L + FL::a_line(t);
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      buf[FL::a_x(t, m) * C::SP + col] = cscale(a[i][m], inv);
    });
  });
  __syncthreads();
  {
    float2* dst = Hn + (size_t)y0 * H + c0 + cc;
    const float2* src = buf + y0 * C::SP + cc;
#pragma unroll
    for (int k = 0; k < SR; ++k)
      if (N % RS == 0 || y0 + k * RS < N) dst[(size_t)k * RS * H] = src[k * RS * C::SP];
  }
  // the warp's error terms: an FP32 pair, FP64 beyond its range.  Each warp adds
  // its own: a barrier and one thread's sum over the warps would be the block's
  // tail (ten iterations, with / without: N = 1024, 300 angles 18.90 / 18.67 ms,
  // 700, 27 angles 1.31 / 1.27, 512, 360 angles 5.06 / 5.05; without the look at
  // the range 5.02)
  float es = 2.0f * err2, ee = 0.0f;
  two_add(es, ee, err1);
  warp_add_pairs(es, ee);
  const double errd = isfinite(es) ? (double)es + (double)ee : warp_sum(2.0 * (double)err2 + (double)err1);
  if (lane == 0) atomicAdd(err_acc + n, errd);
  tc_finish<PREC>(tc);
}

template <int N, int PREC, bool MASKED>
__global__ void __launch_bounds__(ColW<N, PREC>::NT, ColW<N, PREC>::MINB)
k_colpass_w(const JobStatic* __restrict__ js, const JobStep* __restrict__ st,
            const int2* __restrict__ tiles) {
  colpass_tile<N, PREC, MASKED>(js, st, tiles[blockIdx.y], blockIdx.x);
}

// ---------------------------------------------------------------- persistent
// One launch of the warp engine over `iters` iterations of a group of
// reconstructions of one N.  Every CTA takes the next task of a queue
// ordered (iteration, pass, tile, block): the column-pass blocks of every
// (member, angle) tile, then their row-pass blocks.  Before it runs a task
// the CTA waits until the blocks it reads from are done: a column block of
// iteration i needs every row block of its tile at i - 1 (the launch starts
// after the coupling prime), a row block every column block of its tile at
// i.  Dependencies point to earlier tasks, which running CTAs hold, so the
// queue drains whatever the grid size.  A wait longer than `budget` clock
// cycles flags TIMEOUT in every member's status word and the CTA returns.
// Each task computes exactly what the same block of the separate passes
// computes.

template <int N> struct PersistCfg {
  using C = ColW<N, kPrecFP32>;
  using R = RowW<N, kPrecFP32>;
  static constexpr int NT = C::NT;
  static constexpr int RPT = C::NT / (R::WARPS * 32);  // row-pass blocks a task (its warps)
  static constexpr int CB = (N / 2) / C::CB;            // column tasks an angle
  static constexpr int RB = (N / 2) / (R::WARPS * R::FL::L) / (RPT > 0 ? RPT : 1);  // row tasks an angle
  static constexpr size_t RSMEM = sizeof(float2) * (N + (size_t)(RPT > 0 ? RPT : 1) * R::WARPS * R::WARP_F2);
  static constexpr size_t SMEM = col_smem<N, kPrecFP32>() > RSMEM ? col_smem<N, kPrecFP32>() : RSMEM;
  // resident CTAs an SM the register budget is set for: the column pass's,
  // or, for the 4-warp sizes, three (the row pass's) unless shared memory
  // holds fewer anyway (then the registers are not what limits residency)
  static constexpr int SMEM_CTAS = (int)((228u * 1024u) / (SMEM + 1024u));
  static constexpr int MINB = NT == 128 ? (SMEM_CTAS < 3 ? (SMEM_CTAS > 0 ? SMEM_CTAS : 1) : 3) : C::MINB;
  static constexpr bool OK = (RPT == 1 || RPT == 2) && C::NT == RPT * R::WARPS * 32 &&
                             ((N / 2) / (R::WARPS * R::FL::L)) % (RPT > 0 ? RPT : 1) == 0 &&
                             SMEM <= 227 * 1024;
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// add 1 after every write this CTA made before its last barrier
__device__ __forceinline__ void add_release(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;\n" ::"l"(p) : "memory");
}
// wait until *c >= need (acquire); false after `budget` cycles
__device__ __forceinline__ bool wait_count(const unsigned* c, unsigned need, long long budget) {
  if (ld_acquire(c) >= need) return true;
  const long long t0 = clock64();
  unsigned ns = 32;
  while (ld_acquire(c) < need) {
    if (clock64() - t0 > budget) return false;
    __nanosleep(ns);
    if (ns < 2048) ns *= 2;
  }
  return true;
}

template <int N, bool MASKED>
__global__ void __launch_bounds__(PersistCfg<N>::NT, PersistCfg<N>::MINB)
k_persist_w(const PersistArgs a) {
  using P = PersistCfg<N>;
  __shared__ unsigned task_s;
  __shared__ int ok_s;
  // queue order: the tiles in chunks of a.chunk; a chunk runs all of the
  // launch's iterations (each: the column tasks of its tiles, then their row
  // tasks) before the next chunk starts, so that a chunk's iterates, spectra
  // and amplitudes stay in L2 from one pass to the next.  A chunk of every
  // tile is the plain (iteration, pass, tile, block) order.
  constexpr unsigned PT = P::CB + P::RB;  // tasks of one tile and iteration
  const unsigned K = (unsigned)a.chunk, iters = (unsigned)a.iters;
  const unsigned full = (unsigned)a.ntiles / K;  // chunks of K tiles; the last holds the rest
  const unsigned full_tasks = full * K * PT * iters;
  const unsigned total = (unsigned)a.ntiles * PT * iters;
  // thread 0 holds the CTA's next ticket, fetched while the current task
  // runs (a held ticket runs as soon as the current task ends, so the queue
  // still drains: the smallest unfinished task is always running)
  unsigned next = 0;
  if (threadIdx.x == 0) next = atomicAdd(a.ticket, 1u);
  for (;;) {
    __syncthreads();  // the previous task is done with task_s, ok_s and shared memory
    if (threadIdx.x == 0) task_s = next;
    __syncthreads();
    const unsigned task = task_s;
    if (task >= total) return;
    const bool in_full = task < full_tasks;
    const unsigned c = in_full ? task / (K * PT * iters) : full;  // chunk
    const unsigned kc = in_full ? K : (unsigned)a.ntiles - full * K;  // its tiles
    const unsigned r0 = in_full ? task % (K * PT * iters) : task - full_tasks;
    const int it = (int)(r0 / (kc * PT));
    const unsigned r = r0 % (kc * PT);
    const bool col = r < kc * P::CB;
    const unsigned rr = col ? r : r - kc * P::CB;
    const int tile = (int)(c * K + (col ? rr / P::CB : rr / P::RB));
    const int bx = (int)(col ? rr % P::CB : rr % P::RB);
    if (threadIdx.x == 0) {
      const unsigned* c = col ? a.done + 2 * tile + 1 : a.done + 2 * tile;
      unsigned need = col ? (unsigned)(P::RB * it) : (unsigned)(P::CB * (it + 1));
      if (a.hold && task == 0) {
        c = a.ticket + 1;
        need = 1;
      }
      next = atomicAdd(a.ticket, 1u);
      const bool ok = wait_count(c, need, a.budget);
      if (!ok)
        for (int j = 0; j < a.m; ++j) {
          volatile DevStatus* ds = a.js[j].status;
          ds->flags = ds->flags | kStatusTimeout;
        }
      ok_s = ok;
    }
    __syncthreads();
    if (!ok_s) return;
    const int2 tl = a.tiles[tile];
    const JobStep* st = a.st + (size_t)(a.row0 + it) * a.m;
    if (col) colpass_tile<N, kPrecFP32, MASKED, true>(a.js, st, tl, bx);
    else rowpass_tile<N, kPrecFP32>(a.js, st, tl, bx * P::RPT);
    __syncthreads();
    if (threadIdx.x == 0) add_release(a.done + 2 * tile + (col ? 0 : 1));
  }
}

// ---------------------------------------------------------------- launchers
template <int N, int PREC>
cudaError_t prepare_device_w() {
  cudaError_t e = smem_attr(k_rowpass_w<N, PREC>, row_smem<N, PREC>());
  if (e == cudaSuccess) e = smem_attr(k_prime_w<N, PREC>, prime_smem<N, PREC>());
  if constexpr (PREC == kPrecFP32)
    if (e == cudaSuccess) e = smem_attr(k_prime_w<N, PREC, true>, prime_smem<N, PREC, true>());
  if (e == cudaSuccess) e = smem_attr(k_colpass_w<N, PREC, false>, col_smem<N, PREC>());
  if (e == cudaSuccess) e = smem_attr(k_colpass_w<N, PREC, true>, col_smem<N, PREC>());
  if constexpr (PREC != kPrecFP32) {
    // the tensor-memory columns of every CTA that can be resident on an SM
    // must fit its 512 (an allocation beyond them would wait for a release)
    using P = WP<N>;
    auto fits = [&](auto kernel, int threads, size_t smem, uint32_t cols) -> cudaError_t {
      int blocks = 0;
      cudaError_t r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, kernel, threads, smem);
      if (r != cudaSuccess) return r;
      return (uint32_t)blocks * cols <= 512u ? cudaSuccess : cudaErrorNotSupported;
    };
    constexpr uint32_t row_cols = TcLayout<P::E1, P::E2, RowW<N, PREC>::WARPS>::COLS;
    constexpr uint32_t prime_cols = TcLayout<P::E1, P::E2, PrimeW<N, PREC>::WARPS>::COLS;
    constexpr uint32_t col_cols = TcLayout<P::E1, P::E2, ColW<N, PREC>::WARPS>::COLS;
    if (e == cudaSuccess) e = fits(k_rowpass_w<N, PREC>, RowW<N, PREC>::WARPS * 32, row_smem<N, PREC>(), row_cols);
    if (e == cudaSuccess)
      e = fits(k_prime_w<N, PREC>, PrimeW<N, PREC>::WARPS * 32, prime_smem<N, PREC>(), prime_cols);
    if (e == cudaSuccess) e = fits(k_colpass_w<N, PREC, false>, ColW<N, PREC>::NT, col_smem<N, PREC>(), col_cols);
    if (e == cudaSuccess) e = fits(k_colpass_w<N, PREC, true>, ColW<N, PREC>::NT, col_smem<N, PREC>(), col_cols);
  }
  return e;
}

template <int N, int PREC>
cudaError_t prepare_w() {
  static PerDevice<bool> done;
  return once_on_device(done, prepare_device_w<N, PREC>);
}

template <int N, int PREC>
cudaError_t rowpass_w(const Launch& L) {
  using RW = RowW<N, PREC>;
  const size_t smem = row_smem<N, PREC>();
  cudaError_t e = prepare_w<N, PREC>();
  if (e != cudaSuccess) return e;
  dim3 grid((N / 2) / (RW::WARPS * RW::FL::L), L.ntiles);
  g_launches += 1;
  k_rowpass_w<N, PREC><<<grid, RW::WARPS * 32, smem, L.stream>>>(L.js, L.st, L.tiles);
  return cudaGetLastError();
}

template <int N, int PREC>
cudaError_t prime_w(const Launch& L, double* moments) {
  using RW = PrimeW<N, PREC>;
  const size_t smem = prime_smem<N, PREC>();
  cudaError_t e = prepare_w<N, PREC>();
  if (e != cudaSuccess) return e;
  dim3 grid((N / 2) / (RW::WARPS * RW::FL::L), L.ntiles);
  g_launches += 1;
  if constexpr (PREC == kPrecFP32)
    if (moments) {
      k_prime_w<N, PREC, true><<<grid, RW::WARPS * 32, prime_smem<N, PREC, true>(), L.stream>>>(L.js, L.st, L.tiles, moments);
      return cudaGetLastError();
    }
  k_prime_w<N, PREC><<<grid, RW::WARPS * 32, smem, L.stream>>>(L.js, L.st, L.tiles, nullptr);
  return cudaGetLastError();
}

template <int N, int PREC>
cudaError_t colpass_w(const Launch& L) {
  using C = ColW<N, PREC>;
  const size_t smem = col_smem<N, PREC>();
  cudaError_t e = prepare_w<N, PREC>();
  if (e != cudaSuccess) return e;
  dim3 grid((N / 2) / C::CB, L.ntiles);
  g_launches += 1;
  if (L.masked) k_colpass_w<N, PREC, true><<<grid, C::NT, smem, L.stream>>>(L.js, L.st, L.tiles);
  else k_colpass_w<N, PREC, false><<<grid, C::NT, smem, L.stream>>>(L.js, L.st, L.tiles);
  return cudaGetLastError();
}

// sizes of the tensor-core forms
#define CPRA_FOR_EACH_FAST_N(X) X(64) X(128) X(256) X(512) X(1024)
// sizes at which CPRA_ENGINE_WARP can be asked for (and the persistent batch mode)
#define CPRA_FOR_EACH_WARP_N(X) X(64) X(128) X(192) X(256) X(384) X(512) X(1024)

// The FP32 instances of one N, compiled in the translation unit that names
// them (k_fast_*.cu) and only declared elsewhere: nvcc takes about 10 s a size.
#define CPRA_WARP_INSTANCES(NN, EXTERN)                              \
  EXTERN template cudaError_t prepare_w<NN, kPrecFP32>();            \
  EXTERN template cudaError_t rowpass_w<NN, kPrecFP32>(const Launch&); \
  EXTERN template cudaError_t prime_w<NN, kPrecFP32>(const Launch&, double*); \
  EXTERN template cudaError_t colpass_w<NN, kPrecFP32>(const Launch&);

}  // namespace cpra
