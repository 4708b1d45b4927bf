// fftw.cuh - warp-resident two-level FFTs of length N = E1 * E2.
//
// A warp transforms L lines at once.  With n = l + E2 m and k = k1 + E1 k2,
//   X[k1 + E1 k2] = sum_l W_N^(l k1) W_E2^(l k2) [ sum_m x[l + E2 m] W_E1^(m k1) ]
// so a forward transform is: E1-point DFTs in registers (step A, one per
// (line, l)), the cross twiddle W_N^(l k1), one transpose through the warp's
// shared-memory tile, E2-point DFTs in registers (step B, one per
// (line, k1)).  The inverse runs the same steps backwards.  Only __syncwarp
// is needed: a warp owns its lines and its tile.
//
// Register layouts (lane = threadIdx.x % 32, i = task slot of the lane):
//   A layout  a[i][m] = x_line[l + E2 m],      task t = lane + 32 i:
//             line = t / E2, l = t % E2
//   B layout  b[i][k2] = X_line[k1 + E1 k2],   task t = lane + 32 i:
//             line = t / E1, k1 = t % E1
// Where L * E2 or L * E1 is not a multiple of 32 the last slot's upper lanes
// have no task (a_on, b_on): they take part in the warp's barriers only.
// Twiddles inside the register DFTs are compile-time constants (cos and sin
// evaluated from their Taylor series at compile time in FP64, exact at
// multiples of pi/2); the cross twiddles come from a table
// xtw[k1 * E2 + l] = exp(-2 pi i l k1 / N) built in FP64 on the host.
#pragma once
#include <type_traits>

#include "fft.cuh"
#include "fftw_tc.cuh"

namespace cpra {

// exp(DIR * 2 pi i Q / M) as compile-time constants
template <int M, int Q, int DIR> struct TwC {
  static constexpr float re = (float)cx_cos2pi(Q, M);
  static constexpr float im = (float)(DIR * cx_sin2pi(Q, M));
  static constexpr float re_lo = (float)(cx_cos2pi(Q, M) - (double)re);
  static constexpr float im_lo = (float)(DIR * cx_sin2pi(Q, M) - (double)im);
};

// In-register E-point DFT, y_k = sum_j v_j exp(DIR 2 pi i jk / E), as
// self-sorting Stockham passes over compile-time indices.  ACC: the constants
// as pairs of floats (fft.cuh).
template <int E, int DIR, bool ACC = false, int NS = 1>
__device__ __forceinline__ void reg_fft(float2 (&v)[E]) {
  if constexpr (NS < E) {
    constexpr int R = pick_radix(E / NS);
    constexpr int NB = E / R;
    float2 out[E];
    static_for<0, NB>([&](auto J) {
      constexpr int j = decltype(J)::value;
      constexpr int k = j % NS;
      float2 x[R];
      static_for<0, R>([&](auto RR) {
        constexpr int r = decltype(RR)::value;
        float2 t = v[j + r * NB];
        if constexpr (NS > 1 && r > 0 && k > 0) {
          constexpr int M = NS * R, Q = (k * r) % (NS * R);
          if constexpr ((4 * Q) % M == 0) {
            // a multiple of pi/2: exact sign changes and swaps
            constexpr int quarter = (4 * Q) / M;  // exp(DIR * i * pi/2 * quarter)
            if constexpr (quarter == 1) t = mul_i<DIR>(t);
            else if constexpr (quarter == 2) t = make_float2(-t.x, -t.y);
            else if constexpr (quarter == 3) t = mul_i<-DIR>(t);
          } else {
            constexpr float wr = TwC<M, Q, DIR>::re;
            constexpr float wi = TwC<M, Q, DIR>::im;
            if constexpr (ACC)
              t = cmul(t, make_float2(wr, wi), make_float2(TwC<M, Q, DIR>::re_lo, TwC<M, Q, DIR>::im_lo));
            else
              t = make_float2(fmaf(t.x, wr, -t.y * wi), fmaf(t.x, wi, t.y * wr));
          }
        }
        x[r] = t;
      });
      Dft<R, DIR, ACC>::run(x);
      constexpr int base = (j / NS) * NS * R + k;
      static_for<0, R>([&](auto RR) {
        constexpr int r = decltype(RR)::value;
        out[base + r * NS] = x[r];
      });
    });
    static_for<0, E>([&](auto I) { v[decltype(I)::value] = out[decltype(I)::value]; });
    reg_fft<E, DIR, ACC, NS * R>(v);
  }
}

template <int N> struct WarpPlan;
template <> struct WarpPlan<64> { static constexpr int E1 = 8, E2 = 8, L = 4; };
template <> struct WarpPlan<128> { static constexpr int E1 = 8, E2 = 16, L = 4; };
template <> struct WarpPlan<256> { static constexpr int E1 = 16, E2 = 16, L = 2; };
template <> struct WarpPlan<512> { static constexpr int E1 = 16, E2 = 32, L = 2; };
// N = 2^a 3: a radix-3 stage inside the E1-point register DFT
template <> struct WarpPlan<192> { static constexpr int E1 = 24, E2 = 8, L = 4; };
// (two lines a warp at 384: four hold 48 values a lane, 255 registers in the
// column pass and 8 warps an SM: row pass 0.50 us an angle against 0.39)
template <> struct WarpPlan<384> { static constexpr int E1 = 24, E2 = 16, L = 2; };
template <> struct WarpPlan<1024> { static constexpr int E1 = 32, E2 = 32, L = 1; };
// the remaining sizes: E2 even (the halves of a line then split at a whole
// register, see ColW) and as few idle lanes in the last slot as 32 values a
// lane allow.  Column + row pass, us per angle (360 angles; 230, 192, 160 at
// 640, 700, 768), these plans against the block-wide Stockham passes:
//   32: 0.048 / 0.069   48: 0.064 / 0.069    96: 0.095 / 0.185
//   160: 0.187 / 0.395  320: 0.63 / 1.77     640: 2.7 / 12.6
//   700: 4.1 / 9.7      768: 3.8 / 16.0      16: 0.045 / 0.047
template <> struct WarpPlan<16> { static constexpr int E1 = 4, E2 = 4, L = 8; };
template <> struct WarpPlan<32> { static constexpr int E1 = 4, E2 = 8, L = 8; };
template <> struct WarpPlan<48> { static constexpr int E1 = 8, E2 = 6, L = 4; };
template <> struct WarpPlan<96> { static constexpr int E1 = 12, E2 = 8, L = 4; };
template <> struct WarpPlan<160> { static constexpr int E1 = 20, E2 = 8, L = 4; };
template <> struct WarpPlan<320> { static constexpr int E1 = 20, E2 = 16, L = 2; };
template <> struct WarpPlan<640> { static constexpr int E1 = 20, E2 = 32, L = 1; };
template <> struct WarpPlan<700> { static constexpr int E1 = 25, E2 = 28, L = 1; };
template <> struct WarpPlan<768> { static constexpr int E1 = 24, E2 = 32, L = 1; };

template <int N> struct WP {
  static constexpr int E1 = WarpPlan<N>::E1, E2 = WarpPlan<N>::E2, L = WarpPlan<N>::L;
  static constexpr bool POW2 = (N & (N - 1)) == 0;
  static constexpr int NA = L * E2, NB = L * E1;  // step-A and step-B tasks of the warp
  static constexpr int TA = (NA + 31) / 32;       // step-A slots per lane
  static constexpr int TB = (NB + 31) / 32;       // step-B slots per lane
  static constexpr int TP = E2 + 1;       // odd pitch of the transpose tile
  static constexpr int AP = E1 + 1;       // step-A staging pitch (tensor-core path)
  static constexpr int T0 = (L * E1 * TP > L * N) ? L * E1 * TP : L * N;
  static constexpr int TSIZE = (L * E2 * AP > T0) ? L * E2 * AP : T0;  // float2 per warp
  static __device__ __forceinline__ bool a_on(int t) { return NA % 32 == 0 || t < NA; }
  static __device__ __forceinline__ bool b_on(int t) { return NB % 32 == 0 || t < NB; }
  static_assert(E1 * E2 == N && E2 % 2 == 0, "warp plan");
};

// step-A DFTs of every task of this warp through the tensor cores; a[][]
// goes through the warp tile T with pitch E1 + 1
template <int N, int PREC, int DIR>
__device__ __forceinline__ void tc_step_a(float2 (&a)[WP<N>::TA][WP<N>::E1], float2* T,
                                          const TcCtx& tc, int lane) {
  using P = WP<N>;
  static_for<0, P::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    static_for<0, P::E1>([&](auto MM) { T[t * P::AP + decltype(MM)::value] = a[i][decltype(MM)::value]; });
  });
  __syncwarp();
  for (int c = 0; c < P::TA; ++c)
    cta_tc_dft<P::E1, PREC>(T + c * 32 * P::AP, P::AP, tc, DIR < 0 ? 0 : 1, lane);
  static_for<0, P::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    static_for<0, P::E1>([&](auto MM) { a[i][decltype(MM)::value] = T[t * P::AP + decltype(MM)::value]; });
  });
  __syncwarp();
}

// A layout -> B layout (forward, unnormalised).  ACC: constants as pairs of
// floats, XACC: the cross twiddles too (their low parts at xtw + N): see
// WarpLines.
template <int N, int PREC = kPrecFP32, bool ACC = false, bool XACC = false>
__device__ __forceinline__ void warp_fft_fwd(float2 (&a)[WP<N>::TA][WP<N>::E1],
                                             float2 (&b)[WP<N>::TB][WP<N>::E2], float2* T,
                                             const float2* xtw, int lane,
                                             const TcCtx* tc = nullptr) {
  using P = WP<N>;
  if constexpr (PREC != kPrecFP32) tc_step_a<N, PREC, -1>(a, T, *tc, lane);
  if constexpr (PREC == kPrecFP32)
    static_for<0, P::TA>([&](auto II) { reg_fft<P::E1, -1, ACC>(a[decltype(II)::value]); });
  // cross twiddles: k1 outermost so tasks of a lane that share l share the load
  static_for<0, P::E1>([&](auto KK) {
    constexpr int k1 = decltype(KK)::value;
    float2 v[P::TA];
    static_for<0, P::TA>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int l = (lane + 32 * i) % P::E2;
      v[i] = a[i][k1];
      if constexpr (k1 > 0 && XACC) v[i] = cmul(v[i], xtw[k1 * P::E2 + l], xtw[N + k1 * P::E2 + l]);
      else if constexpr (k1 > 0) v[i] = cmul(v[i], xtw[k1 * P::E2 + l]);
    });
    static_for<0, P::TA>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int t = lane + 32 * i;
      const int line = t / P::E2, l = t % P::E2;
      if (P::a_on(t)) T[(line * P::E1 + k1) * P::TP + l] = v[i];
    });
  });
  __syncwarp();
  if constexpr (PREC != kPrecFP32) {
    // rows of T are the step-B tasks (line * E1 + k1 = t)
    for (int c = 0; c < P::TB; ++c)
      cta_tc_dft<P::E2, PREC>(T + c * 32 * P::TP, P::TP, *tc, 2, lane);
  }
  static_for<0, P::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const int line = t / P::E1, k1 = t % P::E1;
    if (P::b_on(t))
      static_for<0, P::E2>([&](auto LL) {
        constexpr int l = decltype(LL)::value;
        b[i][l] = T[(line * P::E1 + k1) * P::TP + l];
      });
    if constexpr (PREC == kPrecFP32) reg_fft<P::E2, -1, ACC>(b[i]);
  });
  __syncwarp();
}

// B layout -> A layout (inverse, unnormalised).  tile_free() runs when the
// warp has read its tile for the last time, before the step-A DFTs: a caller
// can start copies into the tile there (FP32 only).
struct NoHook {
  __device__ __forceinline__ void operator()() const {}
};
template <int N, int PREC = kPrecFP32, bool ACC = false, bool XACC = false, class Hook = NoHook>
__device__ __forceinline__ void warp_fft_inv(float2 (&b)[WP<N>::TB][WP<N>::E2],
                                             float2 (&a)[WP<N>::TA][WP<N>::E1], float2* T,
                                             const float2* xtw, int lane,
                                             const TcCtx* tc = nullptr, Hook&& tile_free = Hook{}) {
  using P = WP<N>;
  static_for<0, P::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    const int line = t / P::E1, k1 = t % P::E1;
    if constexpr (PREC == kPrecFP32) reg_fft<P::E2, +1, ACC>(b[i]);
    if (P::b_on(t))
      static_for<0, P::E2>([&](auto LL) {
        constexpr int l = decltype(LL)::value;
        T[(line * P::E1 + k1) * P::TP + l] = b[i][l];
      });
  });
  __syncwarp();
  if constexpr (PREC != kPrecFP32) {
    for (int c = 0; c < P::TB; ++c)
      cta_tc_dft<P::E2, PREC>(T + c * 32 * P::TP, P::TP, *tc, 3, lane);
  }
  static_for<0, P::E1>([&](auto KK) {
    constexpr int k1 = decltype(KK)::value;
    static_for<0, P::TA>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int t = lane + 32 * i;
      const int line = t / P::E2, l = t % P::E2;
      if (P::a_on(t)) a[i][k1] = T[(line * P::E1 + k1) * P::TP + l];
    });
    static_for<0, P::TA>([&](auto II) {
      constexpr int i = decltype(II)::value;
      const int l = (lane + 32 * i) % P::E2;
      if constexpr (k1 > 0 && XACC)
        a[i][k1] = cmul(a[i][k1], cconj(xtw[k1 * P::E2 + l]), cconj(xtw[N + k1 * P::E2 + l]));
      else if constexpr (k1 > 0) a[i][k1] = cmul(a[i][k1], cconj(xtw[k1 * P::E2 + l]));
    });
  });
  if constexpr (!std::is_same_v<std::decay_t<Hook>, NoHook>) {
    __syncwarp();
    tile_free();
  }
  if constexpr (PREC == kPrecFP32)
    static_for<0, P::TA>([&](auto II) { reg_fft<P::E1, +1, ACC>(a[decltype(II)::value]); });
  __syncwarp();
  if constexpr (PREC != kPrecFP32) tc_step_a<N, PREC, +1>(a, T, *tc, lane);
}

// The L-line plan of N as a line-transform policy: task t = lane + 32 i of
// a layout covers
//   A layout: line a_line(t), points a_x(t, m), m < E1;
//   B layout: line b_line(t), frequencies b_k(t, j), j < E2.
//
// Acc is the plan with accurate constants, for the refinement
// (refine_kernels.cuh), which runs a transform and its inverse over the same
// values hundreds of times, and, unless N is a power of two, for the assembly.
// The rounding of a constant (cos(pi/4) as a float is 1.7e-8 short) is the
// same in every pass and adds up in step; it was more than half of the
// refinement's error.  Where N has an odd factor, and so more terms and more
// twiddles, the XN cross twiddles in xs are pairs too; AccConst leaves them
// single, for the lines of the volume, where they cost more than they give.
// Error against 64 bits, plain / constants / with cross twiddles: refinement,
// N = 256, 180 angles, 50 iterations 8.1e-7 / 4.5e-7 / 3.7e-7 in 8.12 / 8.24 /
// 8.74 ms; N = 384, 90 angles, 10 iterations 4.7e-7 / 3.9e-7 / 3.5e-7 in 7.8 /
// 8.0 / 8.3 ms.
template <int N, bool ACC_ = false, bool XACC_ = ACC_ && !WP<N>::POW2> struct WarpLines {
  using P = WP<N>;
  static constexpr bool ACC = ACC_, XACC = XACC_;
  using Acc = WarpLines<N, true>;
  using AccConst = WarpLines<N, true, false>;
  static constexpr int XN = XACC ? 2 * N : N;
  static constexpr int L = P::L, TA = P::TA, E1 = P::E1, TB = P::TB, E2 = P::E2, TSIZE = P::TSIZE;
  // whether task t exists (else its registers hold nothing)
  static __device__ __forceinline__ bool a_on(int t) { return P::a_on(t); }
  static __device__ __forceinline__ bool b_on(int t) { return P::b_on(t); }
  static __device__ __forceinline__ int a_line(int t) { return t / E2; }
  static __device__ __forceinline__ int a_x(int t, int m) { return t % E2 + E2 * m; }
  static __device__ __forceinline__ int b_line(int t) { return t / E1; }
  static __device__ __forceinline__ int b_k(int t, int j) { return t % E1 + E1 * j; }
  static __device__ __forceinline__ void fwd(float2 (&a)[TA][E1], float2 (&b)[TB][E2], float2* T,
                                             const float2* xs, int lane) {
    warp_fft_fwd<N, kPrecFP32, ACC, XACC>(a, b, T, xs, lane);
  }
  template <class Hook = NoHook>
  static __device__ __forceinline__ void inv(float2 (&b)[TB][E2], float2 (&a)[TA][E1], float2* T,
                                             const float2* xs, int lane, Hook&& tile_free = Hook{}) {
    warp_fft_inv<N, kPrecFP32, ACC, XACC>(b, a, T, xs, lane, nullptr, tile_free);
  }
};
}  // namespace cpra
