// refine_kernels.cuh - line passes over volumes with the warp-resident FFTs of the
// two-pass warp engine, every supported N.
//
// Full complex volumes (the refinement's data set-up, the assembly's y lines):
//   k_xw  x rows: coalesced loads straight into the warp's A layout, FFT,
//         stores from the B layout;
//   k_vw  y or z lines: CB adjacent x columns staged through shared memory
//         (rows of CB * 8 bytes, estride apart), one column a warp or L.
//
// Refinement iterations (k_refine.cu has the method): rho is real, so the
// spectrum is kept as its half kx = 0 .. N/2, X[z][y][HP] (HP: N/2 columns,
// column N/2, padding to a whole block of columns), and every pass moves half
// of what complex volumes would.  X <- V on the measured cells followed by
// rho = Re IFFT(X) is, on the half spectrum, with the Hermitian part of the
// constrained spectrum, s = M(k) + M(-k) of 0, 1 or 2:
//   X <- (1 - s/2) G + W,  W = (M(k) V(k) + M(-k) conj V(-k)) / 2,
// and the error sums over k and -k together:
//   M(k)|G - V(k)|^2 + M(-k)|G - conj V(-k)|^2 = 2|G - W|^2 + K_k (s = 2),
//   |G - 2W|^2 (s = 1), K_k = |V(k) - conj V(-k)|^2 / 2,
// so W is built once with the sums of K_k and of |V|^2 (k_rdata, k_refine_w.cu).
//   k_rx  x rows in pairs (two real rows a complex line): rho on the
//         support-positivity set -> R2C -> X; X -> C2R -> rho; or both at
//         once between two iterations, rho never leaving the registers;
//   k_rv  y or z lines of X; the z pass stages W beside X and applies the
//         constraint between its forward and inverse transforms.
// Bound by HBM and, at N = 256, L2: 36 N^3 bytes an iteration, against
// (72 + 8 f) N^3 with complex volumes (f: measured fraction).  N = 256, 180
// angles: 254 us an iteration with complex volumes, 138 with plain constants (y
// lines 26 each, z lines with the data 56, x rows 30), 141 with their low parts
// (WarpLines::Acc), which more than halve the error.
#pragma once
#include "cpra_internal.h"
#include "fast_kernels.cuh"
#include "tiling.cuh"

namespace cpra {

template <int N> using XW = RowCfg<N, typename WLines<N, kPrecFP32>::type::Acc>;

// columns a block of the line passes: the column pass's, but 8 at N = 1024,
// so that the constraint's data fits beside them
template <int N> struct VW {
  using C = ColW<N, kPrecFP32>;
  using FL = typename C::FL::Acc;
  static constexpr int CB = N == 1024 ? 8 : C::CB;
  static constexpr int WARPS = CB / FL::L, NT = WARPS * 32;
  static constexpr int MINB = N == 1024 ? 1 : C::MINB;
  static constexpr int SP = CB + 1;
  static constexpr int STAGE = N * SP, TILES = WARPS * FL::TSIZE;
  static constexpr int BUF = STAGE > TILES ? STAGE : TILES;
  static constexpr int H = N / 2, HP = H + CB;  // row of the half spectrum
  static constexpr int RS = NT / CB, SR = (N + RS - 1) / RS;
  static_assert(N % CB == 0 && H % CB == 0 && NT % CB == 0 && HP % 2 == 0, "line staging");
};

template <int N>
constexpr size_t xw_smem() { return sizeof(float2) * (XW<N>::FL::XN + XW<N>::WARPS * XW<N>::FL::TSIZE); }
template <int N, class FL = typename VW<N>::FL>
constexpr size_t vw_smem() { return sizeof(float2) * (FL::XN + VW<N>::BUF); }
// the constraint pass also stages the data columns (same rows, same pitch)
template <int N>
constexpr size_t vw_smem_c() { return vw_smem<N>() + sizeof(float2) * VW<N>::STAGE; }

// thread to (row, column) of a block of columns: a warp's rows WARPS apart,
// so its 8-byte pieces fall on distinct banks of the odd-pitch staging rows
// (blocks whose columns do not divide a warp take plain thread order)
template <int N> struct VRows {
  using C = VW<N>;
  int y0, cc;
  __device__ VRows() {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    y0 = 32 % C::CB == 0 ? warp + C::WARPS * (lane / C::CB) : threadIdx.x / C::CB;
    cc = 32 % C::CB == 0 ? lane % C::CB : threadIdx.x % C::CB;
  }
  template <class F>
  __device__ __forceinline__ void each(F&& f) const {
#pragma unroll 4
    for (int k = 0; k < C::SR; ++k) {
      const int y = y0 + k * C::RS;
      if (N % C::RS != 0 && y >= N) break;
      f(y);
    }
  }
};

// staged columns -> registers and back (A or B layout)
template <int N, class FL>
__device__ __forceinline__ void take_a(float2 (&a)[FL::TA][FL::E1], const float2* buf, int col0, int lane) {
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::a_on(t)) return;
    const int col = col0 + FL::a_line(t);
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      a[i][m] = buf[FL::a_x(t, m) * VW<N>::SP + col];
    });
  });
}
// (with 1/N as a constant of FL's accuracy)
template <int N, class FL>
__device__ __forceinline__ void put_a(const float2 (&a)[FL::TA][FL::E1], float2* buf, int col0, int lane) {
  constexpr Const<FL::ACC && !WP<N>::POW2> inv(1.0 / N);
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::a_on(t)) return;
    const int col = col0 + FL::a_line(t);
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      buf[FL::a_x(t, m) * VW<N>::SP + col] = inv.mul(a[i][m]);
    });
  });
}
template <int N, class FL, class F>
__device__ __forceinline__ void each_bv(int lane, F&& f) {  // f(i, j, frequency, line)
  static_for<0, FL::TB>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::b_on(t)) return;
    static_for<0, FL::E2>([&](auto JJ) { f(II, JJ, FL::b_k(t, decltype(JJ)::value), FL::b_line(t)); });
  });
}

// ------------------------------------------------------------ full volumes
// x rows of X in place, forward: WARPS * L rows a CTA, L rows a warp
template <int N>
__global__ void __launch_bounds__(XW<N>::WARPS * 32, 3)
k_xw(float2* X, const float2* __restrict__ xtw, size_t rows) {
  using FL = typename XW<N>::FL;
  constexpr int WARPS = XW<N>::WARPS;
  extern __shared__ float2 smem[];
  float2* xs = smem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* T = smem + FL::XN + warp * FL::TSIZE;
  load_xtw<FL::XN>(xs, xtw, WARPS * 32);
  __syncthreads();
  const size_t row0 = ((size_t)blockIdx.x * WARPS + warp) * FL::L;
  if (row0 >= rows) return;  // L divides the rows
  float2 a[FL::TA][FL::E1], b[FL::TB][FL::E2];
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::a_on(t)) return;
    const float2* src = X + (row0 + FL::a_line(t)) * N;
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      a[i][m] = src[FL::a_x(t, m)];
    });
  });
  FL::fwd(a, b, T, xs, lane);
  each_bv<N, FL>(lane, [&](auto II, auto JJ, int k, int line) {
    X[(row0 + line) * N + k] = b[decltype(II)::value][decltype(JJ)::value];
  });
}

// CB adjacent x columns of one line set (blockIdx.y = z for y lines, = ky for
// z lines), N points estride apart, in place: forward, or inverse with 1/N
// (and a copy of the result, same layout, into out when that is not NULL)
template <int N, bool INV>
__global__ void __launch_bounds__(VW<N>::NT, VW<N>::MINB)
k_vw(float2* X, float2* out, const float2* __restrict__ xtw, size_t outer, size_t estride) {
  using C = VW<N>;
  using FL = std::conditional_t<INV, VolLines<N>, typename C::FL>;
  extern __shared__ float2 smem[];
  float2* xs = smem;
  float2* buf = smem + FL::XN;  // staging, then the warps' transpose tiles
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* base = X + blockIdx.y * outer + blockIdx.x * C::CB;
  const VRows<N> rows;
  rows.each([&](int y) { cp_async8(buf + y * C::SP + rows.cc, base + y * estride + rows.cc); });
  cp_async_commit();
  load_xtw<FL::XN>(xs, xtw, C::NT);
  cp_async_wait_all();
  __syncthreads();
  float2 a[FL::TA][FL::E1], b[FL::TB][FL::E2];
  const int col0 = warp * FL::L;
  if constexpr (INV)
    each_bv<N, FL>(lane, [&](auto II, auto JJ, int k, int line) {
      b[decltype(II)::value][decltype(JJ)::value] = buf[k * C::SP + col0 + line];
    });
  else
    take_a<N, FL>(a, buf, col0, lane);
  __syncthreads();
  float2* T = buf + warp * FL::TSIZE;
  if constexpr (INV) FL::inv(b, a, T, xs, lane);
  else FL::fwd(a, b, T, xs, lane);
  __syncthreads();  // every warp is done with its tile before staging
  if constexpr (INV)
    put_a<N, FL>(a, buf, col0, lane);
  else
    each_bv<N, FL>(lane, [&](auto II, auto JJ, int k, int line) {
      buf[k * C::SP + col0 + line] = b[decltype(II)::value][decltype(JJ)::value];
    });
  __syncthreads();
  float2* copy = INV && out ? out + (base - X) : nullptr;
  rows.each([&](int y) {
    const float2 v = buf[y * C::SP + rows.cc];
    base[y * estride + rows.cc] = v;
    if (INV && copy) copy[y * estride + rows.cc] = v;
  });
}

// ------------------------------------------------------------ half spectrum
// W and the constant sums from V in X (k_refine_w.cu); HP: row of W
cudaError_t launch_refine_w_data(const RefineArgs& a, int HP, cudaStream_t st);

enum { kRFwd = 0, kRInv = 1, kRBoth = 2 };

// Pairs of x rows of one plane, L pairs a warp.  kRFwd: rho on the
// support-positivity set, R2C, into X; kRInv: X, C2R, into R; kRBoth: X, C2R,
// the support-positivity set, R2C, back into X (the same floats as kRInv
// followed by kRFwd).
template <int N, int MODE>
__global__ void __launch_bounds__(XW<N>::WARPS * 32, 3)
k_rx(float2* X, float* R, const uint32_t* __restrict__ S3, const float2* __restrict__ xtw, int W) {
  using FL = typename XW<N>::FL;
  constexpr int WARPS = XW<N>::WARPS, H = N / 2, HP = VW<N>::HP;
  extern __shared__ float2 smem[];
  float2* xs = smem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float2* T = smem + FL::XN + warp * FL::TSIZE;
  const size_t row0 = 2 * (((size_t)blockIdx.x * WARPS + warp) * FL::L);  // first image row of the warp
  if constexpr (MODE != kRFwd) {
    // 2L spectrum rows of H values into the tile, 16 bytes a piece
    constexpr int PR = H / 2;
#pragma unroll
    for (int q = 0; q < (2 * FL::L * PR + 31) / 32; ++q) {
      const int p = lane + 32 * q;
      if ((2 * FL::L * PR) % 32 == 0 || p < 2 * FL::L * PR)
        cp_async16(T + 2 * p, X + (row0 + p / PR) * HP + 2 * (p % PR));
    }
    cp_async_commit();
  }
  load_xtw<FL::XN>(xs, xtw, WARPS * 32);
  if constexpr (MODE != kRFwd) cp_async_wait_all();
  __syncthreads();
  float2 a[FL::TA][FL::E1], b[FL::TB][FL::E2];
  if constexpr (MODE != kRFwd) {
    // Z = H(row 2p) + i H(row 2p+1); k = 0 and N/2 carry real parts only
    each_bv<N, FL>(lane, [&](auto II, auto JJ, int k, int line) {
      const float2* r0 = T + line * N;
      const float2* r1 = r0 + H;
      const bool up = k > H;
      const int c = up ? N - k : k;
      float2 z;
      if (k == H) {
        const float2* n0 = X + (row0 + 2 * line) * HP + H;
        z = make_float2(n0[0].x, n0[HP].x);
      } else {
        const float s = up ? -1.0f : 1.0f;
        const float2 h0 = r0[c], h1 = r1[c];
        z = make_float2(fmaf(-s, h1.y, h0.x), fmaf(s, h0.y, h1.x));
        if (k == 0) z = make_float2(h0.x, h1.x);
      }
      b[decltype(II)::value][decltype(JJ)::value] = z;
    });
    __syncwarp();  // the tile is the transforms' scratch from here on
    FL::inv(b, a, T, xs, lane);
  }
  constexpr Const<!WP<N>::POW2> inv(1.0 / N);
  static_for<0, FL::TA>([&](auto II) {
    constexpr int i = decltype(II)::value;
    const int t = lane + 32 * i;
    if (!FL::a_on(t)) return;
    const size_t row = row0 + 2 * FL::a_line(t);
    const uint32_t* s0 = S3 + row * W;
    static_for<0, FL::E1>([&](auto MM) {
      constexpr int m = decltype(MM)::value;
      const int x = FL::a_x(t, m);
      float v0, v1;
      if constexpr (MODE == kRFwd) {
        v0 = R[row * N + x];
        v1 = R[(row + 1) * N + x];
      } else {
        v0 = inv.mul(a[i][m].x);
        v1 = inv.mul(a[i][m].y);
      }
      if constexpr (MODE == kRInv) {
        R[row * N + x] = v0;
        R[(row + 1) * N + x] = v1;
      } else {
        const bool in0 = ((__ldg(s0 + (x >> 5)) >> (x & 31)) & 1u) && v0 >= 0.0f;
        const bool in1 = ((__ldg(s0 + W + (x >> 5)) >> (x & 31)) & 1u) && v1 >= 0.0f;
        a[i][m] = make_float2(in0 ? v0 : 0.0f, in1 ? v1 : 0.0f);
      }
    });
  });
  if constexpr (MODE != kRInv) {
    __syncwarp();
    FL::fwd(a, b, T, xs, lane);
    each_bv<N, FL>(lane, [&](auto II, auto JJ, int k, int line) {
      T[line * N + k] = b[decltype(II)::value][decltype(JJ)::value];
    });
    __syncwarp();
#pragma unroll
    for (int line = 0; line < FL::L; ++line) {
      const float2* Z = T + line * N;
      float2* r0 = X + (row0 + 2 * line) * HP;
      float2* r1 = r0 + HP;
#pragma unroll
      for (int kk = 0; kk < (H + 31) / 32; ++kk) {
        const int k = lane + 32 * kk;
        if (H % 32 != 0 && k >= H) break;
        const float2 z = Z[k], zm = Z[k == 0 ? 0 : N - k];
        r0[k] = make_float2(0.5f * (z.x + zm.x), 0.5f * (z.y - zm.y));
        r1[k] = make_float2(0.5f * (z.y + zm.y), 0.5f * (zm.x - z.x));
      }
      if (lane == 0) {
        const float2 zn = Z[H];
        r0[H] = make_float2(zn.x, 0.0f);
        r1[H] = make_float2(zn.y, 0.0f);
      }
    }
  }
}

enum { kLFwd = 0, kLInv = 1, kLConstrain = 2 };

// CB columns of the half spectrum (the last block holds column N/2 alone),
// N points estride apart: forward, inverse with 1/N, or (z lines) forward,
// data constraint with the error terms, inverse
template <int N, int MODE>
__global__ void __launch_bounds__(VW<N>::NT, VW<N>::MINB)
k_rv(float2* X, const float2* __restrict__ Wd, const uint8_t* __restrict__ M, const float2* __restrict__ xtw,
     const double* __restrict__ konst, double* err2, size_t outer, size_t estride) {
  using C = VW<N>;
  using FL = typename C::FL;
  constexpr int H = C::H;
  extern __shared__ float2 smem[];
  __shared__ double red[32];
  __shared__ uint8_t sc[C::CB];  // M(k) + M(-k) of the block's columns
  float2* xs = smem;
  float2* buf = smem + FL::XN;
  float2* wbuf = buf + C::BUF;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c0 = blockIdx.x * C::CB;
  const int nc = c0 == H ? 1 : C::CB;
  float2* base = X + blockIdx.y * outer + c0;
  const VRows<N> rows;
  if (rows.cc < nc) {
    bool data = false;
    if constexpr (MODE == kLConstrain) {
      const int ky = blockIdx.y, c = c0 + rows.cc;
      const int s = (M[ky * N + c] != 0) + (M[((N - ky) % N) * N + (N - c) % N] != 0);
      data = s > 0;
      if (rows.y0 == 0) sc[rows.cc] = (uint8_t)s;
    }
    rows.each([&](int y) {
      cp_async8(buf + y * C::SP + rows.cc, base + y * estride + rows.cc);
      if constexpr (MODE == kLConstrain)
        if (data) cp_async8(wbuf + y * C::SP + rows.cc, Wd + blockIdx.y * outer + c0 + y * estride + rows.cc);
    });
  }
  cp_async_commit();
  load_xtw<FL::XN>(xs, xtw, C::NT);
  cp_async_wait_all();
  __syncthreads();
  float2 a[FL::TA][FL::E1], b[FL::TB][FL::E2];
  const int col0 = warp * FL::L;
  const bool mine = col0 < nc;  // the warp has a column
  if (mine) {
    if constexpr (MODE == kLInv)
      each_bv<N, FL>(lane, [&](auto II, auto JJ, int k, int line) {
        b[decltype(II)::value][decltype(JJ)::value] = buf[k * C::SP + col0 + line];
      });
    else
      take_a<N, FL>(a, buf, col0, lane);
  }
  __syncthreads();
  float2* T = buf + warp * FL::TSIZE;
  float ef = 0.0f;  // this thread's at most a few dozen terms; FP64 across threads
  if (mine) {
    if constexpr (MODE != kLInv) FL::fwd(a, b, T, xs, lane);
    if constexpr (MODE == kLConstrain) {
      each_bv<N, FL>(lane, [&](auto II, auto JJ, int k, int line) {
        const int col = col0 + line;
        if (col >= nc) return;
        const int s = sc[col], c = c0 + col;
        if (s == 0) return;
        float2& g = b[decltype(II)::value][decltype(JJ)::value];
        const float2 w = wbuf[k * C::SP + col];
        const float wt = (c == 0 || c == H) ? 0.5f : 1.0f;
        if (s == 2) {
          const float dx = g.x - w.x, dy = g.y - w.y;
          ef = fmaf(2.0f * wt, fmaf(dx, dx, dy * dy), ef);
          g = w;
        } else {
          const float dx = fmaf(-2.0f, w.x, g.x), dy = fmaf(-2.0f, w.y, g.y);
          ef = fmaf(wt, fmaf(dx, dx, dy * dy), ef);
          g = make_float2(fmaf(0.5f, g.x, w.x), fmaf(0.5f, g.y, w.y));
        }
      });
    }
    if constexpr (MODE == kLConstrain) {  // the warp's error terms, while other warps transform
      const double e = warp_sum(ef, 0.0f);
      if (lane == 0) red[warp] = e;
    }
    if constexpr (MODE != kLFwd) {
      if constexpr (MODE == kLConstrain) __syncwarp();
      FL::inv(b, a, T, xs, lane);
    }
  }
  __syncthreads();
  if (mine) {
    if constexpr (MODE == kLFwd)
      each_bv<N, FL>(lane, [&](auto II, auto JJ, int k, int line) {
        buf[k * C::SP + col0 + line] = b[decltype(II)::value][decltype(JJ)::value];
      });
    else
      put_a<N, FL>(a, buf, col0, lane);
  }
  __syncthreads();
  if (rows.cc < nc) rows.each([&](int y) { base[y * estride + rows.cc] = buf[y * C::SP + rows.cc]; });
  if constexpr (MODE == kLConstrain) {
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int w = 0; w < C::WARPS && w * FL::L < nc; ++w) s += red[w];
      if (blockIdx.x == 0 && blockIdx.y == 0) {
        s += konst[0];
        err2[1] = konst[1];
      }
      atomicAdd(err2, s);
    }
  }
}

// ------------------------------------------------------------ launchers
template <int N>
cudaError_t refine_w_attrs() {
  cudaError_t e = smem_attr(k_xw<N>, xw_smem<N>());
  if (e == cudaSuccess) e = smem_attr(k_vw<N, false>, vw_smem<N>());
  if (e == cudaSuccess) e = smem_attr(k_rx<N, kRFwd>, xw_smem<N>());
  if (e == cudaSuccess) e = smem_attr(k_rx<N, kRInv>, xw_smem<N>());
  if (e == cudaSuccess) e = smem_attr(k_rx<N, kRBoth>, xw_smem<N>());
  if (e == cudaSuccess) e = smem_attr(k_rv<N, kLFwd>, vw_smem<N>());
  if (e == cudaSuccess) e = smem_attr(k_rv<N, kLInv>, vw_smem<N>());
  if (e == cudaSuccess) e = smem_attr(k_rv<N, kLConstrain>, vw_smem_c<N>());
  return e;
}

template <int N>
cudaError_t refine_w_prepare() {
  static PerDevice<bool> done;
  return once_on_device(done, refine_w_attrs<N>);
}

// V = FFT3(X) in place (X: the data volume), then W and the constant sums
template <int N>
cudaError_t data_w(const RefineArgs& a, cudaStream_t st) {
  cudaError_t e = refine_w_prepare<N>();
  if (e != cudaSuccess) return e;
  using C = VW<N>;
  const size_t NN = (size_t)N * N;
  constexpr int rows = XW<N>::WARPS * XW<N>::FL::L;
  const dim3 grid(N / C::CB, N);
  g_launches += 3;
  k_xw<N><<<(unsigned)((NN + rows - 1) / rows), XW<N>::WARPS * 32, xw_smem<N>(), st>>>(a.X, a.xtw, NN);
  k_vw<N, false><<<grid, C::NT, vw_smem<N>(), st>>>(a.X, nullptr, a.xtw, NN, (size_t)N);
  k_vw<N, false><<<grid, C::NT, vw_smem<N>(), st>>>(a.X, nullptr, a.xtw, (size_t)N, NN);
  e = cudaGetLastError();
  return e == cudaSuccess ? launch_refine_w_data(a, C::HP, st) : e;
}

template <int N, int MODE>
void rx(const RefineArgs& a, cudaStream_t st) {
  constexpr int pairs = XW<N>::WARPS * XW<N>::FL::L;
  static_assert((N / 2) % pairs == 0, "row pairs of a plane fill whole CTAs");
  g_launches += 1;
  k_rx<N, MODE><<<(unsigned)((size_t)N * (N / 2) / pairs), XW<N>::WARPS * 32, xw_smem<N>(), st>>>(
      a.X, a.R, a.S3, a.xtw, a.W);
}

template <int N, int MODE>
void rv(const RefineArgs& a, double* err2, cudaStream_t st) {
  using C = VW<N>;
  constexpr size_t line = C::HP, plane = (size_t)N * C::HP;
  constexpr bool along_z = MODE == kLConstrain;
  constexpr size_t smem = MODE == kLConstrain ? vw_smem_c<N>() : vw_smem<N>();
  g_launches += 1;
  k_rv<N, MODE><<<dim3(C::H / C::CB + 1, N), C::NT, smem, st>>>(
      a.X, a.Wd, a.M, a.xtw, a.konst, err2, along_z ? line : plane, along_z ? plane : line);
}

template <int N>
cudaError_t iter_w(const RefineArgs& a, double* err2, bool first, bool last, cudaStream_t st) {
  if (first) rx<N, kRFwd>(a, st);
  rv<N, kLFwd>(a, nullptr, st);
  rv<N, kLConstrain>(a, err2, st);
  rv<N, kLInv>(a, nullptr, st);
  if (last) rx<N, kRInv>(a, st);
  else rx<N, kRBoth>(a, st);
  return cudaGetLastError();
}

template <int N>
cudaError_t volume_ylines_n(float2* vol, float2* out, const float2* xtw, cudaStream_t st) {
  using C = VW<N>;
  static PerDevice<bool> attr;
  const cudaError_t e = smem_once(k_vw<N, true>, vw_smem<N, VolLines<N>>(), attr);
  if (e != cudaSuccess) return e;
  g_launches += 1;
  k_vw<N, true><<<dim3(N / C::CB, N), C::NT, vw_smem<N, VolLines<N>>(), st>>>(vol, out, xtw, (size_t)N * N, (size_t)N);
  return cudaGetLastError();
}

// The instances of one N, compiled in the translation unit that names them
// (k_refine_*.cu) and only declared elsewhere.
#define CPRA_REFINE_INSTANCES(NN, EXTERN)                                                                     \
  EXTERN template cudaError_t data_w<NN>(const RefineArgs&, cudaStream_t);                                   \
  EXTERN template cudaError_t iter_w<NN>(const RefineArgs&, double*, bool, bool, cudaStream_t);              \
  EXTERN template cudaError_t volume_ylines_n<NN>(float2*, float2*, const float2*, cudaStream_t);

}  // namespace cpra
