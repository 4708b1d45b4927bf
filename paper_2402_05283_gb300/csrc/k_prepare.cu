// k_prepare.cu - input preparation (Eq. 1-3), support, seeded start, exports.
#include "cpra_internal.h"
#include "fft.cuh"

namespace cpra {

std::atomic<long long> g_launches{0};

// Amplitudes of every loaded angle, FFT order.  A(k) = sqrt(I) at the centred
// index of k; A_sym(k) = (A(k) + A(-k)) / 2 on the half plane kx <= N/2,
// stored column-major (A_main[n][kx][ky], A_nyq[n][ky] for kx = N/2); the
// full-plane sums of ((A(k) - A(-k))/2)^2 and A(k)^2 go to Cn and sumA2.
// With a measured-pixel mask (centred, nonzero = measured; per angle when
// mask_stride is N*N, one for all when 0) only the pairs {k, -k} with both
// pixels measured are constrained: the others get A_sym = -1 (the modulus
// projection leaves them free) and stay out of Cn and sumA2.
//
// A CTA takes a 32 x 32 tile of the half plane with its partners -k, so each
// intensity is read and rooted once, and the tile leaves transposed through
// shared memory.  Each thread sums its terms in FP32 (at most ten), the
// warp FP32 pairs (48 bits), FP64 across warps and CTAs; a warp whose sums
// leave FP32's range takes FP64.  Bound by HBM and
// the square roots.  N = 512, 360 angles: a warp a row over the full plane and
// a transpose pass after it 443 + 143 us, this kernel 296 us.
//
// An invalid pattern (a negative or non-finite intensity) marks bad[n] and
// makes C_n NaN, so the first iteration on it publishes a non-finite error
// and flags the plan's status word: the load itself does not wait for the
// device.
__global__ void __launch_bounds__(256) k_prepare(const float* __restrict__ I, int N, int first, float* A_main,
                                                 float* A_nyq, double* Cn, double* sumA2, uint8_t* bad_angle,
                                                 const uint8_t* __restrict__ mask, size_t mask_stride) {
  __shared__ float tile[32][33];
  __shared__ double sc[8], sa[8];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int h = N / 2, kx0 = blockIdx.x * 32, ky0 = blockIdx.y * 32;
  const int n = first + blockIdx.z;
  const float* In = I + (size_t)blockIdx.z * N * N;
  const uint8_t* Mn = mask ? mask + (size_t)n * mask_stride : nullptr;
  float cf = 0.0f, af = 0.0f;
  int bad = 0;
  // the pair {(ky, kx), (-ky, -kx)}, 0 <= kx <= h: its terms to add(half the
  // difference, A(k), A(-k) or 0, how often); returns A_sym
  auto pair = [&](int ky, int kx, auto&& add) {
    const int ry = ky < h ? ky + h : ky - h;               // centred row of +ky
    const int my = ky <= h ? h - ky : N + h - ky;           // centred row of -ky
    const int rx = kx < h ? kx + h : 0, mx = h - kx;        // centred columns of +kx and -kx
    const size_t p = (size_t)ry * N + rx, q = (size_t)my * N + mx;
    const float ip = __ldg(In + p), im = __ldg(In + q);
    if (!(ip >= 0.0f) || !isfinite(ip) || !(im >= 0.0f) || !isfinite(im)) bad = 1;
    if (Mn && !(Mn[p] && Mn[q])) return -1.0f;
    const float ap = sqrtf(fmaxf(ip, 0.0f)), am = sqrtf(fmaxf(im, 0.0f));
    const float d = 0.5f * (ap - am);
    // in the columns 0 and N/2 the partner is in the same column and has its own turn
    if (kx == 0 || kx == h) add(d, ap, 0.0f, 1.0f);
    else add(d, ap, am, 2.0f);
    return 0.5f * (ap + am);
  };
  auto all = [&](auto&& add) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int ky = ky0 + ty + 8 * j, kx = kx0 + tx;
      if (ky < N && kx < h) tile[ty + 8 * j][tx] = pair(ky, kx, add);
    }
    if (kx0 == 0 && ty == 0 && ky0 + tx < N) A_nyq[(size_t)n * N + ky0 + tx] = pair(ky0 + tx, h, add);
  };
  all([&](float d, float ap, float am, float w) {
    cf = fmaf(w * d, d, cf);
    af = fmaf(ap, ap, fmaf(am, am, af));
  });
  double c_part, a_part;
  if (__all_sync(0xffffffffu, isfinite(cf) && isfinite(af))) {
    c_part = warp_sum(cf, 0.0f);
    a_part = warp_sum(af, 0.0f);
  } else {  // beyond FP32: the terms again in FP64
    c_part = a_part = 0.0;
    all([&](float d, float ap, float am, float w) {
      c_part += (double)w * d * d;
      a_part += (double)ap * ap + (double)am * am;
    });
    c_part = warp_sum(c_part);
    a_part = warp_sum(a_part);
  }
  if (tx == 0) { sc[ty] = c_part; sa[ty] = a_part; }
  const int block_bad = __syncthreads_or(bad);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int kx = kx0 + ty + 8 * j, ky = ky0 + tx;
    if (ky < N && kx < h) A_main[((size_t)n * h + kx) * N + ky] = tile[tx][ty + 8 * j];
  }
  if (threadIdx.x == 0) {
    double c = 0.0, a = 0.0;
    for (int i = 0; i < 8; ++i) { c += sc[i]; a += sa[i]; }
    if (block_bad) {
      c = __longlong_as_double(0x7ff8000000000000ll);  // NaN
      bad_angle[n] = 1;
    }
    atomicAdd(Cn + n, c);
    atomicAdd(sumA2 + n, a);
  }
}

cudaError_t launch_prepare(cpra_plan_s* p, const float* I, int first, int count) {
  cudaError_t e = cudaMemsetAsync(p->Cn + first, 0, sizeof(double) * count, p->stream);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(p->sumA2 + first, 0, sizeof(double) * count, p->stream);
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(p->bad + first, 0, count, p->stream);
  if (e != cudaSuccess) return e;
  const int h = p->N / 2;
  g_launches += 1;
  k_prepare<<<dim3((h + 31) / 32, (p->N + 31) / 32, count), 256, 0, p->stream>>>(
      I, p->N, first, p->A_main, p->A_nyq, p->Cn, p->sumA2, p->bad, p->mask,
      p->mask_per_angle ? (size_t)p->N * p->N : 0);
  return cudaGetLastError();
}

// Support bits from the padded bounding box [N/4, 3N/4)^2 (or from bytes).
__global__ void k_support(uint32_t* S, int N, int W, const uint8_t* src, int per_angle) {
  const int y = blockIdx.x, n = blockIdx.y;
  for (int w = threadIdx.x; w < W; w += blockDim.x) {
    uint32_t bits = 0;
    for (int b = 0; b < 32; ++b) {
      const int x = w * 32 + b;
      if (x >= N) break;
      bool in;
      if (src) {
        const size_t off = (per_angle ? (size_t)n * N * N : 0) + (size_t)y * N + x;
        in = src[off] != 0;
      } else {
        in = (y >= N / 4) && (y < N / 4 + N / 2) && (x >= N / 4) && (x < N / 4 + N / 2);
      }
      if (in) bits |= 1u << b;
    }
    S[((size_t)n * N + y) * W + w] = bits;
  }
}

cudaError_t launch_support_box(cpra_plan_s* p) {
  g_launches += 1;
  k_support<<<dim3(p->N, p->Np), 32, 0, p->stream>>>(p->S, p->N, p->W, nullptr, 0);
  return cudaGetLastError();
}

cudaError_t launch_support_u8(cpra_plan_s* p, const uint8_t* S, int per_angle) {
  g_launches += 1;
  k_support<<<dim3(p->N, p->Np), 32, 0, p->stream>>>(p->S, p->N, p->W, S, per_angle);
  return cudaGetLastError();
}

// Seeded start g0 = u * [x in S], u = (splitmix64(key) >> 40) * 2^-24,
// key = ((seed * Np + n) * N + y) * N + x (mod 2^64).
// the seeded start into both Jacobi buffers (angles outside a present mask
// keep it whichever buffer is current)
__global__ void k_init_guess(float* g, float* g2, const uint32_t* S, int N, int Np, int W,
                             unsigned long long seed) {
  const int y = blockIdx.x, n = blockIdx.y;
  const size_t srow = ((size_t)n * N + y) * W;
  for (int x = threadIdx.x; x < N; x += blockDim.x) {
    const uint64_t key = ((seed * (uint64_t)Np + (uint64_t)n) * (uint64_t)N + (uint64_t)y) *
                             (uint64_t)N + (uint64_t)x;
    const float u = (float)(splitmix64(key) >> 40) * (1.0f / 16777216.0f);
    const float v = sbit(S, srow, x) ? u : 0.0f;
    g[((size_t)n * N + y) * N + x] = v;
    g2[((size_t)n * N + y) * N + x] = v;
  }
}

cudaError_t launch_init_guess(cpra_plan_s* p) {
  int threads = p->N >= 256 ? 256 : p->N;
  g_launches += 1;
  k_init_guess<<<dim3(p->N, p->Np), threads, 0, p->stream>>>(p->g, p->g_alt, p->S, p->N, p->Np,
                                                             p->W, (unsigned long long)p->cfg.seed);
  return cudaGetLastError();
}

// Raw-pointer forms of the two support conversions (count patterns).
cudaError_t launch_bits_from_u8(uint32_t* bits, const uint8_t* src, int N, int count,
                                cudaStream_t st) {
  g_launches += 1;
  k_support<<<dim3(N, count), 32, 0, st>>>(bits, N, (N + 31) / 32, src, 1);
  return cudaGetLastError();
}

__global__ void k_export_po(const float* g, const uint32_t* S, float* out, int N, int W) {
  const int y = blockIdx.x, n = blockIdx.y;
  const size_t srow = ((size_t)n * N + y) * W;
  for (int x = threadIdx.x; x < N; x += blockDim.x) {
    const size_t i = ((size_t)n * N + y) * N + x;
    const float v = g[i];
    out[i] = (sbit(S, srow, x) && v >= 0.0f) ? v : 0.0f;
  }
}

cudaError_t launch_export_po(cpra_plan_s* p, float* out) {
  int threads = p->N >= 256 ? 256 : p->N;
  g_launches += 1;
  k_export_po<<<dim3(p->N, p->Np), threads, 0, p->stream>>>(p->g, p->S, out, p->N, p->W);
  return cudaGetLastError();
}

__global__ void k_export_support(const uint32_t* S, uint8_t* out, int N, int W) {
  const int y = blockIdx.x, n = blockIdx.y;
  const size_t srow = ((size_t)n * N + y) * W;
  for (int x = threadIdx.x; x < N; x += blockDim.x)
    out[((size_t)n * N + y) * N + x] = sbit(S, srow, x) ? 1 : 0;
}

cudaError_t launch_export_support(cpra_plan_s* p, uint8_t* out) {
  int threads = p->N >= 256 ? 256 : p->N;
  g_launches += 1;
  k_export_support<<<dim3(p->N, p->Np), threads, 0, p->stream>>>(p->S, out, p->N, p->W);
  return cudaGetLastError();
}

cudaError_t launch_bits_to_u8(const uint32_t* bits, uint8_t* out, int N, int count,
                              cudaStream_t st) {
  const int threads = N >= 256 ? 256 : N;
  g_launches += 1;
  k_export_support<<<dim3(N, count), threads, 0, st>>>(bits, out, N, (N + 31) / 32);
  return cudaGetLastError();
}

}  // namespace cpra
