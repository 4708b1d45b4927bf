// k_assemble.cu - Step C mass-centre move and merge, Step D assembly.
//
//   moments  FP64 sums of rho = P_{S+} g, rho*z, rho*u per angle
//   ramps    exp(+2 pi i k c / N) of the mass-centre move, per angle along z
//            and u (signed k)
//   spectra  E_n(kz, ku) = DFT2(rho_n) * ramps, then the inverse DFT along kz
//            of the columns ku = 0 .. N/2: F[z / 8][n][ku][z % 8] (z stored
//            fftshifted).  rho is real, so the columns ku < 0 follow:
//            F(-ku, z) = conj F(ku, z) + corr(n, ku) (-1)^z, where corr is
//            what the one row without a partner, kz = -N/2, leaves.  The R2C
//            rows come from the row-pass kernel; this kernel does the columns.
//   grid     a row ky of eight planes or more: V = sum_e w_e F[idx_e][z] over
//            the row's cells, into shared memory, then the inverse FFT along
//            kx, stored as a row of the volume.  The cell lists (bilinear
//            adjoint weights of every sample, normalised by their sum, FP64,
//            rounded once) are built on the host; the sign (-1)^(kx+ky) makes
//            the inverse transform land centred in x and y.
//   y lines  inverse FFT along ky in place (refine_kernels.cuh).
// Step C merge of several guesses (cpra_merge): the spectra kernel stores the
// best guess's E of one PO (REF) and tells for the other guesses whether their
// E or conj E, the spectrum of the centrally inverted PO, is the nearer to it
// (DIST); k_merge then takes a block of columns through all kept
// guesses: mean of E or conj(E), ring sums of |sum E'| / sum |E'| for the
// PRTF, and the inverse DFT along kz of the mean into F.
// The inverse 3D DFT is applied as IDFT_z on each slice before gridding
// (gridding acts on kx, ky only and its weights do not depend on kz), then
// IDFT_xy on each z plane after gridding.
#include "assemble_kernels.cuh"

namespace cpra {

#define CPRA_CASE(NN) CPRA_ASSEMBLE_INSTANCES(NN, extern)
CPRA_FOR_EACH_N(CPRA_CASE)
#undef CPRA_CASE

// ---------------------------------------------------------------- moments
// The moments apart from the rows of rho, for the prime kernels that do not
// take them along and for the refinement.
// One warp per kMomRows rows: each lane sums its pixels of a row in FP32 (at
// most N/32 terms) and its rows as pairs of FP32 (48 bits, with the exact
// products by y; FP64 where that leaves FP32's range); FP64 across warps and
// CTAs.  Bound by HBM: the FP64
// pipe is narrow, and ten FP64 shuffles and adds a row made it the bound
// (N = 256, 144 angles: 44 us, 33 with one reduction of FP32 pairs per 16 rows).
constexpr int kMomRows = 16;
__global__ void k_moments(const float* __restrict__ g, const uint32_t* __restrict__ S,
                          double* moments, int N, int W) {
  __shared__ double red[3][8];
  const int n = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int y0 = (blockIdx.x * (blockDim.x >> 5) + warp) * kMomRows;
  auto rows = [&](auto&& f) {
#pragma unroll 4
    for (int r = 0; r < kMomRows; ++r) {
      const int y = y0 + r;
      if (y >= N) break;
      const float* gy = g + ((size_t)n * N + y) * N;
      const uint32_t* sy = S + ((size_t)n * N + y) * W;
      float p0 = 0.0f, pu = 0.0f;
      for (int x = lane, w = 0; x < N; x += 32, ++w) {
        const float v = gy[x];
        const float q = ((sy[w] >> lane) & 1u) && v >= 0.0f ? v : 0.0f;
        p0 += q;
        pu = fmaf(q, (float)x, pu);
      }
      f(p0, pu, (float)y);
    }
  };
  Moments mom;
  rows([&](float p, float pu, float y) { mom.add(p, pu, y); });
  double m[3];
  if (mom.in_range()) {
    mom.total(m);
  } else {
    double d[3] = {0.0, 0.0, 0.0};
    rows([&](float p, float pu, float y) { add_moments(d, p, pu, y); });
    for (int q = 0; q < 3; ++q) m[q] = warp_sum(d[q]);
  }
  if (lane == 0)
    for (int q = 0; q < 3; ++q) red[q][warp] = m[q];
  __syncthreads();
  if (threadIdx.x < 3) {
    double a = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) a += red[threadIdx.x][i];
    atomicAdd(moments + 3 * n + threadIdx.x, a);
  }
}

// ---------------------------------------------------------------- ramps
// exp(2 pi i turns), the argument reduced to [-1/2, 1/2) turns, FP64
__device__ __forceinline__ double2 unit_phase(double turns) {
  const double r = turns - rint(turns);
  double s, c;
  sincospi(2.0 * r, &s, &c);
  return make_double2(c, s);
}

// Per angle the unit ramps of the mass-centre move (ramp_len).
// k = 32 a + b as the product of two of about N/32 + 32 FP64 phases (the
// FP64 pipe is narrow, and a sine and cosine of every entry in every column
// block were half of the old spectra kernel's time).
__global__ void k_ramps(const double* __restrict__ moments, float2* ramps, int N, int com_align) {
  __shared__ double2 hi[2][17], lo[2][32];
  const int n = blockIdx.x, H = N / 2;
  const double m0 = moments[3 * n];
  double c[2] = {0.5 * N, 0.5 * N};
  if (com_align && m0 > 0.0) {
    c[0] = moments[3 * n + 1] / m0;
    c[1] = moments[3 * n + 2] / m0;
  }
  for (int i = threadIdx.x; i < 2 * 49; i += blockDim.x) {
    const int d = i / 49, q = i - d * 49;
    if (q < 17) hi[d][q] = unit_phase(32.0 * q * c[d] / N);
    else lo[d][q - 17] = unit_phase((q - 17) * c[d] / N);
  }
  __syncthreads();
  float2* rz = ramps + (size_t)n * ramp_len(N);
  float2* ru = rz + N;
  for (int i = threadIdx.x; i < 2 * (H + 1); i += blockDim.x) {
    const int d = i / (H + 1), k = i - d * (H + 1);
    const double2 a = hi[d][k >> 5], b = lo[d][k & 31];
    const float2 w = make_float2((float)(a.x * b.x - a.y * b.y), (float)(a.x * b.y + a.y * b.x));
    if (d == 0) {
      if (k < H) rz[k] = w;
      if (k > 0) rz[N - k] = cconj(w);  // k = H: the row -N/2
    } else {
      ru[k] = k < H ? w : cconj(w);
    }
  }
}

// Q[cell] = sum of w corr over the cell's samples of ku < 0 (see k_spectra): the
// same for every plane but for (-1)^z, so it is summed once and not in every
// chunk of planes.  A warp a cell; the origin's list is thousands long.
__global__ void __launch_bounds__(256) k_grid_corr(const float2* __restrict__ corr,
                                                   const int32_t* __restrict__ cell_ptr,
                                                   const GridEnt* __restrict__ ents, float2* Q, int NN) {
  const int cell = (blockIdx.x * 256 + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (cell >= NN) return;
  const int e0 = cell_ptr[cell], e1 = cell_ptr[cell + 1];
  float2 s = make_float2(0.0f, 0.0f);
  for (int e = e0 + lane; e < e1; e += 32) {
    const GridEnt g = ents[e];
    if (g.at >> 31) {
      const float2 c = __ldg(corr + (g.at & 0x7fffffffu));
      s.x = fmaf(g.w, c.x, s.x);
      s.y = fmaf(g.w, c.y, s.y);
    }
  }
  if (e1 > e0) {  // the whole warp
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
      s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
  }
  if (lane == 0) Q[cell] = s;
}

cudaError_t launch_grid_corr(cpra_plan_s* p) {
  const Assembly& a = p->asmb;
  const int NN = p->N * p->N;
  g_launches += 1;
  k_grid_corr<<<(NN + 7) / 8, 256, 0, p->stream>>>(a.corr, a.cell_ptr, a.ents, a.Q, NN);
  return cudaGetLastError();
}

// PRTF = ring mean (float), from the ring sums and the ring populations
__global__ void k_prtf(const unsigned long long* __restrict__ rings, const unsigned* __restrict__ counts, float* prtf,
                       int H, int total) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  const unsigned c = counts[i % H];
  const unsigned long long s = rings[i];
  prtf[i] = s >= kRingNaN ? __int_as_float(0x7fc00000) : c ? (float)((double)s * kRingUnit / (double)c) : 0.0f;
}

// ------------------------------------------------------------------ launchers
size_t ramps_bytes(int N, int Np) { return sizeof(float2) * ramp_len(N) * (size_t)Np; }
size_t corr_bytes(int N, int Np) { return sizeof(float2) * (N / 2 + 1) * (size_t)Np; }
size_t spectra_bytes(int N, int Np) {
  return sizeof(float2) * 8 * (size_t)((N + 7) / 8) * Np * (N / 2 + 1);
}

cudaError_t launch_prtf(const unsigned long long* rings, const unsigned* counts, float* prtf, int H, int total,
                        cudaStream_t st) {
  g_launches += 1;
  k_prtf<<<(total + 255) / 256, 256, 0, st>>>(rings, counts, prtf, H, total);
  return cudaGetLastError();
}

// moments of rho = P_{S+} g of every angle of p into `moments`
cudaError_t launch_moments(cpra_plan_s* p, double* moments, cudaStream_t st) {
  const int N = p->N, Np = p->Np;
  cudaError_t e = cudaMemsetAsync(moments, 0, sizeof(double) * 3 * Np, st);
  if (e != cudaSuccess) return e;
  g_launches += 1;
  const int warps = (N + kMomRows - 1) / kMomRows, wpb = warps < 8 ? warps : 8;
  k_moments<<<dim3((warps + wpb - 1) / wpb, Np), 32 * wpb, 0, st>>>(p->g, p->S, moments, N, p->W);
  return cudaGetLastError();
}

cudaError_t launch_rho_rows(cpra_plan_s* p, const Launch& L, double* moments, float2* ramps) {
  cudaStream_t st = p->stream;
  cudaError_t e;
  if (L.prec == CPRA_FP32 && L.engine != CPRA_ENGINE_TWO_PASS) {
    e = cudaMemsetAsync(moments, 0, sizeof(double) * 3 * p->Np, st);
    if (e == cudaSuccess) e = launch_prime_fast(L, moments);
  } else {
    e = launch_prime(L);
    if (e == cudaSuccess) e = launch_moments(p, moments, st);
  }
  if (e != cudaSuccess) return e;
  g_launches += 1;
  k_ramps<<<p->Np, 128, 0, st>>>(moments, ramps, p->N, p->cfg.com_align);
  return cudaGetLastError();
}

cudaError_t launch_assemble(cpra_plan_s* p, float2* out) {
#define CPRA_CASE(NN) \
  case NN: return assemble_n<NN>(p, out);
  switch (p->N) { CPRA_FOR_EACH_N(CPRA_CASE) default: return cudaErrorInvalidValue; }
#undef CPRA_CASE
}

// ------------------------------------------------------------ Step C merge
cudaError_t launch_merge_twins(cpra_plan_s* dst, const MergeArgs& ma, int n_l) {
#define CPRA_CASE(NN) \
  case NN: return merge_twins_n<NN>(dst, ma, n_l);
  switch (dst->N) { CPRA_FOR_EACH_N(CPRA_CASE) default: return cudaErrorInvalidValue; }
#undef CPRA_CASE
}

cudaError_t launch_merge(cpra_plan_s* dst, const MergeArgs& ma, int n_l, float2* acc, unsigned long long* rings,
                         float* prtf) {
#define CPRA_CASE(NN) \
  case NN: return merge_n<NN>(dst, ma, n_l, acc, rings, prtf);
  switch (dst->N) { CPRA_FOR_EACH_N(CPRA_CASE) default: return cudaErrorInvalidValue; }
#undef CPRA_CASE
}

}  // namespace cpra
