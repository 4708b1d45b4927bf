// cpra_internal.h - plan layout and kernel launchers shared by the .cu files.
//
// Device data of one plan (all stacks contiguous per angle):
//   g, g_alt   [Np][N][N]    float   iterate (Jacobi double buffer for Eq. 4)
//   Hp         [Np][N][N/2]  float2  row spectra of g, packed: column 0 holds
//                                    (Re H(y,0), Re H(y,N/2)); the two-pass
//                                    engine keeps it between its passes
//   A_main     [Np][N/2][N]  float   Hermitian-symmetrised amplitude, kx < N/2,
//                                    column-major ([kx][ky])
//   A_nyq      [Np][N]       float   the same at kx = N/2
//   Cn, sumA2  [Np]          double  antisymmetric-part energy, sum A^2
//   S          [Np][N][W]    uint32  support bits, W = ceil(N/32) words a row
//   err_acc    [Np]          double  per-iteration error accumulator
//   err_hist   [cap][Np]     double  Fourier error history
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <string>
#include <vector>

#include "cpra.h"
#include "per_device.h"

namespace cpra {

struct JobStatic;
struct JobStep;
struct MergeGuess;

// Device-side status of a plan.  It lives in mapped, pinned host memory, so
// kernels set it with plain stores and the host reads it without waiting
// for the plan's stream.
struct DevStatus {
  unsigned flags;  // kStatusNonFinite
  int angle;       // an angle whose Fourier error was not finite
};
constexpr unsigned kStatusNonFinite = 1u;
constexpr unsigned kStatusTimeout = 2u;  // a bounded device wait gave up

// A sample of a grid cell: its line of F, n * (N/2 + 1) + |ku| (bit 31: ku < 0,
// the conjugate is read), and its bilinear weight (normalised in FP64).
struct GridEnt {
  uint32_t at;
  float w;
};

struct Assembly {
  float2* F = nullptr;        // z-transformed spectra, [z / 8][n][ku = 0 .. N/2][z % 8]
  float2* corr = nullptr;     // [Np][N/2 + 1] what F(-ku) is beside conj F(ku) (k_assemble.cu)
  float2* Q = nullptr;        // [N][N] a cell's sum of weight * corr
  float2* ramps = nullptr;    // per angle the unit ramps of its mass-centre move
  float2* vol = nullptr;      // [N][N][N] grid, then the centred volume
  int32_t* cell_ptr = nullptr;  // [N*N + 1] CSR rows (cells ky*N + kx)
  cpra::GridEnt* ents = nullptr;  // samples of the cells
  double* moments = nullptr;    // [Np][3] sum rho, sum rho*z, sum rho*u
  int64_t n_ent = 0;
  bool ready = false;    // a volume of the current angles may be read
  bool grid_ok = false;  // the gridding lists match the current angles
};

}  // namespace cpra

struct cpra_plan_s {
  cpra_config cfg;
  cudaStream_t stream = nullptr;
  // volume downloads that overlap later work (cpra_assemble_3d_async)
  float2* dl_buf = nullptr;  // staging copy of the volume being downloaded
  cudaStream_t dl_stream = nullptr;
  cudaEvent_t dl_ready = nullptr, dl_done = nullptr;
  bool dl_pending = false;
  // intensity uploads from host memory, on their own stream and buffer, so
  // that they overlap work already queued on the plan's stream
  float* ul_buf = nullptr;  // Np*N*N floats, allocated on the first host upload
  cudaStream_t ul_stream = nullptr;
  cudaEvent_t ul_done = nullptr, ul_free = nullptr;
  bool ul_used = false;  // ul_free has been recorded (the buffer was read)
  int N = 0, Np = 0, W = 0;
  int64_t t = 0;
  bool state_ready = false;
  bool hp_valid = false;
  int n_loaded = 0;
  std::vector<uint8_t> loaded;
  std::vector<double> theta;
  int engine = CPRA_ENGINE_TWO_PASS;

  float* g = nullptr;
  float* g_alt = nullptr;
  float2* Hp = nullptr;
  float* A_main = nullptr;
  float* A_nyq = nullptr;
  double* Cn = nullptr;
  double* sumA2 = nullptr;
  double* err_acc = nullptr;
  uint32_t* S = nullptr;
  double* err_hist = nullptr;
  int64_t err_cap = 0;
  float2* tw = nullptr;        // forward twiddles exp(-2 pi i k/N)
  float2* xtw = nullptr;       // warp-FFT cross twiddles, [k1][l] = exp(-2 pi i l k1/N)
  uint16_t* tcw = nullptr;     // tensor-core DFT matrices (BF16 / FP16 precision)
  float* stage = nullptr;      // staging for host inputs, Np*N*N floats
  uint8_t* bad = nullptr;      // device, Np bytes: 1 where the last load of the angle was invalid
  cpra::DevStatus* status_h = nullptr;  // mapped pinned host memory (cudaHostAlloc)
  cpra::DevStatus* status_d = nullptr;  // its device address
  float* sw_tmp = nullptr;     // shrink-wrap scratch, Np*N*N floats
  unsigned* sw_max = nullptr;  // per-angle max (float bits)
  float* sw_taps = nullptr;    // periodic Gaussian taps
  int sw_ntaps = 0;
  float* po_tmp = nullptr;
  uint8_t* mask = nullptr;     // measured-pixel mask (cpra_load_mask), centred; NULL = all
  bool mask_per_angle = false;
  bool masked = false;         // intensities were loaded under a mask (kernels check A_sym < 0)
  cpra::Assembly asmb;
  // Step C merge scratch (cpra_merge with this plan as destination)
  float2* mg_acc = nullptr;    // [Np][N][N] merged spectra (the mean)
  float2* mg_ref = nullptr;    // [N][N] E of the reference PO of the best guess
  unsigned long long* mg_rings = nullptr;  // [Np][N/2] ring sums of the PRTF, then N/2 ring populations
  int32_t mg_cap = 0;          // kept guesses that mg_guess, mg_dist and mg_ramps hold
  cpra::MergeGuess* mg_guess = nullptr;
  double* mg_dist = nullptr;   // [mg_cap] twin choice (MergeArgs::dist)
  float2* mg_ramps = nullptr;  // [mg_cap] ramps of the kept guesses
  float* mg_prtf = nullptr;    // [Np][N/2] PRTF staging for host outputs
  bool merged = false;         // mg_acc holds the mean of the last merge
  // Step D refinement (cpra_refine_3d)
  int vol_state = 0;           // 0 none, 1 Step D volume (assemble or merge), 2 refined
  float2* rf_X = nullptr;
  float2* rf_W = nullptr;
  double* rf_konst = nullptr;  // [2]
  float* rf_R = nullptr;
  float* rf_B = nullptr;
  uint32_t* rf_S3 = nullptr;
  uint8_t* rf_M = nullptr;
  double* rf_err = nullptr;    // [2 * rf_err_cap] error sums per iteration
  int64_t rf_err_cap = 0;
  double2* rf_cs = nullptr;    // [Np] (cos, sin) of the angles
  int2* rf_shift = nullptr;    // [Np] whole-pixel mass-centre shifts (dz, du)
  float* rf_taps = nullptr;    // [N] periodic Gaussian taps of the last shrink
  unsigned* rf_max = nullptr;
  int64_t rf_t = 0;            // refinement iterations run
  // kernel tables of this plan as a one-job launch
  cpra::JobStatic* d_js = nullptr;
  int2* d_tiles = nullptr;     // (0, angle) of every iterating angle, ascending
  // angles that iterate (cpra_set_present); all of them unless partial
  uint8_t* present = nullptr;  // device, Np bytes
  std::vector<uint8_t> present_h;
  int n_present = 0;
  bool partial = false;
  int64_t present_version = 0;
  cpra::JobStep* d_steps = nullptr;
  int64_t steps_cap = 0;

  // device-time profiling of launches (cpra_set_profiling)
  struct Timed { int kind; cudaEvent_t a, b; };
  bool profiling = false;
  std::vector<Timed> pending;
  std::vector<Timed> spare;
  double kms[CPRA_KERNEL_KINDS] = {0};
  long long kcount[CPRA_KERNEL_KINDS] = {0};

  std::string err;
  std::vector<void*> owned;
};

namespace cpra {

// kernels launched by this library in this process (cpra_launch_count)
extern std::atomic<long long> g_launches;

enum Algo { kHIO = 0, kER = 1, kRAAR = 2 };

// Real-space step of one pixel from the old iterate g, g' = Re IFFT2(P_M G)
// and its support bit.
//   HIO  (Fienup):  g' on V = {in S, g' >= 0}, g - beta g' elsewhere
//   ER:             g' on V, 0 elsewhere
//   RAAR (Luke 2005, T = beta/2 (R_S R_M + I) + (1 - beta) P_M with the
//        reflections R = 2P - I): R_M g = 2g' - g, so g' where 2g' - g lies
//        in the support-positivity set, beta g + (1 - 2 beta) g' elsewhere;
//        c2 = 1 - 2 beta.
template <int ALGO>
__device__ __forceinline__ float update_pixel_t(float g, float gp, bool in_s, float beta, float c2) {
  if constexpr (ALGO == kRAAR) return (in_s && fmaf(2.0f, gp, -g) >= 0.0f) ? gp : fmaf(beta, g, c2 * gp);
  const bool v = in_s && gp >= 0.0f;
  if constexpr (ALGO == kHIO) return v ? gp : fmaf(-beta, gp, g);
  return v ? gp : 0.0f;
}
__device__ __forceinline__ float update_pixel(float g, float gp, bool in_s, int algo, float beta,
                                              float c2) {
  if (algo == kRAAR) return update_pixel_t<kRAAR>(g, gp, in_s, beta, c2);
  if (algo == kHIO) return update_pixel_t<kHIO>(g, gp, in_s, beta, c2);
  return update_pixel_t<kER>(g, gp, in_s, beta, c2);
}

// prepare / state kernels (k_prepare.cu)
cudaError_t launch_prepare(cpra_plan_s* p, const float* I, int first, int count);
cudaError_t launch_support_box(cpra_plan_s* p);
cudaError_t launch_support_u8(cpra_plan_s* p, const uint8_t* S, int per_angle);
cudaError_t launch_init_guess(cpra_plan_s* p);
cudaError_t launch_export_po(cpra_plan_s* p, float* out);
cudaError_t launch_export_support(cpra_plan_s* p, uint8_t* out);
cudaError_t launch_bits_from_u8(uint32_t* bits, const uint8_t* src, int N, int count,
                                cudaStream_t st);
cudaError_t launch_bits_to_u8(const uint32_t* bits, uint8_t* out, int N, int count,
                              cudaStream_t st);

// two-pass iteration (k_twopass.cu, k_fast.cu)
struct CoupleArgs {
  int n_taps;        // 1 = no coupling
  float alpha[CPRA_MAX_TAPS];
  int mirror;
  int object;        // blend P_{S+} g instead of g
  int store_g;       // write the coupled rows to g_dst
  int sweep;         // Gauss-Seidel: taps on angles before n read g_dst
};

// Per-reconstruction pointers and constants, read by the kernels from a
// device table so that one launch can serve many reconstructions.
struct JobStatic {
  float2* Hp;
  const float* A_main;
  const float* A_nyq;
  const double* Cn;
  const double* sumA2;
  double* err_acc;
  const uint32_t* S;
  double* err_hist;
  const float2* tw;
  const float2* xtw;
  const uint16_t* tcw;  // 16-bit block DFT matrices (tensor-core precision)
  const uint8_t* present;  // angles that iterate (coupling renormalises), NULL = all
  DevStatus* status;       // device address of the plan's status word
  int Np, W;
  float beta;
  int pad;
};

// The Fourier error E_F of angle n from its FP64 sums (error terms of the
// column pass + the constant C_n, over sum A^2), as written to the error
// history.  A non-finite sum means a non-finite iterate (a diverged run, a
// NaN or Inf state) or an invalid pattern (the preparation poisons C_n):
// it is flagged in the plan's status word, which the next call reports.
__device__ __forceinline__ double publish_error(double acc, double cn, double den, DevStatus* st,
                                                int n) {
  const double num = acc + cn;
  if (!isfinite(num) || !isfinite(den)) {
    volatile DevStatus* v = st;
    v->angle = n;
    v->flags = kStatusNonFinite;
  }
  return den > 0.0 ? sqrt(num / den) : 0.0;
}

// What one reconstruction does in one iteration (device table, one entry
// per job per iteration).
struct JobStep {
  const float* g_src;  // prime: source stack (coupling reads the neighbours here)
  float* g_dst;        // prime: coupled stack, written when ca.store_g
  float* g;            // the iterate the row pass updates in place
  long long err_slot;  // error-history row, -1 = none
  int prime;           // run the prime kernel (coupling and/or row R2C)
  int algo;            // kHIO / kRAAR / kER; fused engine: the rule of its
                       // first hio_left iterations (ER after them)
  int forward;         // row pass also computes the next row spectra
  int active;          // 0: the column and row passes skip this job
  CoupleArgs ca;
  int n_iters;         // fused engine: iterations of this launch (prime first)
  int hio_left;        // fused engine: how many of them are HIO (the rest ER)
};

// Arguments of the warp engine's persistent work-queue kernel (k_persist_w
// in fast_kernels.cuh).
struct PersistArgs {
  const JobStatic* js;
  const JobStep* st;  // step rows of the call: iteration i of this launch at st + (row0 + i) * m
  const int2* tiles;  // (member, angle) tiles
  int ntiles, m, row0, iters;
  int chunk;          // tiles a chunk: the queue runs chunk by chunk, all iterations each
  unsigned* ticket;   // [2]: next task; [1] is a count that no task increments
  unsigned* done;     // [2 * ntiles]: column and row blocks done in this launch
  long long budget;   // clock64 cycles a wait may take
  int hold;           // testing: the first task waits on ticket[1] >= 1 (never)
};

// One launch over ntiles (job, angle) tiles.
struct Launch {
  int N;
  int engine;
  int prec;  // CPRA_FP32 / CPRA_BF16_TC / CPRA_FP16_TC
  int masked;  // some amplitude carries the missing-data sentinel (A_sym < 0)
  cudaStream_t stream;
  const JobStatic* js;
  const JobStep* st;
  const int2* tiles;
  int ntiles;
};

cudaError_t prepare_kernels(int N, int engine, int prec);  // shared-memory attributes, before capture
cudaError_t launch_prime(const Launch& L);
cudaError_t launch_colpass(const Launch& L);
cudaError_t launch_rowpass(const Launch& L);
cudaError_t launch_shrinkwrap(cpra_plan_s* p);

// the value of the current device (the one that the caller's stream and buffers
// are on)
template <class T, class F>
cudaError_t on_device(PerDevice<T>& facts, T& v, F&& make) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e == cudaSuccess ? facts.get(dev, v, make) : e;
}
// make() once on each device
template <class F>
cudaError_t once_on_device(PerDevice<bool>& done, F&& make) {
  bool v;
  return on_device(done, v, [&](bool&) { return make(); });
}
// opt-in to more than 48 KB of dynamic shared memory
template <class K>
cudaError_t smem_attr(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <class K>
cudaError_t smem_once(K kernel, size_t bytes, PerDevice<bool>& done) {
  return once_on_device(done, [&] { return smem_attr(kernel, bytes); });
}

// assembly (k_assemble.cu)
// spectra, grid and volume from Hp and the ramps (launch_rho_rows); out: NULL,
// or device memory of the plan's device that receives the volume too
cudaError_t launch_assemble(cpra_plan_s* p, float2* out);
size_t spectra_bytes(int N, int Np);  // Assembly::F, ::corr and ::ramps
size_t corr_bytes(int N, int Np);
size_t ramps_bytes(int N, int Np);

// Step C merge (k_assemble.cu): modes of the spectra kernel
enum SpecMode { kSpecF = 0, kSpecRef = 1, kSpecDist = 2 };
// a kept guess: its R2C rows of rho, its ramps, whether it is inverted
struct MergeGuess {
  const float2* Hp;
  const float2* ramps;
  int inv, pad;
};
struct MergeArgs {
  int n0;                   // REF, DIST: the PO
  const MergeGuess* guess;  // device table of the kept guesses, best first
  float2* ref;              // E of PO n0 of the best guess, [kz][ku]
  double* dist;             // [kept] sum Im ref Im E: negative where conj E is the nearer to ref
};
// FP64 moments (sum rho, sum rho z, sum rho u) of rho = P_{S+} g of every angle
cudaError_t launch_moments(cpra_plan_s* p, double* moments, cudaStream_t st);
// R2C rows of rho into Hp (L: the plan's launch of a plain object prime over
// every angle), the moments of rho, and the unit ramps of the mass-centre moves
cudaError_t launch_rho_rows(cpra_plan_s* p, const Launch& L, double* moments, float2* ramps);
// twin choice of the kept guesses (MergeArgs::dist), on dst's stream
cudaError_t launch_merge_twins(cpra_plan_s* dst, const MergeArgs& ma, int n_l);
// acc = mean of the corrected spectra, PRTF (rings and prtf not NULL), its
// IDFT_z, gridding and the plane IFFTs into dst's volume, on dst's stream
cudaError_t launch_merge(cpra_plan_s* dst, const MergeArgs& ma, int n_l, float2* acc, unsigned long long* rings,
                         float* prtf);
// inverse FFT along y of every plane of a volume, in place, and into out when
// that is not NULL (refine_kernels.cuh)
cudaError_t launch_volume_ylines(int N, float2* vol, float2* out, const float2* xtw, cudaStream_t st);

// Step D refinement (k_refine.cu): buffers of one plan's refinement
struct RefineArgs {
  int N, W;            // W = ceil(N/32) words per x row of S3
  float2* X;           // N^3: the data volume, then the half spectrum [z][y][HP]
  float2* Wd;          // N^3: the data of the half spectrum (refine_kernels.cuh), same layout
  float* R;            // [N^3] real iterate rho
  float* Bv;           // [N^3] shrink-wrap blur scratch
  uint32_t* S3;        // [N][N][W] 3D support bits
  uint8_t* M;          // [N][N] measured (ky, kx) cells
  const float2* xtw;   // warp-FFT cross twiddles
  double* konst;       // [2] constant parts of the error sums
};
// X = vol (centred), R = Re vol
cudaError_t launch_refine_setup(const RefineArgs& a, const float2* vol, cudaStream_t st);
// S3 from the 2D supports S2 [Np][N][W] moved by shift[n] = (dz, du), with
// (cos, sin) of every angle; M from the gridding lists
cudaError_t launch_refine_support(const RefineArgs& a, const uint32_t* S2, const double2* cs,
                                  const int2* shift, int Np, const int32_t* cell_ptr, cudaStream_t st);
// Wd and konst from X and M; X is free afterwards
cudaError_t launch_refine_data(const RefineArgs& a, cudaStream_t st);
// one iteration (first: it starts from R; last: it ends in R); err2[0] +=
// sum_M |X - V|^2, err2[1] = sum_M |V|^2
cudaError_t launch_refine_iter(const RefineArgs& a, double* err2, bool first, bool last, cudaStream_t st);
// S3 <- {blur(P_{S3+} R) >= tau max} (mx: one unsigned of scratch)
cudaError_t launch_refine_shrink(const RefineArgs& a, const float* taps, int ntaps, float tau,
                                 unsigned* mx, cudaStream_t st);
// vol = P_{S3+} R
cudaError_t launch_refine_output(const RefineArgs& a, float2* vol, cudaStream_t st);

bool n_supported(int N);

// two-pass engine with warp-resident FFTs (k_fast.cu)
bool warp_engine_listed(int N);      // sizes that CPRA_ENGINE_WARP names (its kernels cover every N)
bool tc_supported(int N);            // tensor-core forms
bool fast_dims(int N, int* E1, int* E2);
cudaError_t prepare_kernels_fast(int N);
cudaError_t prepare_kernels_fast_tc(int N, int prec);
cudaError_t launch_rowpass_fast_tc(const Launch& L);
cudaError_t launch_prime_fast_tc(const Launch& L);
cudaError_t launch_colpass_fast_tc(const Launch& L);
cudaError_t launch_rowpass_fast(const Launch& L);
cudaError_t launch_prime_fast(const Launch& L, double* moments = nullptr);
cudaError_t launch_colpass_fast(const Launch& L);
// persistent work-queue form of the column and row passes (FP32)
bool persist_supported(int N);
cudaError_t prepare_persist(int N, int* blocks_per_sm);
cudaError_t launch_persist(int N, const PersistArgs& a, int masked, int grid, cudaStream_t st);

// cluster-resident fused engine (k_fused.cu): one launch = prime + n_iters
// iterations of every tile, the angle's spectrum held in distributed shared
// memory
bool fused_supported(int N);
cudaError_t prepare_kernels_fused(int N);
cudaError_t launch_fused(const Launch& L);

// One launch for a whole Gauss-Seidel episode (k_sweep.cu at the block-wide
// engine's sizes, k_fused.cu for N = 64, 128, 256): tile j = (member,
// 0), the member's angles in order inside the launch; step row: the coupling
// arguments, g_src, g = g_dst, err_slot, n_iters, hio_left.
bool sweep_supported(int N, int engine, int members);
cudaError_t launch_sweep(const Launch& L);
bool fused_sweep_supported(int N);
cudaError_t launch_fused_sweep(const Launch& L);

// records a failure of a call without a plan (cpra_last_error(NULL))
cpra_status record_error(cpra_status st, const std::string& msg);

}  // namespace cpra
