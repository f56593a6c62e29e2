// gs_internal.h -- parameters shared by the host API and the iteration kernel.
#pragma once

#include <cuda_runtime.h>

#include <initializer_list>

namespace gsk {

// A block of the iteration kernels works on 256 lanes of 32 values, each held
// by one thread or by two (GroupT, gs_fft.cuh).
constexpr int kThreads = 256;
constexpr int kMaxThreads = 2 * kThreads;
// Threads per lane of the FP32 kernel of an nx x ny grid of powers of two.
inline __host__ __device__ constexpr int iteration_split(int nx, int ny) { return (nx > 512 || ny > 512) ? 1 : 2; }
constexpr int kMixedSplit = 1;  // ... of the mixed and serving kernels
constexpr int kLossSplit = 2;   // ... of the loss kernel
constexpr int kMaxIterPerLaunch = 128;          // iterations per persistent launch
constexpr int kSlots = 2 * kMaxIterPerLaunch + 2;  // FP64 partial-sum slots per launch
constexpr int kMaxGrid = 256;                   // upper bound on blocks per launch
constexpr int kMaxBatch = 64;                   // masks per launch
// Pass timestamps (gs_set_trace): rows of kMaxGrid (done, released) pairs,
// row 0 the launch start, row 1 + q pass q of the launch.
constexpr int kTraceRows = 2 * kMaxIterPerLaunch + 4;
// Group exchange buffers: (256 / T) groups of (n + n/32) complex, T = n/32,
// which is 256 * 33 complex whatever n is.
constexpr int kGroupSmemBytes = kThreads * 33 * 8;
// Split-exchange buffers of the kernels with two threads per lane: 16 complex
// values per lane. The FP32 kernels with one thread per lane have a second
// staging buffer for column blocks there.
constexpr int kSplitSmemBytes = kThreads * 16 * 8;
constexpr int kAheadSmemBytes = 8192 * 8;
constexpr int lane_smem_bytes(int split) { return split > 1 ? kSplitSmemBytes : kAheadSmemBytes; }
// Extra shared memory of the tensor-core kernels: stage twiddles [32][32]
// complex and a 32-entry cos/sin table (mma.sync); the two DFT matrices (hi
// and lo parts, 8 KiB each) and an 8 KiB twiddle table (tcgen05, whose
// operands share the exchange buffers).
constexpr int kTcExtraSmemBytes = 32 * 32 * 8 + 32 * 8;
constexpr int kTc5ExtraSmemBytes = 4 * 64 * 64 * 2 + 32 * 32 * 8;
// The mixed launch on tcgen05: the 32-point matrix (hi, lo), the 8-, 16- and
// 32-point matrices (hi, lo) and three twiddle tables.
constexpr int kMixedTc5ExtraSmemBytes = 2 * 64 * 64 * 2 + 2 * (16 * 16 + 32 * 32 + 64 * 64) * 2 + 3 * 32 * 32 * 8;

struct Params {
  int nx, ny;          // grid, powers of two in [32, 4096]
  int lognx, logny;
  float2* B;           // [ny][nx] field between passes (row-transformed)
  float* mT;           // scaled OSP amplitude, transposed: [nx][ny]
  const float* I;      // target intensity [ny][nx]
  const float* phi_in; // initial phase [ny][nx]
  float* phi_out;      // final phase [ny][nx]
  double* partials;    // [kSlots][batch][grid] per-block FP64 sums
  double* r_out;       // r^nu, or null
  double* g_out;       // g^nu, or null
  const float2* twx;   // stage twiddle tables of the row transforms (length nx)
  const float2* twy;   // stage twiddle tables of the column transforms (length ny)
  unsigned* bar;       // grid barrier arrival counter (zeroed before each launch)
  int* status;         // device status word (first error wins)
  int* abort_flag;     // set when a launch failed; later launches of the run return at once
  int* mask_flags;     // [kMaxBatch]: 1 for a mask whose target was rejected (written by the first launch)
  int batch;           // masks in this launch, 1..kMaxBatch, strided in every array
  long long mstride;   // elements of one mask in I, phi_in, phi_out, B and mT (nx*ny)
  int rstride;         // entries of one mask in r_out
  int gstride;         // entries of one mask in g_out
  int it0, it1;        // iterations [it0, it1) of this launch
  int iters;           // total K of the run
  int do_init;         // this launch computes m and u^0
  int do_final;        // this launch ends the run (phase out, final residual)
  int final_resid;     // compute r^K
  const float* p_slm;  // SLM amplitude p [ny][nx] (Eq. slm-constraint), or null for p = 1
  const double* energy;  // sum p^2 (FP64, workspace) when p_slm is set
  int init_target;     // start from P_S(F^{-1} m) instead of p exp(i phi_in)
  unsigned extra_arrivals;  // test hook: arrivals a barrier waits for beyond the grid (0 in use)
  float inv_sqrt_n;    // 1/sqrt(N)
  double inv_n;        // 1/N
  int tensor_core;     // host side: transforms on the FP32 ALUs (0) or the tensor cores (square 256,
                       // 512, 1024): mma.sync (1), tcgen05 with FP16 (2) or BF16 (3) operands
  unsigned long long* trace;  // [kTraceRows][grid][2] globaltimer stamps of block 0's thread 0 per block, or null
  int group;           // masks iterated together, 1..batch: the batch runs group after group
                       // through the whole schedule, so that a group's fields stay in L2
  // Grids with a side that is not a power of two (gs_general.cuh): the
  // radices of the row and column transforms, 3 bits per stage (code c means
  // radix kRadixOf[c]), first stage in the low bits, and the stage counts.
  unsigned planx, plany;
  int nstx, nsty;
  int gen_teams, gen_team_log;  // teams of a block, log2 of a team's threads
  int small_logc;      // log2 of the blocks per mask of the small-grid kernel
};

// Three size classes in one launch: square grids 256, 512 and 1024
// (log2 n = 8 + c), any of them with an empty batch. Every class has the
// same iteration count, flags and chunk; the barrier, status and abort words
// are class 0's. Mask flags and partial sums are per class.
struct MixedParams {
  Params cls[3];
};

// Small grids (power-of-two sides 32 ... 256, at most this many pixels) run on
// a cluster of 2^lc blocks per mask with the whole field in their shared
// memory (gs_small.cuh).
constexpr int kSmallMaxPixels = 32768;
constexpr int kSmallMaxLogC = 3;  // 8 blocks, the largest portable cluster
inline __host__ __device__ bool small_grid(int nx, int ny) {
  const bool px = nx > 0 && (nx & (nx - 1)) == 0, py = ny > 0 && (ny & (ny - 1)) == 0;
  return px && py && nx >= 32 && ny >= 32 && nx <= 256 && ny <= 256 && nx * ny <= kSmallMaxPixels;
}
// Blocks: at most 4096 pixels each (two fields, the amplitude and the exchange
// buffers in shared memory), at least 1024 (one warp of lanes).
inline int small_min_logc(int nx, int ny) {
  int lc = 0;
  while ((nx * ny >> lc) > 4096) ++lc;
  return lc;
}
inline int small_max_logc(int nx, int ny) {
  int lc = 0;
  while (lc < kSmallMaxLogC && (nx * ny >> lc) > 1024) ++lc;
  return lc;
}

// The general kernel serves every grid with a side that is not a power of
// two or is below 32 (the power-of-two kernels need 32 points per thread).
inline __host__ __device__ bool uses_general(int nx, int ny) {
  const bool px = nx > 0 && (nx & (nx - 1)) == 0, py = ny > 0 && (ny & (ny - 1)) == 0;
  return !px || !py || nx < 32 || ny < 32;
}

// Register-resident general-grid kernel (gs_rg.cuh): sides n = T V with a
// line in one warp (T lanes of V points, T, V <= 32). rg_threads(n) is T for
// the sides it serves (600 = 24 x 25, 768 = 32 x 24, 800 = 32 x 25,
// 1024 = 32 x 32), else 0; a grid whose two sides are both served, and not
// both powers of two, runs there (800 x 600, 1024 x 768, ...); any other grid
// with a side that is not a power of two on the shared-memory general kernel.
// Kernel templates take such a side itself in place of log2 nx (is_rg_side).
inline __host__ __device__ constexpr int rg_threads(int n) {
  return n == 600 ? 24 : (n == 768 || n == 800 || n == 1024) ? 32 : 0;
}
inline __host__ __device__ constexpr bool is_rg_side(int lx) { return lx >= 32; }
inline __host__ __device__ bool uses_rg(int nx, int ny) {
  return rg_threads(nx) > 0 && rg_threads(ny) > 0 && !(nx == 1024 && ny == 1024);
}

// Sides of the general kernel: 5-smooth (2^a 3^b 5^c) in [8, kMaxGeneralSide].
constexpr int kMaxGeneralSide = 1536;
constexpr int kMaxGeneralStages = 10;

// The general kernel transforms a row or column with a team of threads; a
// block has at most kGenMaxTeams teams, and one block runs per SM.
constexpr int kGenMinTeams = 4;
constexpr int kGenMaxTeams = 10;
constexpr int kGenMaxThreads = 640;
static_assert(kGenMaxTeams << 6 <= kGenMaxThreads, "teams of two warps fit");
constexpr int kGenSmemLimit = 227 * 1024 - 2048;  // dynamic part; the rest is the block's static arrays

// Shared-memory layout of the general kernel: the two twiddle tables (nx,
// then ny complex), then per team two buffers of max(nx, ny) complex.
inline __host__ __device__ int gen_tw_entries(int nx, int ny) { return (nx + ny + 1) & ~1; }
inline __host__ __device__ int gen_team_stride(int nmax) { return 2 * nmax + 2; }  // complex; 16-byte multiple
inline __host__ __device__ size_t gen_smem_bytes(int nx, int ny, int teams) {
  const int nmax = nx > ny ? nx : ny;
  return (static_cast<size_t>(gen_tw_entries(nx, ny)) + static_cast<size_t>(teams) * gen_team_stride(nmax)) *
         sizeof(float2);
}

// Values that the busiest thread of a team of `threads` threads takes through
// shared memory in a length-n transform: R per butterfly and stage (the radices
// of radix_plan, gs_api.cu).
inline int gen_thread_values(int n, int threads) {
  int left = n, sum = 0;
  for (int r : {3, 5, 8, 4, 2})
    while (left % r == 0) {
      sum += r * ((n / r + threads - 1) / threads);
      left /= r;
    }
  return sum;
}

// Teams per block and log2 of a team's threads for `masks` masks of nx x ny
// on `sms` SMs: the fewest rounds that shared memory allows, then the fewest
// teams that need no more (at least kGenMinTeams, so that column tiles are
// 32-byte row segments).
struct GenGeom {
  int teams;
  int team_log;
};
// The smallest block, the one of which an SM may hold several: kThreads
// threads (iteration_threads) and gen_smem_bytes(nx, ny, kGenMinTeams).
constexpr GenGeom kGenMinGeom{kGenMinTeams, 6};
static_assert(kGenMinGeom.teams << kGenMinGeom.team_log == kThreads, "the block of the occupancy query");
inline GenGeom gen_geom(int nx, int ny, int masks, int sms) {
  const int nmax = nx > ny ? nx : ny;
  int fit = kGenMaxTeams;
  while (fit > kGenMinTeams && gen_smem_bytes(nx, ny, fit) > static_cast<size_t>(kGenSmemLimit)) --fit;
  const long long lines = static_cast<long long>(nmax) * masks;
  const long long rounds = (lines + static_cast<long long>(sms) * fit - 1) / (static_cast<long long>(sms) * fit);
  const long long per = static_cast<long long>(sms) * rounds;
  int teams = static_cast<int>((lines + per - 1) / per);
  if (teams < kGenMinTeams) teams = kGenMinTeams;
  // Two warps per line. Four, where a block has room, if they spare the
  // busiest thread of a row and of a column transform 23 values together: that
  // pays for the wider synchronisation of every stage. Ten iterations with two
  // warps and four, values spared: 320 x 320 (0) 147 and 164 us, 384 x 384 (10)
  // 167 and 179, 480 x 320 (12) 161 and 168, 400 x 300 (21) 168 and 170, 480 x
  // 360 (23) 173 and 172, 600 x 50 (24) 154 and 150, 400 x 400 (28) 180 and
  // 182, 432 x 324 (29) 186 and 182, 500 x 375 (37) 177 and 170, 640 x 480 (37)
  // 204 and 200, 625 x 625 (40) 220 and 207. Sides below 300 keep two (243 x
  // 243, 30 spared: 170 and 171).
  const int saved = gen_thread_values(nx, 64) + gen_thread_values(ny, 64) - gen_thread_values(nx, 128) -
                    gen_thread_values(ny, 128);
  const int tl = nmax >= 300 && saved >= 23 && (teams << 7) <= kGenMaxThreads ? 7 : 6;
  return {teams, tl};
}

// Kernel for log2(nx) = LX and the given log2(ny); defined per LX in gs_inst.cu.
template <int LX>
const void* iterate_kernel_lx(int ly);
// Kernel of runs under a laser amplitude for log2(nx) = LX in 11, 12; null where
// the kernel above serves them.
template <int LX>
const void* iterate_kernel_slm_lx(int ly);
// Kernel with tensor-core transforms for an n x n grid, log2(n) = l in 8..10
// (gs_tc_inst.cu); null otherwise.
const void* iterate_kernel_tc(int l);
// Kernel for grids with a side that is not a power of two (gs_general_inst.cu).
const void* iterate_kernel_general();
// Register-resident kernel for an nx x ny grid with uses_rg (gs_rg_inst.cu),
// its dynamic shared memory, and the layout of its twiddle tables: for a side
// n = T V, n entries W_n^{t q} at [q T + t] (q < V, t < T), then n entries
// W_n^{q j} at [j V + q].
const void* iterate_kernel_rg(int nx, int ny);
size_t rg_smem_bytes(int nx, int ny);
// The kernels and shared memory for one row length, from the object of
// gs_rg_inst.cu compiled for it.
template <int NX>
const void* iterate_kernel_rg_nx(int ny);
template <int NX>
size_t rg_smem_bytes_nx(int ny);
// Stage twiddle tables of a power-of-two length n (the layout stage_c reads),
// kStageTwiddleEntries entries, rounded once from double (gs_api.cu).
constexpr int kStageTwiddleEntries = 31 * 32 + 31 * 1024;
void stage_twiddles_host(int n, float2* out);
// Kernel for three square size classes in one launch (gs_mixed_inst.cu), by
// TcMode.
const void* iterate_kernel_mixed(int tc_mode);
size_t mixed_smem_bytes(int tc_mode);
cudaError_t mixed_occupancy(int tc_mode, int* blocks_per_sm);
cudaError_t launch_mixed(const MixedParams& mp, int grid, int tc_mode, cudaStream_t s);

// Tensor-core modes of Params::tensor_core.
enum TcMode { kTcNone = 0, kTcMmaSync = 1, kTcGen05F16 = 2, kTcGen05Bf16 = 3 };
size_t iteration_smem_bytes(int nx, int ny, int tc_mode = kTcNone);

// Intensity loss and gradient (square grids), see gs_loss.cuh. A launch
// either does everything (fused), or stages the target once (prepare) for
// later launches that run only the transform passes on it (step).
enum LossMode { kLossFused = 0, kLossPrepare = 1, kLossStep = 2 };
struct LossParams {
  int n, logn;             // square grid n x n
  float2* B;               // workspace field (column-blocked layout)
  float* IT;               // workspace: target transposed [n][n]
  const float* I;          // target intensity [n][n]
  const float* phi;        // phase [n][n]
  float* grad;             // dL/dphi [n][n], or null (loss only)
  double* loss;            // [steps]: the loss before each step
  double* phys;            // [2]: physical error (E_l, E_d), or null
  const float* p_slm;      // SLM amplitude [n][n], or null (p = 1)
  const double* energy;    // sum p^2 when p_slm is set
  double* partials;        // rows of LossRow (gs_loss.cuh): six of `grid` values, three of kMaxGrid
  const float2* tw;        // stage twiddle tables (length n)
  unsigned* bar;
  int* status;
  int* abort_flag;
  float inv_n;             // 1/N
  int mode;                // LossMode: fused, prepare the target, or a step on the prepared target
  // A step with the Adam update fused into the gradient pass (grad is then
  // null): phase (the same array as phi) is updated in place with the running
  // moments m, v; state[0] counts the steps done, state[1] the blocks done.
  float* phase;
  float* m;
  float* v;
  int* state;
  float lr, beta1, beta2, eps;
  // Adam steps in this launch (1 unless m is set): the gradient pass of a
  // step also forms the next step's row transforms of exp(i phase).
  int steps;
};

// Adam steps per launch of gs_loss_adam_run (a longer run is split).
constexpr int kMaxAdamStepsPerLaunch = 1024;

cudaError_t launch_loss(const LossParams& p, int grid, cudaStream_t s);
cudaError_t launch_iterations(const Params& p, int grid, cudaStream_t s);
// sum p^2 of an SLM amplitude into *energy (NaN if p has a negative or
// non-finite value); scratch: kMaxGrid doubles
cudaError_t launch_energy(const float* p, long long n, double* energy, double* scratch, cudaStream_t s);
cudaError_t iteration_occupancy(int nx, int ny, int* blocks_per_sm, int tc_mode = kTcNone);
// The tcgen05 kernel of n x n masks, log2(n) = l in 8..10 (gs_tc5_inst.cu);
// FP16 or BF16 operands; null for other sizes.
const void* iterate_kernel_tc5(int l, bool bf16);
// Small grids (small_grid): allow the kernel its shared memory and find how
// many clusters of 2^lc blocks run at once (0 where lc does not apply), and
// launch one cluster of 2^small_logc blocks per mask of p.batch
// (gs_small_inst.cu).
cudaError_t small_prepare(int nx, int ny, int clusters[kSmallMaxLogC + 1]);
cudaError_t launch_small(const Params& p, cudaStream_t s);

}  // namespace gsk
