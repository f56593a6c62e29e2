// gs_launch.cu -- host helpers that select, size and launch the iteration kernel.
#include <cfloat>

#include "gs_internal.h"

namespace gsk {

// sum p^2 in FP64, in a fixed order; NaN if any p is negative or not finite.
// Each block a contiguous share into scratch, eight loads of a thread in
// flight; then one warp adds the blocks. Up to 4096 values are one block, which
// writes the sum itself. Microseconds a call with one block of 1024 threads and
// a load at a time for everything, with two launches for everything, and now:
// 8 x 8 6.2, 8.3, 4.2; 64 x 64 8.3, 10.3, 6.3; 128 x 128 14.5, 10.3, 10.3; 1024 x
// 1024 577, 12.5, 12.5. (One block of 1024 threads up to 128 x 128: 10.4 at 64 x
// 64 and 14.5 at 128 x 128, the FP64 pipe of one SM.)
constexpr int kEnergyThreads = 256;
constexpr int kEnergyBlocks = kMaxGrid;

__global__ void __launch_bounds__(kEnergyThreads) energy_kernel(const float* __restrict__ p, long long n,
                                                               double* __restrict__ to) {
  __shared__ double red[kEnergyThreads / 32];
  const long long lo = blockIdx.x * n / gridDim.x, hi = (blockIdx.x + 1) * n / gridDim.x;
  double acc = 0.0;
  bool bad = false;
  for (long long e0 = lo + threadIdx.x; e0 < hi; e0 += 8 * kEnergyThreads) {
    float x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) x[u] = e0 + u * kEnergyThreads < hi ? p[e0 + u * kEnergyThreads] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      bad |= !(x[u] >= 0.f && x[u] <= FLT_MAX);
      acc += static_cast<double>(x[u]) * static_cast<double>(x[u]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  const int any_bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < kEnergyThreads / 32; ++w) s += red[w];
    to[blockIdx.x] = any_bad ? __longlong_as_double(0x7ff8000000000000ll) : s;
  }
}

__global__ void __launch_bounds__(32) energy_total(const double* __restrict__ scratch, int blocks, double* out) {
  double s = 0.0;
  for (int b = threadIdx.x; b < blocks; b += 32) s += scratch[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (threadIdx.x == 0) out[0] = s;
}

cudaError_t launch_energy(const float* p, long long n, double* energy, double* scratch, cudaStream_t s) {
  const long long want = (n + 4095) / 4096;
  const int blocks = static_cast<int>(want < kEnergyBlocks ? want : kEnergyBlocks);
  energy_kernel<<<blocks, kEnergyThreads, 0, s>>>(p, n, blocks == 1 ? energy : scratch);
  if (blocks > 1) energy_total<<<1, 32, 0, s>>>(scratch, blocks, energy);
  return cudaGetLastError();
}

// Each is defined in the gs_inst.cu object compiled with GS_LX = LX.
extern template const void* iterate_kernel_lx<5>(int);
extern template const void* iterate_kernel_lx<6>(int);
extern template const void* iterate_kernel_lx<7>(int);
extern template const void* iterate_kernel_lx<8>(int);
extern template const void* iterate_kernel_lx<9>(int);
extern template const void* iterate_kernel_lx<10>(int);
extern template const void* iterate_kernel_lx<11>(int);
extern template const void* iterate_kernel_lx<12>(int);
extern template const void* iterate_kernel_slm_lx<11>(int);
extern template const void* iterate_kernel_slm_lx<12>(int);

extern template const void* iterate_kernel_rg_nx<600>(int);
extern template const void* iterate_kernel_rg_nx<768>(int);
extern template const void* iterate_kernel_rg_nx<800>(int);
extern template const void* iterate_kernel_rg_nx<1024>(int);
extern template size_t rg_smem_bytes_nx<600>(int);
extern template size_t rg_smem_bytes_nx<768>(int);
extern template size_t rg_smem_bytes_nx<800>(int);
extern template size_t rg_smem_bytes_nx<1024>(int);

const void* iterate_kernel_rg(int nx, int ny) {
  switch (nx) {
    case 600: return iterate_kernel_rg_nx<600>(ny);
    case 768: return iterate_kernel_rg_nx<768>(ny);
    case 800: return iterate_kernel_rg_nx<800>(ny);
    case 1024: return iterate_kernel_rg_nx<1024>(ny);
    default: return nullptr;
  }
}

size_t rg_smem_bytes(int nx, int ny) {
  switch (nx) {
    case 600: return rg_smem_bytes_nx<600>(ny);
    case 768: return rg_smem_bytes_nx<768>(ny);
    case 800: return rg_smem_bytes_nx<800>(ny);
    case 1024: return rg_smem_bytes_nx<1024>(ny);
    default: return 0;
  }
}

static int log2_exact(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return l;
}

static const void* kernel_for(int nx, int ny, int tc_mode) {
  if (uses_general(nx, ny)) {
    if (tc_mode != kTcNone) return nullptr;
    return uses_rg(nx, ny) ? iterate_kernel_rg(nx, ny) : iterate_kernel_general();
  }
  const int ly = log2_exact(ny);
  if (tc_mode == kTcGen05F16 || tc_mode == kTcGen05Bf16)
    return nx == ny ? iterate_kernel_tc5(ly, tc_mode == kTcGen05Bf16) : nullptr;
  if (tc_mode == kTcMmaSync) return nx == ny ? iterate_kernel_tc(ly) : nullptr;
  switch (log2_exact(nx)) {
    case 5: return iterate_kernel_lx<5>(ly);
    case 6: return iterate_kernel_lx<6>(ly);
    case 7: return iterate_kernel_lx<7>(ly);
    case 8: return iterate_kernel_lx<8>(ly);
    case 9: return iterate_kernel_lx<9>(ly);
    case 10: return iterate_kernel_lx<10>(ly);
    case 11: return iterate_kernel_lx<11>(ly);
    case 12: return iterate_kernel_lx<12>(ly);
    default: return nullptr;
  }
}

// Runs under a laser amplitude whose row passes take seven rounds or more
// (256 / (nx/32) rows per block and round: 4096 x 4096, 4096 x 2048 and 2048 x
// 4096) have a kernel of their own, which fetches the next rows behind the
// transforms as the kernel of p = 1 does and keeps the row's amplitude in the
// second staging buffer. nx x ny x 10 iterations without and with the fetch:
// 4096 x 4096 3.78 and 3.20 ms, 4096 x 2048 1.36 and 1.30, 2048 x 4096 1.72 and
// 1.47; with four rounds it is slower (2048 x 2048 0.696 and 0.700, 4096 x 1024
// 0.632 and 0.639). One kernel that chooses at run time cost p = 1 one per cent
// (4096 x 4096 3.01 and 3.04). Null: the common kernel.
static const void* iterate_kernel_slm(int nx, int ny, int tc_mode) {
  if (tc_mode != kTcNone || uses_general(nx, ny)) return nullptr;
  if (nx == 4096) return iterate_kernel_slm_lx<12>(log2_exact(ny));
  return nx == 2048 ? iterate_kernel_slm_lx<11>(log2_exact(ny)) : nullptr;
}

// threads per block of the kernel of an nx x ny grid (the general kernel's
// block depends on the run: here its smallest one, kGenMinGeom)
static int iteration_threads(int nx, int ny, int tc_mode) {
  return (uses_general(nx, ny) || tc_mode != kTcNone) ? kThreads : kThreads * iteration_split(nx, ny);
}

static int mixed_threads(int tc_mode) { return tc_mode != kTcNone ? kThreads : kThreads * kMixedSplit; }

size_t iteration_smem_bytes(int nx, int ny, int tc_mode) {
  if (uses_rg(nx, ny)) return rg_smem_bytes(nx, ny);
  if (uses_general(nx, ny)) return gen_smem_bytes(nx, ny, kGenMinGeom.teams);
  // group exchange buffers, one column block of the amplitude, one of the
  // field; then the split-exchange buffers, or the tensor-core tables (and,
  // for tcgen05, operands)
  const size_t extra = tc_mode == kTcMmaSync ? kTcExtraSmemBytes
                       : (tc_mode == kTcGen05F16 || tc_mode == kTcGen05Bf16) ? kTc5ExtraSmemBytes
                                                                               : lane_smem_bytes(iteration_split(nx, ny));
  return kGroupSmemBytes + 8192 * 4 + 8192 * 8 + extra;
}

cudaError_t iteration_occupancy(int nx, int ny, int* blocks_per_sm, int tc_mode) {
  const void* k = kernel_for(nx, ny, tc_mode);
  if (k == nullptr) return cudaErrorInvalidValue;
  const size_t smem = iteration_smem_bytes(nx, ny, tc_mode);
  // The general kernel serves every size: allow its largest request, so that
  // contexts of different sizes do not undo each other's setting.
  const size_t allow = (uses_general(nx, ny) && !uses_rg(nx, ny)) ? kGenSmemLimit : smem;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(allow));
  if (e != cudaSuccess) return e;
  if (const void* ks = iterate_kernel_slm(nx, ny, tc_mode)) {  // the same shared memory: one block per SM, as k
    e = cudaFuncSetAttribute(ks, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, iteration_threads(nx, ny, tc_mode), smem);
}

size_t mixed_smem_bytes(int tc_mode) {
  // mma.sync: one twiddle table per class, then the shared cos/sin table;
  // tcgen05: the matrices and twiddle tables of the three lengths
  const size_t extra = tc_mode == kTcMmaSync ? 3 * 32 * 32 * 8 + 32 * 8
                       : (tc_mode == kTcGen05F16 || tc_mode == kTcGen05Bf16) ? kMixedTc5ExtraSmemBytes
                                                                               : lane_smem_bytes(kMixedSplit);
  return kGroupSmemBytes + 8192 * 4 + 8192 * 8 + extra;
}

cudaError_t mixed_occupancy(int tc_mode, int* blocks_per_sm) {
  const void* k = iterate_kernel_mixed(tc_mode);
  const size_t smem = mixed_smem_bytes(tc_mode);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k, mixed_threads(tc_mode), smem);
}

cudaError_t launch_mixed(const MixedParams& mp, int grid, int tc_mode, cudaStream_t s) {
  void* args[] = {const_cast<MixedParams*>(&mp)};
  return cudaLaunchCooperativeKernel(iterate_kernel_mixed(tc_mode), dim3(grid), dim3(mixed_threads(tc_mode)), args,
                                     mixed_smem_bytes(tc_mode), s);
}

cudaError_t launch_iterations(const Params& p, int grid, cudaStream_t s) {
  const void* k = p.p_slm != nullptr ? iterate_kernel_slm(p.nx, p.ny, p.tensor_core) : nullptr;
  if (k == nullptr) k = kernel_for(p.nx, p.ny, p.tensor_core);
  if (k == nullptr) return cudaErrorInvalidValue;
  void* args[] = {const_cast<Params*>(&p)};
  if (p.gen_teams > 0)
    return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(p.gen_teams << p.gen_team_log), args,
                                       gen_smem_bytes(p.nx, p.ny, p.gen_teams), s);
  const size_t smem = iteration_smem_bytes(p.nx, p.ny, p.tensor_core);
  return cudaLaunchCooperativeKernel(k, dim3(grid), dim3(iteration_threads(p.nx, p.ny, p.tensor_core)), args, smem, s);
}

}  // namespace gsk
