// gs_small.cuh -- Gerchberg-Saxton on small grids: one cluster of blocks per
// mask, the whole run in shared memory.
//
// For grids of power-of-two sides 32 ... 256 with at most 32768 pixels (64 x 64,
// 32 x 256, 128 x 256, ...) the field and the scaled amplitude fit in the
// shared memory of a few SMs, so a mask needs neither global round trips
// between passes nor grid barriers: the C blocks of a cluster run
// A0 -> A1 -> (A2, A3) x K -> A4 of Eq. (e:AP) alone, with a cluster barrier
// between passes, and a batch is one cluster per mask. Block r holds the
// columns [r nx/C, (r+1) nx/C) of the field between a row and a column pass,
// and the rows [r ny/C, (r+1) ny/C) between a column and a row pass: a pass
// reads its lines from its own shared memory and stores every result into the
// shared memory of the block that owns it in the next pass. Each row and
// column is transformed by the same group FFT (gs_fft.cuh) and projected by
// the same code (gs_project.cuh) as in the persistent kernel (gs_iterate.cuh),
// so the iterates agree bit for bit; only the order of the gap sums differs.
//
// What bounds it: on one SM a 64 x 64 pass is 1.9 us however its lanes are
// held (128 threads of 32 values, or 512 of 8: the exchanges fill the shared
// memory pipe where the chain of instructions no longer does). C blocks divide
// the exchanges; what is left is the chain of one line, the cluster barrier
// (510 cycles) and the remote stores (20 cycles per warp and store). A lane is
// four threads (GroupT), so that the 32 to 128 lanes of a block are 4 to 16
// warps. 20 iterations, before (one block up to 8192 pixels, the persistent
// kernel above) and now: 64 x 64 105 -> 96 us, 128 x 64 156 -> 105,
// 128 x 128 374 -> 112, 256 x 128 260 -> 167, eight masks of it 824 -> 168.
//
// Shared-memory layout of a block, every line contiguous with element e of
// local line l at l n + (e ^ rev4(l)) (rev4: bit reversal of the low four bits),
// which keeps the accesses of a half-warp (T lanes per line, 16/T lines) on
// distinct 8-byte banks: its rows (ny/C lines of nx), its columns (nx/C lines
// of ny), the amplitude of its columns (row stride ny + T_y), the groups'
// exchange buffers, the teams' split-exchange buffers.
#pragma once

#include <cfloat>
#include <cmath>

#include "gs.h"
#include "gs_fft.cuh"
#include "gs_internal.h"
#include "gs_project.cuh"
#include "gs_tma.cuh"

namespace gsk {

template <int LX, int LY>
struct SmallGeom {
  static constexpr int NX = 1 << LX;
  static constexpr int NY = 1 << LY;
  static constexpr int N = NX * NY;
  static constexpr int TX = NX >> 5;   // lanes per row transform
  static constexpr int TY = NY >> 5;   // lanes per column transform
  static constexpr int S = 4;          // threads per lane
  static constexpr int MLD = NY + TY;  // row stride of the amplitude
  static_assert(LX >= 5 && LY >= 5 && LX <= 8 && LY <= 8 && N <= kSmallMaxPixels, "small grids only");
  // C = 2^lc blocks
  __host__ __device__ static constexpr int lanes(int lc) { return (N >> 5) >> lc; }
  __host__ __device__ static constexpr int rows_at(int) { return 0; }
  __host__ __device__ static constexpr int cols_at(int lc) { return rows_at(lc) + (N >> lc) * 8; }
  __host__ __device__ static constexpr int amp_at(int lc) { return cols_at(lc) + (N >> lc) * 8; }
  __host__ __device__ static constexpr int ex_at(int lc) {
    return amp_at(lc) + (((NX >> lc) * MLD * 4 + 15) / 16) * 16;
  }
  __host__ __device__ static constexpr int split_at(int lc) { return ex_at(lc) + lanes(lc) * 33 * 8; }
  __host__ __device__ static constexpr int smem(int lc) { return split_at(lc) + lanes(lc) * split_values(S) * 8; }
  __device__ static int rev4(int l) { return static_cast<int>(__brev(static_cast<unsigned>(l)) >> 28); }
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// The address of this block's shared-memory location `a` in block `rank` of
// the cluster.
__device__ __forceinline__ unsigned map_rank(unsigned a, unsigned rank) {
  unsigned d;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(rank));
  return d;
}

__device__ __forceinline__ void st_cluster(unsigned a, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster(unsigned a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// Every thread of every block of the cluster; their shared-memory writes
// before it are seen after it.
__device__ __forceinline__ void cluster_sync(int lc) {
  if (lc == 0) {
    __syncthreads();
  } else {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

enum SmallPass { kSmallInit = 0, kSmallRow = 1, kSmallCol = 2, kSmallResid = 3 };

// One pass over this block's lines of length 2^LN, one per group: A1
// (kSmallInit, the rows of u0 = exp(i phi0)), A2 (kSmallCol), A3 (kSmallRow) or
// A4's final residual (kSmallResid, columns). The transforms of a line go
// through one rolled loop and a square grid serves every kind with one
// instantiation, so that the kernel holds a single copy of the unrolled FFT: a
// body with four copies spent most of its time waiting for instructions.
// ROWS / COLS: the kinds this instantiation serves. Returns this thread's
// share of the pass's gap sum.
template <int LX, int LY, int LN, bool ROWS, bool COLS>
__device__ __forceinline__ float small_pass(const Params& p, size_t moff, int kind, bool last, int lc, int rank,
                                            unsigned char* smem, const StageTw<LN, SmallGeom<LX, LY>::S>& stw) {
  using Gm = SmallGeom<LX, LY>;
  using G = GroupT<LN, Gm::S>;
  static_assert(!ROWS || LN == LX, "row transforms have length nx");
  static_assert(!COLS || LN == LY, "column transforms have length ny");
  constexpr int N = G::N;
  constexpr int V = G::V;
  constexpr int STEP = G::STEP;
  const bool rows = ROWS && (!COLS || kind == kSmallRow || kind == kSmallInit);
  const int o = lane_of<Gm::S>();
  const int line = o / G::T;  // local
  G grp;
  grp.t = o & (G::T - 1);
  grp.c = lane_part<Gm::S>();
  grp.bar_id = 1 + o / 32;  // T <= 8: a team is a warp's lanes
  grp.sm = reinterpret_cast<float2*>(smem + Gm::ex_at(lc)) + line * G::SMEM;
  grp.sx = reinterpret_cast<float2*>(smem + Gm::split_at(lc)) + (o / 32) * G::SPLIT + (o & 31);
  grp.tw = rows ? p.twx : p.twy;
  const int t0 = grp.first();
  float2* const src = reinterpret_cast<float2*>(smem + (rows ? Gm::rows_at(lc) : Gm::cols_at(lc))) + line * N;
  const int sw = Gm::rev4(line);
  // lines of the other direction in a block, and this line's index in the grid
  const int log_other = (rows ? LX : LY) - lc;
  const int gline = (rank << ((rows ? LY : LX) - lc)) + line;
  // a pass that ends the run without the final residual stops after the projection
  const int nh = (kind == kSmallInit || kind == kSmallResid || (rows && last && !p.final_resid)) ? 1 : 2;
  float2* const su = grp.sm + t0;  // this thread's elements of the exchange buffer
  float2 v[V];
  if (kind == kSmallInit) {
    const float* ph = p.phi_in + moff + static_cast<size_t>(gline) * N + t0;
#pragma unroll 4
    for (int i = 0; i < V; ++i) {
      float s, c;
      sincosf(ph[STEP * i], &s, &c);
      su[STEP * i] = make_float2(c, s);  // u0 = exp(i phi0)
    }
    // zero iterations: arg exp(i phi0)
    if (last) phase_out<V, STEP>(p.phi_out + moff + static_cast<size_t>(gline) * N + t0, su);
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = su[STEP * i];
    grp.sync();  // the buffer is reused by the transform's exchange
  } else {
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = src[(t0 + STEP * i) ^ sw];
  }
  float part = 0.f;
#pragma unroll 1
  for (int h = 0; h < nh; ++h) {
    group_fft<LN>(v, grp, stw);
    if (h != 0) continue;
    if (!rows) {
      // v = Y = F u^nu along this column: residual and Eq. (e:Mhat)
      const float* const m = reinterpret_cast<const float*>(smem + Gm::amp_at(lc)) + line * Gm::MLD + t0;
      project<kProjTarget, V>(v, p.inv_sqrt_n, m, STEP, part);
    } else if (kind == kSmallRow) {
      // v = swap(IDFT_x(B)) = swap(sqrt(N) P_M u^nu): gap to S and Eq. (e:PS)
      project<kProjUnit, V>(v, p.inv_sqrt_n, nullptr, 0, part);
      if (last) {  // through the exchange buffer: a rolled loop holds the only copy of atan2f
        grp.sync();  // the transform has read the buffer
#pragma unroll
        for (int i = 0; i < V; ++i) su[STEP * i] = v[i];
        phase_out<V, STEP>(p.phi_out + moff + static_cast<size_t>(gline) * N + t0, su);
        grp.sync();
      }
    }
  }
  if (nh == 2 || kind == kSmallInit) {
    // element e of this line is element `gline` of line e of the other
    // direction, in block e >> log_other
    const int dst = rows ? Gm::cols_at(lc) : Gm::rows_at(lc);
    const int nd = rows ? Gm::NY : Gm::NX;
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const int e = t0 + STEP * i;
      const int l = e & ((1 << log_other) - 1);
      unsigned char* const at = smem + dst + (l * nd + (gline ^ Gm::rev4(l))) * 8;
      if (lc == 0) *reinterpret_cast<float2*>(at) = v[i];
      else st_cluster(map_rank(smem_u32(at), e >> log_other), v[i]);
    }
  }
  return part;
}

constexpr int kSmallMaxThreads = 512;

template <int LX, int LY>
__global__ void __launch_bounds__(kSmallMaxThreads, 1) gs_small(const Params p) {
  using Gm = SmallGeom<LX, LY>;
  constexpr int S = Gm::S;
  constexpr int kWarps = kSmallMaxThreads / 32;
  constexpr int kC = 1 << kSmallMaxLogC;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[kWarps];
  __shared__ double totals[kC];      // the blocks' shares of sum I
  __shared__ float redf[2][kWarps];
  __shared__ float gaps[4][kC];      // block 0: the blocks' gap sums of a pass
  const int lc = p.small_logc;
  const int C = 1 << lc;
  const int rank = lc == 0 ? 0 : static_cast<int>(cluster_rank());
  const int nt = blockDim.x, nw = nt >> 5;
  const int mb = blockIdx.x >> lc;
  const size_t moff = static_cast<size_t>(mb) * static_cast<size_t>(p.mstride);
  const float* I = p.I + moff;
  double* r_out = p.r_out ? p.r_out + static_cast<size_t>(mb) * p.rstride : nullptr;
  double* g_out = p.g_out ? p.g_out + static_cast<size_t>(mb) * p.gstride : nullptr;
  const double energy = static_cast<double>(Gm::N);  // sum p^2 with p = 1

  // A0: sum I in FP64, each block a share; a non-finite or negative pixel
  // poisons it with NaN
  double acc = 0.0;
  bool bad = false;
  const int share = Gm::N >> lc;  // 32 values per lane, 8 per thread
  constexpr int kPer = 32 / S;
  {
    float x[kPer];  // every load in flight
#pragma unroll
    for (int u = 0; u < kPer; ++u) x[u] = I[rank * share + threadIdx.x + u * nt];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      bad |= !(x[u] >= 0.f && x[u] <= FLT_MAX);
      acc += static_cast<double>(x[u]);
    }
  }
  if (__syncthreads_or(bad)) acc = __longlong_as_double(0x7ff8000000000000ll);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  // every block has started: its shared memory may be written from here on
  cluster_sync(lc);
  if (threadIdx.x < C) {
    double t = 0.0;
    for (int w = 0; w < nw; ++w) t += red[w];
    if (lc == 0) totals[0] = t;
    else st_cluster(map_rank(smem_u32(&totals[rank]), threadIdx.x), t);
  }
  cluster_sync(lc);
  double total = 0.0;
  for (int k = 0; k < C; ++k) total += totals[k];
  if (!(total > 0.0) || !(total <= DBL_MAX)) {
    // rejected (in every block): phase untouched, gaps NaN, GS_ENUMERIC
    if (rank != 0) return;
    if (threadIdx.x == 0) atomicCAS(p.status, 0, GS_ENUMERIC);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    if (r_out)
      for (int e = threadIdx.x; e < p.iters + (p.final_resid ? 1 : 0); e += nt) r_out[e] = nan;
    if (g_out)
      for (int e = threadIdx.x; e < p.iters; e += nt) g_out[e] = nan;
    return;
  }
  const float s = static_cast<float>(sqrt(energy / total));
  {  // m of this block's columns
    float* const m = reinterpret_cast<float*>(smem + Gm::amp_at(lc));
    const int log_cols = LX - lc;
    float v[kPer];
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int e = threadIdx.x + u * nt;
      v[u] = I[(e >> log_cols) * Gm::NX + (rank << log_cols) + (e & ((1 << log_cols) - 1))];
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
      const int e = threadIdx.x + u * nt;
      m[(e & ((1 << log_cols) - 1)) * Gm::MLD + (e >> log_cols)] = s * sqrtf(v[u]);
    }
  }
  // stage twiddles of both lengths, held for the whole run
  StageTw<LX, S> twr;
  twr.load(p.twx, lane_of<S>() & (Gm::TX - 1), lane_part<S>());
  StageTw<LY, S> twc;
  twc.load(p.twy, lane_of<S>() & (Gm::TY - 1), lane_part<S>());
  __syncthreads();

  const int K = p.iters;
  const int npass = 1 + 2 * K + (p.final_resid ? 1 : 0);
  // The gap of pass q > 0, from the blocks' sums in block 0 (one thread): the
  // raw sum, the normalisation follows after the loop.
  auto put_gap = [&](int q) {
    double t = 0.0;
    for (int k = 0; k < C; ++k) t += static_cast<double>(gaps[q & 3][k]);
    double* const out = (q & 1) ? r_out : g_out;  // the column passes are odd
    if (out) out[(q - 1) >> 1] = t;
  };
  // pass 0: the start; then the column pass of iteration (q - 1)/2 (q odd) or
  // its row pass (q even); at the end the final residual
#pragma unroll 1
  for (int q = 0; q < npass; ++q) {
    const int kind = q == 0 ? kSmallInit : q > 2 * K ? kSmallResid : (q & 1) ? kSmallCol : kSmallRow;
    const bool last = q == 2 * K;
    float a;
    if constexpr (LX == LY) {
      a = small_pass<LX, LY, LX, true, true>(p, moff, kind, last, lc, rank, smem, twr);
    } else {
      a = (kind == kSmallInit || kind == kSmallRow)
              ? small_pass<LX, LY, LX, true, false>(p, moff, kind, last, lc, rank, smem, twr)
              : small_pass<LX, LY, LY, false, true>(p, moff, kind, last, lc, rank, smem, twc);
    }
    // FP32 within the block (a warp's FP64 shuffles would run on the FP64 pipe,
    // 1/64 of the FP32 rate here). One thread adds the warps' totals beside
    // the next pass and hands them to block 0, which adds the blocks' one pass
    // later still. (Forming the warps' totals between the arrival and the wait
    // of the barrier takes a __syncthreads and was slower: 64 x 64 96 -> 104 us.)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if ((threadIdx.x & 31) == 0) redf[q & 1][threadIdx.x >> 5] = a;
    cluster_sync(lc);  // the pass's writes are seen by the next pass
    if (threadIdx.x == nt - 32) {
      float t = 0.f;
      for (int w = 0; w < nw; ++w) t += redf[q & 1][w];
      if (lc == 0) gaps[q & 3][0] = t;
      else st_cluster(map_rank(smem_u32(&gaps[q & 3][rank]), 0), t);
      if (rank == 0 && q > 1) put_gap(q - 1);
    }
  }
  cluster_sync(lc);
  if (rank != 0) return;
  if (threadIdx.x == 0 && npass > 1) put_gap(npass - 1);
  __syncthreads();  // the sums are visible to the block
  const int nr = K + (p.final_resid ? 1 : 0);
  if (r_out)
    for (int e = threadIdx.x; e < nr; e += nt) r_out[e] = sqrt(r_out[e] / energy);
  if (g_out)
    for (int e = threadIdx.x; e < K; e += nt) g_out[e] = sqrt(g_out[e] / energy);
}

}  // namespace gsk
