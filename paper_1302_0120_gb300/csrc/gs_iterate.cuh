// gs_iterate.cuh -- the persistent Gerchberg-Saxton iteration kernel for sm_103a.
//
// The kernel is a template on (log2 nx, log2 ny) and on where the transforms
// run: the FP32 ALUs (gs_fft.cuh; gs_inst.cu instantiates every size) or the
// tensor cores (gs_tc.cuh; gs_tc_inst.cu, square 256, 512 and 1024).
//
// One cooperative launch runs a whole run (or a chunk of up to 128 iterations)
// of Eq. (e:AP), u^{nu+1} = P_S P_M u^nu, as a sequence of passes over the
// field separated by grid barriers:
//
//   A0  sum of I (FP64) -> m = sqrt(I) sqrt(N / sum I), stored transposed
//       (Eq. pattern-constraint: m is the OSP amplitude)
//   A1  init rows:   u^0 = exp(i phi^0), B = DFT_x(u^0)
//   per iteration nu:
//   A2  column pass: Y = DFT_y(B) = F u^nu; r^nu from | |Y|/sqrt(N) - m |;
//                    Yhat = m Y/|Y| (Eq. e:Mhat); B = IDFT_y(Yhat)
//   A3  row pass:    v = IDFT_x(B) = sqrt(N) P_M u^nu (Eq. e:PM); g^nu from
//                    | |v|/sqrt(N) - 1 |; u = v/|v| (Eq. e:PS); B = DFT_x(u)
//                    (the last one writes phi = arg u instead, and B too when
//                    the final residual is requested)
//   A4  column pass, forward only: r^K.
//
// Each pass keeps a row (or column) in the registers of one thread group
// (gs_fft.cuh) from the moment it is loaded to the moment it is stored, so one
// iteration reads and writes the field exactly twice. Columns are staged
// through shared memory so that global accesses stay coalesced. Only forward
// transforms are issued: the inverse transforms are obtained by swapping
// real and imaginary parts, which is folded into the projections, so B holds
// swap(IDFT_y(Yhat)) between a column pass and the next row pass.
//
// FP64 is used only for the sums of the target energy and, across blocks, of the
// two gaps (FP32 within a block); the field is FP32.
#pragma once

#include <cfloat>
#include <cmath>
#include <type_traits>

#include "gs.h"
#include "gs_common.cuh"
#include "gs_fft.cuh"
#include "gs_general.cuh"
#include "gs_rg.cuh"
#include "gs_internal.h"
#include "gs_project.cuh"
#include "gs_tc.cuh"
#include "gs_tc5.cuh"
#include "gs_tma.cuh"

namespace gsk {

// Tensor-core kernels only: the block's stage twiddles and cos/sin table.
constexpr int kTcTwOffset = kBlockSmemOffset + kBlockSmemBytes;
constexpr int kTcCsOffset = kTcTwOffset + kTcTwBytes;
static_assert(kTcTwBytes + kTcCsBytes == kTcExtraSmemBytes, "tensor-core tables match the launch size");

// Stands in for TcFft in the kernels whose transforms run on the FP32 ALUs,
// S threads per lane; AHEAD: the kernel has the second staging buffer; SLM: the
// kernel of runs under a laser amplitude (iterate_kernel_slm).
template <int S, bool AHEAD = S == 1, bool SLM = false>
struct NoTc {
  static_assert(!SLM || AHEAD, "the laser amplitude takes the second staging buffer");
  static constexpr int kThreadsPerLane = S;
  static constexpr bool kAhead = AHEAD;
  static constexpr bool kSlm = SLM;
  static constexpr bool kEnabled = false;
  static constexpr bool kTcgen05 = false;
};

// Column blocks of the next round are loaded during a round.
template <class TCF>
__host__ __device__ constexpr bool loads_ahead() {
  if constexpr (TCF::kEnabled) return false;
  else return TCF::kAhead;
}

template <class TCF>
__host__ __device__ constexpr bool slm_kernel() {
  if constexpr (TCF::kEnabled) return false;
  else return TCF::kSlm;
}

// Threads per lane of a kernel whose transforms are TCF's.
template <class TCF>
__host__ __device__ constexpr int lane_threads() {
  if constexpr (TCF::kEnabled) return 1;
  else return TCF::kThreadsPerLane;
}

// Storage of the field B between passes: column blocks of W adjacent columns,
// each block one contiguous [ny][W] array, with the W elements of each of its
// rows permuted by an XOR swizzle. A column pass moves a whole block with one
// bulk copy each way and reads its columns from shared memory without bank
// conflicts; a row pass reads and writes 8W-byte row segments.
//
// P column blocks are in flight per round of a column pass: P = 2 (4) when a
// block of W = 8 columns fills only a half (a quarter) of the thread block
// (512-point, 256-point columns). Each slot of the threads then loads,
// transforms and stores its own column block on its own mbarrier, so that all
// threads work and the copies of one slot overlap the transforms of the
// others. (Blocks of 4 columns for
// 1024-point columns, two per round, were measured slower: the column pass
// gained 0.26 us, but the row pass, now reading 32-byte segments from twice
// as many lines, lost 0.5 us.) PMAX bounds P: 1 for the loss kernel, 2 for
// tcgen05, where the warps of a half of the block (a slot, then) issue their
// products together and must go through the rounds together.
__host__ __device__ constexpr int cmin(int a, int b) { return a < b ? a : b; }

template <int LX, int LY, int PMAX = kMaxSlots>
struct FieldLayout {
  static constexpr int NX = 1 << LX;
  static constexpr int NY = 1 << LY;
  static constexpr int TY = NY >> 5;          // threads per column transform
  static constexpr int NGY = kThreads / TY;   // column groups per block
  static constexpr int W = cmin(cmin(8, TY), cmin(NGY, NX));
  // blocks in flight per round
  static constexpr int P = (W == 8 && W * TY * PMAX >= kThreads) ? kThreads / (W * TY) : 1;
  // A round of a column pass may keep the next round's blocks in flight in a
  // second staging buffer: every lane owns a column.
  static constexpr bool kAhead = W * TY * P == kThreads;
  static constexpr int LW = ilog2(W);
  static constexpr int S = (W == 1) ? 0 : ilog2(16 / W);
  static constexpr int NBLK = NX / W;
  static constexpr int BLOCK = NY * W;        // elements of one column block
  static_assert(P * BLOCK <= 8192, "the column blocks in flight fit the staging buffer");
  static_assert(P == 1 || W * TY * P == kThreads, "the slots share out the block");
  __device__ static constexpr int swz(int y) { return W > 1 ? ((y >> S) & (W - 1)) : 0; }
  // element (row y, column x) of the field
  __device__ static size_t off(int y, int x) {
    return static_cast<size_t>(x >> LW) * BLOCK + y * W + ((x & (W - 1)) ^ swz(y));
  }
  // element (row y, column k) inside one block
  __device__ static int boff(int y, int k) { return y * W + (k ^ swz(y)); }
};

// One pass over rows [lo, hi) (kInit, kRow; LOGN = log2 nx) or column blocks
// [lo, hi) (kCol, kResid, kInitM; LOGN = log2 ny) of mask mb. Returns this
// thread's contribution to the pass's gap sum (FP32: the lines it holds).
//
// Square grids run rows and columns through this one function body, so that
// the kernel holds a single copy of the unrolled transform (see project).
template <int LOGN, int LX, int LY, bool HOLD, class TCF>
__device__ __forceinline__ float run_pass(const Params& p, int mb, int kind, bool last, int lo, int hi,
                                           unsigned char* smem, Shared& sh, unsigned& mphase,
                                           const StageTw<LOGN, lane_threads<TCF>()>& tw_rows, const TCF& tcf) {
  // this mask's arrays
  const size_t moff = static_cast<size_t>(mb) * static_cast<size_t>(p.mstride);
  float2* const Bm = p.B + moff;
  const float* const mTm = p.mT + moff;
  constexpr int S = lane_threads<TCF>();  // threads per lane
  constexpr int THR = kThreads * S;
  using G = GroupT<LOGN, S>;
  using L = FieldLayout<LX, LY, TCF::kTcgen05 ? 2 : kMaxSlots>;
  constexpr int N = G::N;
  constexpr int T = G::T;
  constexpr int V = G::V;        // elements per thread: t0 + STEP i
  constexpr int STEP = G::STEP;
  constexpr int LOGT = LOGN - 5;
  constexpr int LOGNG = 8 - LOGT;  // log2(kThreads / T)
  constexpr int NG = 1 << LOGNG;   // groups per block
  constexpr bool kRows = LOGN == LX, kCols = LOGN == LY;  // the passes this instantiation serves
  static_assert(kRows || kCols, "lines are rows or columns");
  static_assert(kThreads == 256, "geometry assumes 256 lanes");
  const bool rows = kRows && (!kCols || kind == kInit || kind == kRow);
  const int o = lane_of<S>();  // this thread's lane of the block
  const int g = o >> LOGT;
  G grp;
  grp.t = o & (T - 1);
  grp.c = lane_part<S>();
  grp.bar_id = 1 + (S == 1 ? g : o / G::TT);
  grp.sm = reinterpret_cast<float2*>(smem) + g * G::SMEM;
  grp.sx = S == 1 ? nullptr
                  : reinterpret_cast<float2*>(smem + kSplitSmemOffset) + (o / G::TT) * G::SPLIT + (o & (G::TT - 1));
  grp.tw = rows ? p.twx : p.twy;
  const int t0 = grp.first();
  // stage twiddles: the kernel's register copy for square grids, else
  // loaded once for this pass
  StageTw<LOGN, S> tw_own;
  if constexpr (!HOLD && !TCF::kEnabled) tw_own.load(grp.tw, grp.t, grp.c);
  const StageTw<LOGN, S>& stw = [&]() -> const StageTw<LOGN, S>& {
    if constexpr (HOLD) return tw_rows;
    else return tw_own;
  }();
  float* ms = reinterpret_cast<float*>(smem + kAmpSmemOffset);
  float2* blk = reinterpret_cast<float2*>(smem + kBlockSmemOffset);
  const bool from_m = kind == kInitM;  // transform m itself (the target start)
  const int nfft = (kind == kCol || (kind == kRow && !(last && !p.final_resid))) ? 2 : 1;
  const float inv_sqrt_n = p.inv_sqrt_n;
  float acc = 0.f;
  // Tensor-core transforms: this mask's power-of-two operand scales.
  float tc_in = 1.f, tc_out = 32.f;
  if constexpr (TCF::kEnabled) tc_scales(p.nx > p.ny ? p.nx : p.ny, energy_of(p), tc_in, tc_out);
  // One forward transform of the group's vector: on the FP32 ALUs, on the
  // tensor cores through the warp's slice of the exchange buffers (mma.sync),
  // or on the tensor cores of the block's half (tcgen05, all warps at once).
  auto fft = [&](float2(&x)[V]) {
    if constexpr (TCF::kTcgen05) {
      tcf.run(x, tc_in, tc_out);
    } else if constexpr (TCF::kEnabled) {
      tcf.run(x, smem + (threadIdx.x >> 5) * kTcWarpBytes, tc_in, tc_out);
    } else {
      group_fft<LOGN>(x, grp, stw);
    }
  };
  // the first line of the threads that transform together: of this warp's
  // team, or (tcgen05) of this half of the block
  const int g_first = (TCF::kTcgen05 ? ((o >> 7) << 7) : (o & ~31)) >> LOGT;

  // Column passes: P column blocks (W columns, N = ny rows each) per round,
  // one per slot of THR / P threads.
  constexpr int W = L::W;
  constexpr int P = L::P;
  constexpr int ST = THR / P;           // threads of a slot
  constexpr int GS = kThreads / P / T;  // groups of a slot
  const int slot = P > 1 ? o / (kThreads / P) : 0;
  const int gl = g - slot * GS;                           // group within the slot
  const bool gact = gl < W;                               // this group owns a column
  const int gq = gact ? gl : 0;                           // idle groups read a valid column
  const bool leader = (threadIdx.x & (ST - 1)) == 0;      // issues the slot's copies
  const int bi = P - 1 + slot;                            // index of the slot's mbarrier
  uint64_t* const mbar = &sh.mbar_s[bi];
  const unsigned pbit = 2u << bi;                         // this mbarrier's phase bit in mphase
  float* const msl = ms + slot * L::BLOCK;                // the slot's amplitude block
  float2* bsl = blk + slot * L::BLOCK;                    // the slot's field block
  // the slot's threads only (the whole block when P == 1)
  auto slot_sync = [&]() {
    if constexpr (P > 1) asm volatile("bar.sync %0, %1;" ::"r"(12 + slot), "n"(ST) : "memory");
    else __syncthreads();
  };
  // Rounds after the first find their column block loaded: while a round
  // transforms one staging buffer, the next round's block lands in the other
  // (which the store of the round before last has left), and each warp's
  // amplitude columns are replaced as soon as the warp has projected.
  const bool ahead = L::kAhead && loads_ahead<TCF>() && !rows && !from_m;
  // Start the copy of column block cb to the slot's field block `to`, and of
  // `bytes_m` amplitude bytes that complete on the same phase (leader only).
  auto load_block = [&](int cb, float2* to, unsigned par, unsigned bytes_m) {
    bulk_wait_read_all();  // a previous bulk store has read the destination
    fence_proxy_async_smem();
    mbar_arrive_expect_tx(mbar, (from_m ? 0u : L::BLOCK * 8u) + bytes_m);
    if (!from_m) bulk_g2s(to, Bm + static_cast<size_t>(cb) * L::BLOCK, L::BLOCK * 8u, mbar);
    sh.m_slot[slot] = mTm + static_cast<size_t>(cb) * L::BLOCK;
    sh.pend_s[bi] = 1;
    sh.pend_phase_s[bi] = par;
  };
  if (!rows && sh.m_layout != P) {  // no amplitude block of another layout stays resident
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int s = 0; s < kMaxSlots; ++s) sh.m_slot[s] = nullptr;
      sh.m_layout = P;
    }
    __syncthreads();
  }
  // Row passes of several rounds fetch the next round's rows (16-byte pieces)
  // into the field staging buffer behind the transforms of this round; a
  // group's row sits at its own N elements of the buffer.
  constexpr bool kSlm = slm_kernel<TCF>();
  const bool fetch = !TCF::kEnabled && L::W >= 2 && kind == kRow && (kSlm || p.p_slm == nullptr);
  float2* const next_row = blk + g * N;
  // the laser amplitude of a row, at this thread's elements (in the field
  // staging buffer, free in row passes; in the second one where the first
  // holds the next rows)
  float* const sp = reinterpret_cast<float*>(kSlm ? blk + kBlockElems : blk) + threadIdx.x;

  for (int u0 = lo; u0 < hi; u0 += rows ? NG : P) {
    const int idx = rows ? u0 + g : u0 + slot;  // this group's row, or this slot's column block
    float2 v[V];
    bool work;   // this warp transforms a line in this round
    bool valid;  // ... and this group's is its own (the others work on a valid copy and store nothing)
    if (rows) {
      // Warps without a row leave: transforming copies instead kept the whole
      // block's issue slots and shared memory busy (256 x 256: row pass 4.3 us
      // with 2 of 8 warps on rows of their own).
      if (u0 + g_first >= hi) break;
      work = true;
      valid = idx < hi;
      const int ridx = valid ? idx : u0;
      if (kind == kInit) {
        // exp(i phi) once per run: a rolled loop through the group's exchange
        // buffer keeps a single copy of sincosf (and atan2f) in the kernel.
        // phi (and p) arrive there first by cp.async, all loads in flight.
        const float* ph = p.phi_in + moff + static_cast<size_t>(ridx) * N + t0;
        float2* su = grp.sm + t0;
        if constexpr (S > 1) grp.sync();  // the previous round's transform has read the buffer
        const float* pp = p.p_slm ? p.p_slm + static_cast<size_t>(ridx) * N + t0 : nullptr;
        // rolled: the copies do not wait, so all of them are in flight anyway
#pragma unroll 1
        for (int i = 0; i < V; ++i) cp_async4(&su[STEP * i].x, ph + STEP * i);
        if (pp) {
#pragma unroll 1
          for (int i = 0; i < V; ++i) cp_async4(&su[STEP * i].y, pp + STEP * i);
        }
        cp_async_wait_all();
#pragma unroll 4
        for (int i = 0; i < V; ++i) {
          float s, c;
          const float2 fa = su[STEP * i];
          sincosf(fa.x, &s, &c);
          const float a = pp ? fa.y : 1.f;  // u0 = p exp(i phi0)
          su[STEP * i] = make_float2(a * c, a * s);
        }
        if (last && valid) phase_out<V, STEP>(p.phi_out + moff + static_cast<size_t>(idx) * N + t0, su);
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] = su[STEP * i];
        grp.sync();
      } else {
        if (fetch && u0 != lo) {
          cp_async_wait_all();
          grp.sync();
          const int flip = L::swz(ridx) & 1;
#pragma unroll
          for (int i = 0; i < V; ++i) v[i] = next_row[STEP > 1 ? (t0 ^ flip) + STEP * i : (t0 + i) ^ flip];
          grp.sync();
        } else {
#pragma unroll
          for (int i = 0; i < V; ++i) v[i] = Bm[L::off(ridx, t0 + STEP * i)];
        }
        if (fetch && u0 + NG + g_first < hi) {
          const int nidx = idx + NG;
          const int nrow = nidx < hi ? nidx : u0 + NG;
          // elements x, x + 1 (x even) are 16 bytes of a row segment, in this
          // order when the row's swizzle is even
          const int sw = L::swz(nrow) & ~1;
#pragma unroll 4
          for (int i = 0; i < V / 2; ++i) {
            const int x = 2 * (T * S * i + T * grp.c + grp.t);
            cp_async16(next_row + x, Bm + static_cast<size_t>(x >> L::LW) * L::BLOCK + nrow * L::W +
                                         ((x & (L::W - 1)) ^ sw));
          }
        }
        if (kind == kRow && p.p_slm != nullptr) {
          // the laser amplitude of this row, prefetched behind the first transform
          const float* pp = p.p_slm + static_cast<size_t>(ridx) * N + t0;
#pragma unroll 1
          for (int i = 0; i < V; ++i) cp_async4(sp + THR * i, pp + STEP * i);
        }
      }
    } else {
      if (idx >= hi) break;  // no block left for this slot
      work = g_first - slot * GS < W;
      valid = gact;
      const unsigned par = (mphase & pbit) ? 1u : 0u;
      if (ahead) bsl = blk + slot * L::BLOCK + (((u0 - lo) / P) & 1) * kBlockElems;
      if (!ahead || u0 == lo) {
        slot_sync();  // the previous round is done with this slot's staging buffers
        if (leader) {
          // columns idx W .. idx W + W - 1 of m are contiguous in the transposed
          // amplitude; a block that stays resident is identified by its global
          // address, unique across masks and size classes
          const float* const msrc = mTm + static_cast<size_t>(idx) * L::BLOCK;
          const unsigned bytes_m = sh.m_slot[slot] != msrc ? L::BLOCK * 4u : 0u;
          load_block(idx, bsl, par, bytes_m);
          if (bytes_m) bulk_g2s(msl, msrc, bytes_m, mbar);
        }
      }
      const bool landed = mbar_wait_bounded(mbar, par);
      mphase ^= pbit;
      if (!landed) {
        fail(p, GS_ETIMEOUT);
      } else if (leader) {
        sh.pend_s[bi] = 0;
      }
      if (from_m) {
        // The target start transforms m itself: stage swap((m, 0)) in the field
        // layout, so the forward DFT below yields swap(IDFT_y(m)).
        for (int e = threadIdx.x & (ST - 1); e < L::BLOCK; e += ST) {
          const int k = e % W;
          const int y = e / W;
          bsl[L::boff(y, k)] = make_float2(0.f, msl[k * L::NY + y]);
        }
        slot_sync();
      }
      if (work) {
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] = bsl[L::boff(t0 + STEP * i, gq)];
      }
    }

    if (work) {
      float part = 0.f;
#pragma unroll 1
      for (int h = 0; h < nfft; ++h) {
        fft(v);
        if (h != 0) continue;
        if (rows) {
          if (kind != kRow) continue;
          // v = swap(IDFT_x(B)) = swap(sqrt(N) P_M u^nu). Gap to S and Eq. (e:PS).
          if (p.p_slm == nullptr) {
            project<kProjUnit, V>(v, inv_sqrt_n, nullptr, 0, part);
          } else {
            cp_async_wait_all();
            project<kProjSlm, V>(v, inv_sqrt_n, sp, THR, part);
          }
          if (last) {
            // The mask, once per run: through the group's exchange buffer so
            // that a rolled loop holds the only copy of atan2f.
            float2* su = grp.sm + t0;
            if constexpr (S > 1) grp.sync();  // the transform has read the buffer
#pragma unroll
            for (int i = 0; i < V; ++i) su[STEP * i] = v[i];
            if (valid) phase_out<V, STEP>(p.phi_out + moff + static_cast<size_t>(idx) * N + t0, su);
            grp.sync();
          }
        } else if (!from_m) {
          // v = Y = F u^nu along this column. Residual and Eq. (e:Mhat); the
          // result is swapped, so the next forward DFT acts as the inverse
          // (kResid ends here and ignores it).
          project<kProjTarget, V>(v, inv_sqrt_n, msl + gq * N + t0, STEP, part);
          if (ahead && idx + P < hi) {
            // the next round's block; its amplitude columns replace those of
            // the lines that transform together, which have read theirs
            if (leader) {
              float2* const other = blk + slot * L::BLOCK + ((((u0 - lo) / P) & 1) ^ 1) * kBlockElems;
              load_block(idx + P, other, (mphase & pbit) ? 1u : 0u, L::BLOCK * 4u);
            }
            grp.sync();
            if ((o & (G::TT - 1)) == 0) {
              fence_proxy_async_smem();
              const int k = g_first - slot * GS;  // the team's first column
              bulk_g2s(msl + k * N, mTm + (static_cast<size_t>(idx + P) * W + k) * N, G::TT * 32 * 4u, mbar);
            }
          }
        }
      }
      if (valid) {
        acc += part;
        if (rows) {
          if (kind == kInit || nfft == 2) {
#pragma unroll
            for (int i = 0; i < V; ++i) Bm[L::off(idx, t0 + STEP * i)] = v[i];
          }
        } else if (kind != kResid) {
#pragma unroll
          for (int i = 0; i < V; ++i) bsl[L::boff(t0 + STEP * i, gl)] = v[i];
        }
      }
    }
    if (!rows && (kind != kResid || ahead)) {
      slot_sync();
      if (kind != kResid && leader) {
        fence_proxy_async_smem();
        bulk_s2g(Bm + static_cast<size_t>(idx) * L::BLOCK, bsl, L::BLOCK * 8u);
        bulk_commit();
      }
    }
  }
  // the field must be in global memory before the grid barrier releases the next pass
  if (!rows && kind != kResid && leader) bulk_wait_all();
  return acc;
}

// Before leaving after a failure, give a bulk copy that may still target this
// block's shared memory a bounded time to land.
static __device__ void drain_copies(Shared& sh) {
  if (threadIdx.x == 0 && sh.pending) mbar_wait_bounded(&sh.mbar, sh.pending_phase);
  if (threadIdx.x < kSlotBars && sh.pend_s[threadIdx.x])
    mbar_wait_bounded(&sh.mbar_s[threadIdx.x], sh.pend_phase_s[threadIdx.x]);
  __syncthreads();
}

// m = s sqrt(I) for this block's columns, written transposed ([nx][ny]) so
// that the column pass reads it contiguously.
static __device__ void build_amplitude(const Params& p, int mb, float s, unsigned char* smem) {
  const size_t moff = static_cast<size_t>(mb) * static_cast<size_t>(p.mstride);
  const float* const Im = p.I + moff;
  float* const mTm = p.mT + moff;
  const int logNG = 8 - (p.logny - 5);
  const int W = 1 << logNG;
  float* blk = reinterpret_cast<float*>(smem + kBlockSmemOffset);
  const int lo = split(blockIdx.x, gridDim.x, p.nx);
  const int hi = split(blockIdx.x + 1, gridDim.x, p.nx);
  for (int base = lo; base < hi; base += W) {
    const int wcur = min(W, hi - base);
    __syncthreads();
    // every copy of a thread in flight at once
    for (int e = threadIdx.x; e < p.ny * W; e += blockDim.x) {
      const int k = e & (W - 1);
      const int y = e >> logNG;
      if (k < wcur) cp_async4(blk + y * (W + 1) + k, Im + static_cast<size_t>(y) * p.nx + base + k);
    }
    cp_async_wait_all();
    __syncthreads();
#pragma unroll 4
    for (int e = threadIdx.x; e < wcur * p.ny; e += blockDim.x) {
      const int k = e >> p.logny;
      const int y = e & (p.ny - 1);
      mTm[static_cast<size_t>(base + k) * p.ny + y] = s * sqrtf(blk[y * (W + 1) + k]);
    }
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// The kernels. A launch iterates one or more *size classes*: each class is a
// Params (a batch of masks of one grid, with its own arrays and partial-sum
// region); all classes share the barrier, status and abort words and pass
// through the same schedule, one grid barrier per pass. Shared state of mask
// mb of a class lives at index base + mb of the block's Shared arrays.

// A0, part 1: this block's FP64 share of sum I for every mask of the class.
// A non-finite or negative pixel poisons the sum with NaN.
static __device__ __forceinline__ void a0_partials(const Params& p, Shared& sh) {
  const int G = gridDim.x;
  const int b = blockIdx.x;
  const int r0 = split(b, G, p.ny);
  const int r1 = split(b + 1, G, p.ny);
  const int cnt = (r1 - r0) * p.nx;
  for (int mb = 0; mb < p.batch; ++mb) {
    const float* I = p.I + static_cast<size_t>(mb) * static_cast<size_t>(p.mstride) + static_cast<size_t>(r0) * p.nx;
    double acc = 0.0;
    bool bad = false;
    constexpr int U = 8;  // loads in flight: one at a time, a 2048 x 2048 target took 50 us
    const int step = blockDim.x;
    for (int e0 = threadIdx.x; e0 < cnt; e0 += U * step) {
      float x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) x[u] = e0 + u * step < cnt ? I[e0 + u * step] : 0.f;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        bad |= !(x[u] >= 0.f && x[u] <= FLT_MAX);
        acc += static_cast<double>(x[u]);
      }
    }
    if (__syncthreads_or(bad)) acc = __longlong_as_double(0x7ff8000000000000ll);
    const double tot = block_sum(acc, sh);
    if (threadIdx.x == 0) p.partials[static_cast<size_t>(mb) * G + b] = tot;
  }
}

// A0, part 2 (after a grid barrier): validity and scale sqrt(sum p^2 / sum I)
// of every mask, the same in every block (each reduces the same partials in
// the same order). Rejected masks get NaN gaps and GS_ENUMERIC; they are
// skipped from then on. (The tensor-core forms keep their FP16 operands in
// range with a power-of-two scale per mask, tc_scales, so no energy is too
// large for them.) Returns the number of rejected masks.
static __device__ __forceinline__ int a0_scales(const Params& p, Shared& sh, int base) {
  const int b = blockIdx.x;
  if (threadIdx.x < 32) {
    for (int mb = 0; mb < p.batch; ++mb) {
      const double total = warp_slot_sum(p, mb);
      if (threadIdx.x == 0) {
        const double ep = energy_of(p);
        const bool bad = !(total > 0.0) || !(total <= DBL_MAX) || !(ep > 0.0) || !(ep <= DBL_MAX);
        sh.bad[base + mb] = bad ? 1 : 0;
        if (b == 0) p.mask_flags[mb] = bad ? 1 : 0;  // for later launches of the run
        sh.scale[base + mb] = bad ? 0.f : static_cast<float>(sqrt(ep / total));
      }
    }
  }
  __syncthreads();
  int nbad = 0;
  for (int mb = 0; mb < p.batch; ++mb) nbad += sh.bad[base + mb];
  if (nbad > 0 && b == 0) {
    // Masks with an invalid target are skipped: phase untouched, gaps NaN.
    if (threadIdx.x == 0) fail_status(p, GS_ENUMERIC);
    const double nan = __longlong_as_double(0x7ff8000000000000ll);
    const int nr = p.iters + (p.final_resid ? 1 : 0);
    for (int mb = 0; mb < p.batch; ++mb) {
      if (!sh.bad[base + mb]) continue;
      if (p.r_out)
        for (int e = threadIdx.x; e < nr; e += blockDim.x) p.r_out[static_cast<size_t>(mb) * p.rstride + e] = nan;
      if (p.g_out)
        for (int e = threadIdx.x; e < p.iters; e += blockDim.x) p.g_out[static_cast<size_t>(mb) * p.gstride + e] = nan;
    }
  }
  return nbad;
}

// Later launches of a run: the invalid masks were flagged by the first.
static __device__ __forceinline__ void restore_flags(const Params& p, Shared& sh, int base) {
  if (threadIdx.x == 0)
    for (int mb = 0; mb < p.batch; ++mb) sh.bad[base + mb] = p.mask_flags[mb];
}

template <int LX, int LY = LX>
__device__ __forceinline__ void build_amplitudes(const Params& p, Shared& sh, int base, unsigned char* smem) {
  for (int mb = 0; mb < p.batch; ++mb)
    if (!sh.bad[base + mb]) {
      if constexpr (LX == 0) gen_build_amplitude(p, mb, sh.scale[base + mb], smem);
      else if constexpr (is_rg_side(LX)) rg_build_amplitude<LX, LY>(p, mb, sh.scale[base + mb], smem);
      else build_amplitude(p, mb, sh.scale[base + mb], smem);
    }
}

// Pass q0 of the schedule [init] (col, row) x nit [resid]: its kind, whether
// it ends the run, and the partial-sum slot of its gap (-1: none). Pass q
// after the init passes sums into slot 1 + q.
struct PassInfo {
  int kind;
  int slot;
  bool last;
};

static __device__ __forceinline__ int pass_count(const Params& p) {
  const int nit = p.it1 - p.it0;
  const int resid = (p.do_final && p.final_resid) ? 1 : 0;
  const int ninit = p.do_init ? (p.init_target ? 2 : 1) : 0;  // target start: columns then rows
  return ninit + 2 * nit + resid;
}

static __device__ __forceinline__ PassInfo pass_info(const Params& p, int q0) {
  const int nit = p.it1 - p.it0;
  const int ninit = p.do_init ? (p.init_target ? 2 : 1) : 0;
  const int q = q0 - ninit;
  PassInfo f{kCol, -1, false};
  if (q < 0) {
    f.kind = !p.init_target ? kInit : (q == -2 ? kInitM : kRow);
    f.last = p.do_final && p.iters == 0 && q == -1;
  } else if (q < 2 * nit) {
    f.kind = (q & 1) ? kRow : kCol;
    f.slot = 1 + q;
    f.last = (f.kind == kRow) && p.do_final && (p.it0 + (q >> 1) == p.iters - 1);
  } else {
    f.kind = kResid;
    f.slot = 1 + q;
  }
  return f;
}

// One pass over the valid masks [w0, w1) of a class. The work units of those
// masks (rows, or column blocks) form one sequence split evenly over the
// blocks, so that small masks of a batch do not leave blocks idle; a block
// works through its share mask by mask and writes the FP64 partial of each
// mask's gap to its slot (zero for the masks it does not touch). With `late`
// the last mask's sum is left to the barrier that follows (grid_sync).
struct LateSum {
  float x = 0.f;
  double* to = nullptr;
};
template <int LX, int LY, bool HOLD, class TCF, class TW>
__device__ __forceinline__ LateSum class_pass(const Params& p, Shared& sh, int base, int w0, int w1,
                                              const PassInfo& f, bool late, unsigned char* smem, unsigned& mphase,
                                              const TW& tw_rows, const TCF& tcf) {
  LateSum left;
  const bool rows = (f.kind == kInit || f.kind == kRow);
  int per;  // units of one mask
  if constexpr (LX == 0) per = rows ? p.ny : p.nx;
  else if constexpr (is_rg_side(LX)) per = rows ? p.ny : LX / RgLayout<LX, LY>::W;
  else per = rows ? p.ny : FieldLayout<LX, LY>::NBLK;
  const int G = gridDim.x;
  int lo, hi, m0, m1;
  if (w1 - w0 == 1) {  // one mask: its own share, no mask boundaries
    lo = split(blockIdx.x, G, per);
    hi = split(blockIdx.x + 1, G, per);
    m0 = w0;
    m1 = w1;
  } else {
    const int total = per * (w1 - w0);
    lo = split(blockIdx.x, G, total);
    hi = split(blockIdx.x + 1, G, total);
    m0 = w0 + lo / per;
    m1 = w0 + (hi + per - 1) / per;  // masks [m0, m1) meet [lo, hi)
    if (f.slot >= 0 && threadIdx.x == 0)
      for (int mb = w0; mb < w1; ++mb)
        if (mb < m0 || mb >= m1) p.partials[(static_cast<size_t>(f.slot) * p.batch + mb) * G + blockIdx.x] = 0.0;
  }
  for (int mb = m0; mb < m1; ++mb) {
    if (sh.bad[base + mb]) continue;
    const int slo = max(lo, (mb - w0) * per) - (mb - w0) * per;
    const int shi = min(hi, (mb - w0 + 1) * per) - (mb - w0) * per;
    float a;
    if constexpr (LX == 0) {
      a = p.gen_team_log == 6 ? run_pass_gen<6>(p, mb, f.kind, f.last, slo, shi, smem)
                              : run_pass_gen<7>(p, mb, f.kind, f.last, slo, shi, smem);
    } else if constexpr (is_rg_side(LX)) {
      a = run_pass_rg<LX, LY>(p, mb, f.kind, f.last, slo, shi, smem, sh, mphase);
    } else if constexpr (LX == LY) {
      a = run_pass<LX, LX, LY, HOLD>(p, mb, f.kind, f.last, slo, shi, smem, sh, mphase, tw_rows, tcf);
    } else {
      const StageTw<LY, lane_threads<TCF>()> none{};
      a = rows ? run_pass<LX, LX, LY, false>(p, mb, f.kind, f.last, slo, shi, smem, sh, mphase, tw_rows, tcf)
               : run_pass<LY, LX, LY, false>(p, mb, f.kind, f.last, slo, shi, smem, sh, mphase, none, tcf);
    }
    if (f.slot >= 0) {
      double* const to = p.partials + (static_cast<size_t>(f.slot) * p.batch + mb) * G + blockIdx.x;
      if (late && mb == m1 - 1) {
        left.x = a;
        left.to = to;
      } else {
        const double tot = block_sum_f(a, sh);
        if (threadIdx.x == 0) *to = tot;
      }
    }
  }
  return left;
}

// Gaps: r from column passes, g from row passes, in FP64, for every valid
// mask of a class (block b reduces slots b, b + G, ...).
static __device__ __forceinline__ void final_gaps(const Params& p, Shared& sh, int base) {
  const int G = gridDim.x;
  const int nit = p.it1 - p.it0;
  const int resid = (p.do_final && p.final_resid) ? 1 : 0;
  const int nslots = 2 * nit + resid;
  if (threadIdx.x < 32) {
    for (int s = blockIdx.x; s < nslots * p.batch; s += G) {
      const int slot = 1 + s / p.batch;
      const int mb = s % p.batch;
      if (sh.bad[base + mb]) continue;
      const double sum = warp_slot_sum(p, slot * p.batch + mb);
      if (threadIdx.x == 0) {
        const double val = sqrt(sum / energy_of(p));
        const int q = slot - 1;
        if (q < 2 * nit) {
          const int nu = p.it0 + (q >> 1);
          if ((q & 1) == 0) {
            if (p.r_out) p.r_out[static_cast<size_t>(mb) * p.rstride + nu] = val;
          } else {
            if (p.g_out) p.g_out[static_cast<size_t>(mb) * p.gstride + nu] = val;
          }
        } else if (p.r_out) {
          p.r_out[static_cast<size_t>(mb) * p.rstride + p.iters] = val;
        }
      }
    }
  }
}

static __device__ __forceinline__ void block_setup(Shared& sh) {
  if (threadIdx.x == 0) {
    mbar_init(&sh.mbar, 1);
    for (int s = 0; s < kSlotBars; ++s) {
      mbar_init(&sh.mbar_s[s], 1);
      sh.pend_s[s] = 0;
    }
    fence_barrier_init();
    sh.pending = 0;
    sh.m_block = nullptr;
    for (int s = 0; s < kMaxSlots; ++s) sh.m_slot[s] = nullptr;
    sh.m_layout = 0;
  }
  __syncthreads();
}

// The schedule of one size class (every grid): A0, then the passes, then the
// gaps. Returns early (in every thread of the block) when a grid barrier gave
// up or every mask was rejected.
template <int LX, int LY, bool kHold, class TCF, class TW>
__device__ __forceinline__ void iterate_class(const Params& p, Shared& sh, unsigned char* smem,
                                              const TW& tw_rows, const TCF& tcf) {
  unsigned target = 0;
  unsigned mphase = 0;
  block_setup(sh);
  if constexpr (LX == 0) gen_load_twiddles(p, smem);  // sides that are not powers of two
  if constexpr (is_rg_side(LX)) rg_load_twiddles<LX, LY>(p, smem);

  if (p.do_init) {
    a0_partials(p, sh);
    if (!grid_sync(p, target, sh)) return;
    const int nbad = a0_scales(p, sh, 0);
    if (nbad == p.batch) {
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(p.abort_flag, 1);  // later launches of the run
      return;
    }
    build_amplitudes<LX, LY>(p, sh, 0, smem);
    // the target start transforms m in its first pass, reading columns that
    // other blocks built
    if (p.init_target && !grid_sync(p, target, sh)) return;
  } else {
    restore_flags(p, sh, 0);
  }
  __syncthreads();

  const int npass = pass_count(p);
  const int gsz = p.group > 0 ? p.group : p.batch;
  unsigned long long* const tr = (p.trace != nullptr && threadIdx.x == 0) ? p.trace + 2 * blockIdx.x : nullptr;
  if (tr) tr[0] = tr[1] = global_ns();
  for (int w0 = 0; w0 < p.batch; w0 += gsz) {  // mask groups, each through the whole schedule
    const int w1 = min(p.batch, w0 + gsz);
    for (int q0 = 0; q0 < npass; ++q0) {
      // the sums of the last pass are read right after its barrier
      const LateSum ls =
          class_pass<LX, LY, kHold>(p, sh, 0, w0, w1, pass_info(p, q0), q0 + 1 < npass, smem, mphase, tw_rows, tcf);
      // pass timestamps: work done, then released by the barrier
      unsigned long long* const trq = tr ? tr + static_cast<size_t>(2 * (1 + q0)) * gridDim.x : nullptr;
      if (trq) trq[0] = global_ns();
      if (!grid_sync(p, target, sh, ls.x, ls.to)) {
        drain_copies(sh);
        return;
      }
      if (trq) trq[1] = global_ns();
    }
  }
  final_gaps(p, sh, 0);
}

template <int LX, int LY, bool TC>
__host__ __device__ constexpr int kernel_split() {
  return (TC || LX == 0) ? 1 : iteration_split(1 << LX, 1 << LY);
}

// One size class per launch (every grid). SLM: iterate_kernel_slm.
template <int LX, int LY, bool TC = false, bool SLM = false>
__global__ void __launch_bounds__(LX == 0 ? kGenMaxThreads : kThreads * kernel_split<LX, LY, TC>(), 1) gs_iterate(const Params p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared sh;
  if (*reinterpret_cast<volatile int*>(p.abort_flag) != 0) return;  // an earlier chunk failed
  constexpr bool kHold = LX > 0 && LX == LY && !TC;
  constexpr int S = kernel_split<LX, LY, TC>();
  StageTw<LX, S> tw_rows;  // square grids: stage twiddles held for the whole run
  if constexpr (kHold) {
    tw_rows.load(p.twx, lane_of<S>() & ((1 << (LX - 5)) - 1), lane_part<S>());
  }
  // Tensor-core transforms: the block's tables, then the DFT-matrix fragments
  // held in registers for the whole run.
  static_assert(!TC || LX == LY, "tensor-core kernels are square");
  constexpr int kR = TC ? (1 << (LX > 5 ? LX - 5 : 0)) : 32;
  TcStage1 s1;
  TcStage2<kR> s2;
  const float2* tctw = reinterpret_cast<const float2*>(smem + kTcTwOffset);
  if constexpr (TC) {
    tc_build_tables<LX>(reinterpret_cast<float2*>(smem + kTcTwOffset), reinterpret_cast<float2*>(smem + kTcCsOffset));
    __syncthreads();
    s1.load(reinterpret_cast<const float2*>(smem + kTcCsOffset));
    s2.load(reinterpret_cast<const float2*>(smem + kTcCsOffset));
  }
  const auto tcf = [&]() {
    if constexpr (TC) return TcFft<LX>{s1, s2, tctw};
    else return NoTc<S, S == 1, SLM>{};
  }();
  iterate_class<LX, LY, kHold>(p, sh, smem, tw_rows, tcf);
}

// The tensor-core form on tcgen05 (square 256, 512, 1024): the same schedule
// with every transform issued by the block's halves as products on the
// tensor cores (gs_tc5.cuh). Warp 0 holds the block's TMEM columns from the
// start of the launch to its end, on every exit path.
constexpr int kTc5Offset = kBlockSmemOffset + kBlockSmemBytes;  // after the amplitude and field blocks

template <int L, bool BF16>
__global__ void __launch_bounds__(kThreads, 1) gs_iterate_tc5(const Params p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared sh;
  __shared__ uint64_t tc_mbar[2];
  __shared__ unsigned tc_tmem;
  if (*reinterpret_cast<volatile int*>(p.abort_flag) != 0) return;  // an earlier chunk failed
  static_assert(2 * kTc5HalfStride == kGroupSmemBytes, "the A operands fill the exchange area");
  unsigned char* abuf = smem;  // the exchange area (gs_tc5.cuh)
  unsigned char* tabs = smem + kTc5Offset;
  tc5_build_tables<L, BF16>(tabs, tabs + kTc5B2Offset, reinterpret_cast<float2*>(tabs + kTc5TwOffset));
  if (threadIdx.x == 0) {
    mbar_init(&tc_mbar[0], 1);
    mbar_init(&tc_mbar[1], 1);
    fence_barrier_init();
  }
  if ((threadIdx.x >> 5) == 0) tc5_alloc(&tc_tmem);
  fence_proxy_async_smem();  // the DFT matrices are read by the tensor cores
  tc5_fence_before();
  __syncthreads();
  tc5_fence_after();
  unsigned phase = 0;
  const Tc5Fft<L, BF16> tcf{abuf, smem_u32(tabs), smem_u32(tabs + kTc5B2Offset),
                            reinterpret_cast<const float2*>(tabs + kTc5TwOffset), tc_mbar, tc_tmem, &phase, &p};
  const StageTw<L> none{};
  iterate_class<L, L, false>(p, sh, smem, none, tcf);
  tc5_fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) tc5_dealloc(tc_tmem);
}

template <int C, bool TC>
__device__ __forceinline__ LateSum mixed_class_pass(const MixedParams& mp, Shared& sh, int w0, int w1,
                                                    const PassInfo& f, bool late, unsigned char* smem, unsigned& mphase, const TcStage1& s1,
                                                 const TcStage2<8 << C>& s2) {
  constexpr int L = 8 + C;
  const Params& p = mp.cls[C];
  const int base = (C > 0 ? mp.cls[0].batch : 0) + (C > 1 ? mp.cls[1].batch : 0);
  const StageTw<L, TC ? 1 : kMixedSplit> none{};
  if constexpr (TC) {
    const TcFft<L> tcf{s1, s2, reinterpret_cast<const float2*>(smem + kTcTwOffset + C * kTcTwBytes)};
    return class_pass<L, L, false>(p, sh, base, w0, w1, f, late, smem, mphase, none, tcf);
  } else {
    return class_pass<L, L, false>(p, sh, base, w0, w1, f, late, smem, mphase, none, NoTc<kMixedSplit>{});
  }
}

// The schedule of a mixed launch (the tcgen05 form; gs_iterate_mixed writes
// the same out): A0 for every class, then the classes one after the other,
// each (in mask groups) through the whole schedule of passes;
// `pass(c, w0, w1, f, mphase)` runs one pass of class c. Returns early when a
// barrier gave up or every mask was rejected.
template <class PassFn>
__device__ __forceinline__ void iterate_mixed(const MixedParams& mp, Shared& sh, unsigned char* smem, PassFn&& pass) {
  const Params& p0 = mp.cls[0];  // barrier, status, abort flag, schedule
  unsigned target = 0;
  unsigned mphase = 0;
  block_setup(sh);
  const int total = mp.cls[0].batch + mp.cls[1].batch + mp.cls[2].batch;
  const int base1 = mp.cls[0].batch, base2 = base1 + mp.cls[1].batch;

  if (p0.do_init) {
    for (int c = 0; c < 3; ++c) a0_partials(mp.cls[c], sh);
    if (!grid_sync(p0, target, sh)) return;
    const int nbad = a0_scales(mp.cls[0], sh, 0) + a0_scales(mp.cls[1], sh, base1) + a0_scales(mp.cls[2], sh, base2);
    if (nbad == total) {
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(p0.abort_flag, 1);
      return;
    }
    build_amplitudes<8>(mp.cls[0], sh, 0, smem);
    build_amplitudes<9>(mp.cls[1], sh, base1, smem);
    build_amplitudes<10>(mp.cls[2], sh, base2, smem);
    // the target start transforms m in its first pass, reading columns that
    // other blocks built
    if (p0.init_target && !grid_sync(p0, target, sh)) return;
  } else {
    restore_flags(mp.cls[0], sh, 0);
    restore_flags(mp.cls[1], sh, base1);
    restore_flags(mp.cls[2], sh, base2);
  }
  __syncthreads();

  // Mask groups (each class's group size keeps a group's fields in L2), each
  // through the whole schedule; classes one after the other.
  const int npass = pass_count(p0);
  for (int c = 0; c < 3; ++c) {
    const Params& pc = mp.cls[c];
    const int gsz = pc.group > 0 ? pc.group : pc.batch;
    for (int w0 = 0; w0 < pc.batch; w0 += gsz) {
      const int w1 = min(pc.batch, w0 + gsz);
      for (int q0 = 0; q0 < npass; ++q0) {
        const LateSum ls = pass(c, w0, w1, pass_info(p0, q0), q0 + 1 < npass, mphase);
        if (!grid_sync(p0, target, sh, ls.x, ls.to)) {
          drain_copies(sh);
          return;
        }
      }
    }
  }
  final_gaps(mp.cls[0], sh, 0);
  final_gaps(mp.cls[1], sh, base1);
  final_gaps(mp.cls[2], sh, base2);
}

template <bool TC>
__global__ void __launch_bounds__(TC ? kThreads : kThreads * kMixedSplit, 1) gs_iterate_mixed(const MixedParams mp) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared sh;
  if (*reinterpret_cast<volatile int*>(mp.cls[0].abort_flag) != 0) return;
  TcStage1 s1;
  TcStage2<8> s2a;
  TcStage2<16> s2b;
  TcStage2<32> s2c;
  if constexpr (TC) {
    float2* cs = reinterpret_cast<float2*>(smem + kTcTwOffset + 3 * kTcTwBytes);
    tc_build_tables<8>(reinterpret_cast<float2*>(smem + kTcTwOffset), cs);
    tc_build_tables<9>(reinterpret_cast<float2*>(smem + kTcTwOffset + kTcTwBytes), cs);
    tc_build_tables<10>(reinterpret_cast<float2*>(smem + kTcTwOffset + 2 * kTcTwBytes), cs);
    __syncthreads();
    s1.load(cs);
    s2a.load(cs);
    s2b.load(cs);
  }
  // The schedule of iterate_mixed, written out: passing the register-held
  // DFT fragments through a closure moved them to local memory.
  const Params& p0 = mp.cls[0];
  unsigned target = 0;
  unsigned mphase = 0;
  block_setup(sh);
  const int total = mp.cls[0].batch + mp.cls[1].batch + mp.cls[2].batch;
  const int base1 = mp.cls[0].batch, base2 = base1 + mp.cls[1].batch;
  if (p0.do_init) {
    for (int c = 0; c < 3; ++c) a0_partials(mp.cls[c], sh);
    if (!grid_sync(p0, target, sh)) return;
    const int nbad = a0_scales(mp.cls[0], sh, 0) + a0_scales(mp.cls[1], sh, base1) + a0_scales(mp.cls[2], sh, base2);
    if (nbad == total) {
      if (blockIdx.x == 0 && threadIdx.x == 0) atomicExch(p0.abort_flag, 1);
      return;
    }
    build_amplitudes<8>(mp.cls[0], sh, 0, smem);
    build_amplitudes<9>(mp.cls[1], sh, base1, smem);
    build_amplitudes<10>(mp.cls[2], sh, base2, smem);
    // the target start transforms m in its first pass, reading columns that
    // other blocks built
    if (p0.init_target && !grid_sync(p0, target, sh)) return;
  } else {
    restore_flags(mp.cls[0], sh, 0);
    restore_flags(mp.cls[1], sh, base1);
    restore_flags(mp.cls[2], sh, base2);
  }
  __syncthreads();
  const int npass = pass_count(p0);
  for (int c = 0; c < 3; ++c) {
    const Params& pc = mp.cls[c];
    const int gsz = pc.group > 0 ? pc.group : pc.batch;
    for (int w0 = 0; w0 < pc.batch; w0 += gsz) {
      const int w1 = min(pc.batch, w0 + gsz);
      for (int q0 = 0; q0 < npass; ++q0) {
        const PassInfo f = pass_info(p0, q0);
        const bool late = q0 + 1 < npass;
        LateSum ls;
        if (c == 0) ls = mixed_class_pass<0, TC>(mp, sh, w0, w1, f, late, smem, mphase, s1, s2a);
        else if (c == 1) ls = mixed_class_pass<1, TC>(mp, sh, w0, w1, f, late, smem, mphase, s1, s2b);
        else ls = mixed_class_pass<2, TC>(mp, sh, w0, w1, f, late, smem, mphase, s1, s2c);
        if (!grid_sync(p0, target, sh, ls.x, ls.to)) {
          drain_copies(sh);
          return;
        }
      }
    }
  }
  final_gaps(mp.cls[0], sh, 0);
  final_gaps(mp.cls[1], sh, base1);
  final_gaps(mp.cls[2], sh, base2);
}

// The mixed launch with tcgen05 transforms: one TMEM allocation for the
// launch, the 32-point matrix shared by the three lengths, an R-point matrix
// and a twiddle table per length (kMixedTc5SmemBytes after the kernel's own
// shared memory).
// offset of the R-point matrix of class c (R = 8 << c) in the tables
__host__ __device__ constexpr int mixed_b2_offset(int c) {
  return 2 * tc5_form_bytes(32) + (c > 0 ? 2 * tc5_form_bytes(8) : 0) + (c > 1 ? 2 * tc5_form_bytes(16) : 0);
}
constexpr int kMixedTwOffset = 4 * tc5_form_bytes(32) + 2 * tc5_form_bytes(8) + 2 * tc5_form_bytes(16);
static_assert(kMixedTwOffset + 3 * kTc5TwBytes == kMixedTc5ExtraSmemBytes, "mixed tcgen05 tables match the launch size");

template <int C, bool BF16>
__device__ __forceinline__ LateSum mixed_class_pass_tc5(const MixedParams& mp, Shared& sh, int w0, int w1,
                                                     const PassInfo& f, bool late, unsigned char* smem, unsigned& mphase,
                                                     const Tc5Fft<8 + C, BF16>& tcf) {
  constexpr int L = 8 + C;
  const int base = (C > 0 ? mp.cls[0].batch : 0) + (C > 1 ? mp.cls[1].batch : 0);
  const StageTw<L> none{};
  return class_pass<L, L, false>(mp.cls[C], sh, base, w0, w1, f, late, smem, mphase, none, tcf);
}

template <bool BF16>
__global__ void __launch_bounds__(kThreads, 1) gs_iterate_mixed_tc5(const MixedParams mp) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared sh;
  __shared__ uint64_t tc_mbar[2];
  __shared__ unsigned tc_tmem;
  const Params& p0 = mp.cls[0];
  if (*reinterpret_cast<volatile int*>(p0.abort_flag) != 0) return;
  static_assert(2 * kTc5HalfStride == kGroupSmemBytes, "the A operands fill the exchange area");
  unsigned char* tabs = smem + kTc5Offset;
  float2* tw = reinterpret_cast<float2*>(tabs + kMixedTwOffset);
  tc5_build_tables<8, BF16>(tabs, tabs + mixed_b2_offset(0), tw);
  tc5_build_tables<9, BF16>(nullptr, tabs + mixed_b2_offset(1), tw + 1024);
  tc5_build_tables<10, BF16>(nullptr, tabs + mixed_b2_offset(2), tw + 2048);
  if (threadIdx.x == 0) {
    mbar_init(&tc_mbar[0], 1);
    mbar_init(&tc_mbar[1], 1);
    fence_barrier_init();
  }
  if ((threadIdx.x >> 5) == 0) tc5_alloc(&tc_tmem);
  fence_proxy_async_smem();  // the DFT matrices are read by the tensor cores
  tc5_fence_before();
  __syncthreads();
  tc5_fence_after();
  unsigned phase = 0;  // one parity per half, shared by the three lengths (their products run in turn)
  const unsigned b1 = smem_u32(tabs);
  const Tc5Fft<8, BF16> t8{smem, b1, smem_u32(tabs + mixed_b2_offset(0)), tw, tc_mbar, tc_tmem, &phase, &p0};
  const Tc5Fft<9, BF16> t9{smem, b1, smem_u32(tabs + mixed_b2_offset(1)), tw + 1024, tc_mbar, tc_tmem, &phase, &p0};
  const Tc5Fft<10, BF16> t10{smem, b1, smem_u32(tabs + mixed_b2_offset(2)), tw + 2048, tc_mbar, tc_tmem, &phase, &p0};
  iterate_mixed(mp, sh, smem, [&](int c, int w0, int w1, const PassInfo& f, bool late, unsigned& mphase) {
    if (c == 0) return mixed_class_pass_tc5<0, BF16>(mp, sh, w0, w1, f, late, smem, mphase, t8);
    if (c == 1) return mixed_class_pass_tc5<1, BF16>(mp, sh, w0, w1, f, late, smem, mphase, t9);
    return mixed_class_pass_tc5<2, BF16>(mp, sh, w0, w1, f, late, smem, mphase, t10);
  });
  tc5_fence_before();
  __syncthreads();
  if ((threadIdx.x >> 5) == 0) tc5_dealloc(tc_tmem);
}

}  // namespace gsk
