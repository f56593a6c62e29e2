// gs_loss.cuh -- intensity loss and its adjoint (gradient) in one persistent
// launch, for square grids.
//
// The differentiable form of the same inverse problem (fit |F u|^2 to the
// target intensity over phase-only u, Sec. II):
//   L(phi) = sum_k (|y_k|^2 / N - I_k)^2,   y = F x,  x = exp(i phi)
//   dL/dphi_j = 4 Im(conj(x_j) z_j),        z = F^{-1}(r * y),  r = |y|^2/N - I
// with F the unnormalised 2D DFT and F^{-1} its normalised inverse (from
// dy_k/dphi_j = F_kj i x_j and the symmetry of F). Three passes:
//   rows     x = exp(i phi), B = DFT_x(x)                       (as A1)
//   columns  y = DFT_y(B); r; loss partial; B = IDFT_y(r * y)   (adjoint, swapped)
//   rows     N z = IDFT_x(B); grad = 4 Im(conj(x) z)            (adjoint)
// The target is staged like the amplitude of the iteration kernel
// (transposed [nx][ny], read per column block). FP64 only for the sums.
// With the Adam update fused into the third pass, one launch can run many
// optimiser steps: the third pass of a step, which owns the same rows as the
// first, also forms the next step's x = exp(i phi) and B = DFT_x(x), so every
// step after the first is a column pass and a row pass.
// With a laser amplitude p on the SLM the field is x = p exp(i phi); the
// gradient formula is unchanged (dy_k/dphi_j = F_kj i x_j still holds).
//
// The same column pass can also evaluate the physical error of Eq.
// (phys-error) for u = x (Sec. II): with It = I / max I and the reconstructed
// intensity Ir = |F_u u|^2 (sum I / sum p^2) / max I,
//   E_l = sum_{I > 0} (t_d |It - Ir| / (t_l It) - t_d) Theta(|It - Ir|/It - t_l)
//   E_d = sum_{I = 0} (Ir - t_d) Theta(Ir - t_d),   t_l = 0.1, t_d = 3e-4.
#pragma once

#include "gs_iterate.cuh"

namespace gsk {

constexpr float kTolLit = 0.1f;    // t_l, Sec. II
constexpr float kTolDark = 3e-4f;  // t_d, Sec. II

// partial-sum rows of the loss kernel (each [grid]); row kRowStaged holds the
// reduced target statistics of a prepared target (flag, sum I, max I).
// The loss partials of the steps of a multi-step launch go alternately to the
// two rows behind it (each of kMaxGrid).
enum LossRow { kRowFlag = 0, kRowSumI = 1, kRowMaxI = 2, kRowLoss = 3, kRowEl = 4, kRowEd = 5, kRowStaged = 6, kRowSteps = 7 };

// Record a failure: the first one also adds the abort bit to the barrier
// counter, which releases every waiting block (as fail() in gs_common.cuh).
static __device__ void loss_fail(const LossParams& p, int code) {
  atomicCAS(p.status, 0, code);
  if (atomicExch(p.abort_flag, 1) == 0) atomicAdd(p.bar, kAbortBit);
}

// Grid barrier for the loss kernel (same protocol as grid_sync). With sum_to
// the block's sum of x goes there behind the arrival, to be read after the
// next barrier; `meanwhile` runs on the second warp's first thread while the
// first warp waits.
template <class F>
static __device__ bool loss_sync(const LossParams& p, unsigned& target, Shared& sh, float x, double* sum_to,
                                 F&& meanwhile) {
  __syncthreads();
  target += gridDim.x;
  if (threadIdx.x == 0) asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p.bar) : "memory");
  if (sum_to != nullptr) {  // the same in every thread
    __syncwarp();
    late_sum(x, sum_to, sh);
  }
  if (threadIdx.x == 32) meanwhile();
  if (threadIdx.x == 0) {
    int ok = 1;
    unsigned spins = 0;
    unsigned long long t0 = 0;
    unsigned v;
    while (static_cast<int>((v = ld_acquire_gpu(p.bar)) - target) < 0) {
      ++spins;
      if ((spins & 255u) == 0) {
        const unsigned long long now = global_ns();
        if (t0 == 0) t0 = now;
        if (now - t0 > kBarrierTimeoutNs || spins > kMaxSpins) {
          ok = 0;
          loss_fail(p, GS_ETIMEOUT);
          break;
        }
      }
    }
    asm volatile("fence.proxy.async.global;" ::: "memory");
    if (ok && (v & kAbortBit) != 0) ok = 0;  // a block failed in this launch
    sh.flag = ok;
  }
  __syncthreads();
  return sh.flag != 0;
}

static __device__ __forceinline__ bool loss_sync(const LossParams& p, unsigned& target, Shared& sh) {
  return loss_sync(p, target, sh, 0.f, nullptr, [] {});
}

// The target's statistics from the blocks' partials, by one warp in a fixed
// order (the result in every lane). Every thread adding all of them in turn
// held up each call by the latency of three FP64 chains over the grid.
static __device__ void loss_target_stats(const LossParams& p, double& flag, double& sum_i, double& max_i) {
  const int G = gridDim.x;
  flag = sum_i = max_i = 0.0;
  for (int c = threadIdx.x & 31; c < G; c += 32) {
    flag += p.partials[kRowFlag * G + c];
    sum_i += p.partials[kRowSumI * G + c];
    max_i = fmax(max_i, p.partials[kRowMaxI * G + c]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    flag += __shfl_xor_sync(0xffffffffu, flag, o);
    sum_i += __shfl_xor_sync(0xffffffffu, sum_i, o);
    max_i = fmax(max_i, __shfl_xor_sync(0xffffffffu, max_i, o));
  }
}

// MODE (LossMode, gs_internal.h) kLossFused: validate and stage the target,
// then the three passes (one call does everything). kLossPrepare: validate
// and stage the target only, and reduce its statistics into row kRowStaged.
// kLossStep: the three passes on the staged target (the target of the last
// kLossPrepare launch); with the Adam update, p.steps optimiser steps.

template <int LN, int MODE>
__global__ void __launch_bounds__(kThreads * kLossSplit, 1) gs_loss_kernel(const LossParams p) {
  using G = GroupT<LN, kLossSplit>;  // two threads per lane, as in the iteration kernel
  using L = FieldLayout<LN, LN, 1>;
  constexpr int N = G::N;
  constexpr int T = G::T;
  constexpr int V = G::V;        // elements per thread: t0 + STEP i
  constexpr int STEP = G::STEP;
  constexpr int THR = kThreads * kLossSplit;
  constexpr int LOGT = LN - 5;
  constexpr int NG = kThreads / T;
  constexpr int W = L::W;
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Shared sh;
  __shared__ float adam_c[2];  // Adam: lr / (1 - beta1^t), 1 / sqrt(1 - beta2^t)
  const int b = blockIdx.x;
  const int o = lane_of<kLossSplit>();  // this thread's lane of the block
  const int gidx = o >> LOGT;
  const int team_line = (o & ~31) >> LOGT;  // the first line of this thread's team
  G grp;
  grp.t = o & (T - 1);
  grp.c = lane_part<kLossSplit>();
  grp.bar_id = 1 + (kLossSplit == 1 ? gidx : o / G::TT);
  grp.sm = reinterpret_cast<float2*>(smem) + gidx * G::SMEM;
  grp.sx = reinterpret_cast<float2*>(smem + kSplitSmemOffset) + (o / G::TT) * G::SPLIT + (o & (G::TT - 1));
  grp.tw = p.tw;
  const int t0 = grp.first();
  StageTw<LN, kLossSplit> stw;
  stw.load(p.tw, grp.t, grp.c);
  float* its = reinterpret_cast<float*>(smem + kAmpSmemOffset);
  float2* blk = reinterpret_cast<float2*>(smem + kBlockSmemOffset);
  unsigned target = 0;
  unsigned mphase = 0;
  if (threadIdx.x == 0) {
    mbar_init(&sh.mbar, 1);
    fence_barrier_init();
    sh.pending = 0;
  }
  __syncthreads();

  // Target: validate this block's rows, and stage its columns transposed.
  if constexpr (MODE != kLossStep) {
    const int r0 = split(b, gridDim.x, N);
    const int r1 = split(b + 1, gridDim.x, N);
    bool bad = false;
    double sum_i = 0.0;
    float max_i = 0.f;
    const float* Ib = p.I + static_cast<size_t>(r0) * N;
    const int cnt = (r1 - r0) * N;
    for (int e0 = threadIdx.x; e0 < cnt; e0 += 8 * THR) {
      float xs[8];  // eight loads in flight before they are used
#pragma unroll
      for (int u = 0; u < 8; ++u) xs[u] = (e0 + u * THR < cnt) ? Ib[e0 + u * THR] : 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        bad |= !(fabsf(xs[u]) <= FLT_MAX);
        sum_i += static_cast<double>(xs[u]);
        max_i = fmaxf(max_i, xs[u]);
      }
    }
    const int any_bad = __syncthreads_or(bad);
    const double bsum = block_sum(sum_i, sh);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) max_i = fmaxf(max_i, __shfl_xor_sync(0xffffffffu, max_i, o));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh.red[threadIdx.x >> 5] = static_cast<double>(max_i);
    __syncthreads();
    if (threadIdx.x == 0) {
      double bmax = 0.0;
      for (int w = 0; w < THR / 32; ++w) bmax = fmax(bmax, sh.red[w]);
      const int G = gridDim.x;
      p.partials[kRowFlag * G + b] = any_bad ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;
      p.partials[kRowSumI * G + b] = bsum;
      p.partials[kRowMaxI * G + b] = bmax;
    }
    // transpose this block's column blocks through shared memory (coalesced
    // on both sides): IT[c][y] = I[y][c]
    const int lo = split(b, gridDim.x, L::NBLK);
    const int hi = split(b + 1, gridDim.x, L::NBLK);
    float* tb = reinterpret_cast<float*>(blk);  // [N][W + 1]
    for (int cb = lo; cb < hi; ++cb) {
      __syncthreads();
      for (int e = threadIdx.x; e < N * W; e += THR) {
        const int k = e & (W - 1);
        const int y = e >> L::LW;
        cp_async4(tb + y * (W + 1) + k, p.I + static_cast<size_t>(y) * N + cb * W + k);
      }
      cp_async_wait_all();
      __syncthreads();
      for (int e = threadIdx.x; e < N * W; e += THR) {
        const int k = e >> LN;
        const int y = e & (N - 1);
        p.IT[static_cast<size_t>(cb * W + k) * N + y] = tb[y * (W + 1) + k];
      }
    }
  }
  if constexpr (MODE == kLossPrepare) {
    // the staged target's statistics, reduced once (FP64, fixed order)
    if (!loss_sync(p, target, sh)) return;
    if (b == 0 && threadIdx.x < 32) {
      double flag, sum_i, max_i;
      loss_target_stats(p, flag, sum_i, max_i);
      if (threadIdx.x == 0) {
        double* st = p.partials + kRowStaged * kMaxGrid;  // a fixed place: the step may use another grid
        st[0] = flag;
        st[1] = sum_i;
        st[2] = max_i;
        if (!(flag == 0.0)) atomicCAS(p.status, 0, GS_ENUMERIC);
      }
    }
    return;
  }

  // Pass 1 (rows): x = exp(i phi), B = DFT_x(x).
  {
    const int lo = split(b, gridDim.x, N);
    const int hi = split(b + 1, gridDim.x, N);
    for (int base = lo; base < hi; base += NG) {
      if (base + team_line >= hi) break;  // no row for this team: a copy would only take issue slots
      const int idx = base + gidx;
      const bool valid = idx < hi;
      const int ridx = valid ? idx : base;
      float2 v[V];
      const float* ph = p.phi + static_cast<size_t>(ridx) * N + t0;
      const float* pp = p.p_slm ? p.p_slm + static_cast<size_t>(ridx) * N + t0 : nullptr;
      float2* su = grp.sm + t0;
      grp.sync();  // the previous round's transform has read the buffer
      // phi (and p) by cp.async, all loads in flight, then a rolled loop
#pragma unroll
      for (int i = 0; i < V; ++i) cp_async4(&su[STEP * i].x, ph + STEP * i);
      if (pp) {
#pragma unroll
        for (int i = 0; i < V; ++i) cp_async4(&su[STEP * i].y, pp + STEP * i);
      }
      cp_async_wait_all();
      // four copies of sincosf: independent work for the scheduler, while
      // the code stays small (instruction fetch is this kernel's top stall)
#pragma unroll 4
      for (int i = 0; i < V; ++i) {
        float s, c;
        const float2 fa = su[STEP * i];
        sincosf(fa.x, &s, &c);
        const float a = pp ? fa.y : 1.f;
        su[STEP * i] = make_float2(a * c, a * s);
      }
#pragma unroll
      for (int i = 0; i < V; ++i) v[i] = su[STEP * i];
      grp.sync();
      group_fft<LN>(v, grp, stw);
      if (valid) {
#pragma unroll
        for (int i = 0; i < V; ++i) p.B[L::off(idx, t0 + STEP * i)] = v[i];
      }
    }
  }
  if (!loss_sync(p, target, sh)) return;
  // Scale of the reconstructed intensity for the physical error:
  // Ir = |y|^2/N * (sum I / sum p^2) / max I, It = I / max I.
  float ir_scale = 0.f, it_scale = 0.f;
  {
    double tot = 0.0, sum_i = 0.0, max_i = 0.0;
    if constexpr (MODE == kLossStep) {
      const double* st = p.partials + kRowStaged * kMaxGrid;  // written by the prepare launch
      tot = st[0];
      sum_i = st[1];
      max_i = st[2];
    } else {
      if (threadIdx.x < 32) {
        loss_target_stats(p, tot, sum_i, max_i);
        if (threadIdx.x == 0) {
          sh.red[0] = tot;
          sh.red[1] = sum_i;
          sh.red[2] = max_i;
        }
      }
      __syncthreads();
      tot = sh.red[0];
      sum_i = sh.red[1];
      max_i = sh.red[2];
      __syncthreads();  // sh.red is reused
    }
    const double ep = p.p_slm ? *p.energy : static_cast<double>(N) * N;
    if (max_i > 0.0 && ep > 0.0) {
      ir_scale = static_cast<float>((sum_i / ep) / max_i * p.inv_n);
      it_scale = static_cast<float>(1.0 / max_i);
    }
    if (!(tot == 0.0) || (p.p_slm && !(ep > 0.0 && ep <= DBL_MAX))) {  // a non-finite target or a bad p
      if (b == 0 && threadIdx.x == 0) {
        atomicCAS(p.status, 0, GS_ENUMERIC);
        const double nan = __longlong_as_double(0x7ff8000000000000ll);
        for (int k = 0; k < (p.m != nullptr ? p.steps : 1); ++k) p.loss[k] = nan;
        if (p.phys) p.phys[0] = p.phys[1] = nan;
      }
      return;
    }
  }

  const bool adam = p.m != nullptr;  // the Adam update in place of the gradient output
  const bool want_grad = p.grad != nullptr || adam;  // the adjoint passes
  const bool want_phys = p.phys != nullptr;
  // Adam steps of this launch; every block reads the step count before the
  // last block to finish advances it
  const int steps = adam ? p.steps : 1;
  const int t_done = adam ? p.state[0] : 0;
  for (int k = 0; k < steps; ++k) {
    // Pass 2 (columns): y = DFT_y(B) = F x; r = |y|^2/N - I; loss partial;
    // B = swap(IDFT_y(r y)) for the adjoint.
    float acc = 0.f, acc_l = 0.f, acc_d = 0.f;  // this thread's lines, FP32
    {
      const int lo = split(b, gridDim.x, L::NBLK);
      const int hi = split(b + 1, gridDim.x, L::NBLK);
      const bool gact = gidx < W;
      const bool wact = ((o & ~31) >> LOGT) < W;
      const int gq = gact ? gidx : 0;
      for (int cb = lo; cb < hi; ++cb) {
        __syncthreads();
        if (threadIdx.x == 0) {
          bulk_wait_read_all();
          fence_proxy_async_smem();
          mbar_arrive_expect_tx(&sh.mbar, L::BLOCK * 12u);
          bulk_g2s(blk, p.B + static_cast<size_t>(cb) * L::BLOCK, L::BLOCK * 8u, &sh.mbar);
          bulk_g2s(its, p.IT + static_cast<size_t>(cb) * L::BLOCK, L::BLOCK * 4u, &sh.mbar);
          sh.pending = 1;
          sh.pending_phase = mphase;
        }
        const bool landed = mbar_wait_bounded(&sh.mbar, mphase);
        mphase ^= 1u;
        if (!landed) {
          loss_fail(p, GS_ETIMEOUT);
        } else if (threadIdx.x == 0) {
          sh.pending = 0;
        }
        if (wact) {
          float2 v[V];
#pragma unroll
          for (int i = 0; i < V; ++i) v[i] = blk[L::boff(t0 + STEP * i, gq)];
          group_fft<LN>(v, grp, stw);
          const float* icol = its + gq * N + t0;
          float* sa2 = reinterpret_cast<float*>(grp.sm) + t0;  // |y|^2 for the physical error
          if (want_phys) grp.sync();  // the transform has read the buffer
          float part = 0.f;
#pragma unroll
          for (int i = 0; i < V; ++i) {
            const float2 y = v[i];
            const float a2 = norm2(y.x, y.y);
            const float r = fmaf(a2, p.inv_n, -icol[STEP * i]);
            part = fmaf(r, r, part);
            if (want_phys) sa2[STEP * i] = a2;
            v[i] = make_float2(r * y.y, r * y.x);  // swapped: the next forward DFT acts as the inverse
          }
          if (gact) acc += part;
          if (want_phys) {  // Eq. (phys-error), once per call: a rolled loop
            float el = 0.f, ed = 0.f;
#pragma unroll 1
            for (int i = 0; i < V; ++i) {
              const float ir = sa2[STEP * i] * ir_scale;  // reconstructed intensity
              const float iv = icol[STEP * i];
              if (iv > 0.f) {
                const float it = iv * it_scale;
                const float rel = fabsf(it - ir) / it;
                if (rel - kTolLit > 0.f) el += kTolDark * rel / kTolLit - kTolDark;
              } else if (ir - kTolDark > 0.f) {
                ed += ir - kTolDark;
              }
            }
            if (gact) {
              acc_l += el;
              acc_d += ed;
            }
            grp.sync();
          }
          if (want_grad) {
            group_fft<LN>(v, grp, stw);
            if (gact) {
#pragma unroll
              for (int i = 0; i < V; ++i) blk[L::boff(t0 + STEP * i, gidx)] = v[i];
            }
          }
        }
        if (want_grad) {
          __syncthreads();
          if (threadIdx.x == 0) {
            fence_proxy_async_smem();
            bulk_s2g(p.B + static_cast<size_t>(cb) * L::BLOCK, blk, L::BLOCK * 8u);
            bulk_commit();
          }
        }
      }
      if (want_grad && threadIdx.x == 0) bulk_wait_all();
    }
    // FP32 within the block, FP64 across blocks (below). A step that another
    // follows leaves its sum to the barrier, and block 0 adds the blocks' sums
    // after the next one.
    const bool fuse = k + 1 < steps;
    double* const step_row = p.partials + (kRowSteps + (k & 1)) * kMaxGrid;
    if (!fuse) {
      const int G = gridDim.x;
      const double tot = block_sum_f(acc, sh);
      if (threadIdx.x == 0) p.partials[kRowLoss * G + b] = tot;
      if (want_phys) {
        const double tl = block_sum_f(acc_l, sh);
        if (threadIdx.x == 0) p.partials[kRowEl * G + b] = tl;
        const double td = block_sum_f(acc_d, sh);
        if (threadIdx.x == 0) p.partials[kRowEd * G + b] = td;
      }
    }
    if (!loss_sync(p, target, sh, acc, fuse ? step_row + b : nullptr, [&] {
          if (!adam) return;
          // the step's bias corrections, once per block (in every thread they
          // took 0.5 us of a step)
          const float t = static_cast<float>(t_done + 1 + k);
          const float b1 = 1.f - powf(p.beta1, t);
          const float b2 = 1.f - powf(p.beta2, t);
          adam_c[0] = p.lr / b1;
          adam_c[1] = 1.f / sqrtf(b2);
        })) {
      if (threadIdx.x == 0 && sh.pending) mbar_wait_bounded(&sh.mbar, sh.pending_phase);
      return;
    }
    if (!fuse && b == 0 && threadIdx.x < 32) {
      const int G = gridDim.x;
      for (int row = kRowLoss; row <= (want_phys ? kRowEd : kRowLoss); ++row) {
        double s = 0.0;
        for (int c = threadIdx.x; c < G; c += 32) s += p.partials[row * G + c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) {
          if (row == kRowLoss) p.loss[k] = s;
          else p.phys[row - kRowEl] = s;
        }
      }
    }
    if (!want_grad) return;

    // Pass 3 (rows): N z = IDFT_x(B), grad = 4 Im(conj(x) z) with x = exp(i phi);
    // with the fused update, the Adam step of gs_adam_step on every element
    // instead of its gradient output (the phase of a row is read into shared
    // memory before the thread that owns each element updates it). When
    // another step follows, the same pass also does its pass 1 for the rows it
    // owns (the rows are split over the blocks as in pass 1): exp(i phi) of
    // the updated phase, straight from the update, then B = DFT_x through a
    // second turn of the transform loop.
    const float adam_step = adam ? adam_c[0] : 0.f, adam_rb2 = adam ? adam_c[1] : 0.f;
    {
      const int lo = split(b, gridDim.x, N);
      const int hi = split(b + 1, gridDim.x, N);
      const float scale = 4.f * p.inv_n;
      for (int base = lo; base < hi; base += NG) {
        // No row for this team. A block of the automatic grid has eight rows of
        // 512 points for its 16 groups (of 256 points 8 for 32), so that half of
        // the teams or more leave here: 1.86 -> 1.68 ms per 100 steps at 512 x
        // 512. From 1024 points on it is one or two of eight (1024) or some in
        // the last round, and the compiler's code for a loop that may end early
        // lost more than that won (1024 x 1024 4.26 -> 4.57 ms per 200 steps).
        if (LN <= 9 && base + team_line >= hi) break;
        const int idx = base + gidx;
        const bool valid = idx < hi;
        const int ridx = valid ? idx : base;
        float2 v[V];
#pragma unroll
        for (int i = 0; i < V; ++i) v[i] = p.B[L::off(ridx, t0 + STEP * i)];
        // phi (and p) of this row by cp.async into the field staging buffer
        // (free in this pass), in flight behind the transform
        float* sph = reinterpret_cast<float*>(blk) + threadIdx.x;
        float* spp = sph + V * THR;
        // the fused update with p = 1: the row's moments too, into the laser
        // amplitude's buffer and the staged target's (free in this pass)
        float* const smm = (adam && !p.p_slm) ? spp : nullptr;
        float* const smv = (adam && !p.p_slm) ? its + threadIdx.x : nullptr;
        {
          const size_t r0 = static_cast<size_t>(ridx) * N + t0;
          const float* ph = p.phi + r0;
#pragma unroll
          for (int i = 0; i < V; ++i) cp_async4(sph + THR * i, ph + STEP * i);
          if (p.p_slm) {
            const float* pp = p.p_slm + r0;
#pragma unroll
            for (int i = 0; i < V; ++i) cp_async4(spp + THR * i, pp + STEP * i);
          }
          if (smm != nullptr) {
#pragma unroll
            for (int i = 0; i < V; ++i) {
              cp_async4(smm + THR * i, p.m + r0 + STEP * i);
              cp_async4(smv + THR * i, p.v + r0 + STEP * i);
            }
          }
        }
        // one copy of the transform for both turns (instruction fetch is this
        // kernel's top stall)
#pragma unroll 1
        for (int h = 0; h < (fuse ? 2 : 1); ++h) {
          group_fft<LN>(v, grp, stw);  // h = 0: swap(N z); h = 1: the next step's row DFT
          if (h == 1) {
            if (valid) {
#pragma unroll
              for (int i = 0; i < V; ++i) p.B[L::off(idx, t0 + STEP * i)] = v[i];
            }
            break;
          }
          // Im(conj(x) z) = x.re z.im - x.im z.re, with z = (v.y, v.x) / N
          float2* su = grp.sm + t0;
          grp.sync();  // the transform has read the buffer
#pragma unroll
          for (int i = 0; i < V; ++i) su[STEP * i] = v[i];
          cp_async_wait_all();
          if (valid && !adam) {
            float* gr = p.grad + static_cast<size_t>(idx) * N + t0;
#pragma unroll 4
            for (int i = 0; i < V; ++i) {
              float s, c;
              sincosf(sph[THR * i], &s, &c);
              const float a = p.p_slm ? spp[THR * i] : 1.f;  // x = p exp(i phi)
              const float2 w = su[STEP * i];
              gr[STEP * i] = scale * a * fmaf(c, w.x, -(s * w.y));
            }
          } else if (valid) {
            const size_t e0 = static_cast<size_t>(idx) * N + t0;
#pragma unroll 4
            for (int i = 0; i < V; ++i) {
              float s, c;
              sincosf(sph[THR * i], &s, &c);
              const float a = p.p_slm ? spp[THR * i] : 1.f;
              const float2 w = su[STEP * i];
              const float g = scale * a * fmaf(c, w.x, -(s * w.y));
              const size_t e = e0 + STEP * i;
              const float m0 = smm ? smm[THR * i] : p.m[e];
              const float v0 = smv ? smv[THR * i] : p.v[e];
              const float mi = fmaf(p.beta1, m0, (1.f - p.beta1) * g);
              const float vi = fmaf(p.beta2, v0, (1.f - p.beta2) * g * g);
              p.m[e] = mi;
              p.v[e] = vi;
              const float ph = sph[THR * i] - adam_step * mi / fmaf(sqrtf(vi), adam_rb2, p.eps);
              p.phase[e] = ph;
              if (fuse) {  // x = p exp(i phi) of the next step, in place of w
                sincosf(ph, &s, &c);
                su[STEP * i] = make_float2(a * c, a * s);
              }
            }
          }
          if (fuse) {  // a group with no row of its own transforms what it holds and stores nothing
#pragma unroll
            for (int i = 0; i < V; ++i) v[i] = su[STEP * i];
            grp.sync();
          }
        }
        grp.sync();
      }
    }
    if (fuse) {
      if (!loss_sync(p, target, sh)) return;
      // block 0 reads the step's partials here; their row is written again two
      // steps on, behind a barrier that block 0 reaches after this
      if (b == 0 && threadIdx.x < 32) {
        double s = 0.0;
        for (int c = threadIdx.x; c < static_cast<int>(gridDim.x); c += 32) s += step_row[c];
#pragma unroll
        for (int o2 = 16; o2 > 0; o2 >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o2);
        if (threadIdx.x == 0) p.loss[k] = s;
      }
    }
  }  // steps
  if (adam) {  // the last block to finish advances the step count (every block has read it)
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      if (atomicAdd(p.state + 1, 1) == static_cast<int>(gridDim.x) - 1) {
        p.state[0] = t_done + steps;
        p.state[1] = 0;
      }
    }
  }
}

}  // namespace gsk
