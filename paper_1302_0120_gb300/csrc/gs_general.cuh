// gs_general.cuh -- passes of the iteration kernel for grids whose sides are
// not powers of two or are below 32 (5-smooth sides 2^a 3^b 5^c in [8, 1536],
// also beside a power of two up to 2048), except those of gs_rg.cuh.
//
// The pass structure, projections and FP64 gap sums are those of the
// power-of-two kernel (gs_iterate.cuh); what differs is the transform and the
// data movement:
//   * The field B is stored row-major [ny][nx]; m transposed [nx][ny].
//   * A row or column is transformed by a team of GenTeam::T threads; teams
//     synchronise on their own named barrier. A block has as many teams as an
//     SM has lines to do in one round (GenGeom, gs_internal.h): the passes are
//     chains of dependent stage loops, and a second round costs a whole chain
//     again (1280 x 1024 with four teams per block: 320 column groups on 256
//     blocks, 35 us per column pass, of which the second round half).
//   * A row pass gives each team one row: the row is read coalesced into the
//     team's shared-memory buffer, transformed, projected and transformed
//     again there, and written back coalesced.
//   * A column pass moves one column per team at a time: the block reads the
//     tile of adjacent columns in row segments into the teams' column buffers,
//     each team transforms, projects and transforms its column, and the block
//     writes the tile back the same way.
//   * A length-n transform is a Stockham auto-sort FFT with radices 3 and 5
//     first, then 8, 4 and 2 (gen_fft), each stage read from one of the team's
//     two buffers and written to the other. The twiddles of the stage with sub-transform length ns and radix R sit at
//     entries ns - 1 + (m - 1) ns + r (W_{ns R}^{r m}), so that consecutive
//     butterflies read consecutive entries; the tables are rounded once from
//     double on the host and copied to shared memory per launch.
//   * Rows and column tiles arrive by cp.async, every copy of a thread in
//     flight at once.
#pragma once

#include "gs_common.cuh"
#include "gs_fft.cuh"
#include "gs_tma.cuh"

namespace gsk {

// Radix of stage code c (3 bits per stage in Params::planx / plany).
__host__ __device__ constexpr int radix_of_code(unsigned c) {
  return c == 0 ? 2 : c == 1 ? 3 : c == 2 ? 4 : c == 3 ? 5 : 8;
}

// 3-point DFT, exp(-2 pi i jk/3): with t = a1 + a2 and d = (sqrt3/2)(a1 - a2),
// y1,2 = a0 - t/2 -/+ i d.
__host__ __device__ __forceinline__ void dft3(float2 (&a)[3]) {
  constexpr float h = 0.8660254037844386f;  // sqrt(3)/2
  const float2 t = cadd(a[1], a[2]);
  const float2 d = make_float2(h * (a[1].x - a[2].x), h * (a[1].y - a[2].y));
  const float2 c = make_float2(fmaf(-0.5f, t.x, a[0].x), fmaf(-0.5f, t.y, a[0].y));
  a[0] = cadd(a[0], t);
  a[1] = make_float2(c.x + d.y, c.y - d.x);
  a[2] = make_float2(c.x - d.y, c.y + d.x);
}

// 5-point DFT, exp(-2 pi i jk/5), from the symmetric and antisymmetric pairs
// b1 = a1 + a4, b2 = a2 + a3, d1 = a1 - a4, d2 = a2 - a3:
//   y1,4 = a0 + c1 b1 + c2 b2 -/+ i (s1 d1 + s2 d2)
//   y2,3 = a0 + c2 b1 + c1 b2 -/+ i (s2 d1 - s1 d2)
// with ck = cos(2 pi k/5), sk = sin(2 pi k/5).
__host__ __device__ __forceinline__ void dft5(float2 (&a)[5]) {
  constexpr float c1 = 0.30901699437494745f, c2 = -0.8090169943749475f;
  constexpr float s1 = 0.9510565162951535f, s2 = 0.5877852522924731f;
  const float2 b1 = cadd(a[1], a[4]), b2 = cadd(a[2], a[3]);
  const float2 d1 = csub(a[1], a[4]), d2 = csub(a[2], a[3]);
  const float2 e1 = make_float2(fmaf(c1, b1.x, fmaf(c2, b2.x, a[0].x)), fmaf(c1, b1.y, fmaf(c2, b2.y, a[0].y)));
  const float2 e2 = make_float2(fmaf(c2, b1.x, fmaf(c1, b2.x, a[0].x)), fmaf(c2, b1.y, fmaf(c1, b2.y, a[0].y)));
  const float2 f1 = make_float2(fmaf(s1, d1.x, s2 * d2.x), fmaf(s1, d1.y, s2 * d2.y));
  const float2 f2 = make_float2(fmaf(s2, d1.x, -s1 * d2.x), fmaf(s2, d1.y, -s1 * d2.y));
  a[0] = cadd(a[0], cadd(b1, b2));
  // e - i f = (e.x + f.y, e.y - f.x)
  a[1] = make_float2(e1.x + f1.y, e1.y - f1.x);
  a[4] = make_float2(e1.x - f1.y, e1.y + f1.x);
  a[2] = make_float2(e2.x + f2.y, e2.y - f2.x);
  a[3] = make_float2(e2.x - f2.y, e2.y + f2.x);
}

template <int R>
__host__ __device__ __forceinline__ void small_dft(float2 (&a)[R]) {
  if constexpr (R == 3) dft3(a);
  else if constexpr (R == 5) dft5(a);
  else dft<R>(a);
}

// This thread's team of T = 2^LOG threads (at least a warp). T is known to the
// compiler, so that the steps of every loop over a line are immediate offsets:
// with T read at run time 1280 x 1024 x 10 took 430 us (now 422), 1500 x 1500
// 718 (703), 1536 x 9 205 (196; 200 with fixed teams of two warps before).
template <int LOG>
struct GenTeam {
  static constexpr int T = 1 << LOG;  // threads
  int id;    // team in the block
  int t;     // thread in the team
  int n;     // teams of the block
  __device__ GenTeam() : id(threadIdx.x >> LOG), t(threadIdx.x & (T - 1)), n(blockDim.x >> LOG) {}
  // named barrier 1 + id
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + id), "r"(T) : "memory");
  }
};

// floor(a / b) for 0 <= a < 2^14, 0 < b < 2^14 through the reciprocal: (a + 1/2)/b
// is at least 1/(2b) away from a whole number, further than its rounding
// error. (Each stage of a transform needs four quotients and remainders by a
// run-time length; the integer division sequence took longer than the stage.)
__device__ __forceinline__ int small_div(int a, int b) {
  return static_cast<int>((static_cast<float>(a) + 0.5f) * __fdividef(1.f, static_cast<float>(b)));
}

// One Stockham stage of radix R on a length-n transform whose first stages
// formed sub-transforms of length ns: butterfly j = q ns + r reads
// src[j + m n/R], multiplies by W_{ns R}^{r m} (stage table tw), transforms
// over m and writes dst[q ns R + r + k ns]. Thread t of the team takes
// butterflies t, t + T, ...
template <int R, int LOG>
__device__ __forceinline__ void gen_stage(const float2* __restrict__ src, float2* __restrict__ dst, int n, int ns,
                                          const float2* __restrict__ tw, const GenTeam<LOG>& tm) {
  const int nb = n / R;
  const int tt = tm.t;
  const int qinc = small_div(tm.T, ns), rinc = tm.T - qinc * ns;
  int q = small_div(tt, ns), r = tt - q * ns;
  const float2* const tws = tw + (ns - 1);
  for (int j = tt; j < nb; j += tm.T) {
    float2 a[R];
#pragma unroll
    for (int m = 0; m < R; ++m) a[m] = src[j + m * nb];
    if (ns > 1) {
#pragma unroll
      for (int m = 1; m < R; ++m) a[m] = cmul(a[m], tws[(m - 1) * ns + r]);
    }
    small_dft<R>(a);
    float2* const to = dst + q * ns * R + r;
#pragma unroll
    for (int k = 0; k < R; ++k) to[k * ns] = a[k];
    q += qinc;
    r += rinc;
    if (r >= ns) {
      r -= ns;
      ++q;
    }
  }
}

// Forward unnormalised DFT of the length-n vector in `a` by the team,
// using `b` as the second buffer; returns the buffer that holds the result
// (a for an even number of stages, b for an odd one).
template <int LOG>
__device__ __forceinline__ float2* gen_fft(float2* a, float2* b, int n, unsigned plan, int nst, const float2* tw,
                                           const GenTeam<LOG>& tm) {
  int ns = 1;
#pragma unroll 1
  for (int s = 0; s < nst; ++s) {
    const int R = radix_of_code((plan >> (3 * s)) & 7u);
    switch (R) {
      case 2: gen_stage<2>(a, b, n, ns, tw, tm); break;
      case 3: gen_stage<3>(a, b, n, ns, tw, tm); break;
      case 4: gen_stage<4>(a, b, n, ns, tw, tm); break;
      case 5: gen_stage<5>(a, b, n, ns, tw, tm); break;
      default: gen_stage<8>(a, b, n, ns, tw, tm); break;
    }
    tm.sync();
    ns *= R;
    float2* t = a;
    a = b;
    b = t;
  }
  return a;
}

// Copy the twiddle tables to shared memory (once per launch).
__device__ __forceinline__ void gen_load_twiddles(const Params& p, unsigned char* smem) {
  float2* t = reinterpret_cast<float2*>(smem);
  for (int e = threadIdx.x; e < p.nx; e += blockDim.x) t[e] = p.twx[e];
  for (int e = threadIdx.x; e < p.ny; e += blockDim.x) t[p.nx + e] = p.twy[e];
  __syncthreads();
}

// m = s sqrt(I), transposed ([nx][ny]), for this block's columns: tiles of 8
// columns go through the (still unused) team buffers, so that both sides are
// read and written in segments (lanes striding over rows took 20 us once per
// run at 1280 x 1024).
__device__ __forceinline__ void gen_build_amplitude(const Params& p, int mb, float s, unsigned char* smem) {
  const size_t moff = static_cast<size_t>(mb) * static_cast<size_t>(p.mstride);
  const float* const Im = p.I + moff;
  float* const mTm = p.mT + moff;
  const int ny = p.ny;
  float* const tile = reinterpret_cast<float*>(reinterpret_cast<float2*>(smem) + gen_tw_entries(p.nx, ny));
  const int lo = split(blockIdx.x, gridDim.x, p.nx);
  const int hi = split(blockIdx.x + 1, gridDim.x, p.nx);
  const int k = threadIdx.x & 7;
  for (int c0 = lo; c0 < hi; c0 += 8) {
    const int wc = min(8, hi - c0);
    if (k < wc)
      for (int y = threadIdx.x >> 3; y < ny; y += blockDim.x >> 3)
        cp_async4(tile + k * (ny + 1) + y, Im + static_cast<size_t>(y) * p.nx + c0 + k);
    cp_async_wait_all();
    __syncthreads();
    for (int c = 0; c < wc; ++c)
      for (int y = threadIdx.x; y < ny; y += blockDim.x)
        mTm[static_cast<size_t>(c0 + c) * ny + y] = s * sqrtf(tile[c * (ny + 1) + y]);
    __syncthreads();
  }
}

// Wrap an angle as the power-of-two kernel does: (-pi, pi].
__device__ __forceinline__ float gen_phase(float2 u) {
  const float a = atan2f(u.y, u.x);
  return (a <= -3.14159274f) ? 3.14159274f : a;
}

// One pass over rows [lo, hi) (kInit, kRow) or columns [lo, hi)
// (kCol, kResid, kInitM) of mask mb. Returns this thread's FP32 contribution
// to the pass's gap sum.
template <int LOG>
static __device__ __forceinline__ float run_pass_gen(const Params& p, int mb, int kind, bool last, int lo, int hi,
                                                      unsigned char* smem) {
  const size_t moff = static_cast<size_t>(mb) * static_cast<size_t>(p.mstride);
  float2* const Bm = p.B + moff;
  const float* const mTm = p.mT + moff;
  const int nx = p.nx, ny = p.ny;
  const int nmax = nx > ny ? nx : ny;
  const float2* twx = reinterpret_cast<const float2*>(smem);
  const float2* twy = twx + nx;
  float2* wbase = reinterpret_cast<float2*>(smem) + gen_tw_entries(nx, ny);
  const GenTeam<LOG> tm;
  constexpr int T = GenTeam<LOG>::T;
  const int tt = tm.t;
  float2* const A = wbase + tm.id * gen_team_stride(nmax);
  float2* const Bf = A + nmax + 1;
  const float inv_sqrt_n = p.inv_sqrt_n;
  const bool two = (kind == kCol || (kind == kRow && !(last && !p.final_resid)));
  float acc = 0.f;

  if (kind == kInit || kind == kRow) {
    for (int row = lo + tm.id; row < hi; row += tm.n) {
      float2* src = Bm + static_cast<size_t>(row) * nx;
      const float* pp = p.p_slm ? p.p_slm + static_cast<size_t>(row) * nx : nullptr;
      if (kind == kInit) {
        const float* ph = p.phi_in + moff + static_cast<size_t>(row) * nx;
        float* po = p.phi_out + moff + static_cast<size_t>(row) * nx;
        for (int x0 = tt; x0 < nx; x0 += T * 4) {
          float f[4], a[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int x = x0 + T * k;
            f[k] = x < nx ? ph[x] : 0.f;
            a[k] = (pp && x < nx) ? pp[x] : 1.f;  // u0 = p exp(i phi0)
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            float s, c;
            sincosf(f[k], &s, &c);
            if (x0 + T * k < nx) A[x0 + T * k] = make_float2(a[k] * c, a[k] * s);
          }
        }
        if (last) {  // zero iterations
          tm.sync();
          for (int x = tt; x < nx; x += T) po[x] = gen_phase(A[x]);
        }
      } else {
        for (int x = tt; x < nx; x += T) cp_async8(A + x, src + x);
        cp_async_wait_all();
      }
      tm.sync();
      float2* res = gen_fft(A, Bf, nx, p.planx, p.nstx, twx, tm);
      if (kind == kRow) {
        // res = swap(IDFT_x(B)) = swap(sqrt(N) P_M u^nu): gap to S, Eq. (e:PS)
        float part = 0.f;
        for (int x0 = tt; x0 < nx; x0 += T * 8) {
          float a[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) a[k] = (pp && x0 + T * k < nx) ? pp[x0 + T * k] : 1.f;
          float2 t8[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) t8[k] = (x0 + T * k < nx) ? res[x0 + T * k] : make_float2(1.f, 0.f);
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int x = x0 + T * k;
            if (x < nx) {
              const float2 t = t8[k];
              const float vx = t.y, vy = t.x;
              const float a2 = vx * vx + vy * vy;
              const float rs = rsqrtf(a2);
              const float mag = a2 > 0.f ? a2 * rs : 0.f;
              const float d = mag * inv_sqrt_n - a[k];
              part += d * d;
              const float f = a[k] * rs;
              res[x] = a2 > 0.f ? make_float2(vx * f, vy * f) : make_float2(a[k], 0.f);
            }
          }
        }
        acc += part;
        tm.sync();
        if (last) {
          float* po = p.phi_out + moff + static_cast<size_t>(row) * nx;
          for (int x = tt; x < nx; x += T) po[x] = gen_phase(res[x]);
        }
        if (two) res = gen_fft(res, res == A ? Bf : A, nx, p.planx, p.nstx, twx, tm);
      }
      if (kind == kInit || two) {
        // rolled: unrolled, its code lengthens the rounds of rows of a few points
        // (64 masks of 8 x 1536 2.53 ms, now 2.48) and gains long ones nothing
#pragma unroll 1
        for (int x = tt; x < nx; x += T) src[x] = res[x];
      }
      tm.sync();
    }
    return acc;
  }

  // Column passes: groups of adjacent columns; team k owns column c0 + k.
  const int stride = gen_team_stride(nmax);
  const bool store = (kind == kCol || kind == kInitM);
  // which of a team's buffers holds the stored result: A after two transforms,
  // else A or Bf by the parity of the stage count
  const int out_off = (kind == kCol || (p.nsty & 1) == 0) ? 0 : nmax + 1;
  // the tile's copies: this thread's column of the group, and its first row
  // and row step (T rows per sweep of the block)
  const int cy = small_div(threadIdx.x, tm.n), ck = threadIdx.x - cy * tm.n;
  for (int c0 = lo; c0 < hi; c0 += tm.n) {
    const int wc = min(tm.n, hi - c0);
    __syncthreads();  // the previous group's tile has been written back
    if (ck < wc) {
      float2* const col = wbase + ck * stride;
      if (kind == kInitM) {
        for (int y = cy; y < ny; y += T)  // swap((m, 0))
          col[y] = make_float2(0.f, mTm[static_cast<size_t>(c0 + ck) * ny + y]);
      } else {
        for (int y = cy; y < ny; y += T) cp_async8(col + y, Bm + static_cast<size_t>(y) * nx + c0 + ck);
        cp_async_wait_all();
      }
    }
    __syncthreads();
    if (tm.id < wc) {
      float2* res = gen_fft(A, Bf, ny, p.plany, p.nsty, twy, tm);
      if (kind != kInitM) {
        // res = Y = F u^nu along this column: residual and Eq. (e:Mhat)
        const float* mcol = mTm + static_cast<size_t>(c0 + tm.id) * ny;
        float part = 0.f;
        for (int y0 = tt; y0 < ny; y0 += T * 8) {
          float mv[8];
          float2 yv[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) mv[u] = (y0 + T * u < ny) ? mcol[y0 + T * u] : 0.f;
#pragma unroll
          for (int u = 0; u < 8; ++u) yv[u] = (y0 + T * u < ny) ? res[y0 + T * u] : make_float2(1.f, 0.f);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int y = y0 + T * u;
            if (y < ny) {
              const float m = mv[u];
              const float2 Y = yv[u];
              const float a2 = Y.x * Y.x + Y.y * Y.y;
              const float rs = rsqrtf(a2);
              const float mag = a2 > 0.f ? a2 * rs : 0.f;
              const float d = mag * inv_sqrt_n - m;
              part += d * d;
              if (kind == kCol) {
                const float f = m * rs;
                const float2 Yh = a2 > 0.f ? make_float2(Y.x * f, Y.y * f) : make_float2(m, 0.f);
                res[y] = make_float2(Yh.y, Yh.x);  // swapped: the next forward DFT acts as the inverse
              }
            }
          }
        }
        acc += part;
        tm.sync();
        if (kind == kCol) res = gen_fft(res, res == A ? Bf : A, ny, p.plany, p.nsty, twy, tm);
      }
    }
    if (store) {
      __syncthreads();
      if (ck < wc) {
        const float2* const col = wbase + ck * stride + out_off;
        for (int y = cy; y < ny; y += T) Bm[static_cast<size_t>(y) * nx + c0 + ck] = col[y];
      }
    }
  }
  return acc;
}

}  // namespace gsk
