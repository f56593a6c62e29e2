// gs_fft.cuh -- register/shared-memory FFT building blocks for sm_103a.
//
// A length-n transform (n = 2^logn, 32 <= n <= 4096) is computed by a group
// of T = n/32 lanes, each of one or two threads; lane t holds the 32 elements
// x[t + T*i], i = 0..31, in registers. The transform is a Stockham auto-sort
// FFT: a first radix-32 stage in registers, then further stages of radix 32
// (and one final stage of radix 2..16 when log2(n) is not a multiple of 5),
// each preceded by one exchange through the group's padded shared-memory
// buffer. The output is left in registers in the same layout, in natural order.
//
// Only the forward transform (kernel exp(-2 pi i jk/n), unnormalised) is
// implemented. The inverse is obtained from it by exchanging real and
// imaginary parts before and after: swap(DFT(swap(x))) = n * IDFT(x). The
// kernels fold those swaps into the neighbouring projection code, so they cost
// nothing.
#pragma once

#include <cuda_runtime.h>

namespace gsk {

__host__ __device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// a * w for a twiddle w = (c, s) meaning c + i s. The fused operations are
// written out here and in norm2: left to the compiler, the choice of the
// product that is fused depends on the code around it, and the same
// transform would round differently from kernel to kernel. (cmul_late fuses
// the other product of the imaginary part: the stage after 1024 points, and
// the twiddles of both tensor-core transforms, which then give the same masks
// bit for bit.)
__host__ __device__ __forceinline__ float2 cmul(float2 a, float2 w) {
  return make_float2(fmaf(a.x, w.x, -(a.y * w.y)), fmaf(a.y, w.x, a.x * w.y));
}
__device__ __forceinline__ float2 cmul_late(float2 a, float2 w) {
  return make_float2(fmaf(a.x, w.x, -(a.y * w.y)), fmaf(a.x, w.y, a.y * w.x));
}
// x^2 + y^2
__device__ __forceinline__ float norm2(float x, float y) { return fmaf(x, x, y * y); }

// cos(2 pi e / 32) for e = 0..8, rounded to float.
struct Cos32 {
  static constexpr float v[9] = {1.0f,
                                 9.807852507e-01f,
                                 9.238795042e-01f,
                                 8.314695954e-01f,
                                 7.071067691e-01f,
                                 5.555702448e-01f,
                                 3.826834261e-01f,
                                 1.950903237e-01f,
                                 0.0f};
};

// W_32^E = exp(-2 pi i E/32) = C - i S for 0 <= E < 16.
template <int E>
struct W32 {
  static constexpr float C = (E <= 8) ? Cos32::v[E] : -Cos32::v[16 - E];
  static constexpr float S = (E <= 8) ? Cos32::v[8 - E] : Cos32::v[E - 8];
};

// Pairs of FP32 operations on the two halves of a float2, each rounded as the
// scalar operation. On the device one instruction works on both halves: the
// FP32 rate is the same (128 lanes per cycle and SM, measured for add,
// multiply and fused multiply-add), but it takes half the issue slots and half
// the code, and the kernels are bound by latency and instruction fetch rather
// than by the FP32 pipe (64 mixed masks 15.38 -> 15.05 ms, 4 x 512^2 0.516 ->
// 0.500 ms, 200 Adam steps at 1024^2 4.50 -> 4.37 ms).
__host__ __device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
  return __ffma2_rn(a, b, c);
#else
  return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
#endif
}
__host__ __device__ __forceinline__ float2 add2(float2 a, float2 b) {
#if defined(__CUDA_ARCH__) && __CUDA_ARCH__ >= 1000
  return __fadd2_rn(a, b);
#else
  return cadd(a, b);
#endif
}

// Radix-2 decimation-in-time butterfly (a, b) -> (a + w b, a - w b) with
// w = W_32^E (0 <= E < 16). Trivial factors (1, -i) cost only additions,
// (+-1 - i)/sqrt2 one addition pair less than a general factor, and the
// general case uses fused multiply-adds with a - w b = 2a - (a + w b).
template <int E>
__host__ __device__ __forceinline__ void bfly(float2& a, float2& b) {
  float2 s;
  if constexpr (E == 0) {
    s = add2(a, b);
    b = fma2(b, make_float2(-1.f, -1.f), a);  // a - b, one rounding
  } else if constexpr (E == 8) {  // w = -i: w b = (b.y, -b.x)
    s = make_float2(a.x + b.y, a.y - b.x);
    b = make_float2(a.x - b.y, a.y + b.x);
  } else if constexpr (E == 4 || E == 12) {
    constexpr float c = Cos32::v[4];
    const float t1 = b.x + b.y;
    const float t2 = b.y - b.x;
    // w b = c t1 + i c t2 (E = 4), c t2 - i c t1 (E = 12)
    const float2 u = E == 4 ? make_float2(t1, t2) : make_float2(t2, t1);
    constexpr float cy = E == 4 ? c : -c;
    s = fma2(make_float2(c, cy), u, a);
    b = fma2(make_float2(-c, -cy), u, a);
  } else {
    constexpr float C = W32<E>::C;
    constexpr float S = W32<E>::S;
    // w b = (C b.x + S b.y) + i (C b.y - S b.x)
    s = fma2(make_float2(C, C), b, fma2(make_float2(S, -S), make_float2(b.y, b.x), a));
    b = fma2(make_float2(2.f, 2.f), a, make_float2(-s.x, -s.y));
  }
  a = s;
}

// One decimation-in-time stage with half-span H on an R-array (bit-reversed
// input order): for every block of 2H and k < H,
// (x[k], x[k + H]) -> (x[k] + W_{2H}^k x[k + H], x[k] - W_{2H}^k x[k + H]).
template <int R, int H>
struct DitStage {
  template <int BASE, int K>
  static __host__ __device__ __forceinline__ void k_loop(float2 (&a)[R]) {
    if constexpr (K < H) {
      bfly<K * (16 / H)>(a[BASE + K], a[BASE + K + H]);
      k_loop<BASE, K + 1>(a);
    }
  }
  template <int BASE>
  static __host__ __device__ __forceinline__ void b_loop(float2 (&a)[R]) {
    if constexpr (BASE < R) {
      k_loop<BASE, 0>(a);
      b_loop<BASE + 2 * H>(a);
    }
  }
  static __host__ __device__ __forceinline__ void run(float2 (&a)[R]) { b_loop<0>(a); }
};

template <int R, int H>
__host__ __device__ __forceinline__ void dit_all(float2 (&a)[R]) {
  if constexpr (H < R) {
    DitStage<R, H>::run(a);
    dit_all<R, 2 * H>(a);
  }
}

__host__ __device__ constexpr int bitrev(int i, int bits) {
  int r = 0;
  for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
  return r;
}

__host__ __device__ constexpr int ilog2(int n) { return n <= 1 ? 0 : 1 + ilog2(n >> 1); }

template <int R, int I>
__host__ __device__ __forceinline__ void bitrev_copy(float2 (&dst)[R], const float2 (&src)[R]) {
  if constexpr (I < R) {
    dst[I] = src[bitrev(I, ilog2(R))];
    bitrev_copy<R, I + 1>(dst, src);
  }
}

// In-register forward DFT of size R (power of two, 2 <= R <= 32), natural
// order in and out: bit-reversal permutation (register renaming only), then
// log2(R) radix-2 decimation-in-time stages.
template <int R>
__host__ __device__ __forceinline__ void dft(float2 (&a)[R]) {
  float2 t[R];
  bitrev_copy<R, 0>(t, a);
  dit_all<R, 1>(t);
#pragma unroll
  for (int i = 0; i < R; ++i) a[i] = t[i];
}

// Values per lane of a team's split-exchange buffer.
__host__ __device__ constexpr int split_values(int S) { return S == 2 ? 16 : 32; }

// Per-group state of a distributed transform of length N = 2^LOGN. The
// geometry is a compile-time constant so that every register and
// shared-memory index folds to an immediate offset.
//
// The line is laid out over T = N/32 lanes; lane t owns the 32 elements
// x[t + T i'], i' = 0..31. S = 1: one thread holds all of them. S = 2 or 4:
// S threads share a lane, thread c with the elements i' = S i + c; they sit in
// the same lane of neighbouring warps, so that c is uniform over a warp. The
// transform evaluates the same butterflies on the same operands in each form
// (the results are equal bit for bit): the radix-2 decimation-in-time stages
// of a 32-point DFT work on the inputs of equal i' mod S separately until the
// last log2 S stages, which combine the threads of a lane (split_last). S = 4
// serves lengths up to 256.
//
// Why: a lane's two transforms, projection and copies are a chain of some 2600
// dependent-issue instructions, which one warp alone on its scheduler runs at
// 3.3 cycles each. More threads per lane shorten the chain and put more warps
// in flight, at the price of one more exchange per 32-point DFT. Column pass
// of one mask, from loaded to stored: 256 x 256 6000 cycles with S = 1, 3400
// with S = 2; 512 x 512 6668 and 4720; 1024 x 1024, where a scheduler has two
// warps of S = 1, 8389 and 9131.
template <int LOGN, int S = 1>
struct GroupT {
  static constexpr int N = 1 << LOGN;
  static constexpr int T = N >> 5;         // lanes of a line
  static constexpr int V = 32 / S;         // elements per thread
  static constexpr int SMEM = N + N / 32;  // padded exchange buffer (complex)
  static constexpr int TT = T > 32 ? T : 32;  // lanes that synchronise together (a team)
  static constexpr int SPLIT = split_values(S) * TT;  // a team's split-exchange buffer (complex), S > 1
  static_assert(S == 1 || S == 2 || (S == 4 && LOGN <= 8), "threads per lane");
  int t;                                   // lane in the line, 0..T-1
  int c;                                   // residue of this thread's elements i' mod S
  int bar_id;                              // named barrier id (S = 1: T > 32; S > 1: the team's)
  float2* sm;                              // this line's exchange buffer
  float2* sx;                              // the team's split-exchange buffer at this lane, S > 1
  const float2* __restrict__ tw;           // stage twiddle tables (twiddle_offset)

  __device__ __forceinline__ void sync() const {
    if constexpr (S == 1 && T <= 32) {
      __syncwarp();
    } else {
      asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "n"(S == 1 ? T : S * TT) : "memory");
    }
  }
  // element index of register i is first() + STEP i
  static constexpr int STEP = T * S;
  __device__ __forceinline__ int first() const { return t + T * c; }
};

// This thread's lane of the block, and which of the lane's S threads it is:
// the threads of a lane sit in neighbouring warps.
template <int S>
__device__ __forceinline__ int lane_of() {
  return S == 1 ? threadIdx.x : ((threadIdx.x / (32 * S)) << 5) | (threadIdx.x & 31);
}
template <int S>
__device__ __forceinline__ int lane_part() {
  return S == 1 ? 0 : (threadIdx.x >> 5) & (S - 1);
}

// Twiddle tables. For the stage with Ns = 2^NSL and radix R the factors
// W_{Ns R}^{r m} (1 <= m < R, r < Ns) are stored transposed, entry
// (m - 1) * Ns + r, so that the threads of a warp (consecutive r) read
// consecutive addresses. The stage with NSL = 5 starts at entry 0; the stage
// with NSL = 10 (only for N > 1024, after a radix-32 stage) at entry 31 * 32.
__host__ __device__ constexpr int twiddle_offset(int nsl) { return nsl == 5 ? 0 : 31 * 32; }

// Twiddles of the stage that follows the first 32 points (NSL = 5), held in
// registers: the element i' = b + Q m of a lane (b < Q = 32/R) is multiplied
// by W_{32 R}^{r m}, r = (t + T b) mod 32. Register i holds the factor of
// element i' = S i + c; elements with m = 0 have none. Loaded once and reused
// by every transform of the same length.
template <int LOGN, int S = 1>
struct StageTw {
  static constexpr int R = (LOGN <= 5) ? 1 : ((LOGN - 5 >= 5) ? 32 : (1 << (LOGN - 5)));
  static constexpr int Q = 32 / R;
  static constexpr int V = 32 / S;
  static constexpr int COUNT = (R > 1) ? V : 1;
  float2 w[COUNT];

  __device__ __forceinline__ void load(const float2* __restrict__ tw, int t, int c = 0) {
    if constexpr (R > 1) {
      constexpr int T = (1 << LOGN) >> 5;
#pragma unroll
      for (int i = 0; i < V; ++i) {
        const int ip = S * i + (S > 1 ? c : 0);
        const int b = ip % Q, m = ip / Q;
        const int r = (t + T * b) & 31;
        w[i] = m > 0 ? __ldg(tw + (m - 1) * 32 + r) : make_float2(1.f, 0.f);
      }
    }
  }
};

// The last radix-2 stage (half-span 16) of a 32-point DFT shared by the two
// threads of a lane (S = 2): v holds the 16-point DFT of the thread's own
// inputs, position k = 0..15. The thread of parity c forms the outputs k and
// k + 16 of the positions k of its parity, which gives back the layout
// i' = 2 i + c: it sends the positions of the other parity to its partner.
template <int C, int K>
__device__ __forceinline__ void split_bfly(float2 (&v)[16], float2 (&o)[16], const float2 (&r)[8]) {
  if constexpr (K < 16) {
    float2 a = C == 0 ? v[K] : r[K >> 1];
    float2 b = C == 0 ? r[K >> 1] : v[K];
    bfly<K>(a, b);
    o[K >> 1] = a;
    o[(K >> 1) + 8] = b;
    split_bfly<C, K + 2>(v, o, r);
  }
}

template <int C, class G>
__device__ __forceinline__ void split_last(float2 (&v)[16], const G& g) {
#pragma unroll
  for (int k = 0; k < 8; ++k) g.sx[(2 * k + 1 - C) * G::TT] = v[2 * k + 1 - C];
  g.sync();
  float2 r[8], o[16];
#pragma unroll
  for (int k = 0; k < 8; ++k) r[k] = g.sx[(2 * k + C) * G::TT];
  split_bfly<C, C>(v, o, r);
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = o[i];
}

// The last two stages shared by the four threads of a lane (S = 4): v holds the
// 8-point DFT of the inputs i' = c mod 4, position j = 0..7. The thread forms
// the outputs k = j + 8 b (b < 4) of its positions j = C and C + 4, that is
// k = C mod 4, from the four threads' values at j. Decimation in time pairs
// the inputs of residues 0 and 2 and those of 1 and 3 first (half-span 8), then
// the two pairs (half-span 16).
template <int C, int J, class G>
__device__ __forceinline__ void split_quad(const float2 (&v)[8], float2 (&o)[8], const G& g) {
  float2 u[4];  // by residue
#pragma unroll
  for (int c = 0; c < 4; ++c) u[c] = c == C ? v[J] : g.sx[(8 * c + J) * G::TT];
  bfly<2 * J>(u[0], u[2]);  // positions J, J + 8 of the even inputs
  bfly<2 * J>(u[1], u[3]);  // ... of the odd ones
  bfly<J>(u[0], u[1]);      // outputs J, J + 16
  bfly<J + 8>(u[2], u[3]);  // outputs J + 8, J + 24
  constexpr int I = J / 4;  // register of output k: (k - C) / 4
  o[I] = u[0];
  o[I + 2] = u[2];
  o[I + 4] = u[1];
  o[I + 6] = u[3];
}

template <int C, class G>
__device__ __forceinline__ void split_last(float2 (&v)[8], const G& g) {
#pragma unroll
  for (int j = 0; j < 8; ++j)
    if (j % 4 != C) g.sx[(8 * C + j) * G::TT] = v[j];
  g.sync();
  float2 o[8];
  split_quad<C, C>(v, o, g);
  split_quad<C, C + 4>(v, o, g);
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = o[i];
}

// 32-point DFT over the elements i' of a lane.
template <class G>
__device__ __forceinline__ void dft32(float2 (&v)[G::V], const G& g) {
  dft<G::V>(v);
  if constexpr (G::V == 16) {
    if (g.c == 0) split_last<0>(v, g);
    else split_last<1>(v, g);
  } else if constexpr (G::V == 8) {
    switch (g.c) {
      case 0: split_last<0>(v, g); break;
      case 1: split_last<1>(v, g); break;
      case 2: split_last<2>(v, g); break;
      default: split_last<3>(v, g); break;
    }
  }
}

// Stockham stage of radix R with Ns = 2^NSL: butterflies j = t + T b,
// b < Q = 32/R. Butterfly j reads x[j + m N/R], which is element i' = b + Q m,
// multiplies by W_{Ns R}^{(j mod Ns) m} and transforms over m; the outputs
// land at the same elements.
template <int LOGN, int NSL, int R, int S>
__device__ __forceinline__ void stage_c(float2 (&v)[32 / S], const GroupT<LOGN, S>& g, const StageTw<LOGN, S>& sw) {
  constexpr int Q = 32 / R;
  constexpr int T = GroupT<LOGN>::T;
  constexpr int NS = 1 << NSL;
  // the threads of a lane share a radix-32 butterfly (parities of m); smaller
  // ones stay within a thread (b = S q + c)
  constexpr int QT = Q > S ? Q / S : 1;  // butterflies of this thread
  constexpr int RT = R * Q / (S * QT);   // elements of each
#pragma unroll
  for (int q = 0; q < QT; ++q) {
    float2 a[RT];
#pragma unroll
    for (int m = 0; m < RT; ++m) a[m] = v[q + QT * m];
    if constexpr (NSL == 5) {
      if (S > 1 && Q == 1 && g.c != 0) a[0] = cmul(a[0], sw.w[0]);  // m = 1 here
#pragma unroll
      for (int m = 1; m < RT; ++m) a[m] = cmul(a[m], sw.w[q + QT * m]);
    } else if constexpr (NSL > 0) {
      static_assert(NSL == 0 || R < 32, "lengths up to 4096 end their second radix-32 stage at 1024");
      const int r = (g.t + T * (S * q + (S > 1 ? g.c : 0))) & (NS - 1);
      const float2* __restrict__ w = g.tw + twiddle_offset(NSL) + r;
#pragma unroll
      for (int m = 1; m < R; ++m) a[m] = cmul_late(a[m], __ldg(w + (m - 1) * NS));
    }
    if constexpr (R == 32) dft32(a, g);
    else dft<R>(a);
#pragma unroll
    for (int m = 0; m < RT; ++m) v[q + QT * m] = a[m];
  }
}

// Exchange after a radix-32 stage with Ns = 2^NSL (butterfly j = t): output
// m goes to (t / Ns) 32 Ns + (t mod Ns) + m Ns; then every thread reads back
// its elements x[t + T i']. Index i of the padded buffer lives at i + i/32.
//
// S > 1 needs no second barrier: the buffer is next written behind the
// barrier of the next split exchange, which every thread reaches after its
// reads here.
template <int LOGN, int NSL, int S>
__device__ __forceinline__ void exchange(float2 (&v)[32 / S], const GroupT<LOGN, S>& g) {
  constexpr int T = GroupT<LOGN>::T;
  constexpr int V = 32 / S;
  static_assert(NSL == 0 || NSL >= 5, "exchanges follow radix-32 stages");
  const int c = S > 1 ? g.c : 0;
  if constexpr (NSL == 0) {
    float2* w = g.sm + 33 * g.t + c;
#pragma unroll
    for (int i = 0; i < V; ++i) w[S * i] = v[i];
  } else {
    const int base = ((g.t >> NSL) << (NSL + 5)) + (g.t & ((1 << NSL) - 1));
    constexpr int STR = (1 << NSL) + (1 << (NSL - 5));
    float2* w = g.sm + base + (base >> 5) + c * STR;
#pragma unroll
    for (int i = 0; i < V; ++i) w[S * i * STR] = v[i];
  }
  g.sync();
  if constexpr (T >= 32) {
    const float2* r = g.sm + g.t + (g.t >> 5) + c * (T + T / 32);
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = r[S * i * (T + T / 32)];
  } else if constexpr (S == 1) {
    const float2* r = g.sm + g.t;
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = r[i * T + ((i * T) >> 5)];
  } else {
    // (S i T + c T + t) >> 5 = (S i T) >> 5, since c T + t < S T divides 32
    static_assert(S * T <= 32, "a thread's elements are whole rows of the padding apart");
    const float2* r = g.sm + g.t + c * T;
#pragma unroll
    for (int i = 0; i < V; ++i) v[i] = r[S * i * T + ((S * i * T) >> 5)];
  }
  if constexpr (S == 1) g.sync();
}

template <int LOGN, int DONE, int S>
__device__ __forceinline__ void fft_from(float2 (&v)[32 / S], const GroupT<LOGN, S>& g, const StageTw<LOGN, S>& sw) {
  if constexpr (DONE < LOGN) {
    if constexpr (DONE > 0) exchange<LOGN, DONE - 5, S>(v, g);
    constexpr int REM = LOGN - DONE;
    constexpr int RL = REM >= 5 ? 5 : REM;
    stage_c<LOGN, DONE, (1 << RL), S>(v, g, sw);
    fft_from<LOGN, DONE + RL, S>(v, g, sw);
  }
}

// Forward unnormalised DFT of length N over the group: the thread's registers
// hold x[first() + STEP i] on entry and X[first() + STEP i] on exit. Every
// thread of the team must call it. S > 1: other uses of the exchange buffer
// after it start with a sync() (other threads may still be reading).
template <int LOGN, int S>
__device__ __forceinline__ void group_fft(float2 (&v)[32 / S], const GroupT<LOGN, S>& g, const StageTw<LOGN, S>& sw) {
  // lengths that end in a 32-point DFT: its split exchange may still be read
  if constexpr (S > 1 && LOGN % 5 == 0) g.sync();
  fft_from<LOGN, 0, S>(v, g, sw);
}

}  // namespace gsk
