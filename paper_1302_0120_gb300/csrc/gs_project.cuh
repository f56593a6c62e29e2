// gs_project.cuh -- the projections onto the two constraint sets and the phase
// output, on the values a thread holds of a line (power-of-two kernels).
#pragma once

#include <cfloat>
#include <cmath>

#include "gs_fft.cuh"

namespace gsk {

// The projections of a line's values z, elementwise, after the transform of a
// pass, and their gaps (part += (|z|/sqrt(N) - a)^2):
//   kProjTarget  z = Y:       z <- swap(m Y/|Y|)   (Eq. e:Mhat; a = m)
//   kProjUnit    z = swap(v): z <- v/|v|           (Eq. e:PS with p = 1; a = 1)
//   kProjSlm     z = swap(v): z <- p v/|v|         (Eq. e:PS; a = p)
//   kProjSlmRg   the same in the register-resident general kernels, whose
//                |z|^2 rounds the other product
// with the phase of an exact zero taken as 0. amp[stride i] is the amplitude
// at element i.
//
// While every |z|^2 of the thread is a normal number the reciprocal square
// root is the bare instruction and no zero rule applies: 9-10 instructions per
// element. Otherwise the loop below it scales subnormals and selects zeros
// (16 per element); both give the same bits on normal values.
enum Projection { kProjTarget = 0, kProjUnit = 1, kProjSlm = 2, kProjSlmRg = 3 };

__device__ __forceinline__ float rsqrt_normal(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// (v[0 .. V) of an array of M values)
template <int PROJ, int V, int M>
__device__ __forceinline__ void project(float2 (&v)[M], float inv_sqrt_n, const float* amp, int stride, float& part) {
  static_assert(V <= M, "the values fit the array");
  auto sq = [](float2 z) {
    return PROJ == kProjUnit || PROJ == kProjSlmRg ? norm2(z.y, z.x) : norm2(z.x, z.y);
  };
  bool normal = true;
#pragma unroll
  for (int i = 0; i < V; ++i) normal &= (sq(v[i]) >= FLT_MIN);  // false for NaN
  if (normal) {
#pragma unroll
    for (int i = 0; i < V; ++i) {
      const float a = PROJ == kProjUnit ? 1.f : amp[stride * i];
      const float a2 = sq(v[i]);
      const float rs = rsqrt_normal(a2);
      const float d = fmaf(a2 * rs, inv_sqrt_n, -a);
      part = fmaf(d, d, part);
      const float f = PROJ == kProjUnit ? rs : a * rs;
      v[i] = make_float2(v[i].y * f, v[i].x * f);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < V; ++i) {
    const float a = PROJ == kProjUnit ? 1.f : amp[stride * i];
    const float a2 = sq(v[i]);
    const float rs = rsqrtf(a2);
    const float mag = a2 > 0.f ? a2 * rs : 0.f;
    const float d = fmaf(mag, inv_sqrt_n, -a);
    part = fmaf(d, d, part);
    const float f = PROJ == kProjUnit ? rs : a * rs;
    const float2 zero = PROJ == kProjTarget ? make_float2(0.f, a) : make_float2(a, 0.f);
    v[i] = a2 > 0.f ? make_float2(v[i].y * f, v[i].x * f) : zero;
  }
}

// The phases of a thread's values su[STEP i] in (-pi, pi]; the loop, four values
// at a time, holds the only copies of atan2f.
template <int V, int STEP>
__device__ __forceinline__ void phase_out(float* po, const float2* su) {
#pragma unroll 4
  for (int i = 0; i < V; ++i) {
    const float2 u = su[STEP * i];
    const float ph = atan2f(u.y, u.x);
    po[STEP * i] = (ph <= -3.14159274f) ? 3.14159274f : ph;
  }
}

}  // namespace gsk
