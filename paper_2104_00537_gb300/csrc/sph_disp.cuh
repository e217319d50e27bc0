// sph_disp.cuh -- displacements as the unevaluated sum of two FP32 numbers, for
// device code and (the same operations) for the host.
//
// FP64 runs at 1/74 of the FP32 rate on this chip and, with its conversions, bound
// the predictor (60 us for 1.48M particles) and the corrector (65 us).  dt is split
// once per step, its products with FP32 velocities keep 48 bits (FP64: 53), and the
// sum with an offset is rounded once, as the FP64 form rounds it: over 4.5e7 random
// offsets (also near zero), steps and velocities the stored offset equals the FP64
// form's every time, at most half a unit from the exact sum.  Only where a
// displacement cancels its offset to 2^-21 and less do the products' bits show: the
// error there is 2^-48 of the displacement.
#pragma once
#include <cmath>
#include <cstring>

#include <cuda_runtime.h>

namespace sph {

struct Disp {
  float hi, lo;
};

// a b, not contracted into a sum that uses it
__host__ __device__ __forceinline__ float disp_mul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
__host__ __device__ __forceinline__ int disp_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_int(x);
#else
  int b;
  std::memcpy(&b, &x, 4);
  return b;
#endif
}
__host__ __device__ __forceinline__ float disp_float(int b) {
#ifdef __CUDA_ARCH__
  return __int_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}

// (c[0] + c[1]) v
__host__ __device__ __forceinline__ Disp disp_scaled(const float (&c)[2], float v) {
  Disp d;
  d.hi = disp_mul(c[0], v);
  d.lo = fmaf(c[1], v, fmaf(c[0], v, -d.hi));
  return d;
}

// a + b = s + (returned error), exactly (Knuth's two-sum)
__host__ __device__ __forceinline__ float disp_two_sum(float a, float b, float &s) {
  s = a + b;
  const float t = s - a;
  return (a - (s - t)) + (b - t);
}

__host__ __device__ __forceinline__ Disp disp_sum(const Disp &a, const Disp &b) {
  Disp d;
  const float e = disp_two_sum(a.hi, b.hi, d.hi);
  d.lo = e + (a.lo + b.lo);
  return d;
}
__host__ __device__ __forceinline__ Disp disp_of(double x) {
  Disp d;
  d.hi = (float)x;
  d.lo = (float)(x - (double)d.hi);
  return d;
}

// off + d, rounded once.  The exact error e of off + d.hi and d.lo are added with
// rounding to odd (an inexact sum of even last bit moves one unit towards the exact
// one), so that the last addition sees on which side of a tie the exact sum lies.
// (Rounded to nearest instead, 3 of 6e7 sums came out a unit off.)  Only a sum whose
// own rounding led onto a tie matters: half an odd number of units of s, with s less
// than 2^11 of them away (where d.hi nearly cancels off, e is 0 and nothing was
// rounded), so its last 12 bits are zero; the others skip the second two-sum.
// Predictor and corrector of 1.48M particles with pair_once: 38.4 and 47.4 us
// rounded to nearest, 42.7 and 50.7 with the second two-sum everywhere (and, by its
// registers, four blocks per SM), 39.3 and 47.9 so (five blocks).
__host__ __device__ __forceinline__ float add_disp(float off, const Disp &d) {
  float s;
  const float e = disp_two_sum(off, d.hi, s);
  float u = e + d.lo;
  if ((disp_bits(u) & 0xfff) == 0 && u != 0.f) {
    const float r = disp_two_sum(e, d.lo, u);
    const int b = disp_bits(u);
    if (r != 0.f) u = disp_float(b + ((b ^ disp_bits(r)) < 0 ? -1 : 1));
  }
  return s + u;
}

}  // namespace sph
