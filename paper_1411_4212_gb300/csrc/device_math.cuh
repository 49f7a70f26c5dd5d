// device_math.cuh -- elementary functions that more than one test or kernel wants for themselves.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace rewl {

// e^x for x <= 0 (0 below -708, NaN for NaN) in integer arithmetic: this GPU issues less than two FP64 operations
// per clock and SM, but 64-bit products of integers at a tenth of its FP32 rate.
// -x log2(e) = n + j/64 + r in 2^-53 units, r < 1/64;  e^x = 2^-n 2^(-j/64) 2^-r with the middle factor from a
// table (2^-63 units) and the last by its Taylor polynomial of degree 6 (error 3e-18).
// Lost at most, in units in the last place: 0.5 where -x is cut to 2^-54 (below 1/4), 0.7 where its product with
// log2(e) is cut to 2^-53, 0.25 by log2(e)'s own rounding (at 708; little below 1/4), 0.05 in table and polynomial,
// 0.5 by the result's rounding: less than two.
constexpr int kPow2 = 64;
__device__ __forceinline__ double exp_fixed(double x, const unsigned long long* pow2) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
  if (bits >= 0x4086200000000000ULL) return bits > 0x7ff0000000000000ULL ? x : 0.0;   // |x| >= 708
  const int e = (int)(bits >> 52) - 1023;
  const unsigned long long m = (bits & 0xfffffffffffffULL) | 0x10000000000000ULL;
  // |x| in 2^-54 units (e <= 9); below 2^-54 nothing is left of it
  const unsigned long long q = e >= -2 ? m << (e + 2) : (e >= -54 ? m >> (-2 - e) : 0ULL);
  const unsigned long long t = __umul64hi(q, 0xb8aa3b295c17f0bcULL);     // log2(e) in 2^-63 units
  const unsigned long long u = (t << 17) >> 6;                            // r in 2^-64 units
  unsigned long long v = 0x00050c244be1b1e2ULL;                            // (ln 2)^i / i! in 2^-63 units, i = 6 .. 0
  v = 0x002bb0ffcf14ce62ULL - __umul64hi(u, v);
  v = 0x013b2ab6fba4e773ULL - __umul64hi(u, v);
  v = 0x071ac235c1282fe3ULL - __umul64hi(u, v);
  v = 0x1ebfbdff82c58ea8ULL - __umul64hi(u, v);
  v = 0x58b90bfbe8e7bcd6ULL - __umul64hi(u, v);
  v = 0x8000000000000000ULL - __umul64hi(u, v);
  const unsigned long long w = __umul64hi(pow2[(t >> 47) & 63], v);        // (1/2, 1] in 2^-62 units
  // rounded to 53 bits; a carry into the next power of two is right as it stands
  return __longlong_as_double((long long)(((1021ULL - (t >> 53)) << 52) + ((w + 256) >> 9)));
}

// 2^(-j/64) in 2^-63 units, from the six factors 2^(-1/2) .. 2^(-1/64) in 2^-64 units.
__device__ __forceinline__ unsigned long long pow2_entry(int j) {
  const unsigned long long f[6] = {0xb504f333f9de6484ULL, 0xd744fccad69d6af4ULL,
                                 0xeac0c6e7dd24392fULL, 0xf5257d152486cc2cULL,
                                 0xfa83b2db722a033aULL, 0xfd3e0c0cf486c175ULL};
  unsigned long long v = 0x8000000000000000ULL;
#pragma unroll
  for (int i = 0; i < 6; ++i)
    if ((j >> (5 - i)) & 1) v = __umul64hi(v, f[i]);
  return v;
}

// 1 / d for 1 <= d <= 2^126, by Newton's iteration r' = r + r (1 - d r) from the hardware's estimate (relative
// error e = 2^-23): one step leaves e^2 and its own rounding, so at most one unit in the last place.  Where 1 / d
// is below the smallest normal number it is 0.
__device__ __forceinline__ float reciprocal(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return fmaf(fmaf(-d, r, 1.0f), r, r);
}

}  // namespace rewl
