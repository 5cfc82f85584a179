// Conversions between float64 and float32 on the integer pipes.  GB300's conversion instructions with a float64 side run at the
// float64 rate (2.0 lanes per clock and SM, measured, against ~100 for integer instructions), so a cast costs as
// much as a float64 FMA; these give the same values in about ten integer instructions.
#pragma once

#include <cuda_runtime.h>

namespace hpsi {

// (float)x, rounded to nearest even
__device__ __forceinline__ float f64_to_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x);
  const unsigned ex = (hi >> 20) & 0x7ff;
  if (ex - 897u > 252u) {   // outside float32's normal range (or about to round out of it)
    if (ex == 0) return __uint_as_float(hi & 0x80000000u);
    return (float)x;
  }
  unsigned long long m = ((unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL) - (896ULL << 52);
  m += 0x0fffffffULL + ((m >> 29) & 1);
  return __uint_as_float((unsigned)(m >> 29) | (hi & 0x80000000u));
}
__device__ __forceinline__ float2 f64_to_f32(double2 x) { return make_float2(f64_to_f32(x.x), f64_to_f32(x.y)); }

// (double)f 2^-sh for 0 <= sh < 64, exact but for subnormal f, which give zero: what produces such values here (tensor cores
// on bf16 terms, float32 transforms whose results are 2^sh times what they stand for) has lost as much before.
// Without a branch: one around the cast costs 2% of H|psi> for 160 bands of 1503 plane waves.
__device__ __forceinline__ double f32_to_f64(float f, int sh = 0) {
  const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
  unsigned hi = (a >> 3) + (a >= 0x7f800000u ? 0x70000000u : 0x38000000u - ((unsigned)sh << 20));   // infinity, NaN: all ones
  hi = a < 0x00800000u ? 0u : hi;
  return __hiloint2double((int)((u & 0x80000000u) | hi), (int)(a < 0x00800000u ? 0u : u << 29));
}

// x = h + l + (less than 2^-46 |x|): h the float32 with x's leading 24 bits, l the bits below (same sign)
__device__ __forceinline__ float2 f64_split(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned ex = (hi >> 20) & 0x7ff;
  if (ex - 921u > 228u) {
    if (ex == 0) return make_float2(__uint_as_float(hi & 0x80000000u), 0.f);
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
  }
  const unsigned sign = hi & 0x80000000u;
  const float h = __uint_as_float(sign | ((ex - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29));
  // the 29 bits below as 1.b - 1 at exponent ex - 23 (its leading 23 bits)
  const unsigned base = sign | ((ex - 919u) << 23);
  return make_float2(h, __uint_as_float(base | ((lo & 0x1fffffffu) >> 6)) - __uint_as_float(base));
}

}  // namespace hpsi
