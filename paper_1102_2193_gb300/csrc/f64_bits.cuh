// f64_bits.cuh -- FP32 to FP64 and to fixed point by integer instructions.
//
// GB300 issues one FP64 instruction per 64 cycles and warp, and the FP32 to
// FP64 and to 64-bit integer conversions run at that rate too (84 cycles
// measured, against 17 from FP64 to FP32 and from integers to FP64).
#pragma once
#include <cuda_runtime.h>

// (double)x, exactly: exponent rebiased, mantissa shifted (zeros kept;
// denormals, infinities and NaN by the instruction).
__device__ __forceinline__ double f32_to_f64(float x) {
  const unsigned u = __float_as_uint(x), e = u & 0x7f800000u;
  const bool zero = (u << 1) == 0u;
  if (e == 0x7f800000u || (e == 0u && !zero)) return (double)x;
  const unsigned hi = zero ? u : ((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u));
  return __hiloint2double((int)hi, (int)(u << 29));
}

// s 2^-k rounded to nearest even (|k| < 900: the result is normal).
__device__ __forceinline__ double fixed_to_f64(long long s, int k) {
  if (s == 0) return 0.0;
  unsigned long long u = s < 0 ? 0ull - (unsigned long long)s : (unsigned long long)s;
  const int lz = __clzll((long long)u);
  u <<= lz;
  const unsigned rem = (unsigned)u & 0x7ffu;
  unsigned long long m = u >> 11;
  m += rem > 0x400u || (rem == 0x400u && (m & 1ull)) ? 1ull : 0ull;
  m += (unsigned long long)(1085 - lz - k) << 52;  // the mantissa's leading one adds 1 to the exponent
  return __longlong_as_double((long long)(m | ((unsigned long long)s & 0x8000000000000000ull)));
}

// x 2^k as a 64-bit integer, |x| 2^k < 2^57, bits below 1 dropped.
__device__ __forceinline__ long long f32_to_fixed(float x, int k) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xffu;
  const unsigned m = e ? (u & 0x7fffffu) | 0x800000u : u & 0x7fffffu;
  const int shift = (int)(e ? e : 1u) + k - 150;
  const long long v = shift >= 0 ? (long long)m << shift : (long long)(shift > -32 ? m >> -shift : 0u);
  return (int)u < 0 ? -v : v;
}
