// Conversions between float and double in integer arithmetic on their IEEE 754 bit patterns.
//
// The conversion instructions issue on the FP64 unit, which takes a warp instruction only every 16
// clocks here (1/64 of the FP32 rate), and the solver's mixed form converts three or four values
// per element of every row pass.  These take 6 and 12 integer instructions, which the four
// schedulers of an SM issue in parallel.  The results are those of the casts for every input: the
// common cases (normal numbers and zeros) are formed here, the others are left to the cast.  (Tested on
// host and device for every float and at every boundary between two normal floats.)
#pragma once
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define LORADS_HD __host__ __device__ __forceinline__
#else
#define LORADS_HD inline
#endif

namespace lorads {

// widening (exact).  A normal float has 8 exponent bits (bias 127) and 23 fraction bits, a double 11
// (bias 1023) and 52: the exponent moves by 1023 - 127 = 896 and the fraction to its upper bits.
LORADS_HD double widen(float x) {
  uint32_t u;
#if defined(__CUDA_ARCH__)
  u = __float_as_uint(x);
#else
  memcpy(&u, &x, 4);
#endif
  const uint32_t a = u & 0x7fffffffu;
  if (a - 0x00800000u >= 0x7f000000u && a != 0u) return (double)x;   // subnormal, Inf, NaN
  const uint32_t hi = (u & 0x80000000u) | (a != 0u ? (a >> 3) + (896u << 20) : 0u);
  const uint32_t lo = u << 29;
#if defined(__CUDA_ARCH__)
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

// narrowing, to nearest, ties to even.  For a result in the normal range the upper 23 fraction bits
// are kept and the 29 dropped ones decide the rounding, whose carry runs into the exponent (and
// to Inf) by itself.
LORADS_HD float narrow(double x) {
  uint32_t hi, lo;
#if defined(__CUDA_ARCH__)
  hi = (uint32_t)__double2hiint(x);
  lo = (uint32_t)__double2loint(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  hi = (uint32_t)(b >> 32);
  lo = (uint32_t)b;
#endif
  const uint32_t a = hi & 0x7fffffffu;
  // biased exponent between 897 and 1150: float exponents 1 .. 254
  const bool normal = a - (897u << 20) < (254u << 20);
  if (!normal && (a | lo) != 0u) return (float)x;     // underflow, overflow, Inf, NaN
  uint32_t f = ((a - (896u << 20)) << 3) | (lo >> 29);
  const uint32_t rest = lo << 3;                       // the dropped bits, left-aligned
  f += (rest > 0x80000000u || (rest == 0x80000000u && (f & 1u))) ? 1u : 0u;
  f = (hi & 0x80000000u) | (normal ? f : 0u);
#if defined(__CUDA_ARCH__)
  return __uint_as_float(f);
#else
  float r;
  memcpy(&r, &f, 4);
  return r;
#endif
}

}  // namespace lorads
