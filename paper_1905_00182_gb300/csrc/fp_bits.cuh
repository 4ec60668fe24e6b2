// fp_bits.cuh -- conversions between FP64 and FP32 by integer operations: a conversion instruction
// issues at the FP64 rate (1.8 lanes per clock and SM), these at the integer rate.
#pragma once

namespace ibfsa {

// (double)x and (float)x (to nearest, ties to even) by integer operations and, for subnormal x, one
// FP32 product.  The two conversions and two additions per component of the FP32 form's FP64 update
// made its last stage FP64-bound.
// Subnormal values are common (products of small perturbations), so no case is left to the
// instruction: it would be issued for the whole warp.
__device__ __forceinline__ double widen(float x) {
  const bool sub = (__float_as_uint(x) << 1) < (1u << 24);
  const unsigned b = __float_as_uint(sub ? x * 16777216.f : x), m = b << 1;
  const unsigned bias = sub ? 896u - 24u : m >= (255u << 24) ? 2u * 896u : 896u;
  const unsigned hi = m ? (m >> 4) + (bias << 20) : 0u;
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29));
}

__device__ __forceinline__ float narrow(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned m = hi & 0x7fffffffu, e = m >> 20;
  // the result's bits before rounding and what follows them; a carry runs into the exponent
  unsigned f = __funnelshift_l(lo, m - (896u << 20), 3), rest = lo << 3;
  if (e < 897u) {  // subnormal or zero
    const unsigned full = 0x800000u | (f & 0x7fffffu), shift = 897u - e;
    const bool some = shift <= 24u;
    f = some ? full >> shift : 0u;
    rest = some ? full << (32u - shift) | (rest != 0u) : 0u;
  } else if (e > 1150u) {  // too large, infinite or not a number
    f = m > 0x7ff00000u || (m == 0x7ff00000u && lo) ? 0x7fffffffu : 0x7f800000u;
    rest = 0u;
  }
  const unsigned up = rest > 0x80000000u || (rest == 0x80000000u && (f & 1u));
  return __uint_as_float((f + up) | (hi & 0x80000000u));
}

// (float)x truncated, for tests with a margin: magnitudes below FP32's normal range give 0, above it
// (and non-finite values) NaN.
__device__ __forceinline__ float low_precision(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = hi & 0x7ff00000u;
  unsigned r = ((__funnelshift_l(lo, hi, 3) & 0x7fffffffu) ^ 0x40000000u) | (hi & 0x80000000u);
  r = e < 0x38100000u ? 0u : r;
  r = e >= 0x47f00000u ? 0x7fffffffu : r;
  return __uint_as_float(r);
}

}  // namespace ibfsa
