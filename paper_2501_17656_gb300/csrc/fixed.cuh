// fixed.cuh -- float64 products on the integer pipe.
//
// This part issues 2 float64 FMAs per clock and SM, but 27 32 x 32 -> 64-bit integer
// multiply-adds (both measured), so a dot product whose terms share a scale is cheaper in
// fixed point: a float64 v with |v| < 2^(E - 1022) (E: the biased exponent of the largest
// magnitude of its block or vector) becomes the 56-bit integer
//     V = round(v 2^(1078 - E)) = +-(h 2^28 + l),   h < 2^28, l <= 2^28, and
//     V W = +-(h h' 2^56 + (h l' + l h') 2^28 + l l')
// takes three multiply-adds: l l', at most 2^-56 of the largest product (2^-58 on average),
// is left out. The integer sums are exact: 64 terms of h h' stay below 2^62, 64 middle ones
// below 2^63. A value is off by at most 2^-57 of the largest magnitude of its block, without
// a lean to either side (which would add up over a sum); a float64 sum of the same 64 terms
// rounds at 2^-53 of its partial sums.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace h2mg {

// Biased exponents for which values go through fixed point: Inf, NaN and subnormal
// magnitudes stay outside, and no scale factor below overflows or loses bits.
constexpr int FX_EMIN = 128, FX_EMAX = 2000;
// The same for blocks and vectors whose two scales are multiplied with each other first.
constexpr int FX_VMAX = 1500;
// Marks a block that the float64 path multiplies (see k_block_exponents).
constexpr int FX_NONE = -1;

struct Fx {
  int h, l;
};

// Biased exponent field of |v| (2047: Inf or NaN).
__device__ __forceinline__ int fx_exponent(double v) { return (__double2hiint(v) & 0x7FFFFFFF) >> 20; }

// v as fixed point under the exponent E (in FX_EMIN..FX_EMAX, at least v's own): the 64 bits
// of the significand, shifted so that the leading bit of the scale is bit 59, cut into the
// high word and the 28 bits below it, rounded. Shifts of 32 and more go through the low word.
__device__ __forceinline__ Fx fx_encode(double v, int E) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sh = (((unsigned)(E + 4) << 20) - (hi & 0x7FF00000u)) >> 20;
  const unsigned t = __funnelshift_l(lo, hi, 11) | 0x80000000u, b = lo << 11;
  unsigned h, l;
  asm("shr.u32 %0, %1, %2;" : "=r"(h) : "r"(t), "r"(sh));                        // 0 from 32 on
  l = __funnelshift_rc(b, t, sh);                                                // t from 32 on
  asm("shr.u32 %0, %0, %1;" : "+r"(l) : "r"(max((int)sh, 32) - 29));             // (l >> 3) there, and beyond
  l = (l + 1) >> 1;
  const int s = ((int)hi >> 31) | 1;
  return {(int)h * s, (int)l * s};
}

// acc += a * b (32 x 32 -> 64 bits)
__device__ __forceinline__ void fx_mad(int64_t& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// A sum in units of 2^56 from its two parts; the middle part starts at FX_HALF, so that the
// shift rounds to nearest.
constexpr int64_t FX_HALF = 1ll << 27;
__device__ __forceinline__ int64_t fx_join(int64_t hh, int64_t mid) { return hh + (mid >> 28); }

// A joined sum of products of values under the exponents Ea and Eb is
// join * fx_scale_a(Ea) * fx_scale_b(Eb)  (2^(Ea - 1021) and 2^(Eb - 1079)).
__device__ __forceinline__ double fx_scale_a(int E) { return __hiloint2double((E + 2) << 20, 0); }
__device__ __forceinline__ double fx_scale_b(int E) { return __hiloint2double((E - 56) << 20, 0); }

}  // namespace h2mg
