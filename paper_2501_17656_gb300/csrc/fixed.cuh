// fixed.cuh -- float64 products on the integer pipe.
//
// This part issues 2 float64 FMAs per clock and SM, but 63 32 x 32 -> 64-bit integer
// multiply-adds (both measured, from registers), so a dot product whose terms share a scale
// is cheaper in fixed point. With parts of B bits, a float64 v with |v| < s = 2^(E - 1022) (E:
// the biased exponent of the largest magnitude of its block or vector, which is at least
// s / 2) becomes
//     V = round(v 2^(2 B) / s) = +-(h 2^B + l),   h < 2^B, l <= 2^B, and
//     V W = +-(h h' 2^(2 B) + (h l' + l h') 2^B + l l')
// takes three multiply-adds: l l', below 2^-2B of s s', is left out. V is within 2^-(2 B + 1) of
// s, without a lean to either side (which would add up over a sum). All bounds are relative
// to the scales, up to twice the largest magnitudes, and not to each value: a value k bits
// below s keeps 2 B - k bits.
//
// B = 28 for sums of 64 terms in one accumulator (h h' below 2^62, the middle sums below 2^63);
// B = 29 for sums of 16: 58 bits, so that values within 2^-5 of the scale are exact.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace h2mg {

// Biased exponents for which values go through fixed point: Inf, NaN and subnormal
// magnitudes stay outside, and no scale factor below overflows or loses bits.
constexpr int FX_EMIN = 128, FX_EMAX = 2000;
// The same for blocks and vectors whose two scales are multiplied with each other first, and
// the least sum of the two: the product stays a normal number.
constexpr int FX_VMAX = 1500, FX_VSUM = 1080;
// Marks a block that the float64 path multiplies (see k_block_exponents).
constexpr int FX_NONE = -1;

struct Fx {
  int h, l;
};

// The exponent of a block or vector of zeros, which any would fit.
constexpr int FX_EZERO = 1023;

// Biased exponent field of |v| (2047: Inf or NaN).
__device__ __forceinline__ int fx_exponent(double v) { return (__double2hiint(v) & 0x7FFFFFFF) >> 20; }

// On the integer pipe: a float64 comparison issues like a float64 FMA.
__device__ __forceinline__ bool fx_is_zero(double v) {
  return ((__double2hiint(v) & 0x7FFFFFFF) | __double2loint(v)) == 0;
}

// v as fixed point under the exponent E (in FX_EMIN..FX_EMAX, at least v's own): the 64 bits
// of the significand, shifted so that the leading bit of the scale is bit B + 31, cut into the
// high word and the B bits below it, rounded. Shifts of 32 and more go through the low word.
template <int B = 28>
__device__ __forceinline__ Fx fx_encode(double v, int E) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned sh = (((unsigned)(E + 32 - B) << 20) - (hi & 0x7FF00000u)) >> 20;
  const unsigned t = __funnelshift_l(lo, hi, 11) | 0x80000000u, low = lo << 11;
  unsigned h, l;
  asm("shr.u32 %0, %1, %2;" : "=r"(h) : "r"(t), "r"(sh));                        // 0 from 32 on
  l = __funnelshift_rc(low, t, sh);                                              // t from 32 on
  asm("shr.u32 %0, %0, %1;" : "+r"(l) : "r"(max((int)sh, 32) - B - 1));          // to B + 1 bits there, and beyond
  l = (l + 1) >> 1;
  const int s = ((int)hi >> 31) | 1;
  return {(int)h * s, (int)l * s};
}

// The same value as h 2^B + l with |l| <= 2^(B - 1) (and |h| <= 2^B): the part l l' that a product
// leaves out is then a quarter of that and has no lean either. With l of v's own sign it always
// pulls sums of equal signs towards zero, by 2^-(2 B + 2) of the scales per term, which in the
// update of a factor adds up over all of it.
template <int B = 28>
__device__ __forceinline__ Fx fx_encode_even(double v, int E) {
  Fx f = fx_encode<B>(v, E);
  const int c = (f.l + (1 << (B - 1))) >> B;     // -1, 0 or 1
  return {f.h + c, f.l - (c << B)};
}

// acc += a * b (32 x 32 -> 64 bits)
__device__ __forceinline__ void fx_mad(int64_t& acc, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc) : "r"(a), "r"(b));
}

// A sum in units of 2^(2 B) from its two parts; the middle part starts at fx_half, so that the
// shift rounds to nearest.
template <int B = 28>
constexpr int64_t fx_half() { return 1ll << (B - 1); }
template <int B = 28>
__device__ __forceinline__ int64_t fx_join(int64_t hh, int64_t mid) { return hh + (mid >> B); }

// A joined sum (B = 29) of products of values under the exponents Ea and Eb is
// join * fx_scale_a(Ea) * fx_scale_b(Eb)  (2^(Ea - 1021) and 2^(Eb - 1081)).
__device__ __forceinline__ double fx_scale_a(int E) { return __hiloint2double((E + 2) << 20, 0); }
__device__ __forceinline__ double fx_scale_b(int E) { return __hiloint2double((E - 58) << 20, 0); }

}  // namespace h2mg
