// 64-bit fixed-point arithmetic of the FP64 2D wave solve (wave_fx_kernels.cuh).
//
// On sm_103a the FP64 pipe runs two lanes per SM and cycle, 1/64 of the FP32 rate, while integer
// additions with carry run at about 64 lanes and 32 x 32 -> 64-bit multiply-adds at 50.  The
// levels of a wave solve are kept as integers in units of a quantum 2^e that puts a bound of a
// launch's levels just below 2^59 (fourth order 2^56) and follows it from launch to launch, so
// additions are exact and the only rounding of a step is that of the product with dt^2 c^2 / h^2, to
// the nearest quantum: about 2^-55 of the largest level on the grid, whatever the local one (an FP64
// step rounds several times to 2^-53 of the local values, its float-pair sums to 2^-47).  The
// functions also compile for the host, where tests compare them with exact arithmetic.
#pragma once

#include <cstdint>

namespace mfwh {

// Sums of levels.  Points beyond the valid ring of a tile are stepped too, on values that no bound
// covers; they are never read, and wrap around.
__host__ __device__ __forceinline__ int64_t fx_add(int64_t a, int64_t b) {
  return (int64_t)((uint64_t)a + (uint64_t)b);
}
__host__ __device__ __forceinline__ int64_t fx_sub(int64_t a, int64_t b) {
  return (int64_t)((uint64_t)a - (uint64_t)b);
}
__host__ __device__ __forceinline__ int64_t fx_mul15(int64_t a) {
  return (int64_t)(15ull * (uint64_t)a);
}

// A coefficient A in [0, 1) as an even integer A 2^64 = hi 2^32 + lo, and half = A 2^63.
struct FxCoef {
  uint32_t lo, hi;
  uint64_t half;
};

// d + A x rounded to the nearest integer (halves up), for any x.  x is offset by 2^63 so that every
// partial product is unsigned; the offset's product is the integer half.
__device__ __forceinline__ int64_t fx_mac(int64_t d, int64_t x, const FxCoef& A) {
  const uint32_t xl = (uint32_t)x, xh = (uint32_t)((uint64_t)x >> 32) ^ 0x80000000u;
  const uint64_t t0 = (uint64_t)A.lo * xl;
  const uint64_t t1 = (uint64_t)A.lo * xh + ((t0 >> 32) + 0x80000000u);   // rounds
  const uint64_t t2 = (uint64_t)A.hi * xl + (uint32_t)t1;
  const uint64_t p = (uint64_t)A.hi * xh + (t1 >> 32) + (t2 >> 32);
  return (int64_t)((uint64_t)d + p - A.half);
}

// Sums of products of two 64-bit factors of two signed digits each, hi 2^32 + lo: s1 = sum of hi hi'
// and s2 = sum of hi lo' exactly (two 32 x 32 + 64-bit multiply-adds a term), which stand for
// s1 2^64 + s2 2^32.  The kernel adds lo hi' in FP32, to 2^-24 of terms below 2^-28 of the largest;
// lo lo', at most 2^62 and of either sign, is dropped.
struct FxSum {
  int64_t s1, s2;
};
__device__ __forceinline__ void fx_madd(FxSum& s, int ahi, const int2& b) {
  s.s1 += (int64_t)ahi * b.x;
  s.s2 += (int64_t)ahi * b.y;
}
// v as two signed digits, for |v| < 2^62.
__host__ __device__ __forceinline__ void fx_digits(int64_t v, int& hi, int& lo) {
  lo = (int)(uint32_t)(uint64_t)v;
  hi = (int)(fx_sub(v, lo) >> 32);
}
// The digits of a level as a factor, of W less the constant 2^31 (which makes the low word's
// excess over 2^31 a signed digit); the sums take the constant back once per launch.
__device__ __forceinline__ int2 fx_level_digits(int64_t w) {
  return make_int2((int)(w >> 32), (int)((uint32_t)w ^ 0x80000000u));
}

// v / 2^e rounded to the nearest integer (halves away from zero), for a finite v below 2^(e + 62).
__device__ __forceinline__ int64_t fx_from_bits(uint64_t bits, int e) {
  const int ex = (int)(bits >> 52) & 0x7FF;
  uint64_t m = bits & 0x000FFFFFFFFFFFFFull;
  m |= ex ? 1ull << 52 : 0ull;
  const int sh = (ex ? ex : 1) - 1075 - e;   // |v| / 2^e = m 2^sh
  uint64_t x;
  if (sh >= 0)
    x = sh < 64 ? m << sh : 0ull;   // m = 0 when sh is beyond the range
  else
    x = -sh > 54 ? 0ull : (m + (1ull << (-sh - 1))) >> -sh;
  return (bits >> 63) ? -(int64_t)x : (int64_t)x;
}

// x 2^k rounded to the nearest integer (halves to even: a shift by one bit meets one every other
// time, and a step's increment that is biased by b moves the level n steps on by b n);
// x 2^k below 2^62.
__device__ __forceinline__ int64_t fx_rescale(int64_t x, int k) {
  if (k >= 0) return (int64_t)((uint64_t)x << k);
  return -k > 62 ? 0 : fx_add(x, (((int64_t)1 << (-k - 1)) - 1) + (x >> -k & 1)) >> -k;
}

}  // namespace mfwh
