// Float64 value of one output element from its weight-class sums (tc_pair.cu), in
// integer arithmetic; plain C++ as well, for the host check of its ranges.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define LNO_HD __host__ __device__ __forceinline__
#else
#define LNO_HD inline
#endif

namespace lno {

LNO_HD int round_int(float x) {   // nearest even, |x| < 2^31
#ifdef __CUDA_ARCH__
  return __float2int_rn(x);
#else
  return (int)rintf(x);
#endif
}

// I 2^e as a float64, |I| < 2^53 and the result a normal number (integer
// operations only: a float64 add or conversion of every element would cost
// more than the tile's MMAs, at 1/64 of the float32 rate).
LNO_HD double fixed_to_double(int64_t I, int e) {
  const uint64_t a = (uint64_t)(I < 0 ? -I : I);
  if (a == 0) return 0.0;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = __builtin_clzll(a);
#endif
  const uint64_t m = (a << (lz - 11)) & ((1ull << 52) - 1);
  const uint64_t bits = ((uint64_t)(I < 0) << 63) | ((uint64_t)(1023 + 63 - lz + e) << 52) | m;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double d;
  memcpy(&d, &bits, sizeof d);
  return d;
#endif
}

// Longest contraction whose classes all stay below 2^31 in units of their last digit
// (and class 0 below 2^28): g + 1 products of at most 2^14 each in class g of the
// BF16 slices; of the FP16 slices, whose rows of leading digits have norms of at most
// 2^12 (kExactSum), 2^23 sqrt(K) in class 1 and 2^23 sqrt(K) + 2^20 K in class 2.
constexpr int kWideBF16 = 16384, kWideFP16 = 1536;

// Sum of the classes times 2^e.  Class g is an integer multiple of 2^(-BITS g), or
// (INTS) that integer.  All classes add up to one int64 (at most 2^62 for five
// slices), rounded to nearest from 2^53 on (four slices and FP16 get there only in a
// longer contraction, WIDE).  There a class may also reach 2^30: then they are added in
// float64, smallest first.  A class 0 that is not finite becomes NaN (a NaN operand has
// it in its leading slice, so in class 0).  rest: class 0 plus the float32 sum of the
// others (BF16 only).  WIDE is a template's choice: its checks cost 0.5-0.8% of a
// 140/14/12 domain's central share and of a 60/7/5 gradient, tested by a flag 0.8-2.8%.
template <int S, int BITS, bool INTS, bool WIDE>
LNO_HD double class_sum(const float (&c)[S], int e, bool rest) {
  constexpr float kIntLimit = 1073741824.0f;
  float w;
  bool fits = fabsf(c[0]) < kIntLimit;
  if (WIDE) {
    float big = 0.f;
    w = 1.0f;
#pragma unroll
    for (int g = 1; g < S; ++g) {
      w *= (float)(1 << BITS);
      big = fmaxf(big, fabsf(INTS ? c[g] : c[g] * w));   // exact: a power of two
    }
    fits = fits && big < kIntLimit;
  }
  if (!fits) {
    if (!WIDE || !(fabsf(c[0]) <= 3.402823466e38f)) return (double)NAN;
    double v = 0.0;
    for (int g = S - 1; g >= 0; --g) v += INTS ? ldexp((double)c[g], -BITS * g) : (double)c[g];
    return ldexp(v, e);
  }
  int64_t I = round_int(c[0]);
  if (!INTS && S > 1 && rest) {
    float lo = 0.f;
#pragma unroll
    for (int g = S - 1; g >= 1; --g) lo = lo + c[g];
    constexpr int sh = BITS * (S - 1);      // <= 32
    const float l1 = rintf(lo);             // lo = l1 + l0, both exact
    const float l0 = (lo - l1) * (float)(1ll << (sh < 24 ? sh : 24));
    I = ((I + round_int(l1)) << sh) + ((int64_t)round_int(l0) << (sh < 24 ? 0 : sh - 24));
  } else {
    w = 1.0f;
#pragma unroll
    for (int g = 1; g < S; ++g) {
      w *= (float)(1 << BITS);
      I = (int64_t)((uint64_t)I << BITS) + round_int(INTS ? c[g] : c[g] * w);
    }
  }
  e -= BITS * (S - 1);
  const uint64_t a = (uint64_t)(I < 0 ? -I : I);
  if (e < -960 || e > 960 || ((S == 5 || WIDE) && (a >> 53) != 0)) return ldexp((double)I, e);
  return fixed_to_double(I, e);
}

}  // namespace lno
