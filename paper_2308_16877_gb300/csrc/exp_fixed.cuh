// exp(-a2 s) for s >= 0 in fixed point, on the integer pipes. GB300 issues
// two FP64 operations per SM and clock against 16 to 18 32 x 32 -> 64-bit
// products and 60 to 100 other integer operations, so the fifteen products and
// about fifty simple operations below take the time of three FP64 operations,
// on pipes that are otherwise idle beside FP64 work.
//
// t = s a2 log2(e) as integer part n and 64-bit fraction F, from the
// significand of s times the 64-bit significand C of a2 log2(e). Then
//   2^-t = 2^-(n+1) 2^(G / 2^64), G = 2^64 - 1 - F (2^-64 below 2^64 - F),
// with G's top 11 bits taking 2^(j / 2048) from two tables (2^(i/32) and
// 2^(k/2048), as in Tang's table-driven method, ACM TOMS 15(2), 1989) and the
// rest, r = x 2^-11 with x below 1, from the Taylor polynomial
//   2^r - 1 = sum over k = 1..4 of (r ln 2)^k / k!
// (the fifth term is below 2^-64). Products keep at least 60 bits below the
// leading one, and the result is rounded once to 53: within 0.85 ulp
// of exp(-a2 s) over the whole range (0.25 on average, as correct rounding).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace hpac {

struct ExpFixed {
  uint64_t a[32];  // 2^(i/32) 2^63
  uint64_t b[64];  // 2^(k/2048) 2^63
  uint64_t c;      // a2 log2(e) = c 2^(ex - 64), c's top bit set (c = 0 for a2 = 0)
  int ex;
  uint32_t limit;  // s is taken where its high word is below this: a2 s <= 700, s finite
};

// The tables, then with the scale of a2 >= 0 (finite).
inline ExpFixed exp_fixed_tables() {
  ExpFixed t{};
  for (int i = 0; i < 32; ++i) t.a[i] = (uint64_t)ldexpl(exp2l((long double)i / 32.0L), 63);
  for (int k = 0; k < 64; ++k) t.b[k] = (uint64_t)ldexpl(exp2l((long double)k / 2048.0L), 63);
  return t;
}

inline ExpFixed exp_fixed_constants(double a2) {
  static const ExpFixed tables = exp_fixed_tables();
  ExpFixed t = tables;
  const long double m = frexpl((long double)a2 / logl(2.0L), &t.ex);
  t.c = (uint64_t)ldexpl(m, 64);
  // the high word of 700 / a2: every s with a smaller high word satisfies
  // a2 s <= 700 (infinities and NaN lie above)
  const double most = a2 > 0.0 ? 700.0 / a2 : INFINITY;
  uint64_t bits;
  memcpy(&bits, &most, sizeof bits);
  t.limit = (uint32_t)(bits >> 32);
  // zero and subnormal s are taken with a significand that is not theirs, as
  // numbers below 2^-1022: with a larger scale their t would reach the result
  // (from 2^970 on exp(0) fell below 1), so no s is taken there
  if (t.ex > 900) t.limit = 0;
  return t;
}

// The high 64 bits of a b, without the product of the low words (at most 2
// below the exact value).
__device__ __forceinline__ uint64_t mul_hi64(uint64_t a, uint64_t b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  return (uint64_t)ah * bh + (uint64_t)__umulhi(ah, bl) + (uint64_t)__umulhi(al, bh);
}

// Logical right shift that gives 0 from 32 on, as the hardware's does.
__device__ __forceinline__ uint32_t shr32(uint32_t x, uint32_t s) {
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(s));
  return r;
}

__device__ __forceinline__ bool exp_fixed_in_range(double s, uint32_t limit) {
  return (uint32_t)__double2hiint(s) < limit;  // negative values and NaN compare above
}

// 2^-(n + f 2^-64), rounded to double; ta, tb: the tables (shared memory).
__device__ __forceinline__ double exp_fixed_tail(uint32_t n, uint64_t f, const uint64_t *ta, const uint64_t *tb) {
  const uint64_t g = ~f;
  const uint32_t gh = (uint32_t)(g >> 32);
  const uint64_t t = mul_hi64(ta[gh >> 27], tb[(gh >> 21) & 63u]);  // 2^(j/2048) 2^62
  const uint64_t x = g << 11;
  const uint32_t xh = (uint32_t)(x >> 32);
  // ln2^4/24 2^21, ln2^3/6 2^32, ln2^2/2 2^34, ln2 2^64
  constexpr uint32_t c4 = 20171u, c3 = 238388332u, c2 = 4127059964u;
  constexpr uint64_t c1 = 0xb17217f7d1cf79acull;
  const uint32_t s3 = c3 + __umulhi(xh, c4);
  const uint32_t s2 = c2 + (__umulhi(xh, s3) >> 9);
  const uint64_t s1 = c1 + (((uint64_t)xh * s2) >> 13);
  const uint64_t q = mul_hi64(x, s1);  // (2^r - 1) 2^75
  const uint64_t y = t + (mul_hi64(t, q) >> 11);
  return __longlong_as_double((long long)(((y + 512) >> 10) + ((uint64_t)(1021u - n) << 52)));
}

// exp(-a2 s) for s in range; ta, tb: the tables (shared memory).
__device__ __forceinline__ double exp_fixed(double s, const uint64_t *ta, const uint64_t *tb, uint64_t c, int ex) {
  const uint32_t sh = (uint32_t)__double2hiint(s), sl = (uint32_t)__double2loint(s);
  const int e = (int)(sh >> 20);
  // 64-bit significand (zero and subnormal s: t is below 2^-122 for the scales
  // that take any s, and every significand gives F below 2)
  const uint32_t mh = ((sh << 11) | (sl >> 21)) | 0x80000000u, ml = sl << 11;
  // h: the high 64 bits of the product, l: the next 32
  const uint32_t ch = (uint32_t)(c >> 32), cl = (uint32_t)c;
  const uint64_t p1 = (uint64_t)mh * cl, p2 = (uint64_t)ml * ch;
  const uint64_t mid = (p1 & 0xffffffffu) + (p2 & 0xffffffffu) + __umulhi(ml, cl);
  const uint64_t h = (uint64_t)mh * ch + (p1 >> 32) + (p2 >> 32) + (mid >> 32);
  const uint32_t l = (uint32_t)mid;
  const int k = e - 1022 + ex;  // t = h 2^(k - 64)
  const uint32_t n = shr32((uint32_t)(h >> 32), (uint32_t)(32 - k));
  const int right = k < 0 ? (k < -63 ? 63 : -k) : 0;
  const uint64_t f = k > 0 ? (h << k) | (l >> (32 - k)) : h >> right;
  return exp_fixed_tail(n, f, ta, tb);
}

}  // namespace hpac
