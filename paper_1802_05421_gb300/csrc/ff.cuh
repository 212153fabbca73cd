// Float-float ("double-float") arithmetic on the float32 pipes, built from the
// classical error-free transformations: TwoSum (Knuth, TAOCP vol. 2), FastTwoSum
// (Dekker 1971) and TwoProduct through a fused multiply-add. A value is hi + lo
// with |lo| <= ulp(hi)/2, about 48 significant bits. Used where float64-class
// accuracy is needed in O(n^2) work, because float64 runs at about 1/72 of the
// float32 rate on this GPU.
#pragma once

#include <cstdint>

namespace cdl {

struct ff {
  float hi, lo;
};

__device__ __forceinline__ ff two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return {s, e};
}

// requires |a| >= |b| (or a == 0)
__device__ __forceinline__ ff fast_two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return fast_two_sum(p, e);
}

__device__ __forceinline__ ff ff_add(ff a, ff b) {
  ff s = two_sum(a.hi, b.hi);
  s.lo = __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo));
  return fast_two_sum(s.hi, s.lo);
}

__device__ __forceinline__ ff ff_from_double(double x) {
  const float h = __double2float_rn(x);
  return {h, __double2float_rn(x - (double)h)};
}

__device__ __forceinline__ double ff_to_double(ff a) { return (double)a.hi + (double)a.lo; }

// Conversions between float and double done with integer operations (the
// float64 pipe also executes the hardware conversions, and it is the scarce
// one on this GPU). f2d_bits is exact for normal floats and zero (subnormal
// floats map to zero); d2f_trunc truncates a double to 24 significant bits
// (exact for the top 24 bits; doubles below the float normal range map to
// zero, beyond it the result is meaningless, callers keep |x| < 2^127).
__device__ __forceinline__ double f2d_bits(float f) {
  const uint32_t b = __float_as_uint(f);
  const uint32_t e = (b >> 23) & 0xFFu;
  if (e == 0) return 0.0;
  const unsigned long long sign = (unsigned long long)(b >> 31) << 63;
  const unsigned long long ed = (unsigned long long)(e - 127 + 1023) << 52;
  const unsigned long long m = (unsigned long long)(b & 0x7FFFFFu) << 29;
  return __longlong_as_double((long long)(sign | ed | m));
}

// Split a float64 x >= 0 into floats hi + lo with hi = x truncated to 24 bits
// and lo the remaining 29 mantissa bits rounded to 24 (|x - hi - lo| <=
// 2^-48 x; below 2^-74, where lo falls under the float normal range, lo is
// subnormal and the bound is 2^-149 absolute), by integer operations and two
// exact scalings. Values below 2^-100 give {0, 0}, and so does -0.0 (the sign is
// shifted out).
__device__ __forceinline__ ff split_nonneg(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  if ((uint32_t)(b >> 32) << 1 < (1023u - 100u) << 21) return {0.f, 0.f};
  const uint32_t hi_bits = (uint32_t)(b >> 29) - ((1023u - 127u) << 23);   // x in [2^e, 2^(e+1)), e >= -100
  // lo = low29 2^(e - 52) = (low29 2^-52) 2^e: both factors are normal floats
  // for e >= -100 (2^(e - 52) itself is not, below e = -74)
  const float lo = __fmul_rn(__fmul_rn(__uint2float_rn((uint32_t)b & 0x1FFFFFFFu), 0x1p-52f),
                             __uint_as_float(hi_bits & 0x7F800000u));
  return {__uint_as_float(hi_bits), lo};
}

// The least e >= 0 with x <= 2^e, for the float64 bit pattern of x >= 0
// (zero gives 0).
__device__ __forceinline__ int pow2_exp_above(unsigned long long bits) {
  if (bits == 0) return 0;
  const int e = (int)((bits >> 52) & 0x7FF) - 1023;
  const int up = (bits & 0xFFFFFFFFFFFFFull) != 0 ? e + 1 : e;
  return up > 0 ? up : 0;
}

// Unsigned 64-bit integers to floating point with integer operations only.
// u64_top24: x truncated to its 24 leading bits, as a float (exact for x <
// 2^24). ff_from_u64: x as hi + lo, both truncations (|x - hi - lo| < 2^-47 x).
// u64_to_double_rn: x 2^scale_exp rounded to nearest even, the float64 the
// hardware conversion gives (x 2^scale_exp in the normal range).
__device__ __forceinline__ float u64_top24(unsigned long long x) {
  if (x == 0) return 0.f;
  const int e = 63 - __clzll((long long)x);
  const unsigned long long top = e >= 23 ? (x >> (e - 23)) : (x << (23 - e));
  return __uint_as_float(((uint32_t)(e + 127) << 23) | ((uint32_t)top & 0x7FFFFFu));
}

__device__ __forceinline__ ff ff_from_u64(unsigned long long x) {
  if (x == 0) return {0.f, 0.f};
  const int e = 63 - __clzll((long long)x);
  const unsigned long long rest = e > 23 ? x & ((1ull << (e - 23)) - 1ull) : 0ull;
  return {u64_top24(x), u64_top24(rest)};
}

__device__ __forceinline__ double u64_to_double_rn(unsigned long long x, int scale_exp) {
  if (x == 0) return 0.0;
  int e = 63 - __clzll((long long)x);
  unsigned long long m;
  if (e <= 52) {
    m = x << (52 - e);
  } else {
    const int sh = e - 52;
    unsigned long long q = x >> sh;
    const unsigned long long rem = x & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (q & 1ull))) ++q;
    if (q >> 53) {
      q >>= 1;
      ++e;
    }
    m = q;
  }
  return __longlong_as_double(
      (long long)(((unsigned long long)(e + 1023 + scale_exp) << 52) | (m & 0xFFFFFFFFFFFFFull)));
}

__device__ __forceinline__ float d2f_trunc(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF) - 1023 + 127;
  if (e <= 0) return 0.f;
  const uint32_t sign = (uint32_t)(b >> 32) & 0x80000000u;
  const uint32_t m = (uint32_t)(b >> 29) & 0x7FFFFFu;
  return __uint_as_float(sign | ((uint32_t)e << 23) | m);
}

// sqrt(x) for float64 x >= 0, within one ulp (correctly rounded but within about
// 2^-69 of a rounding midpoint), with three float64 operations: x = m 4^j with m in
// [1, 4) by the exponent field; sqrt(m) in float-float (about 2^-46), one Newton
// correction y + (m - y^2) / (2y) with the residual from one fused multiply-add
// and the quotient in float32; the result rescaled by 2^j through the exponent
// field. Zero and subnormal x take the float64 square root.
__device__ __forceinline__ double sqrt_nonneg(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF) - 1023;
  if (e == -1023) return __dsqrt_rn(x);
  const int j = e >> 1;                                // floor(e / 2)
  const double m = __longlong_as_double((long long)(b - ((unsigned long long)(long long)(2 * j) << 52)));
  const ff a = split_nonneg(m);
  const float sh = __fsqrt_rn(a.hi);
  const float h = __fdiv_rn(0.5f, sh);
  const float sl = __fmul_rn(__fadd_rn(__fmaf_rn(-sh, sh, a.hi), a.lo), h);
  const double y = __dadd_rn(f2d_bits(sh), f2d_bits(sl));
  const double r = __fma_rn(-y, y, m);
  const double ym = __dadd_rn(y, f2d_bits(__fmul_rn(d2f_trunc(r), h)));   // sqrt(m) in [1, 2]
  return __longlong_as_double((long long)((unsigned long long)__double_as_longlong(ym) +
                                          ((unsigned long long)(long long)j << 52)));
}

// exp(-x y) for float64 x >= 0 and a factor y > 0 prepared once per block, with
// integer operations only (float64 and its conversions run on the scarce pipe):
// u = x y log2(e) in fixed point with 54 fractional bits, from the 64-bit product
// of x's mantissa and the 64-bit factor c = y log2(e); 2^-u = 2^-k 2^(-j/256)
// 2^-g with k its integer part, j its next 8 bits and 0 <= g < 2^-8; 2^(-j/256)
// from a table of 64-bit integers; 2^-g = 1 - g (c1 - g (c2 - g (c3 - g c4))), c_i
// = (ln 2)^i / i!, from the exponential series (its degree 5 is below 1.2e-15),
// the inner terms in 32 bits (they are below 2^-10 of c1), the outer product and
// the product with the table in 64. Error at most 2.1e-15 relative, 2.0e-16 on
// average (a host emulation against quad precision over 3.5e6 arguments). About
// 80 instructions; through 128-bit shifts, ln 2 in natural units and a float-float
// series it took about 300, at 1.4e-14.
constexpr int EXP_TABLE = 256;
__constant__ const unsigned long long EXP2_NEG_16[16] = {   // 2^(63 - i / 16)
    0x8000000000000000ull, 0x7a92be8a92436616ull, 0x75606373ee921c97ull, 0x70666f76154a7089ull,
    0x6ba27e656b4eb57aull, 0x6712460a8fc24072ull, 0x62b39508aa836d6full, 0x5e8451cfac061b5full,
    0x5a827999fcef3242ull, 0x56ac1f752150a563ull, 0x52ff6b54d8a89c75ull, 0x4f7a993048d088d7ull,
    0x4c1bf828c6dc54b8ull, 0x48e1e9b9d588e19bull, 0x45cae0f1f545eb73ull, 0x42d561b3e6243d8aull};
__constant__ const unsigned long long EXP2_NEG_256[16] = {  // 2^(63 - i / 256)
    0x8000000000000000ull, 0x7fa765aca88f6453ull, 0x7f4f08ae3dc7c426ull, 0x7ef6e8da4b544f9aull,
    0x7e9f06067a4360baull, 0x7e47600890f223deull, 0x7deff6b672f84e24ull, 0x7d98c9e62113e1faull,
    0x7d41d96db915019dull, 0x7ceb252375c9cf9bull, 0x7c94acddaeea5d3aull, 0x7c3e7072d904a6ceull,
    0x7be86fb985689ddcull, 0x7b92aa886214411cull, 0x7b3d20b6399fc237ull, 0x7ae7d219f329b948ull};

// Threads 0 .. 255 of the block fill the table 2^(63 - j / 256); the caller
// synchronises before use.
__device__ __forceinline__ void exp_table(unsigned long long* tab) {
  for (int j = threadIdx.x; j < EXP_TABLE; j += blockDim.x) {
    const unsigned long long a = EXP2_NEG_16[j >> 4], b = EXP2_NEG_256[j & 15];
    tab[j] = (__umul64hi(a, b) << 1) | ((a * b) >> 63);
  }
}

struct ExpFactor {
  unsigned long long c;   // y log2(e) = c 2^(ey - 1023 - 62)
  int sh;                 // 2053 - ey: u 2^54 = (m c 2^-64) >> (sh - ex), m = x's mantissa with its leading bit at 63
  double y;
};
__device__ __forceinline__ ExpFactor exp_factor(double y) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(y);
  const int ey = (int)((b >> 52) & 0x7FF);
  if (ey == 0) return {0, 1 << 20, y};           // zero and subnormal: u counts as zero
  if (ey == 0x7FF) return {0, -(1 << 20), y};    // every x > 0 to the general path
  return {__umul64hi((b << 11) | (1ull << 63), 0xB8AA3B295C17F0BCull), 2053 - ey, y};   // log2(e) 2^63
}

// The high 64 bits of a b less at most 2 (the product of the low halves is left out).
__device__ __forceinline__ unsigned long long mul64_high(unsigned long long a, unsigned long long b) {
  const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
  return (unsigned long long)ah * bh + __umulhi(ah, bl) + __umulhi(al, bh);
}

__device__ __forceinline__ double exp_neg_prod(double x, const ExpFactor& f, const unsigned long long* __restrict__ tab) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(b >> 52);
  const int sh = ex == 0 ? 63 : min(f.sh - ex, 63);          // x zero or subnormal: u below 2^-54
  const unsigned long long u = mul64_high((b << 11) | (1ull << 63), f.c) >> (sh & 63);
  const uint32_t uh = (uint32_t)(u >> 32), k = uh >> 22;
  if (sh < 0 || k > 1000) return exp(-(x * f.y));            // near and below the normal range; infinities, NaN
  const uint32_t g = (uint32_t)(u >> 14);                    // g 2^40: the 32 bits below j
  const uint32_t c34 = 0xE35846B8u - (__umulhi(g, 0x9D955B7Eu) >> 10);   // c3 2^36, c4 2^38
  const uint32_t c234 = 0xF5FDEFFCu - (__umulhi(g, c34) >> 10);          // c2 2^34
  const unsigned long long s = 0xB17217F7D1CF79ACull - ((unsigned long long)__umulhi(g, c234) << 22);   // c1 2^64
  const unsigned long long t = tab[(uh >> 14) & 255u];
  const unsigned long long v = t - (mul64_high(t, mul64_high(u << 18, s)) >> 8);   // 2^63 2^(-j / 256) 2^-g
  return __longlong_as_double((long long)(((unsigned long long)(1021 - (int)k) << 52) + ((v + 512) >> 10)));
}

}  // namespace cdl
