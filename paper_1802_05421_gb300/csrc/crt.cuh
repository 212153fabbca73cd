// Integer products by residues: the exact product of two integer matrices is
// formed modulo several small pairwise coprime moduli on the bf16 tensor
// cores and put together by the Chinese remainder theorem (the scheme of
// Ozaki, Uchino and Imamura, "Ozaki Scheme II", 2025, with bf16 residues).
//
// Symmetric residues of the moduli below are at most 128 in magnitude: exact in
// bf16, their products at most 2^14, so a float32 accumulator holds a sum of
// 1024 of them exactly. With the first NP moduli, P their product, every
// integer c with |c| <= P / 4 is recovered from its residues. Rows are scaled by
// powers of two so that their rounded integer images have 2-norm at most
// 2^CRT_NORM_BITS(NP) <= sqrt(P / 4); by Cauchy-Schwarz every dot product of two
// of them is then within P / 4.
#pragma once

#include <cstdint>

namespace cdl {

constexpr int CRT_MAX = 16;
// (pairwise coprime: 255 = 3 5 17, 253 = 11 23, 247 = 13 19, 217 = 7 31, the others primes and 2^8)
constexpr int CRT_MOD[CRT_MAX] = {256, 255, 253, 251, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193};

typedef unsigned __int128 u128;

constexpr u128 crt_product(int np) {
  u128 p = 1;
  for (int l = 0; l < np; ++l) p *= (u128)CRT_MOD[l];
  return p;
}

// P / p_l mod p_l, inverted
constexpr int crt_inverse(int np, int l) {
  const int p = CRT_MOD[l];
  int m = 1;
  for (int q = 0; q < np; ++q)
    if (q != l) m = m * (CRT_MOD[q] % p) % p;
  for (int x = 1; x < p; ++x)
    if (m * x % p == 1) return x;
  return 0;
}

constexpr uint32_t crt_magic(int p) {   // ceil(2^39 / p): floor(x / p) = umulhi(x, magic) >> 7 for x < 2^31
  return (uint32_t)(((1ull << 39) + (unsigned)p - 1) / (unsigned)p);
}

constexpr int crt_pow2_mod(int k, int p) {
  int r = 1 % p;
  for (int i = 0; i < k; ++i) r = r * 2 % p;
  return r;
}

// 2^B with 2 B <= log2(P / 4) less a rounding margin: log2 P is 63.575 for 8
// moduli and 125.376 for 16
constexpr float crt_norm_bits(int np) { return np == 8 ? 30.75f : 61.65f; }

constexpr int CRT_ROW_NAN = 0x40000000;   // e_i of a row with a non-finite entry
constexpr int CRT_ROW_ZERO = 0x4000;      // of a zero row, where no other row's units may be coarsened by it

#ifdef __CUDACC__
namespace {

// P / p_l in 20-bit limbs (16 moduli: below 2^118) and 2^23 / p_l
struct CombineTab64 {
  uint32_t limb[6][CRT_MAX];
  uint32_t frac[CRT_MAX];
};
constexpr CombineTab64 make_combine64() {
  CombineTab64 t{};
  const u128 P = crt_product(16);
  for (int l = 0; l < 16; ++l) {
    const u128 m = P / (u128)CRT_MOD[l];
    for (int k = 0; k < 6; ++k) t.limb[k][l] = (uint32_t)(m >> (20 * k)) & 0xFFFFFu;
    t.frac[l] = (uint32_t)(((1u << 24) + (unsigned)CRT_MOD[l]) / (2u * (unsigned)CRT_MOD[l]));
  }
  return t;
}
__constant__ CombineTab64 c_comb64 = make_combine64();
constexpr unsigned long long P64_HI = (unsigned long long)(crt_product(16) >> 64),
                             P64_LO = (unsigned long long)crt_product(16);

// The integer whose 16 t values (k_tc_crt) are the bytes at bit `sh` of the words
__device__ __forceinline__ __int128 crt16_value(const uint32_t (&w)[16], int sh) {
  uint32_t S[6] = {0, 0, 0, 0, 0, 0}, f = 0;
#pragma unroll
  for (int l = 0; l < 16; ++l) {
    const uint32_t t = (w[l] >> sh) & 0xFFu;
#pragma unroll
    for (int k = 0; k < 6; ++k) S[k] += t * c_comb64.limb[k][l];   // 16 terms below 2^28
    f += t * c_comb64.frac[l];
  }
  const uint32_t q = (f + (1u << 22)) >> 23;            // round(sum t_l / p_l): |c| <= P / 4 leaves no doubt
  u128 c = (u128)S[0] + ((u128)S[1] << 20) + ((u128)S[2] << 40) + ((u128)S[3] << 60) + ((u128)S[4] << 80) +
           ((u128)S[5] << 100);
  c -= (u128)q * (((u128)P64_HI << 64) | P64_LO);       // modulo 2^128: |c| < 2^124
  return (__int128)c;
}

// v 2^-e rounded to nearest even, v a signed 128-bit integer
__device__ __forceinline__ double i128_to_double(__int128 v, int e) {
  if (v == 0) return 0.0;
  const bool neg = v < 0;
  const u128 a = neg ? (u128)(-v) : (u128)v;
  const unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
  const int z = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
  const u128 n = a << z;                                  // leading bit 127
  const unsigned long long top = (unsigned long long)(n >> 64);
  const bool sticky = (unsigned long long)n != 0;
  unsigned long long q = top >> 11;
  const unsigned long long rem = top & 0x7FFull;
  if (rem > 0x400ull || (rem == 0x400ull && (sticky || (q & 1)))) ++q;   // may carry to 2^53: exact below
  const int ex = 127 - z - 52 - e;                        // value q 2^ex
  const unsigned long long sign = neg ? 1ull << 63 : 0ull;
  const int field = ex + 52 + 1023;
  if (field > 0 && field < 2046)                          // q in [2^52, 2^53]: adding carries into the exponent
    return __longlong_as_double((long long)(sign | (((unsigned long long)(field - 1) << 52) + q)));
  return ldexp(neg ? -(double)q : (double)q, ex);         // subnormal or out of range
}

}  // namespace
#endif

}  // namespace cdl
