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
// Pairwise coprime (247 = 13 19, 217 = 7 31, the others primes and 2^8), and none of 251 .. 255, for
// which crt_reduce could leave a byte's range.
constexpr int CRT_MOD[CRT_MAX] = {256, 247, 241, 239, 233, 229, 227, 223, 217, 211, 199, 197, 193, 191, 181, 179};

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

// 2^B with 2 B <= log2(P / 4) less a rounding margin: log2 P is 63.09 for 8
// moduli, 101.42 for 13 and 123.98 for 16
constexpr float crt_norm_bits(int np) { return np == 8 ? 30.52f : np == 13 ? 49.68f : 60.96f; }

constexpr int CRT_ROW_NAN = 0x40000000;   // e_i of a row with a non-finite entry
constexpr int CRT_ROW_ZERO = 0x4000;      // of a zero row, where no other row's units may be coarsened by it

#ifdef __CUDACC__
namespace {

// The weights W_l = (P / p_l) ((P / p_l)^-1 mod p_l), 1 modulo p_l and 0 modulo the others
constexpr u128 crt_weight(int np, int l) { return crt_product(np) / (u128)CRT_MOD[l] * (u128)crt_inverse(np, l); }
// round(2^19 W_l / P), without overflow: W_l / P = inv_l / p_l
constexpr uint32_t crt_frac(int np, int l) {
  return (uint32_t)(((unsigned)crt_inverse(np, l) * (1u << 20) + (unsigned)CRT_MOD[l]) / (2u * (unsigned)CRT_MOD[l]));
}

// W_l in 32-bit limbs (16 moduli: below 2^124; 13: below 2^102) and as fractions;
// the constants that take out the bytes' offset of 128
template <int NP>
struct CombineTab {
  uint32_t limb[4][NP];
  uint32_t frac[NP];
};
template <int NP>
constexpr CombineTab<NP> make_combine() {
  CombineTab<NP> t{};
  for (int l = 0; l < NP; ++l) {
    for (int k = 0; k < 4; ++k) t.limb[k][l] = (uint32_t)(crt_weight(NP, l) >> (32 * k));
    t.frac[l] = crt_frac(NP, l);
  }
  return t;
}
constexpr u128 crt_offset(int np) {   // 128 sum W_l modulo 2^128
  u128 s = 0;
  for (int l = 0; l < np; ++l) s += crt_weight(np, l) * 128;
  return s;
}
constexpr uint32_t crt_frac_offset(int np) {
  uint32_t s = 0;
  for (int l = 0; l < np; ++l) s += 128 * crt_frac(np, l);
  return s;
}
__constant__ CombineTab<16> c_comb16 = make_combine<16>();
__constant__ CombineTab<13> c_comb13 = make_combine<13>();

// v modulo p as the nearest representative, v an integer of at most 2^24 in
// magnitude: the quotient is off by at most 2 / p from v / p, so the result is
// within 0.511 p of zero (p <= 247: 126; p = 256: 128, exactly).
__device__ __forceinline__ float crt_reduce(float v, float p, float rp) {
  const float q = __fsub_rn(__fadd_rn(__fmul_rn(v, rp), 12582912.0f), 12582912.0f);   // rint, |q| < 2^17
  return __fmaf_rn(-q, p, v);
}
// r + 128 in the low byte
__device__ __forceinline__ uint32_t crt_byte(float r) { return __float_as_uint(__fadd_rn(r, 12582912.0f + 128.0f)); }
__device__ __forceinline__ uint32_t crt_pack(uint32_t b0, uint32_t b1, uint32_t b2, uint32_t b3) {
  return __byte_perm(__byte_perm(b0, b1, 0x0040), __byte_perm(b2, b3, 0x0040), 0x5410);
}

// The integer c, |c| <= P / 4, from the bytes (residue + 128) at bit `sh` of the words
template <int NP>
__device__ __forceinline__ __int128 crt_value(const uint32_t (&w)[NP], int sh) {
  static_assert(NP == 16 || NP == 13, "tables of 16 and 13 moduli");
  constexpr u128 P = crt_product(NP), off = crt_offset(NP);
  constexpr unsigned long long PH = (unsigned long long)(P >> 64), PL = (unsigned long long)P,
                               OH = (unsigned long long)(off >> 64), OL = (unsigned long long)off;
  constexpr uint32_t f0 = crt_frac_offset(NP);
  unsigned long long S[4] = {0, 0, 0, 0};
  uint32_t f = 0;
#pragma unroll
  for (int l = 0; l < NP; ++l) {
    const uint32_t t = (w[l] >> sh) & 0xFFu;
#pragma unroll
    for (int k = 0; k < 4; ++k)   // below 2^44
      S[k] += (unsigned long long)t * (NP == 16 ? c_comb16.limb[k][l] : c_comb13.limb[k][l]);
    f += t * (NP == 16 ? c_comb16.frac[l] : c_comb13.frac[l]);
  }
  const int q = (int)(f - f0 + (1u << 18)) >> 19;   // round(sum r_l W_l / P): |c| <= P / 4 leaves no doubt
  u128 c = (u128)S[0] + ((u128)S[1] << 32) + ((u128)S[2] << 64) + ((u128)S[3] << 96);
  c -= (((u128)OH << 64) | OL) + (u128)(__int128)q * (((u128)PH << 64) | PL);   // modulo 2^128: |c| < 2^122
  return (__int128)c;
}

// v >> s for 0 <= s < 32, the sign kept
__device__ __forceinline__ __int128 i128_shr(__int128 v, int s) {
  const unsigned w0 = (unsigned)v, w1 = (unsigned)(v >> 32), w2 = (unsigned)(v >> 64), w3 = (unsigned)(v >> 96);
  const unsigned long long lo =
      (unsigned long long)__funnelshift_r(w1, w2, s) << 32 | __funnelshift_r(w0, w1, s);
  const unsigned long long hi = (unsigned long long)(unsigned)((int)w3 >> s) << 32 | __funnelshift_r(w2, w3, s);
  return (__int128)(((u128)hi << 64) | lo);
}

// v 2^-e rounded to nearest even, v a signed 128-bit integer
__device__ __forceinline__ double i128_to_double(__int128 v, int e) {
  if (v == 0) return 0.0;
  const bool neg = v < 0;
  const u128 a = neg ? (u128)(-v) : (u128)v;
  unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
  int z = 0;
  if (hi == 0) {
    hi = lo;
    lo = 0;
    z = 64;
  }
  const int y = __clzll((long long)hi);                   // leading bit to 127
  z += y;
  const unsigned long long top = (hi << y) | ((lo >> 1) >> (63 - y));
  const bool sticky = (lo << y) != 0;
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
