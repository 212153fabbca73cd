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

}  // namespace cdl
