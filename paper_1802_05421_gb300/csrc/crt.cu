// Float64 and float32 chain squarings S~_{i+1} = S~_i^2 (Alg. 2, ChainProduct)
// on the bf16 tensor cores, by integer products through residues (crt.cuh):
//
//   k_crt_residues  row i of the level, scaled by the power of two 2^{e_i}
//                   that brings its 2-norm to 2^(B-1) .. 2^B (B =
//                   crt_norm_bits) and rounded to integers, as NP planes of
//                   symmetric residues in bf16;
//   k_tc_crt        the NP residue products (tc_gemm.cu);
//   k_crt_combine   c_ij 2^{e_i + e_j} from its NP residues (exact), rounded
//                   once to the level's type, and its mirror.
//
// The only errors are the rounding of the scaled rows, at most half a unit of
// 2^-B of the row's norm per entry (B = 60.9 bits with 16 moduli for float64
// levels, 30.5 with 8 for float32 ones), and the final rounding; a float64 or
// float32 dot product rounds every partial sum. Rows with a non-finite entry
// give NaN rows and columns.
//
// Bounds: the products by the tensor cores, 16 (8) times n^2 (n + 1) flop;
// the other two kernels by instruction issue (about 8 instructions per entry
// and plane in the first, 7 in the second). Measured, one squaring: float32 n =
// 8192 13.1 ms on the CUDA cores, here 2.52 ms of products (1.75 PFLOP/s) + 0.36
// + 0.12; float64 n = 1024 1.07 ms on the CUDA cores (1 TFLOP/s of the float64
// pipes), here 30 + 15 + 13 us. Relative error (Frobenius) of a square, n =
// 300 .. 4096: float64 4.7e-17 (5e-16 .. 1.9e-15 before), float32 2.5e-8 (5e-7
// .. 1e-6 before). One modulus less (15, 7) would pass on those graphs and
// save 1/16 (1/8) of the products, but for levels near a multiple of the
// identity the rounding of the rows would then exceed a dot product's.
#include <algorithm>

#include <cuda_bf16.h>

#include "crt.cuh"
#include "internal.h"
#include "score_ab.cuh"
#include "tiles.cuh"

namespace cdl {
namespace {

// 2^16, 2^32, 2^48 modulo p_l, nearest to zero, and 1 / p_l
struct ResidueTab {
  float c[3][CRT_MAX], mod[CRT_MAX], rmod[CRT_MAX];
};
constexpr ResidueTab make_residue_tab() {
  ResidueTab t{};
  for (int l = 0; l < CRT_MAX; ++l) {
    const int p = CRT_MOD[l];
    for (int k = 0; k < 3; ++k) {
      const int r = crt_pow2_mod(16 * (k + 1), p);
      t.c[k][l] = (float)(2 * r > p ? r - p : r);
    }
    t.mod[l] = (float)p;
    t.rmod[l] = 1.0f / (float)p;
  }
  return t;
}
__constant__ ResidueTab c_res = make_residue_tab();

struct CombineTab32 {
  uint32_t lo[8], hi[8], frac[8];
};
constexpr CombineTab32 make_combine32() {
  CombineTab32 t{};
  for (int l = 0; l < 8; ++l) {
    t.lo[l] = (uint32_t)crt_weight(8, l);
    t.hi[l] = (uint32_t)(crt_weight(8, l) >> 32);
    t.frac[l] = crt_frac(8, l);
  }
  return t;
}
__constant__ CombineTab32 c_comb32 = make_combine32();

// The two types' bit patterns: magnitude bits, exponent field and mantissa
// (value = m 2^(e - BIAS)), moduli.
template <typename T>
struct LevelType;
template <>
struct LevelType<double> {
  static constexpr int NP = 16, BIAS = 1075;
  static __device__ __forceinline__ unsigned long long mag(double x) {
    return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
  }
  static __device__ __forceinline__ int exponent(unsigned long long m) { return max((int)(m >> 52), 1); }
  static __device__ __forceinline__ unsigned long long mantissa(unsigned long long m) {
    return (m & 0xFFFFFFFFFFFFFull) | (m >> 52 ? 1ull << 52 : 0ull);
  }
  static __device__ __forceinline__ bool negative(double x) { return __double_as_longlong(x) < 0; }
  static __device__ __forceinline__ bool finite(unsigned long long m) { return (m >> 52) != 0x7FF; }
};
template <>
struct LevelType<float> {
  static constexpr int NP = 8, BIAS = 150;
  static __device__ __forceinline__ unsigned long long mag(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
  static __device__ __forceinline__ int exponent(unsigned long long m) { return max((int)(m >> 23), 1); }
  static __device__ __forceinline__ unsigned long long mantissa(unsigned long long m) {
    return (m & 0x7FFFFFull) | (m >> 23 ? 1ull << 23 : 0ull);
  }
  static __device__ __forceinline__ bool negative(float x) { return __float_as_int(x) < 0; }
  static __device__ __forceinline__ bool finite(unsigned long long m) { return (m >> 23) != 0xFF; }
};

// round(x 2^e) for |x 2^e| < 2^62, ties away from zero
template <typename T>
__device__ __forceinline__ long long scaled_int(T x, int e) {
  const unsigned long long mg = LevelType<T>::mag(x);
  const unsigned long long m = LevelType<T>::mantissa(mg);
  const int sh = LevelType<T>::exponent(mg) - LevelType<T>::BIAS + e;
  unsigned long long v;
  if (sh >= 0)
    v = m << min(sh, 63);
  else
    v = sh > -60 ? (m + (1ull << (-sh - 1))) >> -sh : 0;
  return LevelType<T>::negative(x) ? -(long long)v : (long long)v;
}

// x = d_0 + 2^16 d_1 + .. in ND balanced digits of 16 bits, as floats (|x| < 2^(16
// ND - 2)): the unsigned digits of x + 0x8000.. through the float 2^23 + u.
template <int ND>
__device__ __forceinline__ void digits16(long long x, float (&d)[ND]) {
  const unsigned long long w = (unsigned long long)x + (ND == 4 ? 0x8000800080008000ull : 0x80008000ull);
  const uint32_t lo = (uint32_t)w, hi = (uint32_t)(w >> 32);
#pragma unroll
  for (int k = 0; k < ND; ++k) {
    const uint32_t u = __byte_perm(k < 2 ? lo : hi, 0x4B000000u, k & 1 ? 0x7632u : 0x7610u);
    d[k] = __fsub_rn(__uint_as_float(u), 8421376.0f);   // 2^23 + 2^15
  }
}

// The residue modulo p_l as float bits (an integer of magnitude at most 128: the
// upper half is its bf16): sum d_k (2^16k mod p) is exact in float32 (three
// terms of at most 2^15 123, below 2^24), then as crt_reduce. All at the
// float32 rate; 32-bit multiplications and their high halves run at half of it
// and less.
template <int ND>
__device__ __forceinline__ uint32_t residue_bits(const float (&d)[ND], int l) {
  float r = d[0];
#pragma unroll
  for (int k = 1; k < ND; ++k) r = __fmaf_rn(d[k], c_res.c[k - 1][l], r);
  const float q = __fsub_rn(__fmaf_rn(r, c_res.rmod[l], 12582912.0f), 12582912.0f);
  return __float_as_uint(__fmaf_rn(-q, c_res.mod[l], r));
}

// The power of two next to sqrt(d) as its exponent (0 for zero and non-finite d)
__device__ __forceinline__ int sqrt_exponent(double d) {
  const int e = (int)(LevelType<double>::mag(d) >> 52);
  return e == 0 || e == 0x7FF ? 0 : (e - 1023) >> 1;
}

// One block per row of a rows x cols matrix (zero beyond, to gridDim.x x np):
// the row's largest exponent, then its 2-norm relative to it (float32, a
// margin covers its rounding), e_i, and the residues. Columns in pairs; np a
// multiple of 64. W: column j is first scaled by the power of two next to
// w_j^{-1/2}.
template <typename T, bool W = false>
__global__ void __launch_bounds__(256) k_crt_residues(const T* __restrict__ X, int rows, int cols, int ldx, int np,
                                                       const double* __restrict__ w, int* __restrict__ ex,
                                                       uint32_t* __restrict__ planes) {
  follow();
  typedef LevelType<T> LT;
  constexpr unsigned BIG = ~0u;                           // key of a non-finite entry
  constexpr int OFF = 4096;                               // keys of the others: exponent + OFF; of zeros: 0
  __shared__ unsigned wmax[8];
  __shared__ float wsum[8];
  const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const T* x = X + (size_t)row * ldx;
  if (row >= rows) cols = 0;
  auto shift = [&](int j) { return W ? sqrt_exponent(w[j]) : 0; };
  unsigned mx = 0;
  for (int j = tid; j < cols; j += 256) {
    const unsigned long long m = LT::mag(x[j]);
    mx = max(mx, m == 0 ? 0u : LT::finite(m) ? (unsigned)(LT::exponent(m) - shift(j) + OFF) : BIG);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) wmax[warp] = mx;
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) mx = max(mx, wmax[q]);
  const bool fin = mx != BIG;
  // |x| 2^-emax in [0, 2): emax = exponent of the largest
  const int emax = fin ? (int)mx - OFF - LT::BIAS + (sizeof(T) == 8 ? 52 : 23) : 0;
  float s = 0.f;
  for (int j = tid; j < cols; j += 256) {
    const float v = (float)(int)scaled_int(x[j], 22 - emax - shift(j));   // magnitude up to 2^23, exact in float32
    s = __fmaf_rn(v, v, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) wsum[warp] = s;
  __syncthreads();
  s = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) s += wsum[q];
  // norm 2^(e + 22 - emax) = sqrt(s); rounding and truncation within the 0.02 bits of margin
  // (s < 1: zero, or so far below the smallest normal number that every square underflows)
  const int e = s >= 1.f ? (int)floorf(crt_norm_bits(LT::NP) - 0.02f - 0.5f * log2f(s)) + 22 - emax : 0;
  if (tid == 0) ex[row] = fin ? e : CRT_ROW_NAN;
  const size_t plane = (size_t)gridDim.x * np / 2;
  uint32_t* out = planes + (size_t)row * np / 2;
  for (int j = tid; j < np / 2; j += 256) {
    constexpr int ND = sizeof(T) == 8 ? 4 : 2;
    float d[2][ND];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      digits16<ND>(fin && 2 * j + h < cols ? scaled_int(x[2 * j + h], e - shift(2 * j + h)) : 0, d[h]);
#pragma unroll
    for (int l = 0; l < LT::NP; ++l)
      out[l * plane + j] = __byte_perm(residue_bits<ND>(d[0], l), residue_bits<ND>(d[1], l), 0x7632);
  }
}

template <typename T>
struct Combine;
template <>
struct Combine<double> {
  static constexpr int NP = 16;
  // c from the bytes at bit `sh` of the 16 words
  static __device__ __forceinline__ double value(const uint32_t (&w)[16], int sh, int e) {
    return i128_to_double(crt_value<16>(w, sh), e);
  }
  static __device__ __forceinline__ double nan() { return __longlong_as_double(0x7FF8000000000000ll); }
};
template <>
struct Combine<float> {
  static constexpr int NP = 8;
  static __device__ __forceinline__ float value(const uint32_t (&w)[8], int sh, int e) {
    constexpr unsigned long long P = (unsigned long long)crt_product(8), off = (unsigned long long)crt_offset(8);
    constexpr uint32_t f0 = crt_frac_offset(8);
    unsigned long long c = 0;
    uint32_t hi = 0, f = 0;
#pragma unroll
    for (int l = 0; l < 8; ++l) {
      const uint32_t t = (w[l] >> sh) & 0xFFu;
      c += (unsigned long long)t * c_comb32.lo[l];
      hi += t * c_comb32.hi[l];
      f += t * c_comb32.frac[l];
    }
    const int q = (int)(f - f0 + (1u << 18)) >> 19;
    c += ((unsigned long long)hi << 32) - off - (unsigned long long)(long long)q * P;   // modulo 2^64: |c| < 2^62
    return ldexpf(__ll2float_rn((long long)c), -e);
  }
  static __device__ __forceinline__ float nan() { return __int_as_float(0x7FC00000); }
};

// C (np x np) from the residues t (NP planes of np x np bytes, valid on and
// above the diagonal blocks): 64 x 64 tiles of the upper block triangle, each
// thread four columns of a row at a time (one word per plane), the mirror
// through shared memory.
template <typename T>
__global__ void __launch_bounds__(256) k_crt_combine(const uint8_t* __restrict__ t, int np,
                                                      const int* __restrict__ ex, T* __restrict__ C) {
  follow();
  constexpr int NP = Combine<T>::NP;
  __shared__ T tile[64][65];
  int bi, bj;
  block_tri_index(np / 64, bi, bj);
  const int r0 = bi * 64, c0 = bj * 64;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const size_t plane = (size_t)np * np;
  int ec[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) ec[e] = ex[c0 + tx * 4 + e];
#pragma unroll 1
  for (int m = 0; m < 4; ++m) {
    const int r = ty + 16 * m;
    const int er = ex[r0 + r];
    const uint8_t* src = t + (size_t)(r0 + r) * np + c0 + tx * 4;
    uint32_t w[NP];
#pragma unroll
    for (int l = 0; l < NP; ++l) w[l] = *reinterpret_cast<const uint32_t*>(src + l * plane);
    T v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      v[e] = (er == CRT_ROW_NAN || ec[e] == CRT_ROW_NAN) ? Combine<T>::nan() : Combine<T>::value(w, 8 * e, er + ec[e]);
    T* dst = C + (size_t)(r0 + r) * np + c0 + tx * 4;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      dst[e] = v[e];
      tile[tx * 4 + e][r] = v[e];
    }
  }
  if (bi == bj) return;
  __syncthreads();
  for (int e = threadIdx.x; e < 64 * 64; e += 256) C[(size_t)(c0 + e / 64) * np + r0 + e % 64] = tile[e / 64][e % 64];
}

// The median of five values in the order of their bit patterns as signed numbers
// (NaNs at the ends), 0 where that is not finite.
__device__ __forceinline__ double median5(double a, double b, double c, double d, double e) {
  auto key = [](double v) {
    const long long x = __double_as_longlong(v);
    return x ^ (x >> 63 & 0x7FFFFFFFFFFFFFFFll);
  };
  const long long ka = key(a), kb = key(b), kc = key(c), kd = key(d), ke = key(e);
  const long long f = max(min(ka, kb), min(kc, kd)), g = min(max(ka, kb), max(kc, kd));
  const long long m = max(min(ke, f), min(max(ke, f), g));
  const long long x = m ^ (m >> 63 & 0x7FFFFFFFFFFFFFFFll);
  const double v = __longlong_as_double(x);
  return LevelType<double>::finite(LevelType<double>::mag(v)) ? v : 0.0;
}

// Node series for the residue distances (k_tc_gramr): row i less one common
// series (distances do not change, and the common part of all nodes costs no
// bits), scaled by the power of two 2^{e_i} that brings its 2-norm to 2^60.96
// at most and keeps both series below 2^61, rounded to integers (each entry
// within one unit), as 16 residue planes (rows x kp, zero padded), with its
// exact squared norm. The common series is the median, sample by sample, of five
// nodes spread over the rows: one or two of them may be far off or not finite
// (fill values, a dead instrument). With node 0 in its place such a value there put
// every distance below 2^-6 of the distances to it, and all went through the
// float64 kernel (n = 8192, T = 128: 26.6 ms instead of 1.3). One block of 128
// threads per row, the common series in T doubles of shared memory; also clears the
// tile flags. Series of fewer than DIST_RES_MIN_T samples flag every tile instead:
// they stay with the float64 kernel. Nothing on the grid inputs of
// the other kernel.
__global__ void __launch_bounds__(128) k_series_residues(const double* __restrict__ X, int n, int T, int rows, int kp,
                                                          const int* __restrict__ offgrid, int* __restrict__ ex,
                                                          ulonglong2* __restrict__ norms,
                                                          uint32_t* __restrict__ planes, uint32_t* __restrict__ bad,
                                                          int bad_words) {
  follow();
  if (!(*offgrid & 1)) return;
  typedef LevelType<double> LT;
  __shared__ unsigned long long wmax[2][4];
  __shared__ float wsum[4];
  __shared__ ulonglong2 wn[4];
  const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t flags = T < DIST_RES_MIN_T ? 0x01010101u : 0u;
  for (int w = row * 128 + tid; w < bad_words; w += gridDim.x * 128) bad[w] = flags;
  if (flags) return;
  const bool real = row < n;
  const double* x = X + (size_t)(real ? row : 0) * T;
  extern __shared__ double org[];
  for (int t = tid; t < T; t += 128) {
    auto at = [&](int q) { return X[(size_t)((long long)q * (n - 1) / 4) * T + t]; };
    org[t] = median5(at(0), at(1), at(2), at(3), at(4));
  }
  __syncthreads();
  unsigned long long mx = 0, md = 0;
  for (int t = tid; t < T; t += 128) {
    mx = max(mx, max(LT::mag(x[t]), LT::mag(org[t])));
    md = max(md, LT::mag(__dsub_rn(x[t], org[t])));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    md = max(md, __shfl_xor_sync(0xffffffffu, md, o));
  }
  if (lane == 0) {
    wmax[0][warp] = mx;
    wmax[1][warp] = md;
  }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    mx = max(mx, wmax[0][w]);
    md = max(md, wmax[1][w]);
  }
  const bool fin = LT::finite(mx) && LT::finite(md);
  const int emax = LT::exponent(md) - LT::BIAS + 52;
  float s = 0.f;
  if (fin)
    for (int t = tid; t < T; t += 128) {
      const float v = (float)(int)scaled_int(__dsub_rn(x[t], org[t]), 22 - emax);
      s = __fmaf_rn(v, v, s);
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) wsum[warp] = s;
  __syncthreads();
  s = wsum[0] + wsum[1] + wsum[2] + wsum[3];
  const bool any = real && fin && s >= 1.f;
  int e = CRT_ROW_ZERO;
  if (any) {
    e = (int)floorf(crt_norm_bits(16) - 0.02f - 0.5f * log2f(s)) + 22 - emax;
    e = min(e, 60 - (LT::exponent(mx) - LT::BIAS + 52));
  }
  if (tid == 0) ex[row] = fin ? e : CRT_ROW_NAN;
  const size_t plane = (size_t)rows * kp / 2;
  uint32_t* out = planes + (size_t)row * kp / 2;
  u128 nn = 0;
  for (int j = tid; j < kp / 2; j += 128) {
    float d[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int t = 2 * j + h;
      const long long v = any && t < T ? scaled_int(x[t], e) - scaled_int(org[t], e) : 0;
      nn += (u128)((__int128)v * v);
      digits16<4>(v, d[h]);
    }
#pragma unroll
    for (int l = 0; l < 16; ++l)
      out[l * plane + j] = __byte_perm(residue_bits<4>(d[0], l), residue_bits<4>(d[1], l), 0x7632);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)nn, o);
    const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)(nn >> 64), o);
    nn += ((u128)hi << 64) | lo;
  }
  if (lane == 0) wn[warp] = make_ulonglong2((unsigned long long)nn, (unsigned long long)(nn >> 64));
  __syncthreads();
  if (tid == 0) {
    nn = 0;
    for (int w = 0; w < 4; ++w) nn += ((u128)wn[w].y << 64) | wn[w].x;
    norms[row] = make_ulonglong2((unsigned long long)nn, (unsigned long long)(nn >> 64));
  }
}

// ---- CAD scores (k_tc_gramr) on a and b of score_ab.

// What g is chosen from (zeroed before): the largest |a| and |b| as exponent
// fields, and over the rows' largest |a| and |b| the sums of the exponents and
// the rows that have one. A warp per row, one set of global atomics per block
// (per warp they took 20 us at n = 8192).
struct ScoreScale {
  int amax, bmax;
  int gexp;               // log2 g, left by k_score_residues
  int asum, acnt, bsum, bcnt;
  int pad;
};

__global__ void __launch_bounds__(256) k_score_maxima(const double* __restrict__ Z1, const double* __restrict__ Z2,
                                                       const double* __restrict__ vol1,
                                                       const double* __restrict__ vol2, int n, int k,
                                                       ScoreScale* __restrict__ sc) {
  follow();
  __shared__ ScoreScale bl;
  const double s1 = sqrt(*vol1), s2 = sqrt(*vol2);
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) bl = ScoreScale{};
  __syncthreads();
  int ma = 0, mb = 0, asum = 0, acnt = 0, bsum = 0, bcnt = 0;
  for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < n; i += gridDim.x * 8) {
    int ea = 0, eb = 0;
    for (int r = lane; r < k; r += 32) {
      double a, b;
      score_ab(Z1, Z2, s1, s2, (size_t)i * k + r, a, b);
      ea = max(ea, (int)(LevelType<double>::mag(a) >> 52));
      eb = max(eb, (int)(LevelType<double>::mag(b) >> 52));
    }
    ea = __reduce_max_sync(0xffffffffu, ea);
    eb = __reduce_max_sync(0xffffffffu, eb);
    ma = max(ma, ea);
    mb = max(mb, eb);
    if (ea > 0 && ea < 0x7FF) {
      asum += ea - 1023;
      ++acnt;
    }
    if (eb > 0 && eb < 0x7FF) {
      bsum += eb - 1023;
      ++bcnt;
    }
  }
  auto add = [](ScoreScale* t, int a, int b, int as, int ac, int bs, int bc) {
    atomicMax(&t->amax, a);
    atomicMax(&t->bmax, b);
    atomicAdd(&t->asum, as);
    atomicAdd(&t->acnt, ac);
    atomicAdd(&t->bsum, bs);
    atomicAdd(&t->bcnt, bc);
  };
  if (lane == 0) add(&bl, ma, mb, asum, acnt, bsum, bcnt);
  __syncthreads();
  if (threadIdx.x == 0) add(sc, bl.amax, bl.bmax, bl.asum, bl.acnt, bl.bsum, bl.bcnt);
}

// log2 g: g brings the largest |a| to the binade of the largest |b|, or of three
// binades above the rows' mean exponent of |b| where that is less (g > 1; for g <
// 1 the halves change places): a few rows far above the others (nodes of tiny
// degree) must not scale the other rows' a up until their b has no bits left. With
// g = 1 every row keeps both halves to 2^-B of its own size, which is within the
// rounding of a and b themselves. One node of 200 with |Z| 1e9 times the others',
// equal volumes, float64 scores: 5e-10 relative by the largest alone, 8e-16 so.
__device__ __forceinline__ int score_gexp(const ScoreScale& s) {
  auto mean = [](int sum, int cnt) { return cnt > 0 ? sum / cnt + (sum % cnt > 0) : 0; };   // rounded up
  const int ea = s.amax, eb = s.bmax;
  if (ea == 0 || eb == 0 || ea >= 0x7FF || eb >= 0x7FF) return 0;   // zero or non-finite maxima: no balancing
  if (eb > ea) return min(eb - ea, max(0, mean(s.bsum, s.bcnt) + 3 - (ea - 1023)));
  return max(eb - ea, min(0, (eb - 1023) - mean(s.asum, s.acnt) - 3));
}

// Row i: u_i = [g a_i | b_i] of 2-norm 2^B at most (B = crt_norm_bits) after the
// power of two 2^{e_i}, rounded to integers, as NP residue planes of u and of v
// = [b_i | g a_i] (rows x kp, zero padded), and d'_i = (g a_i) . b_i of the
// integers, exact; g from score_gexp. A block of 128 per row.
template <int NP>
__global__ void __launch_bounds__(128) k_score_residues(const double* __restrict__ Z1, const double* __restrict__ Z2,
                                                         const double* __restrict__ vol1,
                                                         const double* __restrict__ vol2, int n, int k, int rows,
                                                         int kp, ScoreScale* __restrict__ sc, int* __restrict__ ex,
                                                         ulonglong2* __restrict__ dself,
                                                         __nv_bfloat16* __restrict__ up,
                                                         __nv_bfloat16* __restrict__ vp) {
  follow();
  typedef LevelType<double> LT;
  __shared__ unsigned long long wmax[4];
  __shared__ float wsum[4];
  __shared__ ulonglong2 wn[4];
  const int row = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double s1 = sqrt(*vol1), s2 = sqrt(*vol2);
  const int ge = score_gexp(*sc);
  if (row == 0 && tid == 0) sc->gexp = ge;
  const int cols = row < n ? k : 0;
  // magnitudes as exponents relative to g: |g a| is compared through the exponent field
  unsigned long long m = 0;
  for (int r = tid; r < cols; r += 128) {
    double a, b;
    score_ab(Z1, Z2, s1, s2, (size_t)row * k + r, a, b);
    m = max(m, max(LT::mag(scalbn(a, ge)), LT::mag(b)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) wmax[warp] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 4; ++w) m = max(m, wmax[w]);
  const bool fin = LT::finite(m);
  const int emax = LT::exponent(m) - LT::BIAS + 52;
  float s = 0.f;
  if (fin)
    for (int r = tid; r < cols; r += 128) {
      double a, b;
      score_ab(Z1, Z2, s1, s2, (size_t)row * k + r, a, b);
      const float x = (float)(int)scaled_int(a, 22 - emax + ge), y = (float)(int)scaled_int(b, 22 - emax);
      s = __fmaf_rn(x, x, __fmaf_rn(y, y, s));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) wsum[warp] = s;
  __syncthreads();
  s = wsum[0] + wsum[1] + wsum[2] + wsum[3];
  const bool any = fin && s >= 1.f;
  const int e = any ? (int)floorf(crt_norm_bits(NP) - 0.02f - 0.5f * log2f(s)) + 22 - emax : CRT_ROW_ZERO;
  if (tid == 0) ex[row] = fin ? e : CRT_ROW_NAN;
  const size_t plane = (size_t)rows * kp;
  __nv_bfloat16 *u = up + (size_t)row * kp, *v = vp + (size_t)row * kp;
  __int128 dd = 0;
  for (int r = tid; r < k; r += 128) {
    long long x = 0, y = 0;
    if (any && r < cols) {
      double a, b;
      score_ab(Z1, Z2, s1, s2, (size_t)row * k + r, a, b);
      x = scaled_int(a, e + ge);
      y = scaled_int(b, e);
      dd += (__int128)x * y;
    }
    float dx[4], dy[4];
    digits16<4>(x, dx);
    digits16<4>(y, dy);
#pragma unroll
    for (int l = 0; l < NP; ++l) {
      const uint32_t rx = residue_bits<4>(dx, l), ry = residue_bits<4>(dy, l);
      const __nv_bfloat16 bx = __ushort_as_bfloat16((unsigned short)(rx >> 16)),
                          by = __ushort_as_bfloat16((unsigned short)(ry >> 16));
      u[l * plane + r] = bx;
      u[l * plane + k + r] = by;
      v[l * plane + r] = by;
      v[l * plane + k + r] = bx;
    }
  }
  for (int r = 2 * k + tid; r < kp; r += 128)
    for (int l = 0; l < NP; ++l) u[l * plane + r] = v[l * plane + r] = __ushort_as_bfloat16(0);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)(u128)dd, o);
    const unsigned long long hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)((u128)dd >> 64), o);
    dd += (__int128)(((u128)hi << 64) | lo);
  }
  if (lane == 0) wn[warp] = make_ulonglong2((unsigned long long)(u128)dd, (unsigned long long)((u128)dd >> 64));
  __syncthreads();
  if (tid == 0) {
    u128 t = 0;
    for (int w = 0; w < 4; ++w) t += ((u128)wn[w].y << 64) | wn[w].x;
    dself[row] = make_ulonglong2((unsigned long long)t, (unsigned long long)(t >> 64));
  }
}

// X (rows x cols, leading dimension ldx) transposed to out (gridDim.y 32 rows x
// np), zero beyond; 32 x 32 tiles. With w (may be null) row i is scaled by the
// power of two next to w_i^{1/2} (exactly).
__global__ void __launch_bounds__(256) k_transpose_pad(const double* __restrict__ X, int rows, int cols, int ldx,
                                                        int np, const double* __restrict__ w,
                                                        double* __restrict__ out) {
  follow();
  __shared__ double tile[32][33];
  const int i0 = blockIdx.x * 32, c0 = blockIdx.y * 32, tx = threadIdx.x & 31;
  for (int a = threadIdx.x >> 5; a < 32; a += 8) {
    const int i = i0 + a;
    double v = (i < rows && c0 + tx < cols) ? X[(size_t)i * ldx + c0 + tx] : 0.0;
    if (w && i < rows) v *= __longlong_as_double((long long)(1023 + sqrt_exponent(w[i])) << 52);
    tile[a][tx] = v;
  }
  __syncthreads();
  for (int a = threadIdx.x >> 5; a < 32; a += 8) out[(size_t)(c0 + a) * np + i0 + tx] = tile[tx][a];
}

// (M x)_ir of four consecutive columns r from the residues t (16 planes of np x kpb bytes).
__device__ __forceinline__ void product4(const uint8_t* __restrict__ t, int np, int kpb, const int* __restrict__ erow,
                                         const int* __restrict__ ecol, int i, int r, double (&v)[4]) {
  const uint8_t* src = t + (size_t)i * kpb + r;
  uint32_t w[16];
#pragma unroll
  for (int l = 0; l < 16; ++l) w[l] = *reinterpret_cast<const uint32_t*>(src + (size_t)l * np * kpb);
  const int er = erow[i];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int ec = ecol[r + e];
    v[e] = (er == CRT_ROW_NAN || ec == CRT_ROW_NAN) ? Combine<double>::nan()
                                                    : Combine<double>::value(w, 8 * e, er + ec);
  }
}

// x += M x (x: np x kp, kp a multiple of 4)
__global__ void __launch_bounds__(128) k_crt_add(const uint8_t* __restrict__ t, int np, int kpb, int kp,
                                                  const int* __restrict__ erow, const int* __restrict__ ecol,
                                                  double* __restrict__ x) {
  follow();
  const int q = kp / 4;
  const size_t idx = blockIdx.x * (size_t)128 + threadIdx.x;
  if (idx >= (size_t)np * q) return;
  const int i = (int)(idx / q), r = (int)(idx % q) * 4;
  double v[4];
  product4(t, np, kpb, erow, ecol, i, r, v);
#pragma unroll
  for (int e = 0; e < 4; ++e) x[(size_t)i * kp + r + e] += v[e];
}

// R = (Y - D o Z) + A Z, and per-block sums of R^2 (fixed order).
__global__ void __launch_bounds__(128) k_crt_residual(const uint8_t* __restrict__ t, int np, int kpb,
                                                       const int* __restrict__ erow, const int* __restrict__ ecol,
                                                       const double* __restrict__ Y, const double* __restrict__ Z,
                                                       const double* __restrict__ D, int n, int k,
                                                       double* __restrict__ R, double* __restrict__ part) {
  follow();
  __shared__ double red[4];
  const int q = (k + 3) / 4;
  double sq = 0.0;
  for (size_t idx = blockIdx.x * (size_t)128 + threadIdx.x; idx < (size_t)n * q; idx += (size_t)gridDim.x * 128) {
    const int i = (int)(idx / q), r = (int)(idx % q) * 4;
    double v[4];
    product4(t, np, kpb, erow, ecol, i, r, v);
    const double d = D[i];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (r + e < k) {
        const size_t o = (size_t)i * k + r + e;
        const double x = (Y[o] - d * Z[o]) + v[e];
        R[o] = x;
        sq = fma(x, x, sq);
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sq;
  __syncthreads();
  if (threadIdx.x == 0) part[blockIdx.x] = ((red[0] + red[1]) + red[2]) + red[3];
}

template <typename T>
int square_impl(cdl_ctx* ctx, cdl_chain* ch, int level, void* planes, uint8_t* t, int* ex) {
  constexpr int NP = Combine<T>::NP;
  const int np = (int)ch->npad;
  {
    Launch L(ctx, CDL_KC_SQUARE, 0);
    launch_next(k_crt_residues<T>, np, 256, 0, ctx->stream, static_cast<const T*>(ch->level(level)), np, np, np, np,
                nullptr, ex, static_cast<uint32_t*>(planes));
    CDL_TRY(L.done());
  }
  CDL_TRY(crt_gemm(ctx, planes, np, nullptr, 0, np, NP, t, CDL_KC_SQUARE, (double)ch->n * ch->n * (ch->n + 1.0)));
  const int nb = np / 64;
  Launch L(ctx, CDL_KC_SQUARE, 0);
  launch_next(k_crt_combine<T>, nb * (nb + 1) / 2, 256, 0, ctx->stream, t, np, ex,
              static_cast<T*>(ch->level(level + 1)));
  return L.done();
}

}  // namespace

// Squares a float64 or float32 level. CDL_ERR_UNSUPPORTED (nothing launched)
// when the order is past the exact sums' range, the device lacks the
// tensor-core path, or its workspace (3 NP bytes per entry) is not to be had.
int chain_square_crt(cdl_ctx* ctx, cdl_chain* ch, int level) {
  const size_t cnt = (size_t)ch->npad * ch->npad;
  const int planes = ch->dtype == CDL_F64 ? 16 : 8;
  if ((ch->dtype != CDL_F64 && ch->dtype != CDL_F32) || !crt_gemm_supported(ctx, (int)ch->npad))
    return CDL_ERR_UNSUPPORTED;
  CDL_TRY(crt_gemm_prepare(ctx, (int)ch->npad, 0));
  void *vp, *vt, *ve;
  if (ws_get_opt(ctx, {{"crt.planes", planes * cnt * 2, &vp},
                       {"crt.t", planes * cnt, &vt},
                       {"crt.e", (size_t)ch->npad * sizeof(int), &ve}}) != CDL_OK)
    return CDL_ERR_UNSUPPORTED;
  if (ch->dtype == CDL_F64)
    return square_impl<double>(ctx, ch, level, vp, static_cast<uint8_t*>(vt), static_cast<int*>(ve));
  return square_impl<float>(ctx, ch, level, vp, static_cast<uint8_t*>(vt), static_cast<int*>(ve));
}

// ---------------------------------------------------------------- products with right-hand sides
// M x for a float64 matrix M (a chain level, or the graph in the residual) and
// k right-hand sides, through 16 residues as the squaring: the rows of M and
// the columns of x are scaled by their 2-norms, the product is exact, one
// rounding per entry. With weights w (the residual's degrees D) it is formed as
// (M w^{-1/2}) (w^{1/2} x), the roots as powers of two, so exactly the same: A
// D^{-1/2} and D^{1/2} Z have entries of one size also where degrees span many
// orders of magnitude (Z is about D^{-1/2}), and no bits go to a few huge entries
// of Z. Without, one node of degree 5e-18 of the others' left a relative residual of
// 3e-12 that no further step made smaller, with it 1.8e-16 (n = 600, float64 chain). The float64
// pipe's dot products took 0.52 ms per level at n = 2000, k = 32 (its FMA rate);
// here the residues of M take most of the time (8 n^2 bytes read, 32 n^2 written).
int crt_apply_begin(cdl_ctx* ctx, int np, int k, CrtApply* a) {
  if (!crt_gemm_supported(ctx, np)) return CDL_ERR_UNSUPPORTED;
  a->np = np;
  a->kpb = (int)round_up(k, k <= 256 ? 64 : 256);
  CDL_TRY(crt_gemm_prepare(ctx, np, a->kpb));
  const size_t kx = (size_t)a->kpb * np;
  void *vp, *vx, *vxp, *vt, *ve;
  if (ws_get_opt(ctx, {{"crt.planes", (size_t)16 * np * np * 2, &vp},
                       {"crt.xt", kx * sizeof(double), &vx},
                       {"crt.xplanes", 16 * kx * 2, &vxp},
                       {"crt.xprod", 16 * kx, &vt},
                       {"crt.xe", (size_t)(np + a->kpb) * sizeof(int), &ve}}) != CDL_OK)
    return CDL_ERR_UNSUPPORTED;
  a->planes = static_cast<uint32_t*>(vp);
  a->xt = static_cast<double*>(vx);
  a->xplanes = static_cast<uint32_t*>(vxp);
  a->t = static_cast<uint8_t*>(vt);
  a->erow = static_cast<int*>(ve);
  a->ecol = a->erow + np;
  return CDL_OK;
}

int crt_apply_matrix(cdl_ctx* ctx, const CrtApply& a, const double* M, int n, const double* w, int kc) {
  Launch L(ctx, kc, 0);
  if (w)
    launch_next(k_crt_residues<double, true>, a.np, 256, 0, ctx->stream, M, n, n, n, a.np, w, a.erow, a.planes);
  else
    launch_next(k_crt_residues<double>, a.np, 256, 0, ctx->stream, M, n, n, n, a.np, nullptr, a.erow, a.planes);
  return L.done();
}

int crt_apply_product(cdl_ctx* ctx, const CrtApply& a, const double* x, int rows, int cols, int ldx, const double* w,
                      int kc, double work) {
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_transpose_pad, dim3(a.np / 32, a.kpb / 32), 256, 0, ctx->stream, x, rows, cols, ldx, a.np, w, a.xt);
    CDL_TRY(L.done());
  }
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_crt_residues<double>, a.kpb, 256, 0, ctx->stream, a.xt, a.kpb, a.np, a.np, a.np, nullptr, a.ecol,
                a.xplanes);
    CDL_TRY(L.done());
  }
  return crt_gemm(ctx, a.planes, a.np, a.xplanes, a.kpb, a.np, 16, a.t, kc, work);
}

int crt_apply_add(cdl_ctx* ctx, const CrtApply& a, double* x, int kp) {
  Launch L(ctx, CDL_KC_MISC, 0);
  launch_next(k_crt_add, (unsigned)(((size_t)a.np * (kp / 4) + 127) / 128), 128, 0, ctx->stream, a.t, a.np, a.kpb, kp,
              a.erow, a.ecol, x);
  return L.done();
}

int crt_apply_residual(cdl_ctx* ctx, const CrtApply& a, const double* Y, const double* Z, const double* D, int n, int k,
                       double* R, double* part, int nblocks) {
  Launch L(ctx, CDL_KC_RESIDUAL, 0);
  launch_next(k_crt_residual, nblocks, 128, 0, ctx->stream, a.t, a.np, a.kpb, a.erow, a.ecol, Y, Z, D, n, k, R, part);
  return L.done();
}

int series_residues(cdl_ctx* ctx, const double* X, int n, int T, int rows, int kp, const int* offgrid, int* ex,
                    void* norms, void* planes, void* bad, int bad_words) {
  Launch L(ctx, CDL_KC_DISTANCE, 0);
  launch_next(k_series_residues, rows, 128, (size_t)T * sizeof(double), ctx->stream, X, n, T, rows, kp, offgrid, ex,
              static_cast<ulonglong2*>(norms), static_cast<uint32_t*>(planes), static_cast<uint32_t*>(bad), bad_words);
  return L.done();
}

int score_pairs_residues(cdl_ctx* ctx, const double* Z1, const double* Z2, const double* vol1, const double* vol2,
                         int n, int k, bool fp64, const double* A1, const double* A2, double* contrib, double* E) {
  const int planes = fp64 ? 16 : 13;
  const int rows = (n + 127) / 128 * 128, kp = (2 * k + 63) / 64 * 64;
  if (!tc_supported(ctx)) return CDL_ERR_UNSUPPORTED;
  const size_t cnt = (size_t)planes * rows * kp;
  void *vu, *vv, *vd, *ve, *vm;
  // the planes lie where the squarings and the solve of this context put theirs
  if (ws_get_opt(ctx, {{"crt.planes", cnt * 2, &vu},
                       {"crt.t", cnt * 2, &vv},
                       {"crt.score.d", (size_t)rows * 16, &vd},
                       {"crt.score.e", (size_t)rows * sizeof(int), &ve},
                       {"crt.score.max", sizeof(ScoreScale), &vm}}) != CDL_OK)
    return CDL_ERR_UNSUPPORTED;
  ScoreScale* sc = static_cast<ScoreScale*>(vm);
  int* ex = static_cast<int*>(ve);
  CDL_CUDA_TRY(cudaMemsetAsync(sc, 0, sizeof(ScoreScale), ctx->stream));
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_score_maxima, std::min((n + 7) / 8, ctx->sm_count * 4), 256, 0, ctx->stream, Z1, Z2, vol1, vol2, n, k,
                sc);
    CDL_TRY(L.done());
  }
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    if (fp64)
      launch_next(k_score_residues<16>, rows, 128, 0, ctx->stream, Z1, Z2, vol1, vol2, n, k, rows, kp, sc, ex,
                  static_cast<ulonglong2*>(vd), static_cast<__nv_bfloat16*>(vu), static_cast<__nv_bfloat16*>(vv));
    else
      launch_next(k_score_residues<13>, rows, 128, 0, ctx->stream, Z1, Z2, vol1, vol2, n, k, rows, kp, sc, ex,
                  static_cast<ulonglong2*>(vd), static_cast<__nv_bfloat16*>(vu), static_cast<__nv_bfloat16*>(vv));
    CDL_TRY(L.done());
  }
  return score_residues_tc(ctx, vu, vv, planes, ex, vd, &sc->gexp, n, rows, kp, A1, A2, contrib, E,
                           8.0 * (double)n * (n - 1));
}

}  // namespace cdl
