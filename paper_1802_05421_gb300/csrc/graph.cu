// Graph build (Sec. 2; kernel of Sec. 4.2.1; D = A 1 of Sec. 3.2):
//   1. squared distances ||x_i - x_j||^2 for all pairs (upper-triangle tiles,
//      mirrored), exact in int64 when X lies on the 2^-16 grid, otherwise in
//      float64 with one rounding per subtraction, product and sum;
//   2. sigma = lower median of the distances over i < j by an exact radix
//      select on the float64 bit patterns (distances are >= 0, so their bit
//      patterns order like the values);
//   3. A_ij = exp(-d2_ij / (2 sigma^2)), A_ii = 0, D_i = sum_j A_ij, vol.
#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>

#include <cuda_bf16.h>

#include "ff.cuh"

#include "internal.h"
#include "tiles.cuh"

namespace cdl {
namespace {

constexpr int DT = 64;          // distance tile (rows and columns)
constexpr int DTK = 32;         // samples per smem chunk
constexpr int RADIX_BITS = 12;
constexpr int RADIX_BINS = 1 << RADIX_BITS;

struct SelectState {
  unsigned long long prefix;    // selected high bits so far
  unsigned long long mask;      // which bits are selected
  long long rank;               // rank within the still-matching keys
  int flags;                    // bit 0: input off the 2^-16 grid; bit 1: a top digit above 64 in magnitude
  unsigned done;                // blocks of the running pass that have finished
  unsigned long long ncomp;     // keys copied to the buffer
  unsigned long long below;     // keys below the bracket
  uint32_t lo, hi;              // bracket of the wanted key, from a sample: the ends' high words
  int bracket;                  // BRACKET_TRY: lo, hi are set; BRACKET_HELD: the buffer holds the wanted key
  int pad;
};
// Keys from which on a graph by itself takes the bracket form (n >= 4900; the
// buffer then holds the samples): n = 4100 60 us by radix passes, 69 by a bracket;
// n = 5003 85 and 77; n = 8192 160 and 109.
constexpr long long SELECT_BRACKET_MIN = 12000000;
enum { BRACKET_NONE = 0, BRACKET_HELD = 1, BRACKET_TRY = 2 };
constexpr size_t SELECT_STATE_BYTES = 64;    // in front of the histogram in the batched form
static_assert(sizeof(SelectState) <= SELECT_STATE_BYTES, "the batched form's room for the state");

// X (float64, n x T) -> int32 fixed point a = x * 2^16, stored transposed
// (T x n) for coalesced tile loads; flags input off the grid.
__global__ void k_to_fixed(const double* __restrict__ X, int* __restrict__ Xt, int n, int T,
                           SelectState* st) {
  follow();
  const size_t total = (size_t)n * T;
  size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  size_t stride = (size_t)gridDim.x * blockDim.x;
  bool off = false;
  for (; idx < total; idx += stride) {
    double a = X[idx] * 65536.0;   // exact scaling by a power of two
    bool ok = (a == rint(a)) && fabs(a) < 8388608.0;
    off |= !ok;
    size_t i = idx / T, t = idx % T;
    Xt[t * n + i] = ok ? (int)a : 0;
  }
  if (__syncthreads_or(off) && threadIdx.x == 0) atomicOr(&st->flags, 1);
}

// For the tensor-core distances, one warp per row and one pass over X: three
// signed base-256 digit planes of a = x 2^16 (rows x tp bf16 each, zero padded: a
// = d0 + 2^8 d1 + 2^16 d2 with |d| <= 128, exact in bf16), |a_i|^2 = sum_t a_it^2 in
// int64 (exact), and the flag of input off the grid (whose digits are zero:
// other kernels handle it). Bound by memory: 8 bytes read and 6 written per
// sample; three kernels with a pass each (one an int32 copy that nothing
// read) took 238 us at n = 20011, T = 365.
__device__ __forceinline__ void prepare_series_row(const double* __restrict__ X, int n, int T, int row, int rows, int tp,
                                                   __nv_bfloat162* __restrict__ planes, long long* __restrict__ norms,
                                                   SelectState* st) {
  const int lane = threadIdx.x & 31;
  const size_t plane = (size_t)rows * tp / 2;
  const double* x = X + (size_t)min(row, n - 1) * T;
  long long acc = 0;
  bool off = false, wide = false;
  for (int t2 = lane; t2 < tp / 2; t2 += 32) {
    int d[3][2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int t = 2 * t2 + h;
      int a = 0;
      if (row < n && t < T) {
        const double v = x[t] * 65536.0;                    // exact scaling by a power of two
        if (v == rint(v) && fabs(v) < 8388608.0)
          a = (int)v;
        else
          off = true;
      }
      acc += (long long)a * a;
      d[0][h] = ((a + 128) & 255) - 128;
      const int a1 = (a - d[0][h]) >> 8;                    // exact: a - d0 is a multiple of 256
      d[1][h] = ((a1 + 128) & 255) - 128;
      d[2][h] = (a1 - d[1][h]) >> 8;
      wide |= d[2][h] > 64 || d[2][h] < -64;
    }
    const size_t o = (size_t)row * tp / 2 + t2;
#pragma unroll
    for (int q = 0; q < 3; ++q) planes[q * plane + o] = __floats2bfloat162_rn((float)d[q][0], (float)d[q][1]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) norms[row] = acc;
  const int bits = (__any_sync(0xffffffffu, off) ? 1 : 0) | (__any_sync(0xffffffffu, wide) ? 2 : 0);
  if (lane == 0 && bits & ~*reinterpret_cast<volatile int*>(&st->flags)) atomicOr(&st->flags, bits);
}

__global__ void __launch_bounds__(256) k_prepare_series(const double* __restrict__ X, int n, int T, int rows, int tp,
                                                         __nv_bfloat162* __restrict__ planes,
                                                         long long* __restrict__ norms, SelectState* st) {
  follow();
  const int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (row < rows) prepare_series_row(X, n, T, row, rows, tp, planes, norms, st);
}

// Exact squared distances on the 2^-16 grid: int64 sums of squared int32
// differences, written as float64 multiples of 2^-32 to both (i,j) and (j,i).
__device__ __forceinline__ void dist_int_tile(const int* __restrict__ Xt, int n, int T, double* __restrict__ A,
                                              int bi, int bj) {
  __shared__ __align__(16) int As[DTK][DT];
  __shared__ __align__(16) int Bs[DTK][DT];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int r0 = bi * DT, c0 = bj * DT;
  long long acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = 0;
  for (int t0 = 0; t0 < T; t0 += DTK) {
    // load 32 samples x 64 nodes of each side from the transposed copy
    for (int e = threadIdx.x; e < DT * DTK; e += 256) {
      int row = e % DT, tt = e / DT;
      int ia = r0 + row, ib = c0 + row, t = t0 + tt;
      As[tt][row] = (ia < n && t < T) ? Xt[(size_t)t * n + ia] : 0;
      Bs[tt][row] = (ib < n && t < T) ? Xt[(size_t)t * n + ib] : 0;
    }
    __syncthreads();
#pragma unroll 4
    for (int tt = 0; tt < DTK; ++tt) {
      int4 a = *reinterpret_cast<const int4*>(&As[tt][ty * 4]);
      int4 b = *reinterpret_cast<const int4*>(&Bs[tt][tx * 4]);
      int av[4] = {a.x, a.y, a.z, a.w};
      int bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          int dd = av[u] - bv[v];
          acc[u][v] += (long long)dd * dd;
        }
    }
    __syncthreads();
  }
  const double q = 1.0 / 4294967296.0;   // 2^-32
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    int i = r0 + ty * 4 + u;
    if (i >= n) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      int j = c0 + tx * 4 + v;
      if (j >= n) continue;
      double d2 = (double)acc[u][v] * q;
      A[(size_t)i * n + j] = d2;
      if (bi != bj) A[(size_t)j * n + i] = d2;
    }
  }
}

__global__ void __launch_bounds__(256) k_dist_int(const int* __restrict__ Xt, int n, int T,
                                                   double* __restrict__ A, const SelectState* st) {
  follow();
  if (st->flags & 1) return;   // off-grid input: the float64 kernel handles it
  const int nb = (n + DT - 1) / DT;
  int bi, bj;
  block_tri_index(nb, bi, bj);
  dist_int_tile(Xt, n, T, A, bi, bj);
}

// Float64 squared distances for inputs off the grid: same tiling, samples in
// ascending order, explicit round-to-nearest operations (no contraction).
__device__ __forceinline__ void dist_f64_tile(const double* __restrict__ X, int n, int T, double* __restrict__ A,
                                              int bi, int bj) {
  __shared__ double As[DTK][DT + 1];
  __shared__ double Bs[DTK][DT + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int r0 = bi * DT, c0 = bj * DT;
  double acc[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v] = 0.0;
  for (int t0 = 0; t0 < T; t0 += DTK) {
    for (int e = threadIdx.x; e < DT * DTK; e += 256) {
      int row = e / DTK, tt = e % DTK;
      int ia = r0 + row, ib = c0 + row, t = t0 + tt;
      As[tt][row] = (ia < n && t < T) ? X[(size_t)ia * T + t] : 0.0;
      Bs[tt][row] = (ib < n && t < T) ? X[(size_t)ib * T + t] : 0.0;
    }
    __syncthreads();
    const int tmax = min(DTK, T - t0);
    for (int tt = 0; tt < tmax; ++tt) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          double dd = __dsub_rn(As[tt][ty * 4 + u], Bs[tt][tx * 4 + v]);
          acc[u][v] = __dadd_rn(acc[u][v], __dmul_rn(dd, dd));
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    int i = r0 + ty * 4 + u;
    if (i >= n) continue;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      int j = c0 + tx * 4 + v;
      if (j >= n) continue;
      A[(size_t)i * n + j] = acc[u][v];
      if (bi != bj) A[(size_t)j * n + i] = acc[u][v];
    }
  }
}

// `bad` (may be null: every tile): only the 64 x 64 tiles that dist_residues_tc flagged.
__global__ void __launch_bounds__(256) k_dist_f64(const double* __restrict__ X, int n, int T,
                                                   double* __restrict__ A, const SelectState* st,
                                                   const unsigned char* __restrict__ bad, int bad_stride) {
  follow();
  if (!(st->flags & 1)) return;
  __shared__ int tile[2];
  const int nb = (n + DT - 1) / DT;
  const long long tiles = (long long)nb * (nb + 1) / 2;
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    if (threadIdx.x == 0) tri_index(t, nb, tile[0], tile[1]);
    __syncthreads();
    const int bi = tile[0], bj = tile[1];
    if (!bad || bad[(size_t)bi * bad_stride + bj]) dist_f64_tile(X, n, T, A, bi, bj);
    __syncthreads();
  }
}

// The median of the m = n (n - 1) / 2 squared distances, exactly, over their
// float64 bit patterns (for x >= 0 these order like the values).
//
// Radix form: six passes, digits from the top, each a histogram of the keys that
// match the digits selected before; the pass's last block picks the bin with the
// wanted rank. The third pass also copies the matching keys (about 2^-12 of the
// value range around the median) to a buffer, which the later passes read
// instead of A where they all fitted. Three passes over A, each bound by DRAM.
//
// Bracket form: one pass over A. SAMPLE keys, drawn at hashed positions, give two
// of them SAMPLE_MARGIN ranks (4.5 standard deviations) to either side of the
// wanted rank; a pass over A counts the keys below that bracket and copies those
// inside (2.5 % of all) to the buffer; the radix passes then read the buffer
// alone. Where the wanted rank is not inside, or the keys do not fit (many equal
// distances: seen in the sample, then the pass over A is left out too), the radix
// form runs instead. n = 20011 (2.0e8 keys, 1.6 GB): 1088 -> 400 us, of which the
// pass over A 298 (5.4 TB/s); 128 batched graphs (2.2e8 keys): 2.53 -> 0.43 ms.
constexpr int SELECT_THREADS = 512;
constexpr int SELECT_WARPS = SELECT_THREADS / 32;
constexpr int SELECT_STAGE = 256;                        // keys a warp gathers before it takes buffer space
constexpr int SELECT_FINISH = 8192;                      // keys one block looks through for the rest
constexpr int SAMPLE_THREADS = 1024;
constexpr int SAMPLE = 32768;
constexpr int SAMPLE_MARGIN = 407;                       // 4.5 sqrt(SAMPLE) / 2

__device__ __forceinline__ void select_init(SelectState* st, long long rank) {
  st->prefix = 0;
  st->mask = 0;
  st->rank = rank;
  st->flags = 0;
  st->done = 0;
  st->ncomp = 0;
  st->below = 0;
  st->bracket = BRACKET_NONE;
}

__global__ void __launch_bounds__(1024) k_select_init(SelectState* st, long long rank,
                                                      unsigned long long* __restrict__ hist) {
  follow();
  if (threadIdx.x == 0) select_init(st, rank);
  for (int b = threadIdx.x; b < RADIX_BINS; b += blockDim.x) hist[b] = 0;
}

// f(key) for `len` consecutive keys by the lanes of a warp, eight loads in flight
// each (one at a time left half of the DRAM bandwidth idle); every lane calls f
// for every step, with ok = false past the end.
template <class F>
__device__ __forceinline__ void warp_keys(const unsigned long long* __restrict__ k, int len, F&& f) {
  const int lane = threadIdx.x & 31;
  for (int v0 = 0; v0 < len; v0 += 256) {
    unsigned long long key[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int v = v0 + lane + 32 * e;
      key[e] = v < len ? k[v] : 0;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (v0 + 32 * e < len) f(key[e], v0 + lane + 32 * e < len);
  }
}

// The warps of a group of `warps` (this one `warp`) over the upper triangle of
// rows r0 .. r1 - 1 (A holds rows roff ..: row i at A + (i - roff) n).
template <class F>
__device__ __forceinline__ void triangle_keys(const double* __restrict__ A, int n, int r0, int r1, int warp, int warps,
                                              int roff, F&& f) {
  const unsigned long long* K = reinterpret_cast<const unsigned long long*>(A);
  for (int i = r0 + warp; i < r1; i += warps) warp_keys(K + (size_t)(i - roff) * n + i + 1, n - 1 - i, f);
}

// The same over the whole triangle for an even load: rows i and n - 2 - i
// together hold n keys; segments of 256 keys of such pairs of rows go around the
// warps.
template <class F>
__device__ __forceinline__ void folded_keys(const double* __restrict__ A, int n, F&& f) {
  const unsigned long long* K = reinterpret_cast<const unsigned long long*>(A);
  const unsigned segs = (n + 255) / 256, items = (unsigned)(n / 2) * segs;   // n / 2 pairs of rows 0 .. n - 2
  for (unsigned q = blockIdx.x * SELECT_WARPS + (threadIdx.x >> 5); q < items; q += gridDim.x * SELECT_WARPS) {
    const int i = (int)(q / segs), v0 = (int)(q % segs) * 256, v1 = min(v0 + 256, n);
    const int first = n - 1 - i, i2 = n - 2 - i;         // keys of row i; the partner row
    if (v0 < first) warp_keys(K + (size_t)i * n + i + 1 + v0, min(v1, first) - v0, f);
    if (v1 > first && i2 != i) {
      const int w0 = max(v0, first) - first;
      warp_keys(K + (size_t)i2 * n + i2 + 1 + w0, v1 - first - w0, f);
    }
  }
}

struct SelectShared {
  union {
    unsigned int h[RADIX_BINS];
    unsigned long long cnt[RADIX_BINS + SELECT_THREADS];   // one pad word per run: no bank conflicts
    unsigned long long stage[SELECT_WARPS][SELECT_STAGE];
  };
  unsigned long long wsum[SELECT_WARPS];
  unsigned long long bin;                                  // keys in the bin that the last step picked
  int last;
};

// True in every thread of the last of `blocks` blocks to get here, after all
// their writes before this are visible to it.
__device__ __forceinline__ bool select_last_block(SelectState* st, unsigned blocks, int* flag) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) *flag = atomicAdd(&st->done, 1u) == blocks - 1;
  __syncthreads();
  if (!*flag) return false;
  __threadfence();
  return true;
}

// Pick the bin holding the remaining rank; extend the prefix; clear hist. One
// block: every thread sums its run of 8 bins, a block scan of the sums finds the
// run holding the rank, and its thread walks the run. Bound by latency (32 KB of
// counts, one block): 3 us, where one thread walking all 4096 bins took 56 us;
// run by the last block of the histogram it costs no launch of its own.
__device__ __forceinline__ void select_step(SelectState* st, unsigned long long* hist, int shift, int bits,
                                            double* sigma_out, int last, SelectShared& sm) {
  constexpr int RUN = RADIX_BINS / SELECT_THREADS;
  const int nbins = 1 << bits, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll
  for (int e = 0; e < RUN; ++e) {
    const int b = tid + e * SELECT_THREADS;
    sm.cnt[b + b / RUN] = b < nbins ? __ldcg(hist + b) : 0;
    if (b < nbins) hist[b] = 0;
  }
  const unsigned long long r = (unsigned long long)st->rank;
  __syncthreads();
  const unsigned long long* run = sm.cnt + tid * (RUN + 1);
  unsigned long long own = 0;
#pragma unroll
  for (int e = 0; e < RUN; ++e) own += run[e];
  unsigned long long incl = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) sm.wsum[warp] = incl;
  __syncthreads();
  for (int w = 0; w < warp; ++w) incl += sm.wsum[w];
  const unsigned long long before = incl - own;
  if (before <= r && r < incl) {   // exactly one thread: the histogram counts every key that still matches
    unsigned long long below = before;
    int e = 0;
    while (r - below >= run[e]) below += run[e++];
    st->prefix |= (unsigned long long)(tid * RUN + e) << shift;
    st->mask |= (unsigned long long)(nbins - 1) << shift;
    st->rank = (long long)(r - below);
    if (last) *sigma_out = sqrt(__longlong_as_double((long long)st->prefix));
    sm.bin = run[e];
  }
  if (tid == 0) st->done = 0;
}

// The rest of the selection in the block that made the step: of the nc keys in the
// buffer the sm.bin (at most SELECT_THREADS) that match, each ranked among them by
// counting. The later passes then find every digit selected and return: on small
// graphs they took 8 us each.
__device__ __forceinline__ void select_finish(SelectState* st, const unsigned long long* buf, unsigned long long nc,
                                              double* sigma_out, SelectShared& sm) {
  unsigned long long* list = &sm.stage[0][0];
  const unsigned long long prefix = st->prefix, mask = st->mask;
  const int r = (int)st->rank, c = (int)sm.bin;
  __syncthreads();
  if (threadIdx.x == 0) sm.last = 0;
  __syncthreads();
  for (unsigned long long q = threadIdx.x; q < nc; q += SELECT_THREADS) {
    const unsigned long long key = __ldcg(buf + q);
    if ((key & mask) == prefix) list[atomicAdd(&sm.last, 1)] = key;
  }
  __syncthreads();
  if ((int)threadIdx.x >= c) return;
  const unsigned long long key = list[threadIdx.x];
  int less = 0, upto = 0;
  for (int e = 0; e < c; ++e) {
    less += list[e] < key;
    upto += list[e] <= key;
  }
  if (less <= r && r < upto) {   // equal keys write the same
    st->prefix = key;
    st->mask = ~0ull;
    *sigma_out = sqrt(__longlong_as_double((long long)key));
  }
}

__global__ void __launch_bounds__(SELECT_THREADS, 2) k_select_step(SelectState* st, unsigned long long* hist, int shift,
                                                                int bits, double* sigma_out, int last) {
  follow();
  __shared__ SelectShared sm;
  select_step(st, hist, shift, bits, sigma_out, last, sm);
}

// Histogram of the digit at `shift` in shared memory around `keys`, a function
// that calls its argument for this block's keys.
template <class K>
__device__ __forceinline__ void select_hist(const SelectState* st, int shift, int bits, unsigned long long* hist,
                                            SelectShared& sm, K&& keys) {
  for (int b = threadIdx.x; b < RADIX_BINS; b += blockDim.x) sm.h[b] = 0;
  __syncthreads();
  const unsigned long long prefix = st->prefix, mask = st->mask, dmask = (1ull << bits) - 1ull;
  keys([&](unsigned long long key, bool ok) {
    const bool hit = ok && (key & mask) == prefix;
    if (hit) atomicAdd(&sm.h[(key >> shift) & dmask], 1u);
    return hit;
  });
  __syncthreads();
  for (int b = threadIdx.x; b < RADIX_BINS; b += blockDim.x)
    if (sm.h[b]) atomicAdd(&hist[b], (unsigned long long)sm.h[b]);
}

// The digit at `shift` over rows r0 .. r1 - 1 of a panel holding rows r0 .. (the
// regenerated graphs; the step is a launch of its own after the last panel)
__global__ void __launch_bounds__(SELECT_THREADS, 2) k_select_hist_panel(const double* __restrict__ P, int n, int shift,
                                                                      int bits, const SelectState* __restrict__ st,
                                                                      unsigned long long* __restrict__ hist, int r0,
                                                                      int r1) {
  follow();
  __shared__ SelectShared sm;
  select_hist(st, shift, bits, hist, sm, [&](auto&& f) {
    triangle_keys(P, n, r0, r1, blockIdx.x * SELECT_WARPS + (threadIdx.x >> 5), gridDim.x * SELECT_WARPS, r0, f);
  });
}

// Digit p of the selection and its step. Block `block` of `blocks`; rows(f) calls
// f for the block's share of the triangle.
template <class R>
__device__ __forceinline__ void select_pass(SelectState* st, unsigned long long* hist, int p, double* sigma_out,
                                            unsigned long long* buf, unsigned long long cap, unsigned block,
                                            unsigned blocks, SelectShared& sm, R&& rows) {
  const int shift = p < 5 ? 52 - 12 * p : 0, bits = p < 5 ? 12 : 4;
  const unsigned long long dmask = (1ull << bits) - 1ull;
  if (((st->mask >> shift) & dmask) == dmask) return;    // the bracket's common leading digit
  const unsigned long long nc = st->ncomp;
  if (st->bracket == BRACKET_HELD || (p > 2 && cap && nc <= cap)) {
    const size_t step = (size_t)blocks * SELECT_WARPS * 256;
    const size_t w0 = ((size_t)block * SELECT_WARPS) * 256;
    if (w0 < nc)
      select_hist(st, shift, bits, hist, sm, [&](auto&& f) {
        for (size_t q = w0 + (threadIdx.x >> 5) * 256; q < nc; q += step)
          warp_keys(buf + q, (int)min((size_t)256, (size_t)(nc - q)), f);
      });
  } else if (p == 2 && cap) {
    bool full = false;
    select_hist(st, shift, bits, hist, sm, [&](auto&& f) {
      rows([&](unsigned long long key, bool ok) {
        const bool hit = f(key, ok);
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (m == 0 || full) return;
        const int lane = threadIdx.x & 31;
        unsigned long long pos = 0;
        if (lane == 0) pos = atomicAdd(&st->ncomp, (unsigned long long)__popc(m));
        pos = __shfl_sync(0xffffffffu, pos, 0);
        full = pos > cap;                               // ncomp is above cap for good
        pos += __popc(m & ((1u << lane) - 1u));
        if (hit && pos < cap) buf[pos] = key;
      });
    });
  } else {
    select_hist(st, shift, bits, hist, sm, rows);
  }
  if (!select_last_block(st, blocks, &sm.last)) return;
  select_step(st, hist, shift, bits, sigma_out, p == 5, sm);
  if (p != 2 || cap == 0 || st->bracket == BRACKET_HELD) return;
  __syncthreads();
  const unsigned long long got = __ldcg(&st->ncomp);
  if (got <= min(cap, (unsigned long long)SELECT_FINISH) && sm.bin <= SELECT_THREADS)
    select_finish(st, buf, got, sigma_out, sm);
}

// One pass over A for the keys below the bracket and those inside.
template <class R>
__device__ __forceinline__ void select_bracket(SelectState* st, unsigned long long* buf, unsigned long long cap,
                                               unsigned blocks, SelectShared& sm, R&& rows) {
  if (st->bracket != BRACKET_TRY) return;
  const unsigned long long lo = (unsigned long long)st->lo << 32, hi = (unsigned long long)st->hi << 32 | 0xFFFFFFFFull;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long* stage = sm.stage[warp];
  unsigned below = 0;
  int cnt = 0;
  auto flush = [&]() {
    __syncwarp();
    unsigned long long pos = 0;
    if (lane == 0) pos = atomicAdd(&st->ncomp, (unsigned long long)cnt);
    pos = __shfl_sync(0xffffffffu, pos, 0);
    for (int e = lane; e < cnt; e += 32)
      if (pos + e < cap) buf[pos + e] = stage[e];
    __syncwarp();
    cnt = 0;
  };
  rows([&](unsigned long long key, bool ok) {
    below += ok && key < lo;
    const bool in = ok && key >= lo && key <= hi;
    const unsigned m = __ballot_sync(0xffffffffu, in);
    if (m) {
      if (in) stage[cnt + __popc(m & ((1u << lane) - 1u))] = key;
      cnt += __popc(m);
      if (cnt > SELECT_STAGE - 32) flush();
    }
  });
  if (cnt) flush();
  below = __reduce_add_sync(0xffffffffu, below);
  if (lane == 0 && below) atomicAdd(&st->below, (unsigned long long)below);
  if (!select_last_block(st, blocks, &sm.last) || threadIdx.x != 0) return;
  const unsigned long long nc = __ldcg(&st->ncomp), nb = __ldcg(&st->below);
  const unsigned long long r = (unsigned long long)st->rank;
  const bool held = nb <= r && r < nb + nc && nc <= cap;
  if (held) {
    st->rank = (long long)(r - nb);
    if ((lo >> 52) == (hi >> 52)) {
      st->prefix = lo >> 52 << 52;
      st->mask = 0xFFFull << 52;
    }
  } else {
    st->ncomp = 0;
  }
  st->bracket = held ? BRACKET_HELD : BRACKET_NONE;
  st->done = 0;
}

// Sample q: the high word of the key at a hashed position (the finaliser of
// splitmix64: Steele, Lea and Flood, "Fast splittable pseudorandom number
// generators", 2014, applied to q + 1).
__device__ __forceinline__ uint32_t sample_key(const double* __restrict__ A, int n, uint32_t q) {
  unsigned long long x = (q + 1) * 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  x ^= x >> 31;
  const uint32_t i = __umulhi((uint32_t)(x >> 32), (uint32_t)n);
  uint32_t j = __umulhi((uint32_t)x, (uint32_t)(n - 1));
  j += j >= i;
  return reinterpret_cast<const uint32_t*>(A + (size_t)min(i, j) * n + max(i, j))[1];
}

__global__ void __launch_bounds__(256) k_sample_keys(const double* __restrict__ A, int n, uint32_t* __restrict__ out) {
  follow();
  const uint32_t q = blockIdx.x * 256 + threadIdx.x;
  out[q] = sample_key(A, n, q);
}

// The bracket from SAMPLE keys (their high words; positions by a fixed hash, with
// repetitions): two ranks found at once by three histograms in shared memory. One
// block: 15 us, bound by the latency of its passes (with the scattered loads and one
// histogram update per sample at the top digit, where most meet in one bin: 50).
struct SampleShared {
  uint32_t key[SAMPLE];
  unsigned h[2][2048];
  unsigned wsum[32];
  uint32_t prefix[2];
  int rank[2];
  int open[2];                  // the bracket has no end on this side
  int inside;
};
template <class K>
__device__ __forceinline__ void select_sample(int n, SelectState* st, unsigned long long cap, SampleShared& sm,
                                              K&& sample) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll 16
  for (int e = 0; e < SAMPLE / SAMPLE_THREADS; ++e)
    sm.key[tid + e * SAMPLE_THREADS] = sample((uint32_t)(tid + e * SAMPLE_THREADS));
  if (tid == 0) {
    // where the wanted key falls among the samples
    const int at = (int)(((double)st->rank + 0.5) / (0.5 * (double)n * (double)(n - 1)) * SAMPLE);
    sm.rank[0] = at - SAMPLE_MARGIN;
    sm.rank[1] = at + SAMPLE_MARGIN;
    sm.open[0] = at < SAMPLE_MARGIN;
    sm.open[1] = at + SAMPLE_MARGIN >= SAMPLE;
    sm.prefix[0] = sm.prefix[1] = 0;
    sm.inside = 0;
  }
  const int t = tid >> 9, u = tid & 511;                 // half of the block per rank, 4 bins a thread
  uint32_t mask = 0;
  for (int p = 0; p < 3; ++p) {
    const int shift = p == 0 ? 21 : p == 1 ? 10 : 0, bits = p < 2 ? 11 : 10;
    for (int b = tid; b < 4096; b += SAMPLE_THREADS) (&sm.h[0][0])[b] = 0;
    __syncthreads();
    const uint32_t p0 = sm.prefix[0], p1 = sm.prefix[1], dmask = (1u << bits) - 1u;
    const bool same = p0 == p1;                        // one histogram serves both ranks
#pragma unroll 4
    for (int e = 0; e < SAMPLE / SAMPLE_THREADS; ++e) {
      const uint32_t k = sm.key[tid + e * SAMPLE_THREADS], d = (k >> shift) & dmask;
      if (p == 0) {                                      // exponents: most of a warp falls into one bin or two
        const unsigned m = __match_any_sync(0xffffffffu, d);
        if (lane == __ffs(m) - 1) atomicAdd(&sm.h[0][d], (unsigned)__popc(m));
        continue;
      }
      if ((k & mask) == p0) atomicAdd(&sm.h[0][d], 1u);
      if (!same && (k & mask) == p1) atomicAdd(&sm.h[1][d], 1u);
    }
    __syncthreads();
    unsigned c[4], own = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) own += c[e] = sm.h[same ? 0 : t][4 * u + e];
    unsigned incl = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    if (lane == 31) sm.wsum[warp] = incl;
    const int r = sm.rank[t];
    __syncthreads();
    for (int w = t * 16; w < warp; ++w) incl += sm.wsum[w];
    unsigned b0 = incl - own;
    if (r >= 0 && b0 <= (unsigned)r && (unsigned)r < incl) {
      int e = 0;
      while ((unsigned)r - b0 >= c[e]) b0 += c[e++];
      sm.prefix[t] |= (uint32_t)(4 * u + e) << shift;
      sm.rank[t] = r - (int)b0;
    }
    mask |= dmask << shift;
    __syncthreads();
  }
  const uint32_t lo = sm.open[0] ? 0u : sm.prefix[0], hi = sm.open[1] ? 0xFFFFFFFFu : sm.prefix[1];
  int in = 0;
#pragma unroll 4
  for (int e = 0; e < SAMPLE / SAMPLE_THREADS; ++e) {
    const uint32_t k = sm.key[tid + e * SAMPLE_THREADS];
    in += k >= lo && k <= hi;
  }
  in = __reduce_add_sync(0xffffffffu, in);
  if (lane == 0) atomicAdd(&sm.inside, in);
  __syncthreads();
  if (tid == 0) {
    st->lo = lo;
    st->hi = hi;
    const double expected = (double)sm.inside / SAMPLE * (0.5 * (double)n * (double)(n - 1));
    st->bracket = expected < 0.95 * (double)cap + 4.0 ? BRACKET_TRY : BRACKET_NONE;
  }
}

__global__ void __launch_bounds__(SAMPLE_THREADS) k_select_sample(const uint32_t* __restrict__ keys, int n,
                                                                  SelectState* st, unsigned long long cap) {
  follow();
  extern __shared__ __align__(16) unsigned char sample_smem[];
  select_sample(n, st, cap, *reinterpret_cast<SampleShared*>(sample_smem), [&](uint32_t q) { return keys[q]; });
}

__global__ void __launch_bounds__(SELECT_THREADS, 2)
    k_select_bracket(const double* __restrict__ A, int n, SelectState* st, unsigned long long* __restrict__ buf,
                     unsigned long long cap) {
  follow();
  __shared__ SelectShared sm;
  select_bracket(st, buf, cap, gridDim.x, sm, [&](auto&& f) {
    folded_keys(A, n, f);
  });
}

__global__ void __launch_bounds__(SELECT_THREADS, 2) k_select_pass(const double* __restrict__ A, int n, int p,
                                                                SelectState* st, unsigned long long* __restrict__ hist,
                                                                double* sigma_out, unsigned long long* __restrict__ buf,
                                                                unsigned long long cap) {
  follow();
  __shared__ SelectShared sm;
  select_pass(st, hist, p, sigma_out, buf, cap, blockIdx.x, gridDim.x, sm, [&](auto&& f) {
    folded_keys(A, n, f);
  });
}

__global__ void k_set_scalar(double* p, double v) {
  follow();
  *p = v;
}

// A_ij = exp(-d2_ij / (2 sigma^2)) (KERN = KERNEL_GAUSSIAN) or
// A_ij = exp(-sqrt(d2_ij) / sigma) (KERN = KERNEL_EXP, the synthetic-data
// kernel of Sec. 4.2.1), A_ii = 0, D_i = row sum. One block per row (panels of
// a regenerated graph and the graphs without workspace; whole graphs take
// k_kernel_tiles). The exponential is exp_neg_prod: integer operations only, the
// argument d2 * (1 / (2 sigma^2)), or sqrt(d2) (sqrt_nonneg: within one ulp)
// times 1 / sigma, in 64-bit fixed point. The row sum is accumulated in
// float-float (terms below 2^-100 are dropped from the sum, not from A).
enum { KERNEL_GAUSSIAN = 0, KERNEL_EXP = 1 };

__device__ __forceinline__ double kernel_rcp(double sigma, int kern) {
  return kern == KERNEL_EXP ? 1.0 / sigma : 1.0 / (2.0 * (sigma * sigma));
}

// (hi, lo) + a split exactly into floats, lo left unnormalised.
__device__ __forceinline__ void ff_acc(ff& acc, ff q) {
  const ff t = two_sum(acc.hi, q.hi);
  acc.hi = t.hi;
  acc.lo = __fadd_rn(acc.lo, __fadd_rn(t.lo, q.lo));
}

template <int KERN = KERNEL_GAUSSIAN>
__device__ __forceinline__ void kernel_row(double* __restrict__ A, int n, const ExpFactor& f, double* __restrict__ D,
                                           int i, const unsigned long long* __restrict__ tab, int roff = 0) {
  __shared__ double red[8];
  double* row = A + (size_t)(i - roff) * n;
  ff acc = {0.f, 0.f};
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    double a = 0.0;
    if (j != i) {
      a = exp_neg_prod(KERN == KERNEL_EXP ? sqrt_nonneg(row[j]) : row[j], f, tab);
      ff_acc(acc, split_nonneg(a));
    }
    row[j] = a;
  }
  double accd = (double)acc.hi + (double)acc.lo;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) accd += __shfl_xor_sync(0xffffffffu, accd, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = accd;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    D[i] = t;
  }
  __syncthreads();
}

template <int KERN = KERNEL_GAUSSIAN>
__global__ void __launch_bounds__(256) k_kernel_rows(double* __restrict__ A, int n,
                                                      const double* __restrict__ sigma,
                                                      double* __restrict__ D) {
  follow();
  __shared__ unsigned long long tab[EXP_TABLE];
  exp_table(tab);
  const ExpFactor f = exp_factor(kernel_rcp(*sigma, KERN));
  __syncthreads();
  for (int i = blockIdx.x; i < n; i += gridDim.x) kernel_row<KERN>(A, n, f, D, i, tab);
}

// Rows r0 .. r1 - 1 of a panel holding rows r0 .. (squared distances in,
// kernel values out), their degrees into D[i].
__global__ void __launch_bounds__(256) k_kernel_rows_panel(double* __restrict__ P, int n,
                                                            const double* __restrict__ sigma, double* __restrict__ D,
                                                            int r0, int r1) {
  follow();
  __shared__ unsigned long long tab[EXP_TABLE];
  exp_table(tab);
  const ExpFactor f = exp_factor(kernel_rcp(*sigma, KERNEL_GAUSSIAN));
  __syncthreads();
  for (int i = r0 + blockIdx.x; i < r1; i += gridDim.x) kernel_row<KERNEL_GAUSSIAN>(P, n, f, D, i, tab, r0);
}

// Kernel values over the upper block triangle of 64 x 64 tiles (A is
// symmetric, so half the exponentials of the row-by-row pass): a block
// evaluates tile (bi, bj), bj >= bi (a diagonal tile all of its entries),
// writes it and, off the diagonal, its mirror through shared memory (both
// writes coalesced), and leaves the tile's row and column sums of A
// (float-float, the entries split with integer operations) in the slots of
// the 64-node partner blocks: part[bj][i] for its rows, part[bi][j] for its
// columns (rows only on the diagonal). D_i is the fixed-order sum of node i's
// slots (part_sum). Same entry arithmetic as kernel_row.
// Warp w holds rows 8 w .. 8 w + 7, a lane the columns lane and lane + 32: both
// sums start from the registers; the rows' lanes are combined by halving
// exchanges (9 additions for 8 rows instead of 40), the columns' warps through
// shared memory. Bound by instruction issue (125 a weight; float64 sums, two additions a
// weight on a pipe of two lanes a cycle, were no faster): n = 20011 1211 us, 4.0 TB/s;
// with 128-bit exponentials and sums read back from shared memory 2315.
struct KernelTileShared {
  double tt[DT][DT + 1];                                // tt[c][r] = A(i0 + r, j0 + c)
  float2 col[8][DT];
  unsigned long long tab[EXP_TABLE];
};

// FULL: every row and column of the tile lies inside the matrix.
template <int KERN, bool FULL>
__device__ __forceinline__ void kernel_tile(double* __restrict__ A, int n, const ExpFactor& f, double* __restrict__ part,
                                            int bi, int bj, KernelTileShared& sm) {
  const int i0 = bi * DT, j0 = bj * DT;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  ff rs[8], cs[2] = {{0.f, 0.f}, {0.f, 0.f}};
  double* base = A + (size_t)(i0 + 8 * warp) * n + j0 + lane;
#pragma unroll
  for (int m0 = 0; m0 < 8; m0 += 4) {
    double x[4][2];
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = i0 + 8 * warp + m0 + m, j = j0 + lane + 32 * h;
        x[m][h] = FULL || (i < n && j < n) ? base[(size_t)(m0 + m) * n + 32 * h] : 0.0;
      }
#pragma unroll
    for (int m = 0; m < 4; ++m) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = 8 * warp + m0 + m, c = lane + 32 * h, i = i0 + r, j = j0 + c;
        double a = 0.0;
        if (FULL || (i < n && j < n)) {
          if (i != j) a = exp_neg_prod(KERN == KERNEL_EXP ? sqrt_nonneg(x[m][h]) : x[m][h], f, sm.tab);
          base[(size_t)(m0 + m) * n + 32 * h] = a;
        }
        sm.tt[c][r] = a;
        const ff v = split_nonneg(a);
        ff_acc(cs[h], v);
        if (h == 0)
          rs[m0 + m] = v;
        else
          ff_acc(rs[m0 + m], v);
      }
    }
  }
  // lane l ends with the sum of row l >> 2 of the warp's eight
#pragma unroll
  for (int w = 4; w > 0; w >>= 1) {
    const bool up = (lane & (4 * w)) != 0;
#pragma unroll
    for (int m = 0; m < w; ++m) {
      const ff keep = up ? rs[m + w] : rs[m], give = up ? rs[m] : rs[m + w];
      rs[m] = ff_add(
          keep, ff{__shfl_xor_sync(0xffffffffu, give.hi, 4 * w), __shfl_xor_sync(0xffffffffu, give.lo, 4 * w)});
    }
  }
#pragma unroll
  for (int o = 2; o > 0; o >>= 1)
    rs[0] = ff_add(rs[0], ff{__shfl_xor_sync(0xffffffffu, rs[0].hi, o), __shfl_xor_sync(0xffffffffu, rs[0].lo, o)});
  const int ri = i0 + 8 * warp + (lane >> 2);
  if ((lane & 3) == 0 && (FULL || ri < n)) part[(size_t)bj * n + ri] = (double)rs[0].hi + (double)rs[0].lo;
#pragma unroll
  for (int h = 0; h < 2; ++h) sm.col[warp][lane + 32 * h] = make_float2(cs[h].hi, cs[h].lo);
  __syncthreads();
  if (bi != bj) {
    const int r = threadIdx.x & (DT - 1), rg = threadIdx.x >> 6;
    double* mirror = A + (size_t)(j0 + rg) * n + i0 + r;
#pragma unroll 8
    for (int m = 0; m < DT / 4; ++m)                    // lanes write consecutive columns of row j
      if (FULL || (j0 + rg + 4 * m < n && i0 + r < n)) mirror[(size_t)(4 * m) * n] = sm.tt[rg + 4 * m][r];
    if (threadIdx.x < DT && (FULL || j0 + (int)threadIdx.x < n)) {   // column sums (the mirror's row sums)
      ff acc = {0.f, 0.f};
#pragma unroll
      for (int w = 0; w < 8; ++w) acc = ff_add(acc, ff{sm.col[w][threadIdx.x].x, sm.col[w][threadIdx.x].y});
      part[(size_t)bi * n + j0 + threadIdx.x] = (double)acc.hi + (double)acc.lo;
    }
  }
}

template <int KERN>
__device__ __forceinline__ void kernel_tile_any(double* __restrict__ A, int n, const ExpFactor& f,
                                                double* __restrict__ part, int bi, int bj, KernelTileShared& sm) {
  if ((bj + 1) * DT <= n)                                // bi <= bj
    kernel_tile<KERN, true>(A, n, f, part, bi, bj, sm);
  else
    kernel_tile<KERN, false>(A, n, f, part, bi, bj, sm);
}

template <int KERN>
__global__ void __launch_bounds__(256, 4) k_kernel_tiles(double* __restrict__ A, int n, const double* __restrict__ sigma,
                                                          double* __restrict__ part) {
  follow();
  __shared__ KernelTileShared sm;
  __shared__ int tile_s[2];
  const int nb = (n + DT - 1) / DT;
  const long long tiles = (long long)nb * (nb + 1) / 2;
  exp_table(sm.tab);
  const ExpFactor f = exp_factor(kernel_rcp(*sigma, KERN));
  for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
    if (threadIdx.x == 0) tri_index(t, nb, tile_s[0], tile_s[1]);
    __syncthreads();
    kernel_tile_any<KERN>(A, n, f, part, tile_s[0], tile_s[1], sm);
    __syncthreads();
  }
}

__device__ __forceinline__ double part_sum(const double* __restrict__ part, int nb, int n, int i) {
  double s = 0.0;
  for (int b = 0; b < nb; ++b) s += part[(size_t)b * n + i];
  return s;
}

__global__ void k_part_sums(const double* __restrict__ part, int nb, int n, double* __restrict__ D) {
  follow();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) D[i] = part_sum(part, nb, n, i);
}

// vol = sum_i D_i (single block, fixed order per thread then tree).
__device__ __forceinline__ void block_sum_to(const double* __restrict__ v, int n, double* __restrict__ out) {
  __shared__ double red[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += v[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    *out = t;
  }
}

__global__ void k_sum(const double* __restrict__ v, int n, double* __restrict__ out) {
  follow();
  block_sum_to(v, n, out);
}

// ---------------------------------------------------------------- batched form
// The same steps for every graph of a batch, one launch per step; a block
// finds its graph and work item in a tile table.
__global__ void k_g_select_init(const GGraph* __restrict__ gs) {
  const GGraph& G = gs[blockIdx.x];
  select_init(static_cast<SelectState*>(G.sel), ((long long)G.n * (G.n - 1) / 2 - 1) / 2);
}

__global__ void k_g_to_fixed(const uint32_t* __restrict__ tiles, const GGraph* __restrict__ gs) {
  const uint32_t t = tiles[blockIdx.x];
  const GGraph& G = gs[t & 0xFFFu];
  const size_t total = (size_t)G.n * G.T;
  const size_t base = (size_t)(t >> 12) * 1024;
  bool off = false;
  for (size_t idx = base + threadIdx.x; idx < total && idx < base + 1024; idx += blockDim.x) {
    const double a = G.X[idx] * 65536.0;
    const bool ok = (a == rint(a)) && fabs(a) < 8388608.0;
    off |= !ok;
    const size_t i = idx / G.T, tt = idx % G.T;
    G.Xt[tt * G.n + i] = ok ? (int)a : 0;
  }
  if (__syncthreads_or(off) && threadIdx.x == 0) atomicOr(&static_cast<SelectState*>(G.sel)->flags, 1);
}

// tiles: (b << 12) | g, rows 8 b .. of the graph's digit planes
__global__ void __launch_bounds__(256) k_g_prepare_series(const uint32_t* __restrict__ tiles,
                                                           const GGraph* __restrict__ gs) {
  const uint32_t t = tiles[blockIdx.x];
  const GGraph& G = gs[t & 0xFFFu];
  prepare_series_row(G.X, G.n, G.T, (int)(t >> 12) * 8 + (threadIdx.x >> 5), G.npad, G.tp,
                     static_cast<__nv_bfloat162*>(G.planes), G.norms, static_cast<SelectState*>(G.sel));
}

// tiles: g | bi << 12 | bj << 22 (64-node blocks, bi <= bj); what the tensor-core
// distances leave over (128 graphs, T = 64: all by int64 tiles 2.44 ms, through the
// digit planes 0.59 and 0.19 for the planes and the blocks that return here)
__global__ void __launch_bounds__(256) k_g_dist(const uint32_t* __restrict__ tiles, const GGraph* __restrict__ gs) {
  const uint32_t t = tiles[blockIdx.x];
  const GGraph& G = gs[t & 0xFFFu];
  const int bi = (int)((t >> 12) & 0x3FFu), bj = (int)(t >> 22);
  if (static_cast<const SelectState*>(G.sel)->flags & 1)
    dist_f64_tile(G.X, G.n, G.T, G.A, bi, bj);
  else if (!G.planes)
    dist_int_tile(G.Xt, G.n, G.T, G.A, bi, bj);
}

// The buffer is the graph's `part` (as many keys), which is not formed yet.
__device__ __forceinline__ unsigned long long g_select_cap(const GGraph& G) {
  return (unsigned long long)((G.n + DT - 1) / DT) * G.n;
}

__global__ void __launch_bounds__(SAMPLE_THREADS) k_g_select_sample(const GGraph* __restrict__ gs) {
  extern __shared__ __align__(16) unsigned char sample_smem[];
  const GGraph& G = gs[blockIdx.x];
  select_sample(G.n, static_cast<SelectState*>(G.sel), g_select_cap(G), *reinterpret_cast<SampleShared*>(sample_smem),
                [&](uint32_t q) { return sample_key(G.A, G.n, q); });
}

// tiles: (g, first row, end row, b | blocks << 16): block b of the graph's `blocks`
__global__ void __launch_bounds__(SELECT_THREADS, 2) k_g_select_bracket(const int4* __restrict__ tiles,
                                                                     const GGraph* __restrict__ gs) {
  __shared__ SelectShared sm;
  const int4 t = tiles[blockIdx.x];
  const GGraph& G = gs[t.x];
  select_bracket(static_cast<SelectState*>(G.sel), reinterpret_cast<unsigned long long*>(G.part), g_select_cap(G),
                 (unsigned)t.w >> 16, sm,
                 [&](auto&& f) { triangle_keys(G.A, G.n, t.y, t.z, threadIdx.x >> 5, SELECT_WARPS, 0, f); });
}

__global__ void __launch_bounds__(SELECT_THREADS, 2) k_g_select_pass(const int4* __restrict__ tiles,
                                                                  const GGraph* __restrict__ gs, int p) {
  __shared__ SelectShared sm;
  const int4 t = tiles[blockIdx.x];
  const GGraph& G = gs[t.x];
  unsigned long long* hist =
      reinterpret_cast<unsigned long long*>(static_cast<char*>(G.sel) + SELECT_STATE_BYTES);
  select_pass(static_cast<SelectState*>(G.sel), hist, p, G.sigma, reinterpret_cast<unsigned long long*>(G.part),
              g_select_cap(G), (unsigned)t.w & 0xFFFFu, (unsigned)t.w >> 16, sm,
              [&](auto&& f) { triangle_keys(G.A, G.n, t.y, t.z, threadIdx.x >> 5, SELECT_WARPS, 0, f); });
}

__global__ void k_g_set_sigma(const GGraph* __restrict__ gs, double sigma) { *gs[blockIdx.x].sigma = sigma; }

// kernel_tile for every graph (tiles as k_g_dist's)
__global__ void __launch_bounds__(256, 4) k_g_kernel_tiles(const uint32_t* __restrict__ tiles,
                                                            const GGraph* __restrict__ gs) {
  const uint32_t t = tiles[blockIdx.x];
  const GGraph& G = gs[t & 0xFFFu];
  __shared__ KernelTileShared sm;
  exp_table(sm.tab);
  const ExpFactor f = exp_factor(kernel_rcp(*G.sigma, KERNEL_GAUSSIAN));
  __syncthreads();
  kernel_tile_any<KERNEL_GAUSSIAN>(G.A, G.n, f, G.part, (int)((t >> 12) & 0x3FFu), (int)(t >> 22), sm);
}

// D of graph blockIdx.x from its tiles' sums
__global__ void k_g_part_sums(const GGraph* __restrict__ gs) {
  const GGraph& G = gs[blockIdx.x];
  const int nb = (G.n + DT - 1) / DT;
  for (int i = blockIdx.y * blockDim.x + threadIdx.x; i < G.n; i += gridDim.y * blockDim.x)
    G.D[i] = part_sum(G.part, nb, G.n, i);
}

__global__ void k_g_sum(const GGraph* __restrict__ gs) {
  const GGraph& G = gs[blockIdx.x];
  block_sum_to(G.D, G.n, G.vol);
}

}  // namespace

const int* graph_select_flags(const void* sel) { return &static_cast<const SelectState*>(sel)->flags; }

size_t graph_select_bytes() { return SELECT_STATE_BYTES + RADIX_BINS * sizeof(unsigned long long); }

void graph_grouped_tiles(const std::vector<int>& n, const std::vector<char>& tc, int T, GraphTiles& out) {
  std::vector<int> order(n.size());
  for (size_t g = 0; g < n.size(); ++g) order[g] = (int)g;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return n[a] > n[b]; });
  for (int g : order) {
    const int nn = n[g], nb = (nn + DT - 1) / DT;
    const size_t total = (size_t)nn * T;
    if (tc[g]) {
      const int nb128 = (nn + 127) / 128;
      for (int b = 0; b < nb128 * 16; ++b) out.prep.push_back(((uint32_t)b << 12) | (uint32_t)g);
      for (int I = 0; I < nb128; ++I)
        for (int J = 2 * I; J < 2 * nb128; ++J) out.tc.push_back((uint32_t)g | ((uint32_t)I << 12) | ((uint32_t)J << 22));
    } else {
      for (size_t b = 0; b * 1024 < total; ++b) out.fixed.push_back(((uint32_t)b << 12) | (uint32_t)g);
    }
    for (int bi = 0; bi < nb; ++bi)
      for (int bj = bi; bj < nb; ++bj) out.dist.push_back((uint32_t)g | ((uint32_t)bi << 12) | ((uint32_t)bj << 22));
    // selection: consecutive rows holding about 2^17 upper-triangle keys
    int r0 = 0;
    long long acc = 0;
    const size_t sel0 = out.sel.size();
    for (int i = 0; i < nn - 1; ++i) {
      acc += nn - 1 - i;
      if (acc >= (1 << 17) || i == nn - 2) {
        out.sel.push_back(make_int4(g, r0, i + 1, (int)(out.sel.size() - sel0)));
        r0 = i + 1;
        acc = 0;
      }
    }
    for (size_t e = sel0; e < out.sel.size(); ++e) out.sel[e].w |= (int)((out.sel.size() - sel0) << 16);
  }
}

int graph_build_grouped(cdl_ctx* ctx, const GraphBatch& B) {
  cudaStream_t s = ctx->stream;
  CDL_CUDA_TRY(cudaMemsetAsync(B.sel_all, 0, B.sel_bytes, s));
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    k_g_select_init<<<B.G2, 1, 0, s>>>(B.gs);
    CDL_TRY(L.done());
  }
  if (B.prep.count > 0) {
    Launch L(ctx, CDL_KC_DISTANCE, 0);
    k_g_prepare_series<<<B.prep.count, 256, 0, s>>>(B.prep.p, B.gs);
    CDL_TRY(L.done());
  }
  if (B.fixed.count > 0) {
    Launch L(ctx, CDL_KC_DISTANCE, 0);
    k_g_to_fixed<<<B.fixed.count, 256, 0, s>>>(B.fixed.p, B.gs);
    CDL_TRY(L.done());
  }
  if (B.tc.count > 0) CDL_TRY(dist_tc_grouped(ctx, B.dist_groups, B.tc.p, B.tc.count, B.tp, B.dist_terms));
  {
    Launch L(ctx, CDL_KC_DISTANCE, B.tc.count > 0 ? 0 : B.dist_terms);
    k_g_dist<<<B.dist.count, 256, 0, s>>>(B.dist.p, B.gs);
    CDL_TRY(L.done());
  }
  if (B.sigma > 0) {
    Launch L(ctx, CDL_KC_MISC, 0);
    k_g_set_sigma<<<B.G2, 1, 0, s>>>(B.gs, B.sigma);
    CDL_TRY(L.done());
  } else {
    CDL_TRY(allow_smem(ctx, k_g_select_sample, (int)sizeof(SampleShared)));
    {
      Launch L(ctx, CDL_KC_SELECT, 0);
      k_g_select_sample<<<B.G2, SAMPLE_THREADS, sizeof(SampleShared), s>>>(B.gs);
      CDL_TRY(L.done());
    }
    {
      Launch L(ctx, CDL_KC_SELECT, B.select_bytes);
      k_g_select_bracket<<<B.sel_count, SELECT_THREADS, 0, s>>>(B.sel, B.gs);
      CDL_TRY(L.done());
    }
    for (int p = 0; p < 6; ++p) {
      Launch L(ctx, CDL_KC_SELECT, 0);
      k_g_select_pass<<<B.sel_count, SELECT_THREADS, 0, s>>>(B.sel, B.gs, p);
      CDL_TRY(L.done());
    }
  }
  {
    Launch L(ctx, CDL_KC_KERNEL, B.kernel_bytes);
    k_g_kernel_tiles<<<B.dist.count, 256, 0, s>>>(B.dist.p, B.gs);
    CDL_TRY(L.done());
  }
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    k_g_part_sums<<<dim3(B.G2, 8), 256, 0, s>>>(B.gs);
    CDL_TRY(L.done());
  }
  Launch L(ctx, CDL_KC_MISC, 0);
  k_g_sum<<<B.G2, 1024, 0, s>>>(B.gs);
  return L.done();
}

int graph_build(cdl_ctx* ctx, const double* X, int64_t n64, int T, double sigma, double* A,
                double* D, double* vol, double* sigma_out, int kernel) {
  const int n = (int)n64;
  cudaStream_t s = ctx->stream;
  void *wsSt, *wsHist;
  CDL_TRY(ws_get(ctx, "graph.state", sizeof(SelectState), &wsSt));
  CDL_TRY(ws_get(ctx, "graph.hist", RADIX_BINS * sizeof(unsigned long long), &wsHist));
  SelectState* st = static_cast<SelectState*>(wsSt);
  unsigned long long* hist = static_cast<unsigned long long*>(wsHist);
  const long long m = (long long)n * (n - 1) / 2;
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_select_init, 1, 1024, 0, s, st, (m - 1) / 2, hist);
    CDL_TRY(L.done());
  }
  const int nb = (n + DT - 1) / DT;
  const long long tiles = (long long)nb * (nb + 1) / 2;
  if (tiles > 0x7fffffffLL) return CDL_ERR_INVALID_ARG;
  {
    // grid inputs: exact Gram on the tensor cores (three bf16 digit planes)
    const int rows = (n + 127) / 128 * 128, tp = (T + 63) / 64 * 64;
    void *wsPl, *wsNo;
    CDL_TRY(ws_get(ctx, "graph.xplanes", 3 * (size_t)rows * tp * 2, &wsPl));
    CDL_TRY(ws_get(ctx, "graph.norms", (size_t)rows * sizeof(long long), &wsNo));
    {
      Launch L(ctx, CDL_KC_DISTANCE, 0);
      launch_next(k_prepare_series, rows / 8, 256, 0, s, X, n, T, rows, tp, static_cast<__nv_bfloat162*>(wsPl),
                  static_cast<long long*>(wsNo), st);
      CDL_TRY(L.done());
    }
    CDL_TRY(dist_tc(ctx, wsPl, static_cast<const long long*>(wsNo), n, rows, tp, A, &st->flags,
                    0.5 * (double)n * (double)(n - 1) * T));
  }
  void* wsPart;
  CDL_TRY(ws_get(ctx, "graph.dpart", (size_t)nb * n * sizeof(double), &wsPart));
  double* part = static_cast<double*>(wsPart);
  // off the grid: through residues on the tensor cores, and what that leaves over in float64
  const unsigned char* bad = nullptr;
  const int rows = (n + 127) / 128 * 128, kp = (T + 63) / 64 * 64, nb64 = rows / 64;
  const size_t bad_bytes = ((size_t)nb64 * nb64 + 3) / 4 * 4;
  void *wsRp, *wsRn, *wsRe, *wsBad;
  if (ws_get_opt(ctx, {{"crt.planes", T < DIST_RES_MIN_T ? 256 : (size_t)16 * rows * kp * 2, &wsRp},
                       {"crt.dist.norms", (size_t)rows * 16, &wsRn},
                       {"crt.dist.e", (size_t)rows * sizeof(int), &wsRe},
                       {"crt.dist.bad", bad_bytes, &wsBad}}) == CDL_OK) {
    CDL_TRY(series_residues(ctx, X, n, T, rows, kp, &st->flags, static_cast<int*>(wsRe), wsRn, wsRp, wsBad,
                            (int)(bad_bytes / 4)));
    CDL_TRY(dist_residues_tc(ctx, wsRp, static_cast<const int*>(wsRe), wsRn, n, T, rows, kp, A, &st->flags, wsBad));
    bad = static_cast<const unsigned char*>(wsBad);
  }
  {
    Launch L(ctx, CDL_KC_DISTANCE, 0);
    launch_next(k_dist_f64, (unsigned)std::min<long long>(tiles, ctx->sm_count * 6), 256, 0, s, X, n, T, A, st, bad,
                nb64);
    CDL_TRY(L.done());
  }
  if (sigma > 0) {
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_set_scalar, 1, 1, 0, s, sigma_out, sigma);
    CDL_TRY(L.done());
  } else {
    // one buffer for the selection's keys and the kernel values' partial sums after it
    unsigned long long* sbuf = reinterpret_cast<unsigned long long*>(part);
    const unsigned long long cap = (unsigned long long)nb * n;
    if (m >= SELECT_BRACKET_MIN) {
      CDL_TRY(allow_smem(ctx, k_select_sample, (int)sizeof(SampleShared)));
      {
        // the samples into the buffer first: one block's scattered loads took 25 us
        Launch L(ctx, CDL_KC_SELECT, 0);
        launch_next(k_sample_keys, SAMPLE / 256, 256, 0, s, A, n, reinterpret_cast<uint32_t*>(sbuf));
        CDL_TRY(L.done());
      }
      {
        Launch L(ctx, CDL_KC_SELECT, 0);
        launch_next(k_select_sample, 1, SAMPLE_THREADS, sizeof(SampleShared), s,
                    reinterpret_cast<const uint32_t*>(sbuf), n, st, cap);
        CDL_TRY(L.done());
      }
      Launch L(ctx, CDL_KC_SELECT, 8.0 * (double)m);
      launch_next(k_select_bracket, ctx->sm_count * 2, SELECT_THREADS, 0, s, A, n, st, sbuf, cap);
      CDL_TRY(L.done());
    }
    const unsigned hblocks = (unsigned)std::min<long long>((m + 4095) / 4096, ctx->sm_count * 2);
    for (int p = 0; p < 6; ++p) {
      // work: bytes of the triangle for the full passes (the later ones read the copied keys)
      Launch L(ctx, CDL_KC_SELECT, p < 3 && m < SELECT_BRACKET_MIN ? 8.0 * (double)m : 0.0);
      launch_next(k_select_pass, hblocks, SELECT_THREADS, 0, s, A, n, p, st, hist, sigma_out, sbuf, cap);
      CDL_TRY(L.done());
    }
  }
  {
    {
      Launch L(ctx, CDL_KC_KERNEL, 16.0 * (double)n * n);
      const unsigned blocks = (unsigned)std::min<long long>(tiles, ctx->sm_count * 4);
      if (kernel == KERNEL_EXP)
        launch_next(k_kernel_tiles<KERNEL_EXP>, blocks, 256, 0, s, A, n, sigma_out, part);
      else
        launch_next(k_kernel_tiles<KERNEL_GAUSSIAN>, blocks, 256, 0, s, A, n, sigma_out, part);
      CDL_TRY(L.done());
    }
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_part_sums, (n + 255) / 256, 256, 0, s, part, nb, n, D);
    CDL_TRY(L.done());
  }
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_sum, 1, 1024, 0, s, D, n, vol);
    CDL_TRY(L.done());
  }
  return CDL_OK;
}

// ---------------------------------------------------------------------------
// Graphs too large to keep: the Gaussian-kernel graph regenerated from the
// node series in row panels of P rows wherever it is needed. The series'
// digit planes and squared norms are formed once (distances exact on the
// tensor cores; inputs must lie on the 2^-16 grid), sigma by the same exact
// radix select as graph_build with every histogram pass streaming the
// upper-triangle part of each panel's distances, then the degrees from the
// panels' kernel rows. The panel A values equal graph_build's (exact
// distances, the same exponential), the degrees up to summation order.
int graph_regen_init(cdl_ctx* ctx, RegenGraph& g, const double* X, int64_t n64, int T, double sigma, double* panel,
                     int P) {
  const int n = (int)n64;
  cudaStream_t s = ctx->stream;
  g.X = X;
  g.n = n;
  g.T = T;
  g.rows = (n + 127) / 128 * 128;
  g.tp = (T + 63) / 64 * 64;
  const std::string tag = "regen." + std::to_string(g.id) + ".";
  void *wsSt, *wsHist, *wsPl, *wsNo, *wsSc;
  CDL_TRY(ws_get(ctx, (tag + "state").c_str(), sizeof(SelectState), &wsSt));
  CDL_TRY(ws_get(ctx, (tag + "hist").c_str(), RADIX_BINS * sizeof(unsigned long long), &wsHist));
  CDL_TRY(ws_get(ctx, (tag + "planes").c_str(), 3 * (size_t)g.rows * g.tp * 2, &wsPl));
  CDL_TRY(ws_get(ctx, (tag + "norms").c_str(), (size_t)g.rows * sizeof(long long), &wsNo));
  CDL_TRY(ws_get(ctx, (tag + "scalars").c_str(), 2 * sizeof(double), &wsSc));
  SelectState* st = static_cast<SelectState*>(wsSt);
  unsigned long long* hist = static_cast<unsigned long long*>(wsHist);
  g.planes = wsPl;
  g.norms = static_cast<const long long*>(wsNo);
  g.offgrid = &st->flags;
  g.sigma = static_cast<double*>(wsSc);
  const long long m = (long long)n * (n - 1) / 2;
  {
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_select_init, 1, 1024, 0, s, st, (m - 1) / 2, hist);
    CDL_TRY(L.done());
  }
  {
    Launch L(ctx, CDL_KC_DISTANCE, 0);
    launch_next(k_prepare_series, g.rows / 8, 256, 0, s, X, n, T, g.rows, g.tp, static_cast<__nv_bfloat162*>(wsPl),
                static_cast<long long*>(wsNo), st);
    CDL_TRY(L.done());
  }
  int flags = 0;
  CDL_CUDA_TRY(cudaMemcpyAsync(&flags, &st->flags, sizeof(int), cudaMemcpyDeviceToHost, s));
  CDL_CUDA_TRY(cudaStreamSynchronize(s));
  if (flags & 1) {
    set_last_error("graph regeneration needs inputs on the 2^-16 grid", __FILE__, __LINE__);
    return CDL_ERR_UNSUPPORTED;
  }
  if (sigma > 0) {
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_set_scalar, 1, 1, 0, s, g.sigma, sigma);
    CDL_TRY(L.done());
  } else {
    const int shifts[6] = {52, 40, 28, 16, 4, 0};
    const int widths[6] = {12, 12, 12, 12, 12, 4};
    for (int p = 0; p < 6; ++p) {
      for (int r0 = 0; r0 < g.rows; r0 += P) {
        const int pr = std::min(P, g.rows - r0);
        CDL_TRY(dist_tc_panel(ctx, g.planes, g.norms, n, g.rows, g.tp, panel, r0, pr, true, g.offgrid));
        const int r1 = std::min(n - 1, r0 + pr);
        if (r1 <= r0) continue;
        Launch L(ctx, CDL_KC_SELECT, 8.0 * (double)pr * n);
        launch_next(k_select_hist_panel, std::min((r1 - r0 + SELECT_WARPS - 1) / SELECT_WARPS, ctx->sm_count * 4),
                    SELECT_THREADS, 0, s, panel, n, shifts[p], widths[p], st, hist, r0, r1);
        CDL_TRY(L.done());
      }
      Launch L(ctx, CDL_KC_SELECT, 0);
      launch_next(k_select_step, 1, SELECT_THREADS, 0, s, st, hist, shifts[p], widths[p], g.sigma, p == 5);
      CDL_TRY(L.done());
    }
  }
  // degrees: every panel's kernel rows once
  for (int r0 = 0; r0 < n; r0 += P) {
    const int pr = std::min(P, n - r0);
    CDL_TRY(regen_panel(ctx, g, panel, r0, pr, g.D));
  }
  Launch L(ctx, CDL_KC_MISC, 0);
  launch_next(k_sum, 1, 1024, 0, s, g.D, n, g.vol);
  return L.done();
}

int regen_panel(cdl_ctx* ctx, const RegenGraph& g, double* panel, int r0, int rows, double* D) {
  const int pr = (int)std::min<long long>(round_up(rows, 128), g.rows - r0);
  CDL_TRY(dist_tc_panel(ctx, g.planes, g.norms, g.n, g.rows, g.tp, panel, r0, pr, false, g.offgrid));
  const int r1 = std::min(g.n, r0 + rows);
  Launch L(ctx, CDL_KC_KERNEL, 16.0 * (double)(r1 - r0) * g.n);
  launch_next(k_kernel_rows_panel, std::min(r1 - r0, ctx->sm_count * 8), 256, 0, ctx->stream, panel, g.n, g.sigma, D,
              r0, r1);
  return L.done();
}

// ---------------------------------------------------------------------------
// Given graphs: degrees of a caller's adjacency matrix and symmetric edge
// weights added to it (the second graph of the synthetic experiments,
// A_2 = Q + (R + R^T) / 2, Sec. 4.2.1).

// D_i = sum_j A_ij, one block (256 threads) per row: each thread adds its
// strided terms in float64 with a running compensation (Neumaier's TwoSum
// form), the (sum, compensation) pairs are combined the same way across the
// warp and the block; D_i = sum + compensation (within a few units in the
// last place of the exact row sum).
__device__ __forceinline__ void neumaier_add(double& s, double& c, double a) {
  const double t = s + a;
  c += fabs(s) >= fabs(a) ? (s - t) + a : (a - t) + s;
  s = t;
}

__global__ void __launch_bounds__(256) k_degrees(const double* __restrict__ A, int n, double* __restrict__ D) {
  follow();
  __shared__ double red_s[8], red_c[8];
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const double* row = A + (size_t)i * n;
    double s = 0.0, c = 0.0;
    for (int j = threadIdx.x; j < n; j += 256) neumaier_add(s, c, row[j]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double s2 = __shfl_xor_sync(0xffffffffu, s, o);
      const double c2 = __shfl_xor_sync(0xffffffffu, c, o);
      neumaier_add(s, c, s2);
      c += c2;
    }
    if ((threadIdx.x & 31) == 0) {
      red_s[threadIdx.x >> 5] = s;
      red_c[threadIdx.x >> 5] = c;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = red_s[0], tc = red_c[0];
      for (int w = 1; w < 8; ++w) {
        neumaier_add(t, tc, red_s[w]);
        tc += red_c[w];
      }
      D[i] = t + tc;
    }
    __syncthreads();
  }
}

// A_ij += w_e and A_ji += w_e for each pair e = (i, j) of ij (m x 2, row-major).
// Invalid entries (an index outside [0, n), i == j, w negative, infinite or
// NaN) are skipped and counted in *bad. Each listed unordered pair touches its
// two entries once, so distinct pairs give exact, order-free results.
__global__ void k_add_edges(double* __restrict__ A, int n, long long m, const long long* __restrict__ ij,
                            const double* __restrict__ w, unsigned long long* __restrict__ bad) {
  follow();
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += stride) {
    const long long i = ij[2 * e], j = ij[2 * e + 1];
    const double v = w[e];
    if (i < 0 || i >= n || j < 0 || j >= n || i == j || !(v >= 0.0) || isinf(v)) {
      atomicAdd(bad, 1ull);
      continue;
    }
    atomicAdd(A + (size_t)i * n + j, v);
    atomicAdd(A + (size_t)j * n + i, v);
  }
}

int graph_degrees(cdl_ctx* ctx, const double* A, int64_t n64, double* D, double* vol) {
  const int n = (int)n64;
  cudaStream_t s = ctx->stream;
  {
    Launch L(ctx, CDL_KC_KERNEL, 8.0 * (double)n * n);
    launch_next(k_degrees, std::min(n, ctx->sm_count * 8), 256, 0, s, A, n, D);
    CDL_TRY(L.done());
  }
  Launch L(ctx, CDL_KC_MISC, 0);
  launch_next(k_sum, 1, 1024, 0, s, D, n, vol);
  return L.done();
}

int graph_add_edges(cdl_ctx* ctx, double* A, int64_t n, int64_t m, const int64_t* ij, const double* w,
                    int64_t* n_bad) {
  cudaStream_t s = ctx->stream;
  void* wsBad;
  CDL_TRY(ws_get(ctx, "graph.bad", sizeof(unsigned long long), &wsBad));
  unsigned long long* bad = static_cast<unsigned long long*>(wsBad);
  CDL_CUDA_TRY(cudaMemsetAsync(bad, 0, sizeof(unsigned long long), s));
  if (m > 0) {
    const long long blocks = std::min<long long>((m + 255) / 256, (long long)ctx->sm_count * 16);
    Launch L(ctx, CDL_KC_MISC, 0);
    launch_next(k_add_edges, (unsigned)blocks, 256, 0, s, A, (int)n, (long long)m,
                reinterpret_cast<const long long*>(ij), w, bad);
    CDL_TRY(L.done());
  }
  unsigned long long h = 0;
  CDL_CUDA_TRY(cudaMemcpyAsync(&h, bad, sizeof(h), cudaMemcpyDeviceToHost, s));
  CDL_CUDA_TRY(cudaStreamSynchronize(s));
  if (n_bad) *n_bad = (int64_t)h;
  return h ? CDL_ERR_INVALID_ARG : CDL_OK;
}

// ---------------------------------------------------------------------------
// Graph build without any device allocation.
//
// Some callers cannot let a library call cudaMalloc: a process that has
// handed (almost) all device memory to its own pool allocator, where an extra
// allocation would fail or fragment the pool, or a service that must not
// allocate once it is running. For them cdl_build_graph_static runs the same
// kernels as cdl_build_graph, with all of their scratch (the fixed-point copy
// of X, the radix-select state and histogram) in the statically allocated
// device array below, which every GPU that loads the library holds until the
// process exits. The caller still owns X and the outputs.

constexpr size_t STATIC_XT_ELEMS = size_t(1) << 20;   // n * T limit (4 MiB of int32)
constexpr size_t STATIC_HIST_OFF = STATIC_XT_ELEMS * sizeof(int);
constexpr size_t STATIC_STATE_OFF = STATIC_HIST_OFF + RADIX_BINS * sizeof(unsigned long long);
constexpr size_t STATIC_SCRATCH_BYTES = STATIC_STATE_OFF + 256;

static __device__ __align__(256) unsigned char g_graph_scratch[STATIC_SCRATCH_BYTES];

namespace {

// The device address of g_graph_scratch belongs to the CUDA context that was
// current when it was looked up: another context on the same device (one the
// caller made current through the driver API, or the primary context
// re-created after cudaDeviceReset) has its own copy of the array at another
// address. So the address is cached per context, keyed by the context's
// unique ID (cuCtxGetId: IDs are never reused within a process), and the
// host-side name of the array, which is only a stand-in for the symbol, is
// never passed to a kernel.
constexpr int MAX_CONTEXTS = 64;
std::mutex g_static_mu;
unsigned long long g_static_ctx_id[MAX_CONTEXTS] = {0};
void* g_static_addr[MAX_CONTEXTS] = {nullptr};
int g_static_used = 0;

typedef int (*PFN_ctx_get_current)(void** ctx);
typedef int (*PFN_ctx_get_id)(void* ctx, unsigned long long* id);

// ID of the current CUDA context. Driver entry points are taken through the
// runtime, so the library does not link libcuda itself.
int current_context_id(unsigned long long* id) {
  static PFN_ctx_get_current get_current = nullptr;
  static PFN_ctx_get_id get_id = nullptr;
  if (!get_current || !get_id) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !p)
      return CDL_ERR_CUDA;
    get_current = reinterpret_cast<PFN_ctx_get_current>(p);
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !p)
      return CDL_ERR_CUDA;
    get_id = reinterpret_cast<PFN_ctx_get_id>(p);
  }
  // the pointer checks before this call have already made the runtime's
  // context current when the caller had none
  void* c = nullptr;
  if (get_current(&c) != 0 || !c) {
    set_last_error("no current CUDA context", __FILE__, __LINE__);
    return CDL_ERR_CUDA;
  }
  if (get_id(c, id) != 0) {
    set_last_error("cuCtxGetId failed", __FILE__, __LINE__);
    return CDL_ERR_CUDA;
  }
  return CDL_OK;
}

// Device address of g_graph_scratch in the current context, looked up with
// that context current on the first call in it and cached.
int static_scratch(void** out) {
  unsigned long long id = 0;
  CDL_TRY(current_context_id(&id));
  std::lock_guard<std::mutex> lock(g_static_mu);
  for (int i = 0; i < g_static_used; ++i)
    if (g_static_ctx_id[i] == id) {
      *out = g_static_addr[i];
      return CDL_OK;
    }
  void* p = nullptr;
  CDL_CUDA_TRY(cudaGetSymbolAddress(&p, g_graph_scratch));
  // a full table starts over: the contexts it names may be gone, and a
  // lookup costs one symbol query
  if (g_static_used == MAX_CONTEXTS) g_static_used = 0;
  g_static_ctx_id[g_static_used] = id;
  g_static_addr[g_static_used] = p;
  ++g_static_used;
  *out = p;
  return CDL_OK;
}

// Device or managed memory reachable from the current device (the same
// rule as the context-based entry points).
int on_current_device(const void* p) {
  if (!p) return CDL_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(p) % 8) return CDL_ERR_INVALID_ARG;
  int dev = 0;
  CDL_CUDA_TRY(cudaGetDevice(&dev));
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return CDL_ERR_INVALID_ARG;
  }
  if (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) return CDL_ERR_INVALID_ARG;
  if (at.type == cudaMemoryTypeDevice && at.device != dev) return CDL_ERR_INVALID_ARG;
  return CDL_OK;
}

int launched() {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_error(cudaGetErrorString(e), __FILE__, __LINE__);
    return CDL_ERR_CUDA;
  }
  return CDL_OK;
}

}  // namespace

int graph_build_static(const double* X, int64_t n64, int T, double sigma, double* A, double* D,
                       double* vol, double* sigma_out, cudaStream_t s) {
  if (n64 < 2 || n64 > (1 << 20) || T < 1 || T > 4096) return CDL_ERR_INVALID_ARG;
  if ((size_t)n64 * (size_t)T > STATIC_XT_ELEMS) {
    set_last_error("n * T exceeds the static scratch limit of 2^20 samples", __FILE__, __LINE__);
    return CDL_ERR_INVALID_ARG;
  }
  CDL_TRY(on_current_device(X));
  CDL_TRY(on_current_device(A));
  CDL_TRY(on_current_device(D));
  CDL_TRY(on_current_device(vol));
  CDL_TRY(on_current_device(sigma_out));
  void* base = nullptr;
  CDL_TRY(static_scratch(&base));
  int dev = 0, sm_count = 0;
  CDL_CUDA_TRY(cudaGetDevice(&dev));
  CDL_CUDA_TRY(cudaDeviceGetAttribute(&sm_count, cudaDevAttrMultiProcessorCount, dev));
  const int n = (int)n64;
  int* Xt = static_cast<int*>(base);
  unsigned long long* hist = reinterpret_cast<unsigned long long*>(static_cast<char*>(base) + STATIC_HIST_OFF);
  SelectState* st = reinterpret_cast<SelectState*>(static_cast<char*>(base) + STATIC_STATE_OFF);
  const long long m = (long long)n * (n - 1) / 2;
  // The array keeps the previous call's contents: the select state and the
  // histogram must start from zero, Xt is fully overwritten.
  launch_next(k_select_init, 1, 1024, 0, s, st, (m - 1) / 2, hist);
  CDL_TRY(launched());
  const size_t total = (size_t)n * T;
  launch_next(k_to_fixed, (int)std::min<size_t>((total + 255) / 256, (size_t)sm_count * 8), 256, 0, s, X, Xt, n, T, st);
  CDL_TRY(launched());
  const int nb = (n + DT - 1) / DT;
  const long long tiles = (long long)nb * (nb + 1) / 2;
  launch_next(k_dist_int, (unsigned)tiles, 256, 0, s, Xt, n, T, A, st);
  CDL_TRY(launched());
  launch_next(k_dist_f64, (unsigned)std::min<long long>(tiles, sm_count * 6), 256, 0, s, X, n, T, A, st, nullptr, 0);
  CDL_TRY(launched());
  if (sigma > 0) {
    launch_next(k_set_scalar, 1, 1, 0, s, sigma_out, sigma);
    CDL_TRY(launched());
  } else {
    const unsigned hblocks = (unsigned)std::min<long long>((m + 4095) / 4096, sm_count * 2);
    for (int p = 0; p < 6; ++p) {   // no buffer: every pass over A
      launch_next(k_select_pass, hblocks, SELECT_THREADS, 0, s, A, n, p, st, hist, sigma_out, nullptr, 0);
      CDL_TRY(launched());
    }
  }
  launch_next(k_kernel_rows<KERNEL_GAUSSIAN>, std::min(n, sm_count * 8), 256, 0, s, A, n, sigma_out, D);
  CDL_TRY(launched());
  launch_next(k_sum, 1, 1024, 0, s, D, n, vol);
  return launched();
}

}  // namespace cdl
