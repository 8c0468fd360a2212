// FP64 product C = A.B emulated on the e4m3 tensor cores (Ozaki scheme).
//
// Method: K. Ozaki, T. Ogita, S. Oishi, S. M. Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix
// multiplication and its applicability", Numer. Algorithms 59 (2012): split
// every operand into slices whose pairwise products a low-precision matrix
// unit computes without rounding, then add the slice products in the working
// precision.  This library's variant (not in the paper, whose double-precision
// kernels use FP64 arithmetic directly):
//
//   * Row i of A is scaled by 2^-sigma_i, sigma_i = ilogb(max_r |a_ir|) + 2,
//     so |a_ir| 2^-sigma_i < 1/2; column j of B by 2^-tau_j likewise.  The
//     scaled magnitude, truncated to 5S fraction bits, is the integer
//     F = floor(|a| 2^(5S - sigma)) < 2^(5S - 1) (S <= 12: 59 bits), written
//     in balanced base 32: G = F + 16 (32^S - 1) / 31 (16 added to every
//     base-32 position), then d_t = g_t - 16 with g_t = (G >> 5(S-1-t)) & 31
//     for t >= 1 and g_0 = G >> 5(S-1) unmasked, so d_t lies in [-16, 15]
//     (t >= 1), d_0 in [0, 16], and sum_t d_t 32^(S-1-t) = F.  With the sign
//     of a on every digit:
//         a 2^-sigma = sum_t d_t 32^-(t+1) + delta,  |delta| < 2^(-5S).
//     Every digit (|d| <= 16) is exact in e4m3; five bits per slice instead
//     of four cut the slices (and the S(S+1)/2 level products) for the same
//     precision.
//   * Level L = 0..S-1 collects the slice products of equal weight:
//         D_L = sum_{t+u=L} A_t B_u,
//     one tensor-core product along a K of (L+1) slices: A's slices 0..L
//     against B's slices L..0.  Each term is at most 256, a level at most
//     256 S mc, so with K cut into chunks of mc <= (2^24 - 1) / (256 S)
//     columns (a multiple of 128) every D_L is an integer below 2^24 and
//     FP32 accumulation (and the tail split's FP32 partial sums) is exact.
//     Pairs with t + u >= S are dropped.
//   * c_ij = 2^(sigma_i + tau_j) * sum_L 32^-(L+2) D_L[i][j] (summed over
//     the chunks too), formed exactly in 128-bit integers and rounded once
//     to FP64: the double nearest to the kept digit products.
//
// Error: a term a_ir b_rj loses at most (S + 2) 2^(sigma_i + tau_j - 5S - 1)
// (both truncations and the dropped pairs), and zero entries lose nothing,
// so |c^_ij - c_ij| <= (S + 2) 2^(sigma_i + tau_j - 5S - 1) #{r : a_ir b_rj != 0}
// plus the final rounding (half an ulp of c^_ij).  Relative to (|A||B|)_ij this is
// data dependent: ~8 (S + 2) 2^(-5S) for rows and columns without a wide
// spread of magnitudes (uniform data), much more where a row's largest entry
// dwarfs the entries that meet the column's mass.  The accuracy gate (on by
// default) bounds P_ij = (|A||B|)_ij 2^-(sigma_i + tau_j) from below with one
// more e4m3 slice per operand (the scaled magnitudes truncated onto the e4m3
// grid) and one more tensor-core product per K chunk, and where any entry's
// bound could exceed 1e-14 sqrt(m) (|A||B|)_ij, recomputes C with the FP64
// FMA kernel.
//
// Data layout in the library's scratch ("pack region" first, 128-byte rows,
// as the tensor-core kernel's tensor map requires):
//   A digits of chunk c: tile (mt, slice t, kb) at rows
//       a0_c + ((mt*SS + t)*kt_c + kb)*128, one row per row of A (128 k);
//   B digits of chunk c: tile (nt, slot, kb) at rows
//       b0_c + ((nt*SS + slot)*kt_c + kb)*bn, slot = S-1-u for slice u, one
//       row per column of B, so that B's slices L..0 are contiguous;
//   SS = S, or S + 1 with the gate, whose slice is t = slot = S;
//   then the row/column maxima (bit patterns), zero scale words, the level
//   sums D (FP32, [chunk][level] planes of n x p, padded so that planes are
//   not a power of two apart) followed by the gate's planes [chunk], the
//   problem table with the work units of each CTA, the unit map and the
//   gate's flag.
// The level problem (c, L) reads A's K blocks [0, (L+1) kt_c) and B's
// [(S-1-L) kt_c, S kt_c) of each tile through the table's K stride SS kt_c;
// the gate's problem c reads [S kt_c, (S+1) kt_c) of both.
// Rows (columns) holding a NaN or an infinity give NaN rows (columns) of C.
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "ctx.h"
#include "split_common.cuh"

namespace mm {

constexpr int kOzakiMaxChunks = 1024;  // K chunks (the sum's int64 parts stay exact)

namespace {

constexpr int kRowsPerItem = 8;   // maxima: warps per block, one row of A each
constexpr int kColStrip = 128;    // maxima: columns of B per strip
constexpr int kRowChunk = 64;     // maxima: rows of B per strip item
constexpr int kSeg = 16;          // digits: consecutive k per thread
constexpr int kDigRows = 32;      // digits: rows of A (columns of B) per block

// Four consecutive doubles at a 32-byte boundary in one load.
__device__ __forceinline__ void load4(const double *src, double (&v)[4]) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];"
               : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
               : "l"(src));
}
__device__ __forceinline__ bool aligned32(const void *p) {
  return (reinterpret_cast<uintptr_t>(p) & 31u) == 0;
}
__device__ __forceinline__ uint64_t max64(uint64_t a, uint64_t b) { return a > b ? a : b; }

__device__ __forceinline__ uint64_t abs_bits64(double x) {
  return (uint64_t)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// sigma = ilogb(max) + 2 from the bit pattern of a row's largest magnitude;
// 0 for an all-zero row; finite = false for a NaN or an infinity.
__device__ __forceinline__ int slice_exponent(uint64_t max_bits, bool &finite) {
  const int e_raw = (int)(max_bits >> 52);
  finite = e_raw != 0x7ff;
  if (max_bits == 0 || !finite) return 0;
  if (e_raw == 0) return (63 - __clzll((long long)max_bits)) - 1074 + 2;  // subnormal
  return e_raw - 1023 + 2;
}

// Truncated fixed-point magnitude F = floor(|x| 2^(5S - sigma)) (< 2^(5S-1)
// for |x| < 2^(sigma-1)) and the sign of x.
__device__ __forceinline__ uint64_t fixed_magnitude(double x, int sigma, int S, bool &neg) {
  const uint64_t bits = (uint64_t)__double_as_longlong(x);
  neg = (bits >> 63) != 0;
  const int e_raw = (int)((bits >> 52) & 0x7ff);
  const uint64_t frac = bits & 0xfffffffffffffull;
  uint64_t mant;
  int ex;
  if (e_raw == 0) {
    mant = frac;
    ex = -1022;
  } else {
    mant = frac | (1ull << 52);
    ex = e_raw - 1023;
  }
  const int sh = ex - 52 + 5 * S - sigma;  // |x| = mant 2^(ex - 52)
  if (mant == 0 || sh <= -64) return 0;
  return sh >= 0 ? (mant << sh) : (mant >> -sh);
}

// G = F + 16 (32^S - 1) / 31: 16 added to every base-32 position of F, so
// that g_t - 16 are the balanced digits (below 2^60 for S <= 12).
template <int S>
__device__ __forceinline__ uint64_t balanced_offset() {
  static_assert(S >= 2 && S <= 12, "slices");
  uint64_t o = 0;
#pragma unroll
  for (int t = 0; t < S; t++) o = (o << 5) | 16u;
  return o;
}

// Slice digits of 16 values (one per k) -> 16 e4m3 bytes, in pairs of fp16:
// 1024 + g is the fp16 with g in its low bits, and (1024 + g) s - 1040 s = s (g - 16)
// is exact there, s = +-1 the value's sign (0 comes out +0), so a digit of two
// values costs a shift, a mask, one fused multiply-add and one conversion.  The
// digits lie five bits apart in 30-bit words of G (lo: the six lowest ones, hi:
// the others); `word` holds sixteen bits, three digits, of a pair.
struct PairSigns {
  __half2 mul, add;  // (s0, s1) and -1040 (s0, s1)
};
__device__ __forceinline__ uint32_t digit_pair(uint32_t word, int pos, uint32_t mask, const PairSigns &sg) {
  const uint32_t e = ((word >> (5 * pos)) & mask) | 0x64006400u;
  const __half2 d = __hfma2(*reinterpret_cast<const __half2 *>(&e), sg.mul, sg.add);
  return (uint32_t)__nv_cvt_halfraw2_to_fp8x2(static_cast<__half2_raw>(d), __NV_SATFINITE, __NV_E4M3);
}

// The accuracy gate's slice: 16 |x| 2^-sigma truncated toward zero onto the
// e4m3 grid (4 significant bits at 2^-6 and above, multiples of 2^-9 below;
// 0 under 2^-9), so the value is exact in e4m3 and never above 16 |x| 2^-sigma.
// Formed from the truncated fixed-point magnitude F = floor(|x| 2^(5S-sigma))
// in integer and FP32 arithmetic (16 |x| 2^-sigma >= F 2^(4-5S)): F's top four
// bits times a power of two (below 8, since |x| 2^-sigma < 1/2).
__device__ __forceinline__ float gate_value(uint64_t F, int S) {
  if (F == 0) return 0.0f;
  const int b = 64 - __clzll((long long)F);  // bit length, 1..5S-1
  const int sh = b > 4 ? b - 4 : 0;
  const float top = (float)(uint32_t)(F >> sh);  // 1..15, exact
  // 2^(sh + 4 - 5S) >= 2^(4 - 60): a normal float
  const float v = top * __int_as_float((sh + 4 - 5 * S + 127) << 23);
  return v >= 0x1p-6f ? v : floorf(v * 512.0f) * 0x1p-9f;
}

// The same as an e4m3 byte from the double's own bits, for S >= 4 and a normal x
// (F then holds every bit that the e4m3 grid keeps): its leading four
// significant bits m8, with the exponent field E = ex - sigma + 11 of 16 |x| 2^-sigma
// (at most 9), shifted out below 2^-6.
__device__ __forceinline__ uint32_t gate_byte(uint32_t hi, int sigma) {
  const int E = (int)((hi >> 20) & 0x7ff) - 1023 - sigma + 11;
  const uint32_t m8 = 8u | ((hi >> 17) & 7u);
  return E >= 1 ? ((uint32_t)E << 3) | (m8 & 7u) : (E > -3 ? m8 >> (1 - E) : 0u);
}

// One thread's 16 consecutive k of a row (column): S digit slices and, with
// GATE, the gate's slice as 16-byte groups; put(t, bytes) stores slice t (S: the
// gate's).  `live` values are within the matrix and `finite` its row's maximum.
template <int S, bool GATE, typename Get, typename Put>
__device__ __forceinline__ void emit_digits(int live, bool finite, int sigma, Get get, Put put) {
  uint32_t lo[kSeg], hi[S > 6 ? kSeg : 1];
  uint32_t negmask = 0, gate[4] = {0, 0, 0, 0};
#pragma unroll
  for (int e = 0; e < kSeg; e++) {
    uint64_t F = 0;
    if (e < live && finite) {
      const double x = get(e);
      bool neg;
      F = fixed_magnitude(x, sigma, S, neg);
      negmask |= (uint32_t)neg << e;
      if (GATE) {
        const uint32_t xh = (uint32_t)__double2hiint(x);
        uint32_t b;
        if (S >= 4 && (xh & 0x7ff00000u) != 0) {
          b = gate_byte(xh, sigma);
        } else {
          b = (uint32_t)__nv_cvt_float_to_fp8(gate_value(F, S), __NV_SATFINITE, __NV_E4M3);
        }
        gate[e >> 2] |= b << (8 * (e & 3));
      }
    }
    const uint64_t G = F + balanced_offset<S>();  // padding and zeros: all digits 0
    // (the top digit may take a sixth bit)
    lo[e] = (uint32_t)G;
    if (S > 6) hi[e] = (uint32_t)(G >> 30);
  }
  PairSigns sg[kSeg / 2];
#pragma unroll
  for (int q = 0; q < kSeg / 2; q++) {
    // fp16 +-1 and -+1040 (0x3c00, 0xe410) with the pair's signs
    const uint32_t sb = ((negmask >> (2 * q)) & 1u) << 15 | ((negmask >> (2 * q + 1)) & 1u) << 31;
    const uint32_t mu = 0x3c003c00u ^ sb, ad = 0xe410e410u ^ sb;
    sg[q].mul = *reinterpret_cast<const __half2 *>(&mu);
    sg[q].add = *reinterpret_cast<const __half2 *>(&ad);
  }
#pragma unroll
  for (int g = 0; g < (S + 2) / 3; g++) {  // groups of three digits, lowest first
    uint32_t word[kSeg / 2];
#pragma unroll
    for (int q = 0; q < kSeg / 2; q++) {
      const uint32_t a = g < 2 ? lo[2 * q] : hi[S > 6 ? 2 * q : 0];
      const uint32_t b = g < 2 ? lo[2 * q + 1] : hi[S > 6 ? 2 * q + 1 : 0];
      word[q] = (g & 1) ? __byte_perm(a >> 15, b >> 15, 0x5410) : __byte_perm(a, b, 0x5410);
    }
#pragma unroll
    for (int pos = 0; pos < 3; pos++) {
      const int t = S - 1 - (3 * g + pos);  // slice
      if (t < 0) break;
      const uint32_t mask = t == 0 ? 0x003f003fu : 0x001f001fu;
      uint32_t w[4];
#pragma unroll
      for (int q = 0; q < 4; q++)
        w[q] = digit_pair(word[2 * q], pos, mask, sg[2 * q]) |
               digit_pair(word[2 * q + 1], pos, mask, sg[2 * q + 1]) << 16;
      put(t, make_uint4(w[0], w[1], w[2], w[3]));
    }
  }
  if (GATE) put(S, make_uint4(gate[0], gate[1], gate[2], gate[3]));
}

// Maxima: items [0, ceil(n/8)) take 8 rows of A (a warp per row); the next ones
// strips of 128 columns x 64 rows of B, merged into colmax with atomicMax on
// the bit patterns (which order like the magnitudes); the rest write 256
// entries each of the level launch's unit -> problem map (unit u belongs to
// problem u / tiles).  Bound by reading A and B once: 32-byte loads where the
// rows allow them, eight in flight (268 MB at 4096^3 in 72 us).
__global__ void __launch_bounds__(256)
ozaki_max_kernel(const double *__restrict__ A, const double *__restrict__ B, int64_t n, int64_t m,
                 int64_t p, uint64_t *__restrict__ rowmax, unsigned long long *__restrict__ colmax,
                 int64_t max_items, int *__restrict__ map, int64_t units, int64_t tiles) {
  pdl_wait();
  const int64_t items_a = (n + kRowsPerItem - 1) / kRowsPerItem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if ((int64_t)blockIdx.x >= max_items) {
    const int64_t u = ((int64_t)blockIdx.x - max_items) * 256 + threadIdx.x;
    if (u < units) map[u] = (int)(u / tiles);
    return;
  }
  if ((int64_t)blockIdx.x < items_a) {
    const int64_t i = (int64_t)blockIdx.x * kRowsPerItem + warp;
    if (i >= n) return;
    const double *row = A + i * m;
    uint64_t mx = 0;
    if (aligned32(A) && (m & 3) == 0) {
#pragma unroll 8
      for (int64_t k = 4 * lane; k < m; k += 128) {
        double v[4];
        load4(row + k, v);
        mx = max64(mx, max64(max64(abs_bits64(v[0]), abs_bits64(v[1])), max64(abs_bits64(v[2]), abs_bits64(v[3]))));
      }
    } else {
#pragma unroll 8
      for (int64_t k = lane; k < m; k += 32) mx = max64(mx, abs_bits64(row[k]));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max64(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) rowmax[i] = mx;
    return;
  }
  __shared__ uint64_t part[8][kColStrip];
  const int64_t b = (int64_t)blockIdx.x - items_a;
  const int64_t strips = (p + kColStrip - 1) / kColStrip;
  const int64_t c0 = (b % strips) * kColStrip, r0 = (b / strips) * kRowChunk;
  uint64_t mx[4] = {0, 0, 0, 0};
  // four columns a lane: neighbouring ones where a 32-byte load takes them,
  // else 32 apart
  const bool vec = aligned32(B) && (p & 3) == 0;
  if (vec) {
    const int64_t col = c0 + 4 * lane;
#pragma unroll
    for (int r = 0; r < kRowChunk / 8; r++) {
      const int64_t k = r0 + warp + 8 * r;
      if (k < m && col < p) {
        double v[4];
        load4(B + k * p + col, v);
#pragma unroll
        for (int e = 0; e < 4; e++) mx[e] = max64(mx[e], abs_bits64(v[e]));
      }
    }
  } else {
#pragma unroll 2
    for (int r = 0; r < kRowChunk / 8; r++) {
      const int64_t k = r0 + warp + 8 * r;
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const int64_t col = c0 + lane + 32 * e;
        if (k < m && col < p) mx[e] = max64(mx[e], abs_bits64(B[k * p + col]));
      }
    }
  }
#pragma unroll
  for (int e = 0; e < 4; e++) part[warp][vec ? 4 * lane + e : lane + 32 * e] = mx[e];
  __syncthreads();
  if (threadIdx.x < kColStrip) {
    uint64_t v = 0;
#pragma unroll
    for (int w = 0; w < 8; w++) v = max64(v, part[w][threadIdx.x]);
    if (c0 + threadIdx.x < p) atomicMax(&colmax[c0 + threadIdx.x], (unsigned long long)v);
  }
}

// Digits of one K chunk [k0, k0 + mc): blocks [0, blocks_a) take 32 rows of A by
// one K block of 128, the others 32 columns of B; a thread writes 16
// consecutive k of its row (column), eight threads a 128-byte pack row of each
// slice.  B's 128 x 32 doubles are turned in shared memory: entry (kk, c) at
// column (c + 4 (kk / 16)) mod 32 of row kk, so that the eight threads of a
// column, 16 rows apart, meet two on a bank.  SS = S slices per tile, or S + 1
// with the accuracy gate's slice after them.
//
// Bound by instruction issue until the digits went in fp16 pairs (digit_pair;
// through FP32 they cost 321 us at 4096^3 for 0.77 GB, now 197); blocks of a
// quarter of a tile, since one of 256 columns by 128 k kept a small product's
// few blocks busy for 100 us (192 served requests, 43 of them emulated: 12.0 ->
// 8.9 ms).
template <int S, bool GATE>
__global__ void __launch_bounds__(256)
ozaki_digits_kernel(const double *__restrict__ A, const double *__restrict__ B, int64_t n, int64_t m,
                    int64_t p, int64_t k0, int64_t mc, int kt, int bn, unsigned blocks_a,
                    const uint64_t *__restrict__ rowmax, const unsigned long long *__restrict__ colmax,
                    uint4 *__restrict__ pack, int64_t a0, int64_t b0) {
  constexpr int SS = S + (GATE ? 1 : 0);
  __shared__ double tile[128 * 32];
  pdl_wait();
  const int tid = threadIdx.x, r = tid / 8, sg = tid % 8;
  if (blockIdx.x < blocks_a) {
    const int64_t o = blockIdx.x / kt, kb = blockIdx.x % kt;  // group of 32 rows, K block
    const int64_t i = o * kDigRows + r;
    bool finite = true;
    const int sigma = i < n ? slice_exponent(rowmax[i], finite) : 0;
    const int64_t kk = kb * 128 + sg * kSeg;  // within the chunk
    const int live = i < n ? (int)max((int64_t)0, min((int64_t)kSeg, mc - kk)) : 0;
    const double *src = A + i * m + k0 + kk;
    double v[kSeg];
    if (live == kSeg && aligned32(A) && (m & 3) == 0) {
#pragma unroll
      for (int e = 0; e < kSeg; e += 4) load4(src + e, *reinterpret_cast<double(*)[4]>(&v[e]));
    } else {
#pragma unroll
      for (int e = 0; e < kSeg; e++) v[e] = e < live ? src[e] : 0.0;
    }
    const int64_t mt = o / (kTcBM / kDigRows), rr = (o % (kTcBM / kDigRows)) * kDigRows + r;
    emit_digits<S, GATE>(live, finite, sigma, [&](int e) { return v[e]; }, [&](int t, uint4 w) {
      const int64_t row = a0 + ((mt * SS + t) * kt + kb) * kTcBM + rr;
      pack[row * (kPackRowBytes / 16) + sg] = w;
    });
    return;
  }
  const unsigned b = blockIdx.x - blocks_a;
  const int64_t o = b / kt, kb = b % kt;  // group of 32 columns, K block
  const int64_t c0 = o * kDigRows;
  double x[16];
#pragma unroll
  for (int q = 0; q < 16; q++) {
    const int kk = tid / 32 + 8 * q, c = tid % 32;
    const int64_t k = kb * 128 + kk, j = c0 + c;
    x[q] = (k < mc && j < p) ? B[(k0 + k) * p + j] : 0.0;
  }
#pragma unroll
  for (int q = 0; q < 16; q++) {
    const int kk = tid / 32 + 8 * q, c = tid % 32;
    tile[kk * 32 + ((c + 4 * (kk / 16)) & 31)] = x[q];
  }
  __syncthreads();
  const int64_t j = c0 + r;
  bool finite = true;
  const int tau = j < p ? slice_exponent(colmax[j], finite) : 0;
  const double *col = tile + sg * kSeg * 32 + ((r + 4 * sg) & 31);
  const int64_t nt = c0 / bn, rr = c0 % bn + r;
  emit_digits<S, GATE>(j < p ? kSeg : 0, finite, tau, [&](int e) { return col[e * 32]; }, [&](int u, uint4 w) {
    // slices in descending order, then the gate's
    const int64_t row = b0 + ((nt * SS + (u == S ? S : S - 1 - u)) * kt + kb) * bn + rr;
    pack[row * (kPackRowBytes / 16) + sg] = w;
  });
}

// The double nearest to hi:lo (ties to even), times 2^k.
__device__ __forceinline__ double int128_scaled(uint64_t lo, int64_t hi, int k) {
  const bool neg = hi < 0;
  uint64_t mlo = lo, mhi = (uint64_t)hi;
  if (neg) {  // magnitude
    mlo = ~lo + 1;
    mhi = ~(uint64_t)hi + (mlo == 0 ? 1 : 0);
  }
  double d;
  if (mhi == 0) {
    d = __ull2double_rn(mlo);
  } else {
    // keep the top 64 bits, with the bits shifted out as a sticky bit far
    // below the 53-bit rounding position, then round once
    const int sh = 64 - __clzll((long long)mhi);  // 1..64
    const uint64_t top = sh == 64 ? mhi : ((mhi << (64 - sh)) | (mlo >> sh));
    const uint64_t lost = sh == 64 ? mlo : (mlo << (64 - sh));
    d = __ull2double_rn(top | (lost != 0 ? 1ull : 0ull));
    k += sh;
  }
  d = neg ? -d : d;
  // times 2^k: one multiplication by the power of two when it is a normal
  // double (correctly rounded, as scalbn), scalbn otherwise
  if (k >= -1022 && k <= 1023) return d * __longlong_as_double((long long)(k + 1023) << 52);
  return scalbn(d, k);
}

// The digit kernel of one K chunk, instantiated per S and gate (the slice loops
// unroll with constant shifts).
cudaError_t launch_ozaki_digits(int S, bool gate, int64_t blocks_a, int64_t blocks_b, cudaStream_t s,
                                const double *A, const double *B, int64_t n, int64_t m,
                                int64_t p, int64_t k0, int64_t mc, int kt, int bn,
                                const uint64_t *rowmax, const unsigned long long *colmax,
                                uint4 *pack, int64_t a0, int64_t b0) {
  if (blocks_a + blocks_b > 0x7fffffffLL) return cudaErrorInvalidValue;
  auto launch = [&](auto kernel) {
    return launch_pdl_if(blocks_a + blocks_b <= sm_count() * 4, kernel, (unsigned)(blocks_a + blocks_b), 256, 0,
                         s, A, B, n, m, p, k0, mc, kt, bn, (unsigned)blocks_a, rowmax, colmax, pack, a0, b0);
  };
  switch (S) {
#define MM_OZ_DIG(V) \
  case V: return gate ? launch(ozaki_digits_kernel<V, true>) : launch(ozaki_digits_kernel<V, false>);
    MM_OZ_DIG(2) MM_OZ_DIG(3) MM_OZ_DIG(4) MM_OZ_DIG(5) MM_OZ_DIG(6) MM_OZ_DIG(7) MM_OZ_DIG(8)
    MM_OZ_DIG(9) MM_OZ_DIG(10) MM_OZ_DIG(11) MM_OZ_DIG(12)
#undef MM_OZ_DIG
    default: return cudaErrorInvalidValue;
  }
}

// The double nearest to M 2^k (M > 0 a 128-bit integer; ties to even) in
// integer arithmetic: the top 53 bits of M, rounded on the bits below them,
// and the exponent placed directly.  Returns false where the result is not a
// normal double (the caller then takes int128_scaled).
__device__ __forceinline__ bool round_to_double(unsigned __int128 M, int k, uint64_t &bits) {
  const uint64_t mh = (uint64_t)(M >> 64), ml = (uint64_t)M;
  const int L = mh ? 128 - __clzll((long long)mh) : 64 - __clzll((long long)ml);  // bit length
  int e = L - 1 + k;
  uint64_t top;
  if (L <= 53) {
    top = ml << (53 - L);  // exact
  } else {
    const int sh = L - 53;  // 1..75
    top = (uint64_t)(M >> sh);
    const unsigned __int128 rem = M - ((unsigned __int128)top << sh);
    const unsigned __int128 half = (unsigned __int128)1 << (sh - 1);
    if (rem > half || (rem == half && (top & 1u))) {
      if (++top == (1ull << 53)) {
        top >>= 1;
        e++;
      }
    }
  }
  if (e < -1022 || e > 1023) return false;
  bits = ((uint64_t)(e + 1023) << 52) | (top & ((1ull << 52) - 1));
  return true;
}

// c_ij = 2^(sigma_i + tau_j - 5(S+1)) sum_c sum_L D[c][L][i][j] 32^(S-1-L):
// the level sums are integers below 2^24, so their weighted sum is formed
// exactly in 128-bit integers and rounded once to FP64 (then scaled by a
// power of two, which rounds again only in the subnormal range); NaN where
// row i of A or column j of B is not finite.  A thread takes column j of the
// rows blockIdx.y, blockIdx.y + gridDim.y, ...; the S level values of a chunk
// are loaded together, for V neighbouring columns at once (V = 2 halves the
// loads where p is even; 211 -> 185 us at 4096^3).  One instantiation per S, so the level
// loop unrolls without predicates.  The epilogue epi is applied to each entry; skip_if
// (the accuracy gate's flag, when given) set: the FP64 FMA product writes C
// instead and this kernel writes nothing.
template <int S, int V>
__global__ void __launch_bounds__(256, V == 2 ? 3 : 4)
ozaki_sum_kernel(const float *__restrict__ D, int64_t plane, int64_t n, int64_t p, int chunks,
                 const uint64_t *__restrict__ rowmax, const unsigned long long *__restrict__ colmax,
                 double *C, const int *skip_if, EpiT<double> epi) {
  if (skip_if != nullptr && *reinterpret_cast<const volatile int *>(skip_if) != 0) return;
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * V;
  if (j >= p) return;
  bool fb[V];
  int tau[V];
#pragma unroll
  for (int q = 0; q < V; q++) tau[q] = slice_exponent(colmax[j + q], fb[q]);
  // Horner by 32 over levels 0..h-1 into X and h..S-1 into Y (int64: each
  // part at most (2^24 - 1)(32^6 - 1)/31 < 2^49.1 per chunk, below 2^63 over
  // at most kOzakiMaxChunks = 2^10 chunks), then v = X 32^(S-h) + Y once in
  // 128 bits
  constexpr int h = (S + 1) / 2;
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
    bool fa;
    const int sigma = slice_exponent(rowmax[i], fa);
    const int64_t x = i * p + j;
    int64_t X[V] = {}, Y[V] = {};
    for (int c = 0; c < chunks; c++) {
      const float *d = D + (int64_t)c * S * plane + x;
      float v[S][V];
#pragma unroll
      for (int L = 0; L < S; L++) {
        if constexpr (V == 2) {
          const float2 t = __ldcs(reinterpret_cast<const float2 *>(d + (int64_t)L * plane));
          v[L][0] = t.x;
          v[L][1] = t.y;
        } else {
          v[L][0] = __ldcs(d + (int64_t)L * plane);
        }
      }
#pragma unroll
      for (int q = 0; q < V; q++) {
        int64_t xc = 0, yc = 0;
#pragma unroll
        for (int L = 0; L < S; L++) {
          const int64_t g = __float2int_rn(v[L][q]);
          if (L < h) xc = xc * 32 + g;
          else yc = yc * 32 + g;
        }
        X[q] += xc;
        Y[q] += yc;
      }
    }
    constexpr int sh = 5 * (S - h);  // 5..30
#pragma unroll
    for (int q = 0; q < V; q++) {
      uint64_t lo = (uint64_t)X[q] << sh;
      int64_t hi = X[q] >> (64 - sh);
      const uint64_t r = lo + (uint64_t)Y[q];
      hi += (Y[q] < 0 ? -1 : 0) + (r < lo ? 1 : 0);
      lo = r;
      const int k = sigma + tau[q] - 5 * (S + 1);
      double out;
      if (!(fa && fb[q])) {
        out = __longlong_as_double(0x7ff8000000000000ll);
      } else {
        const bool neg = hi < 0;
        unsigned __int128 M = ((unsigned __int128)(uint64_t)hi << 64) | lo;
        if (neg) M = ~M + 1;
        uint64_t bits;
        if (M == 0) out = 0.0;
        else if (round_to_double(M, k, bits)) out = __longlong_as_double((long long)(bits | ((uint64_t)neg << 63)));
        else out = int128_scaled(lo, hi, k);
      }
      C[x + q] = epi_apply(epi, out, x + q);
    }
  }
}

// One wave of blocks (three or four a SM, the launch bounds); pairs of columns
// where p is even and wide enough to fill the blocks.
cudaError_t launch_ozaki_sum(int S, cudaStream_t s, const float *D, int64_t plane, int64_t n, int64_t p,
                             int chunks, const uint64_t *rowmax, const unsigned long long *colmax,
                             double *C, const int *skip_if, const EpiT<double> &epi) {
  const int v = (p & 1) == 0 && p >= 512 ? 2 : 1;
  const int64_t gx = ceil_div(p, 256 * v);
  const int64_t gy = std::max<int64_t>(
      1, std::min<int64_t>({n, 65535, ceil_div((int64_t)sm_count() * (v == 2 ? 3 : 4), gx)}));
  if (gx > 0x7fffffffLL) return cudaErrorInvalidValue;
  auto launch = [&](auto kernel) {
    kernel<<<dim3((unsigned)gx, (unsigned)gy), 256, 0, s>>>(D, plane, n, p, chunks, rowmax, colmax, C,
                                                            skip_if, epi);
    return cudaGetLastError();
  };
  switch (S) {
#define MM_OZ_SUM(W) \
  case W: return v == 2 ? launch(ozaki_sum_kernel<W, 2>) : launch(ozaki_sum_kernel<W, 1>);
    MM_OZ_SUM(2) MM_OZ_SUM(3) MM_OZ_SUM(4) MM_OZ_SUM(5) MM_OZ_SUM(6) MM_OZ_SUM(7) MM_OZ_SUM(8)
    MM_OZ_SUM(9) MM_OZ_SUM(10) MM_OZ_SUM(11) MM_OZ_SUM(12)
#undef MM_OZ_SUM
    default: return cudaErrorInvalidValue;
  }
}

// Accuracy gate.  Every term a_ir b_rj of the emulated product is off by at
// most (S + 2) 2^(sigma_i + tau_j - 5S - 1), so entry (i, j) is off by at most
// m (S + 2) 2^(sigma_i + tau_j - 5S - 1); the product meets e_ij <= 1e-14 sqrt(m)
// wherever P_ij = sum_r |a_ir| 2^-sigma_i |b_rj| 2^-tau_j is at least
// sqrt(m) (S + 2) 2^(-5S-1) 1e14.  A lower bound of 256 P comes from the
// emulation's own machinery: one more slice per operand holds gate_value
// (16 |x| 2^-sigma truncated toward zero onto the e4m3 grid), and one more
// tensor-core product per K chunk multiplies the two (products exact in
// FP32; the FP32 accumulation of nonnegative terms is off by at most m 2^-23
// relative, which the host's threshold absorbs: it divides by 0.98 - m 2^-23,
// the 2% also covering the final rounding to a double, 2^-53 relative, below
// 1.2% of 1e-14; where m 2^-23 reaches 1/2 the threshold is infinite and
// every product falls back).  Truncation only lowers the bound, so entries
// whose magnitudes fall below the e4m3 grid cause a fallback, never a miss.
// The check kernel adds the chunks' planes in FP32 (at most 1024 nonnegative
// terms), lowers the sum by 2^-10 (more than that addition's rounding) and
// sets a flag where any entry with a finite, non-zero row and column misses
// the threshold; the FP64 FMA product then recomputes C.
// A block takes 1024 columns of the rows blockIdx.y, + gridDim.y, ...; a thread
// columns 256 apart, whose maxima it reads once.
// (43 -> 20 us at 4096^3 against a row per block and a column per thread and turn.)
constexpr int kGateCols = 4;
__global__ void __launch_bounds__(256)
ozaki_gate_check_kernel(const float *__restrict__ G, int64_t plane, int chunks, int64_t n,
                        int64_t p, const uint64_t *__restrict__ rowmax,
                        const unsigned long long *__restrict__ colmax, float thr256, int *flag) {
  const int64_t j0 = (int64_t)blockIdx.x * (256 * kGateCols) + threadIdx.x;
  bool live[kGateCols];
#pragma unroll
  for (int q = 0; q < kGateCols; q++) {
    const int64_t j = j0 + 256 * q;
    bool fj = false;
    if (j < p) slice_exponent(colmax[j], fj);
    live[q] = fj && colmax[j] != 0;
  }
  bool fail = false;
#pragma unroll 2
  for (int64_t i = blockIdx.y; i < n; i += gridDim.y) {
    bool fi;
    slice_exponent(rowmax[i], fi);
    // a row with a NaN or an infinity gives NaN by design; an all-zero row
    // gives exact zeros
    const bool row = fi && rowmax[i] != 0;
    const float *g = G + i * p + j0;
    float v[kGateCols];
#pragma unroll
    for (int q = 0; q < kGateCols; q++) v[q] = live[q] && row ? __ldcs(g + 256 * q) : INFINITY;
    for (int c = 1; c < chunks; c++)
#pragma unroll
      for (int q = 0; q < kGateCols; q++)
        if (live[q] && row) v[q] += __ldcs(g + (int64_t)c * plane + 256 * q);
#pragma unroll
    for (int q = 0; q < kGateCols; q++) fail |= !(v[q] * (1.0f - 0x1p-10f) >= thr256);
  }
  if (__syncthreads_or(fail) && threadIdx.x == 0) atomicOr(flag, 1);
}

// Scratch offsets of one call.
struct OzLayout {
  int S, SS, chunks, bn, mt, nt;
  int64_t mc;
  std::vector<int64_t> k0, kc, kt, a0, b0;
  int64_t rows = 0, plane = 0;
  size_t max_off, zero_off, flag_off, zero_end, d_off, tab_off, map_off, simt_off, need;
  int64_t units = 0;
};

}  // namespace

int64_t ozaki_chunk(int S) {
  const int64_t mc = ((int64_t)((1 << 24) - 1) / (256 * (int64_t)S)) / 128 * 128;
  return mc;
}

mm_status run_ozaki(Scratch &ws, int64_t n, int64_t m, int64_t p, const double *A,
                    const double *B, double *C, int S, bool gate, cudaStream_t s, const Epi *epi) {
  if (S < kOzakiMinSlices || S > kOzakiMaxSlices) return MM_EINVAL;
  if (n == 0 || p == 0) return MM_OK;
  if (m == 0) return note_cuda(cudaMemsetAsync(C, 0, (size_t)(n * p) * sizeof(double), s));
  OzLayout lay;
  lay.S = S;
  lay.SS = S + (gate ? 1 : 0);  // slices per tile in the packs (the gate's last)
  lay.mc = ozaki_chunk(S);
  if (ceil_div(m, lay.mc) > kOzakiMaxChunks) return MM_EINVAL;
  lay.chunks = (int)ceil_div(m, lay.mc);
  TcChoice ch = tune_choose(n, std::min(m, lay.mc), p);
  lay.bn = tc_bn(kTcE4m3, ch.bn);
  lay.mt = (int)ceil_div(n, kTcBM);
  lay.nt = (int)ceil_div(p, lay.bn);
  for (int c = 0; c < lay.chunks; c++) {
    const int64_t k0 = (int64_t)c * lay.mc, kc = std::min(lay.mc, m - k0);
    const int64_t kt = ceil_div(kc, 128);
    lay.k0.push_back(k0);
    lay.kc.push_back(kc);
    lay.kt.push_back(kt);
    lay.a0.push_back(lay.rows);
    lay.rows += (int64_t)lay.mt * lay.SS * kt * kTcBM;
    lay.b0.push_back(lay.rows);
    lay.rows += (int64_t)lay.nt * lay.SS * kt * lay.bn;
  }
  if (lay.rows > 0x7fffffffLL) return MM_EINVAL;
  // S level problems per chunk, then the gate's product per chunk
  const int nprobs = lay.chunks * lay.SS;
  const int64_t tiles = (int64_t)lay.mt * lay.nt;
  // level planes of D, padded so that the planes of one entry do not sit a
  // power of two apart (128-byte aligned)
  lay.plane = (n * p + 31) / 32 * 32 + 32;
  std::vector<SplitProb> tab((size_t)nprobs);
  // level problems, longest K first (the persistent grid takes units in
  // order, so the short ones fill the last wave); problem g = (S-1-L) *
  // chunks + c holds units [g T, (g+1) T) of the T tiles.  (Interleaving the
  // levels tile by tile was measured slower: 19 GB of DRAM reads per 4096^3
  // launch instead of 11, 5.4 ms instead of 4.6.)
  int g = 0;
  for (int L = S - 1; L >= 0; L--)
    for (int c = 0; c < lay.chunks; c++, g++) {
      SplitProb &sp = tab[(size_t)g];
      std::memset(&sp, 0, sizeof(sp));
      const int64_t kt = lay.kt[(size_t)c];
      sp.n = (int32_t)n;
      sp.p = (int32_t)p;
      sp.kt = (int32_t)((L + 1) * kt);
      sp.m = sp.kt * 128;  // padded K of the level: zero digits past the chunk
      sp.mt = lay.mt;
      sp.nt = lay.nt;
      sp.bn = lay.bn;
      sp.group_m = ch.group_m;
      sp.a_row0 = lay.a0[(size_t)c];
      sp.b_row0 = lay.b0[(size_t)c] + (int64_t)(S - 1 - L) * kt * lay.bn;
      sp.a_kstride = (int32_t)(lay.SS * kt);
      sp.b_kstride = (int32_t)(lay.SS * kt);
      sp.unit_start = (int32_t)lay.units;
      lay.units += tiles;
      sp.split_from = (int32_t)tiles;
      sp.split_s = 1;
      sp.C = reinterpret_cast<float *>((uintptr_t)(((int64_t)c * S + L) * lay.plane));  // offset
    }
  // the gate's products (one slice against one slice: as short as level 0,
  // so they run last), planes after the level planes
  for (int c = 0; gate && c < lay.chunks; c++, g++) {
    SplitProb &sp = tab[(size_t)g];
    std::memset(&sp, 0, sizeof(sp));
    const int64_t kt = lay.kt[(size_t)c];
    sp.n = (int32_t)n;
    sp.p = (int32_t)p;
    sp.kt = (int32_t)kt;
    sp.m = sp.kt * 128;
    sp.mt = lay.mt;
    sp.nt = lay.nt;
    sp.bn = lay.bn;
    sp.group_m = ch.group_m;
    sp.a_row0 = lay.a0[(size_t)c] + (int64_t)S * kt * kTcBM;
    sp.b_row0 = lay.b0[(size_t)c] + (int64_t)S * kt * lay.bn;
    sp.a_kstride = (int32_t)(lay.SS * kt);
    sp.b_kstride = (int32_t)(lay.SS * kt);
    sp.unit_start = (int32_t)lay.units;
    lay.units += tiles;
    sp.split_from = (int32_t)tiles;
    sp.split_s = 1;
    sp.C = reinterpret_cast<float *>((uintptr_t)(((int64_t)lay.chunks * S + c) * lay.plane));
  }
  if (lay.units > 0x7fffffffLL) return MM_EINVAL;
  const size_t pack_bytes = (size_t)lay.rows * kPackRowBytes;
  lay.max_off = (pack_bytes + 255) & ~(size_t)255;  // row maxima (n) + column maxima (p)
  lay.zero_off = lay.max_off;
  // + zero scale words, the gate's fallback flag
  lay.flag_off = lay.max_off + (size_t)(n + p) * 8 + (size_t)(n + p) * 4;
  lay.zero_end = lay.flag_off + sizeof(int);
  lay.d_off = (lay.zero_end + 255) & ~(size_t)255;
  lay.tab_off = (lay.d_off + (size_t)nprobs * lay.plane * sizeof(float) + 255) & ~(size_t)255;
  // the table, then the work units of each CTA (the levels differ in length)
  TcConfig cfg{128, 4, ch.grid};
  cfg.max_bn = lay.bn;
  std::vector<int> order;
  tc_unit_order(tab.data(), nprobs, tc_launch_grid(cfg, lay.units), order);
  const size_t tab_bytes = ((size_t)nprobs * sizeof(SplitProb) + 15) & ~(size_t)15;
  lay.map_off = (lay.tab_off + tab_bytes + order.size() * sizeof(int) + 255) & ~(size_t)255;
  // the fallback's K-slice partials (under-filled products)
  lay.simt_off = (lay.map_off + (size_t)lay.units * sizeof(int) + 255) & ~(size_t)255;
  lay.need = lay.simt_off + simt_scratch_bytes(true, n, m, p);
  cudaError_t e = ws.reserve(lay.need, s);
  if (e != cudaSuccess) return note_cuda(e);
  uint8_t *base = static_cast<uint8_t *>(ws.ptr);
  uint64_t *rowmax = reinterpret_cast<uint64_t *>(base + lay.max_off);
  unsigned long long *colmax = reinterpret_cast<unsigned long long *>(rowmax + n);
  uint32_t *zero_words = reinterpret_cast<uint32_t *>(colmax + p);
  float *D = reinterpret_cast<float *>(base + lay.d_off);
  for (auto &sp : tab) {
    sp.C = D + (uintptr_t)sp.C;
    sp.sA = zero_words;      // scale exponent 0: the digits are not rescaled
    sp.tB = zero_words + n;
  }
  SplitProb *d_tab = reinterpret_cast<SplitProb *>(base + lay.tab_off);
  const int *d_order = reinterpret_cast<const int *>(base + lay.tab_off + tab_bytes);
  {
    std::vector<uint8_t> blob(tab_bytes + order.size() * sizeof(int), 0);
    std::memcpy(blob.data(), tab.data(), tab.size() * sizeof(SplitProb));
    std::memcpy(blob.data() + tab_bytes, order.data(), order.size() * sizeof(int));
    e = ws.stage.copy_to_device(d_tab, blob.data(), blob.size(), s);
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(base + lay.zero_off, 0, lay.zero_end - lay.zero_off, s);
  if (e != cudaSuccess) return note_cuda(e);
  int *unit_map = reinterpret_cast<int *>(base + lay.map_off);
  {
    TraceScope ts("ozaki_max", s);
    const int64_t items = ceil_div(n, kRowsPerItem) + ceil_div(p, kColStrip) * ceil_div(m, kRowChunk);
    const int64_t blocks = items + ceil_div(lay.units, 256);
    if (blocks > 0x7fffffffLL) return MM_EINVAL;
    e = launch_pdl_if(blocks <= sm_count() * 4, ozaki_max_kernel, (unsigned)blocks, 256, 0, s, A, B, n, m, p,
                      rowmax, colmax, items, unit_map, lay.units, tiles);
    if (e != cudaSuccess) return note_cuda(e);
  }
  {
    TraceScope ts("ozaki_digits", s);
    uint4 *pk = static_cast<uint4 *>(ws.ptr);
    for (int c = 0; c < lay.chunks; c++) {
      const int kt = (int)lay.kt[(size_t)c];
      e = launch_ozaki_digits(S, gate, (int64_t)lay.mt * (kTcBM / kDigRows) * kt,
                              (int64_t)lay.nt * (lay.bn / kDigRows) * kt, s, A, B, n, m, p,
                              lay.k0[(size_t)c], lay.kc[(size_t)c], kt, lay.bn, rowmax, colmax, pk,
                              lay.a0[(size_t)c], lay.b0[(size_t)c]);
      if (e != cudaSuccess) return note_cuda(e);
    }
  }
  e = launch_tc(kTcE4m3, device_table(d_tab, nprobs), (int)lay.units, unit_map, nullptr, ws.ptr, lay.rows, cfg,
                g_ctx.d_err, s, d_order);
  if (e != cudaSuccess) return note_cuda(e);
  // the gate reads the level sums only, so it runs before the sum kernel:
  // where it fails, the sum writes nothing and the FP64 FMA product below
  // reads the epilogue's D (which may be C) untouched
  int *flag = gate ? reinterpret_cast<int *>(base + lay.flag_off) : nullptr;
  if (gate) {
    TraceScope ts("ozaki_gate", s);
    const double room = 0.98 - (double)m * 0x1p-23;
    const double thr256 = room < 0.5 ? (double)INFINITY
                                     : 256.0 * std::sqrt((double)m) * (S + 2) *
                                           std::ldexp(1.0, -5 * S - 1) * 1e14 / room;
    float thr = (float)thr256;  // rounded up to a float
    if ((double)thr < thr256) thr = std::nextafter(thr, (float)INFINITY);
    const int64_t gx = ceil_div(p, 256 * kGateCols);
    const int64_t gy = std::max<int64_t>(1, std::min<int64_t>({n, 65535, ceil_div((int64_t)sm_count() * 8, gx)}));
    if (gx > 0x7fffffffLL) return MM_EINVAL;
    // (not as a dependent: its blocks would wait beside the level products for
    // all of their time)
    ozaki_gate_check_kernel<<<dim3((unsigned)gx, (unsigned)gy), 256, 0, s>>>(
        D + (int64_t)lay.chunks * S * lay.plane, lay.plane, lay.chunks, n, p, rowmax, colmax, thr, flag);
    if ((e = cudaGetLastError()) != cudaSuccess) return note_cuda(e);
  }
  {
    TraceScope ts("ozaki_sum", s);
    e = launch_ozaki_sum(S, s, D, lay.plane, n, p, lay.chunks, rowmax, colmax, C, flag, epi_of<double>(epi));
    if (e != cudaSuccess) return note_cuda(e);
  }
  if (!gate) return MM_OK;
  // the FP64 FMA product replaces C where the flag is set: the same kernels
  // and K slices as MM_MODE_DGEMM, so the bits are that mode's
  const SimtPlan pl = simt_plan(true, n, m, p);
  if (pl.S >= 1)
    return note_cuda(launch_simt_splitk_f64(
        n, m, p, A, B, C, pl.S > 1 ? reinterpret_cast<double *>(base + lay.simt_off) : nullptr, pl, s,
        flag, epi));
  return note_cuda(launch_simt_f64(n, m, p, A, B, C, s, flag, epi));
}

size_t ozaki_scratch_bytes(int64_t n, int64_t m, int64_t p, int S) {
  if (n <= 0 || p <= 0 || m <= 0) return 0;
  const int64_t mc = ozaki_chunk(S);
  const int64_t chunks = ceil_div(m, mc);
  const int64_t kt_all = ceil_div(m, 128) + chunks;  // K blocks over all chunks (bound)
  // S digit slices per operand and the accuracy gate's slice (counted whether
  // or not the gate is on), their level sums and the gate's planes, maxima,
  // table, the CTAs' unit lists and the unit map
  const int64_t SS = S + 1;
  const int64_t rows = (ceil_div(n, kTcBM) * kTcBM + ceil_div(p, 128) * 256) * SS * kt_all;
  return (size_t)rows * kPackRowBytes + (size_t)chunks * SS * (n * p + 64) * sizeof(float) +
         (size_t)(n + p) * 12 + (size_t)chunks * SS * ceil_div(n, kTcBM) * ceil_div(p, 128) * 4 +
         (size_t)chunks * SS * sizeof(SplitProb) +
         (size_t)chunks * SS * ceil_div(n, kTcBM) * ceil_div(p, 128) * 4 + ((size_t)1 << 20) +
         simt_scratch_bytes(true, n, m, p);
}

}  // namespace mm

extern "C" mm_status mm_ozaki_plan(int64_t n, int64_t m, int64_t p, int slices,
                                   int64_t *chunk_columns, int *chunks, size_t *scratch_bytes) {
  using namespace mm;
  if (n < 0 || m < 0 || p < 0 || slices < kOzakiMinSlices || slices > kOzakiMaxSlices ||
      !chunk_columns || !chunks || !scratch_bytes)
    return MM_EINVAL;
  const int64_t mc = ozaki_chunk(slices);
  const int64_t q = ceil_div(m, mc);
  if (q > kOzakiMaxChunks) return MM_EINVAL;
  *chunk_columns = mc;
  *chunks = (int)q;
  *scratch_bytes = ozaki_scratch_bytes(n, m, p, slices);
  return MM_OK;
}

namespace mm {

}  // namespace mm
