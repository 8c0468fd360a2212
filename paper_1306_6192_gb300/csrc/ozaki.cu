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

// The kernels beside the level products take up to kOzItems products a launch, their
// arguments in the launch's parameters: item g has the blocks from it[g].start.
constexpr int kOzItems = 32;
template <typename Item>
struct OzItems {
  int count;
  Item it[kOzItems];
};
template <typename Item>
__device__ __forceinline__ const Item &item_of(const OzItems<Item> &t, int block) {
  int lo = 0, hi = t.count - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (t.it[mid].start <= block) lo = mid;
    else hi = mid - 1;
  }
  return t.it[lo];
}
// launch(items, blocks) over the items, kOzItems at a time; an item's start
// holds its block count until then.
template <typename Item, typename Launch>
cudaError_t launch_items(const std::vector<Item> &items, Launch launch) {
  for (size_t i = 0; i < items.size();) {
    OzItems<Item> t{};
    int64_t blocks = 0;
    for (; i < items.size() && t.count < kOzItems; i++) {
      const int64_t more = items[i].start;
      if (blocks + more > 0x7fffffffLL) break;
      Item &x = t.it[t.count++] = items[i];
      x.start = (int32_t)blocks;
      blocks += more;
    }
    const cudaError_t e = launch(t, (unsigned)blocks);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}
struct OzMaxItem {
  const double *A, *B;
  uint64_t *rowmax;  // n, then the column maxima
  int64_t n, m, p;
  int32_t start;
};
struct OzDigitItem {  // one K chunk [k0, k0 + mc)
  const double *A, *B;
  const uint64_t *rowmax;
  int64_t n, m, p, k0, mc, a0, b0;
  int32_t kt, bn, blocks_a, start;
};
struct OzSumItem {
  const float *D;
  const uint64_t *rowmax;
  double *C;
  const int *skip_if;
  EpiT<double> epi;
  int64_t plane, n, p;
  int32_t chunks, gx, gy, start;
};
struct OzGateItem {
  const float *G;
  const uint64_t *rowmax;
  int *flag;
  int64_t plane, n, p;
  float thr256;
  int32_t chunks, gx, gy, start;
};

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

// Maxima: blocks [0, ceil(n/8)) take 8 rows of A (a warp per row); the next ones
// strips of 128 columns x 64 rows of B, merged into colmax with atomicMax on
// the bit patterns (which order like the magnitudes).
// Bound by reading A and B once: 32-byte loads where the
// rows allow them, eight in flight (268 MB at 4096^3 in 72 us).
__global__ void __launch_bounds__(256)
ozaki_max_kernel(const __grid_constant__ OzItems<OzMaxItem> items) {
  pdl_wait();
  const OzMaxItem &it = item_of(items, blockIdx.x);
  const double *__restrict__ A = it.A, *__restrict__ B = it.B;
  uint64_t *rowmax = it.rowmax;
  const int64_t n = it.n, m = it.m, p = it.p, block = (int)blockIdx.x - it.start;
  unsigned long long *colmax = reinterpret_cast<unsigned long long *>(rowmax + n);
  const int64_t items_a = (n + kRowsPerItem - 1) / kRowsPerItem;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (block < items_a) {
    const int64_t i = block * kRowsPerItem + warp;
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
  const int64_t b = block - items_a;
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
// through FP32 they cost 321 us at 4096^3 for 0.77 GB, now 165); blocks of a
// quarter of a tile, since one of 256 columns by 128 k kept a small product's
// few blocks busy for 100 us (192 served requests, 43 of them emulated: 12.0 ->
// 8.9 ms).
template <int S, bool GATE>
__global__ void __launch_bounds__(256)
ozaki_digits_kernel(const __grid_constant__ OzItems<OzDigitItem> items, uint4 *__restrict__ pack) {
  constexpr int SS = S + (GATE ? 1 : 0);
  __shared__ double tile[128 * 32];
  pdl_wait();
  const OzDigitItem &it = item_of(items, blockIdx.x);
  const double *__restrict__ A = it.A, *__restrict__ B = it.B;
  const uint64_t *__restrict__ rowmax = it.rowmax;
  const int64_t n = it.n, m = it.m, p = it.p, k0 = it.k0, mc = it.mc, a0 = it.a0, b0 = it.b0;
  const int kt = it.kt, bn = it.bn, block = (int)blockIdx.x - it.start;
  const uint64_t *__restrict__ colmax = rowmax + n;
  const int tid = threadIdx.x, r = tid / 8, sg = tid % 8;
  if (block < it.blocks_a) {
    const int64_t o = block / kt, kb = block % kt;  // group of 32 rows, K block
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
  const int b = block - it.blocks_a;
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

// The digit kernel, instantiated per S and gate (the slice loops unroll with
// constant shifts).
cudaError_t launch_ozaki_digits(int S, bool gate, const std::vector<OzDigitItem> &items, uint4 *pack,
                                cudaStream_t s) {
  auto launch = [&](auto kernel) {
    return launch_items(items, [&](const OzItems<OzDigitItem> &t, unsigned blocks) {
      return launch_pdl_if(blocks <= sm_count() * 4u, kernel, blocks, 256, 0, s, t, pack);
    });
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
// row i of A or column j of B is not finite.  A thread takes column j of
// every gy-th row; the S level values of a chunk
// are loaded together, for V neighbouring columns at once (V = 2 halves the
// loads where p is even; 211 -> 185 us at 4096^3).  One instantiation per S, so the level
// loop unrolls without predicates.  The epilogue epi is applied to each entry; skip_if
// (the accuracy gate's flag, when given) set: the FP64 FMA product writes C
// instead and this kernel writes nothing.
template <int S, int V>
__global__ void __launch_bounds__(256, V == 2 ? 3 : 4)
ozaki_sum_kernel(const __grid_constant__ OzItems<OzSumItem> items) {
  const OzSumItem &it = item_of(items, blockIdx.x);
  if (it.skip_if != nullptr && *reinterpret_cast<const volatile int *>(it.skip_if) != 0) return;
  const float *__restrict__ D = it.D;
  double *C = it.C;
  const int64_t plane = it.plane, n = it.n, p = it.p;
  const int chunks = it.chunks, block = (int)blockIdx.x - it.start, by = block / it.gx;
  const uint64_t *__restrict__ rowmax = it.rowmax, *__restrict__ colmax = rowmax + n;
  const EpiT<double> epi = it.epi;
  const int64_t j = ((int64_t)(block % it.gx) * blockDim.x + threadIdx.x) * V;
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
  for (int64_t i = by; i < n; i += it.gy) {
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

// Pairs of columns where p is even and wide enough to fill the blocks.
int sum_columns(int64_t p) { return (p & 1) == 0 && p >= 512 ? 2 : 1; }

// The sum kernel over products of one S and one V = sum_columns.
cudaError_t launch_ozaki_sum(int S, int v, const std::vector<OzSumItem> &items, cudaStream_t s) {
  auto launch = [&](auto kernel) {
    return launch_items(items, [&](const OzItems<OzSumItem> &t, unsigned blocks) {
      kernel<<<blocks, 256, 0, s>>>(t);
      return cudaGetLastError();
    });
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

// Blocks of a product in a kernel whose blocks take gx column groups and, each,
// every gy-th row: a wave of `per_sm` a SM, or, among other products, at least
// eight rows a block.
template <typename Item>
bool row_blocks(Item &it, int64_t columns, int per_sm, bool alone) {
  const int64_t gx = ceil_div(it.p, columns);
  const int64_t rows = alone ? it.n : ceil_div(it.n, 8);
  const int64_t gy = std::max<int64_t>(1, std::min<int64_t>({rows, 65535, ceil_div((int64_t)sm_count() * per_sm, gx)}));
  if (gx * gy > 0x7fffffffLL) return false;
  it.gx = (int32_t)gx;
  it.gy = (int32_t)gy;
  it.start = (int32_t)(gx * gy);
  return true;
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
// A block takes 1024 columns of every gy-th row; a thread
// columns 256 apart, whose maxima it reads once.
// (43 -> 20 us at 4096^3 against a row per block and a column per thread and turn.)
constexpr int kGateCols = 4;
__global__ void __launch_bounds__(256)
ozaki_gate_check_kernel(const __grid_constant__ OzItems<OzGateItem> items) {
  const OzGateItem &it = item_of(items, blockIdx.x);
  const float *__restrict__ G = it.G;
  const int64_t plane = it.plane, n = it.n, p = it.p;
  const int chunks = it.chunks, block = (int)blockIdx.x - it.start, by = block / it.gx;
  const uint64_t *__restrict__ rowmax = it.rowmax, *__restrict__ colmax = rowmax + n;
  const float thr256 = it.thr256;
  const int64_t j0 = (int64_t)(block % it.gx) * (256 * kGateCols) + threadIdx.x;
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
  for (int64_t i = by; i < n; i += it.gy) {
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
  if (__syncthreads_or(fail) && threadIdx.x == 0) atomicOr(it.flag, 1);
}

// Scratch offsets of one product (pack rows and bytes from the scratch's start).
struct OzLayout {
  int S, SS, chunks, bn, mt, nt;
  int64_t mc, tiles;
  std::vector<int64_t> k0, kc, kt, a0, b0;
  int64_t plane = 0;
  size_t max_off, flag_off, d_off;
};

}  // namespace

int64_t ozaki_chunk(int S) {
  const int64_t mc = ((int64_t)((1 << 24) - 1) / (256 * (int64_t)S)) / 128 * 128;
  return mc;
}

// Lays one product out behind `rows` pack rows and appends its level and gate
// problems to the table (C: the plane's index; unit_start unset).
static mm_status ozaki_layout(const OzCall &q, int64_t &rows, OzLayout &lay, TcChoice &ch,
                              std::vector<SplitProb> &tab) {
  const int S = q.S;
  if (S < kOzakiMinSlices || S > kOzakiMaxSlices) return MM_EINVAL;
  lay.S = S;
  lay.SS = S + (q.gate ? 1 : 0);  // slices per tile in the packs (the gate's last)
  lay.mc = ozaki_chunk(S);
  if (ceil_div(q.m, lay.mc) > kOzakiMaxChunks) return MM_EINVAL;
  lay.chunks = (int)ceil_div(q.m, lay.mc);
  ch = tune_choose(q.n, std::min(q.m, lay.mc), q.p);
  lay.bn = tc_bn(kTcE4m3, ch.bn);
  lay.mt = (int)ceil_div(q.n, kTcBM);
  lay.nt = (int)ceil_div(q.p, lay.bn);
  for (int c = 0; c < lay.chunks; c++) {
    const int64_t k0 = (int64_t)c * lay.mc, kc = std::min(lay.mc, q.m - k0);
    const int64_t kt = ceil_div(kc, 128);
    lay.k0.push_back(k0);
    lay.kc.push_back(kc);
    lay.kt.push_back(kt);
    lay.a0.push_back(rows);
    rows += (int64_t)lay.mt * lay.SS * kt * kTcBM;
    lay.b0.push_back(rows);
    rows += (int64_t)lay.nt * lay.SS * kt * lay.bn;
  }
  if (rows > 0x7fffffffLL) return MM_EINVAL;
  lay.tiles = (int64_t)lay.mt * lay.nt;
  // level planes of D, padded so that the planes of one entry do not sit a
  // power of two apart (128-byte aligned)
  lay.plane = (q.n * q.p + 31) / 32 * 32 + 32;
  // level problems, longest K first (the persistent grid takes units in
  // order, so the short ones fill the last wave).  (Interleaving the
  // levels tile by tile was measured slower: 19 GB of DRAM reads per 4096^3
  // launch instead of 11, 5.4 ms instead of 4.6.)  The gate's products (one
  // slice against one slice: as short as level 0) come last, planes after the
  // level planes.
  auto add = [&](int c, int64_t levels, int64_t a_slice, int64_t b_slice, int64_t plane) {
    SplitProb sp;
    std::memset(&sp, 0, sizeof(sp));
    const int64_t kt = lay.kt[(size_t)c];
    sp.n = (int32_t)q.n;
    sp.p = (int32_t)q.p;
    sp.kt = (int32_t)(levels * kt);
    sp.m = sp.kt * 128;  // padded K of the level: zero digits past the chunk
    sp.mt = lay.mt;
    sp.nt = lay.nt;
    sp.bn = lay.bn;
    sp.group_m = ch.group_m;
    sp.a_row0 = lay.a0[(size_t)c] + a_slice * kt * kTcBM;
    sp.b_row0 = lay.b0[(size_t)c] + b_slice * kt * lay.bn;
    sp.a_kstride = (int32_t)(lay.SS * kt);
    sp.b_kstride = (int32_t)(lay.SS * kt);
    sp.split_from = (int32_t)lay.tiles;
    sp.split_s = 1;
    sp.C = reinterpret_cast<float *>((uintptr_t)(plane * lay.plane));  // offset
    tab.push_back(sp);
  };
  for (int L = S - 1; L >= 0; L--)
    for (int c = 0; c < lay.chunks; c++) add(c, L + 1, 0, S - 1 - L, (int64_t)c * S + L);
  for (int c = 0; q.gate && c < lay.chunks; c++) add(c, 1, S, S, (int64_t)lay.chunks * S + c);
  return MM_OK;
}

mm_status run_ozaki(Scratch &ws, int64_t n, int64_t m, int64_t p, const double *A,
                    const double *B, double *C, int S, bool gate, cudaStream_t s, const Epi *epi) {
  const OzCall q{n, m, p, A, B, C, S, gate, epi};
  return run_ozaki_many(ws, &q, 1, s);
}

mm_status run_ozaki_many(Scratch &ws, const OzCall *calls, int count, cudaStream_t s) {
  std::vector<OzCall> qs;
  for (int g = 0; g < count; g++) {
    const OzCall &q = calls[g];
    if (q.S < kOzakiMinSlices || q.S > kOzakiMaxSlices) return MM_EINVAL;
    if (q.n == 0 || q.p == 0) continue;
    if (q.m > 0) {
      qs.push_back(q);
      continue;
    }
    const cudaError_t e = cudaMemsetAsync(q.C, 0, (size_t)(q.n * q.p) * sizeof(double), s);
    if (e != cudaSuccess) return note_cuda(e);
  }
  if (qs.empty()) return MM_OK;
  const size_t nq = qs.size();
  std::vector<OzLayout> lays(nq);
  std::vector<SplitProb> tab;
  std::vector<int> owner;  // problem -> product
  TcConfig cfg{128, 4, 0};
  int64_t rows = 0;
  for (size_t g = 0; g < nq; g++) {
    TcChoice ch;
    const mm_status st = ozaki_layout(qs[g], rows, lays[g], ch, tab);
    if (st != MM_OK) return st;
    owner.resize(tab.size(), (int)g);
    cfg.max_bn = std::max(cfg.max_bn, lays[g].bn);
    if (nq == 1) cfg.grid = ch.grid;
  }
  auto align256 = [](size_t x) { return (x + 255) & ~(size_t)255; };
  // row maxima (n) + column maxima (p), zero scale words and the gate's fallback
  // flag of each product, then the planes
  size_t off = align256((size_t)rows * kPackRowBytes), simt_bytes = 0;
  const size_t zero_off = off;
  for (size_t g = 0; g < nq; g++) {
    const OzCall &q = qs[g];
    lays[g].max_off = off;
    lays[g].flag_off = off + (size_t)(q.n + q.p) * 12;
    off = (lays[g].flag_off + sizeof(int) + 7) & ~(size_t)7;
    simt_bytes = std::max(simt_bytes, simt_scratch_bytes(true, q.n, q.m, q.p));
  }
  const size_t zero_end = off;
  for (size_t g = 0; g < nq; g++) {
    lays[g].d_off = align256(off);
    off = lays[g].d_off + (size_t)lays[g].chunks * lays[g].SS * lays[g].plane * sizeof(float);
  }
  const size_t tab_off = align256(off);
  const int nprobs = (int)tab.size();
  // several products in one launch: longest units first over all of them
  std::vector<int> by_length((size_t)nprobs);
  for (int g = 0; g < nprobs; g++) by_length[(size_t)g] = g;
  if (nq > 1)
    std::stable_sort(by_length.begin(), by_length.end(), [&](int a, int b) {
      return (int64_t)tab[(size_t)a].kt * tab[(size_t)a].bn > (int64_t)tab[(size_t)b].kt * tab[(size_t)b].bn;
    });
  int64_t units = 0;
  std::vector<SplitProb> sorted;
  std::vector<int> map;  // unit -> problem
  for (int g : by_length) {
    SplitProb sp = tab[(size_t)g];
    const int64_t tiles = lays[(size_t)owner[(size_t)g]].tiles;
    if (units + tiles > 0x7fffffffLL) return MM_EINVAL;
    sp.unit_start = (int32_t)units;
    map.insert(map.end(), (size_t)tiles, (int)sorted.size());
    units += tiles;
    sorted.push_back(sp);
  }
  // the table, then the work units of each CTA (the levels differ in length), the
  // unit map
  const int grid = tc_launch_grid(cfg, units);
  const size_t tab_bytes = ((size_t)nprobs * sizeof(SplitProb) + 15) & ~(size_t)15;
  const size_t order_end = (tab_bytes + ((size_t)grid + 1 + (size_t)units) * sizeof(int) + 255) & ~(size_t)255;
  const size_t map_off = tab_off + order_end;
  // the fallbacks' K-slice partials (under-filled products)
  const size_t simt_off = align256(map_off + (size_t)units * sizeof(int));
  cudaError_t e = ws.reserve(simt_off + simt_bytes, s);
  if (e != cudaSuccess) return note_cuda(e);
  uint8_t *base = static_cast<uint8_t *>(ws.ptr);
  for (int k = 0; k < nprobs; k++) {
    const size_t g = (size_t)owner[(size_t)by_length[(size_t)k]];
    SplitProb &sp = sorted[(size_t)k];
    sp.C = reinterpret_cast<float *>(base + lays[g].d_off) + (uintptr_t)sp.C;
    // scale exponent 0: the digits are not rescaled
    sp.sA = reinterpret_cast<uint32_t *>(base + lays[g].max_off + (size_t)(qs[g].n + qs[g].p) * 8);
    sp.tB = sp.sA + qs[g].n;
  }
  SplitProb *d_tab = reinterpret_cast<SplitProb *>(base + tab_off);
  const int *d_order = reinterpret_cast<const int *>(base + tab_off + tab_bytes);
  int *unit_map = reinterpret_cast<int *>(base + map_off);
  e = cudaMemsetAsync(base + zero_off, 0, zero_end - zero_off, s);
  if (e != cudaSuccess) return note_cuda(e);
  auto rowmax = [&](size_t g) { return reinterpret_cast<uint64_t *>(base + lays[g].max_off); };
  auto planes = [&](size_t g) { return reinterpret_cast<const float *>(base + lays[g].d_off); };
  auto flag = [&](size_t g) { return reinterpret_cast<int *>(base + lays[g].flag_off); };
  {
    TraceScope ts("ozaki_max", s);
    std::vector<OzMaxItem> items;
    for (size_t g = 0; g < nq; g++) {
      const OzCall &q = qs[g];
      const int64_t blocks = ceil_div(q.n, kRowsPerItem) + ceil_div(q.p, kColStrip) * ceil_div(q.m, kRowChunk);
      if (blocks > 0x7fffffffLL) return MM_EINVAL;
      items.push_back({q.A, q.B, rowmax(g), q.n, q.m, q.p, (int32_t)blocks});
    }
    e = launch_items(items, [&](const OzItems<OzMaxItem> &t, unsigned blocks) {
      return launch_pdl_if(blocks <= sm_count() * 4u, ozaki_max_kernel, blocks, 256, 0, s, t);
    });
    if (e != cudaSuccess) return note_cuda(e);
  }
  // products of one slice count (gate, column pairing) share a launch
  for (int S = kOzakiMinSlices; S <= kOzakiMaxSlices; S++)
    for (int gate = 0; gate < 2; gate++) {
      std::vector<OzDigitItem> items;
      for (size_t g = 0; g < nq; g++) {
        const OzCall &q = qs[g];
        const OzLayout &lay = lays[g];
        if (q.S != S || q.gate != (gate != 0)) continue;
        for (size_t c = 0; c < (size_t)lay.chunks; c++) {
          const int64_t blocks_a = (int64_t)lay.mt * (kTcBM / kDigRows) * lay.kt[c];
          const int64_t blocks = blocks_a + (int64_t)lay.nt * (lay.bn / kDigRows) * lay.kt[c];
          if (blocks > 0x7fffffffLL) return MM_EINVAL;
          items.push_back({q.A, q.B, rowmax(g), q.n, q.m, q.p, lay.k0[c], lay.kc[c], lay.a0[c], lay.b0[c],
                           (int32_t)lay.kt[c], lay.bn, (int32_t)blocks_a, (int32_t)blocks});
        }
      }
      if (items.empty()) continue;
      TraceScope ts("ozaki_digits", s);
      e = launch_ozaki_digits(S, gate != 0, items, static_cast<uint4 *>(ws.ptr), s);
      if (e != cudaSuccess) return note_cuda(e);
    }
  // while the digits are made: the units' order (alone 0.2 ms at 4096^3)
  {
    std::vector<int> order;
    tc_unit_order(sorted.data(), nprobs, grid, order);
    std::vector<uint8_t> blob(order_end + map.size() * sizeof(int), 0);
    std::memcpy(blob.data(), sorted.data(), sorted.size() * sizeof(SplitProb));
    std::memcpy(blob.data() + tab_bytes, order.data(), order.size() * sizeof(int));
    std::memcpy(blob.data() + order_end, map.data(), map.size() * sizeof(int));
    e = ws.stage.copy_to_device(d_tab, blob.data(), blob.size(), s);
    if (e != cudaSuccess) return note_cuda(e);
  }
  e = launch_tc(kTcE4m3, device_table(d_tab, nprobs), (int)units, unit_map, nullptr, ws.ptr, rows, cfg,
                g_ctx.d_err, s, d_order);
  if (e != cudaSuccess) return note_cuda(e);
  // the gate reads the level sums only, so it runs before the sum kernel:
  // where it fails, the sum writes nothing and the FP64 FMA product below
  // reads the epilogue's D (which may be C) untouched
  std::vector<OzGateItem> gates;
  for (size_t g = 0; g < nq; g++) {
    const OzCall &q = qs[g];
    const OzLayout &lay = lays[g];
    if (!q.gate) continue;
    const double room = 0.98 - (double)q.m * 0x1p-23;
    const double thr256 = room < 0.5 ? (double)INFINITY
                                     : 256.0 * std::sqrt((double)q.m) * (q.S + 2) *
                                           std::ldexp(1.0, -5 * q.S - 1) * 1e14 / room;
    float thr = (float)thr256;  // rounded up to a float
    if ((double)thr < thr256) thr = std::nextafter(thr, (float)INFINITY);
    OzGateItem it{planes(g) + (int64_t)lay.chunks * q.S * lay.plane, rowmax(g), flag(g), lay.plane, q.n, q.p, thr,
                  lay.chunks, 0, 0, 0};
    if (!row_blocks(it, 256 * kGateCols, 8, nq == 1)) return MM_EINVAL;
    gates.push_back(it);
  }
  if (!gates.empty()) {
    TraceScope ts("ozaki_gate", s);
    // (not as a dependent: its blocks would wait beside the level products for
    // all of their time)
    e = launch_items(gates, [&](const OzItems<OzGateItem> &t, unsigned blocks) {
      ozaki_gate_check_kernel<<<blocks, 256, 0, s>>>(t);
      return cudaGetLastError();
    });
    if (e != cudaSuccess) return note_cuda(e);
  }
  for (int S = kOzakiMinSlices; S <= kOzakiMaxSlices; S++)
    for (int v = 1; v <= 2; v++) {
      std::vector<OzSumItem> items;
      for (size_t g = 0; g < nq; g++) {
        const OzCall &q = qs[g];
        if (q.S != S || sum_columns(q.p) != v) continue;
        OzSumItem it{planes(g), rowmax(g), q.C, q.gate ? flag(g) : nullptr, epi_of<double>(q.epi),
                     lays[g].plane, q.n, q.p, lays[g].chunks, 0, 0, 0};
        // one wave of blocks: three or four a SM, the launch bounds
        if (!row_blocks(it, 256 * v, v == 2 ? 3 : 4, nq == 1)) return MM_EINVAL;
        items.push_back(it);
      }
      if (items.empty()) continue;
      TraceScope ts("ozaki_sum", s);
      e = launch_ozaki_sum(S, v, items, s);
      if (e != cudaSuccess) return note_cuda(e);
    }
  // the FP64 FMA product replaces C where the flag is set: the same kernels
  // and K slices as MM_MODE_DGEMM, so the bits are that mode's
  for (size_t g = 0; g < nq; g++) {
    const OzCall &q = qs[g];
    if (!q.gate) continue;
    const SimtPlan pl = simt_plan(true, q.n, q.m, q.p);
    if (pl.S >= 1)
      e = launch_simt_splitk_f64(q.n, q.m, q.p, q.A, q.B, q.C,
                                 pl.S > 1 ? reinterpret_cast<double *>(base + simt_off) : nullptr, pl, s, flag(g),
                                 q.epi);
    else
      e = launch_simt_f64(q.n, q.m, q.p, q.A, q.B, q.C, s, flag(g), q.epi);
    if (e != cudaSuccess) return note_cuda(e);
  }
  return MM_OK;
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
