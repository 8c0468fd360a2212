// Split-BF16x3 operand preparation.
//
// Method: an FP32 operand x is written as x = 2^s (hi + lo + d) with
// hi = bf16_rn(x 2^-s), lo = bf16_rn(x 2^-s - hi) and |d| <= 2^-16 |x 2^-s|
// (three parts: hi + mid + lo, |d| <= 2^-24 |x 2^-s|)
// (G. Henry, P. T. P. Tang, A. Heinecke, "Leveraging the bfloat16 artificial
// intelligence datatype for higher-precision computations", ARITH 2019).  The
// power-of-two scale 2^s is chosen per row of A and per column of B from the
// largest magnitude of that row/column, so operands far from 1 keep all their
// significant bits in the bf16 range; scaling by 2^s is exact.  Not part of
// the paper, whose kernels compute in the input type directly.
//
// Kernels:
//   split_pack_kernel   one block per 128 x 64 tile of A or bn x 64 tile of
//                       B^T: scale, split, write the bf16 parts (hi, lo - or
//                       hi, mid, lo for the three-part split) of the pack
//                       (layout in mm_internal.h); zero outside the matrix
//                       so the tensor-core kernel needs no edge checks.
//
// The split path packs in one pass over A and B (kPackUnscaled): scaling by
// a power of two commutes with rounding to bf16 and with the FP32 sums as long
// as nothing leaves the normal range, so for rows/columns whose largest
// magnitude lies in [2^-40, 2^40] the unscaled split gives the same bits as
// the scaled one.  That pass also writes each tile's row/column maxima;
// split_verify_kernel reduces them to the maxima of whole rows/columns and
// flags, per problem, an operand with a row/column outside the range, and a
// second pack launch (kPackFix) re-packs only the flagged operands with their
// scales.  The epilogue applies 2^(s_i + t_j) only for flagged operands.
//
// kTcSplitF16x3 tables (short inner dimensions, where two bf16 parts miss the
// tolerance): x 2^e = hi + 2^-11 lo with hi = fp16_rn(x 2^e) and lo =
// fp16_rn(2^11 (x 2^e - hi)), one e per operand of a product.  fp16 carries
// eleven bits a part against bf16's eight, so two parts hold what three bf16
// parts hold and three products
// replace six; keeping lo scaled by 2^11 (R. Ootomo, R. Yokota, "Recovering
// single precision accuracy from Tensor Cores while surpassing the FP32
// theoretical peak performance", IJHPCA 36, 2022) keeps it out of fp16's
// subnormals.  e comes from a sample of the operand (split_maps_kernel, or
// the pack itself in a table of one product), the pack tests every entry against
// the window of |x 2^e| (zeros pass), and a product with an entry outside is packed
// again by the fix pass as three bf16 parts, scaled where it must be; one
// whose sample already spreads too far is packed so from the start.
//
// The window, by what the two parts lose.  |x 2^e| from 2^-14 to 61440: hi is a normal
// fp16 number, hi + 2^-11 lo is within 2^-22 of the entry and lo within 2^-11 of
// it, so a term of C (both operands, and the product of the two low parts, which is
// dropped) is within 3 * 2^-22 = 7.2e-7.  Below, hi is a subnormal: at 2^-16 the
// entry is within 2^-20 and lo reaches 2^-9 of it, so a term of two such entries
// is off by up to 2^-18 + 2^-19 = 5.7e-6, all terms of an entry of C alike where a whole
// row of A and column of B lie there.  The tolerance 1e-6 sqrt(m) covers that, with
// 2.3e-6 left for the sums, from m = 64 on: the window starts at 2^-16 there, and at
// 2^-14 below (2 more of the 29 binades under the largest sampled entry then turn a
// product to three parts).  m <= 16 always takes three parts: K in one MMA of
// sixteen leaves the sums nothing to lose, and the six products are the
// more accurate ones (1000 x 16 x 1000, largest error over |A||B| 1.1e-7 against
// 1.8e-7; m = 1 1.5e-7 against 4.6e-7; m = 24 4.5e-7 against 2.2e-7).
#include <algorithm>

#include <cuda_fp16.h>

#include "split_common.cuh"

namespace mm {
namespace {

// Window of |x 2^e| that the two fp16 parts take (its ends as FP32 bit
// patterns; the lower one by the inner dimension), and the exponent that the largest
// sampled magnitude is brought to (a factor of at least 3.75 of room above
// it, 2^29 or 2^27 below).  kHalfExpMax bounds |e| so that 2^e, the window's ends
// divided by 2^e and the products stay normal FP32 numbers.
constexpr int kHalfTopExp = 13, kHalfExpMax = 100;
constexpr uint32_t kHalfHighBits = 0x47700000u;  // 61440
constexpr int kHalfMinK = 17;                    // fewer K values take three parts
__device__ __forceinline__ uint32_t half_low_bits(int m) {
  return m >= 64 ? 0x37800000u : 0x38800000u;  // 2^-16, 2^-14
}
constexpr int kHalfSamples = 256;  // entries sampled per operand

__device__ __forceinline__ uint32_t abs_bits(float x) { return __float_as_uint(x) & 0x7fffffffu; }

__device__ __forceinline__ uint32_t umax(uint32_t a, uint32_t b) { return a > b ? a : b; }

__device__ __forceinline__ bool aligned16(const void *p) {
  return (reinterpret_cast<uintptr_t>(p) & 15u) == 0;
}

// Splits four values scaled by 2^-s (SCALED; unscaled: s = 0, no multiply)
// into PARTS groups of four bf16 (two bf16x2 words each): part 0 = RN(y),
// part q = RN(y - part 0 - ... - part q-1).  Every remainder is exact in FP32
// (the difference of a float and its rounding to fewer bits), so y = sum of
// parts + d, |d| <= 2^(-8*PARTS) |y|.
template <int PARTS, bool SCALED>
__device__ __forceinline__ void split4(float4 x, int s, uint2 (&out)[PARTS]) {
  float y[4] = {x.x, x.y, x.z, x.w};
  if (SCALED) {
#pragma unroll
    for (int e = 0; e < 4; e++) y[e] = scale_pow2(y[e], -s);
  }
#pragma unroll
  for (int q = 0; q < PARTS; q++) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(y[0], y[1]);
    const __nv_bfloat162 b = __floats2bfloat162_rn(y[2], y[3]);
    const float2 fa = __bfloat1622float2(a), fb = __bfloat1622float2(b);
    y[0] -= fa.x;
    y[1] -= fa.y;
    y[2] -= fb.x;
    y[3] -= fb.y;
    out[q] = make_uint2(*reinterpret_cast<const uint32_t *>(&a),
                        *reinterpret_cast<const uint32_t *>(&b));
  }
}

// Two fp16 parts of four values times mul = 2^e: hi = RN(y), lo = RN((y - hi)
// 2^11); y - hi is exact in FP32, and so is its scaling.
__device__ __forceinline__ void split4_half(float4 x, float mul, uint2 (&out)[2]) {
  const float y[4] = {x.x * mul, x.y * mul, x.z * mul, x.w * mul};
  const __half2 a = __floats2half2_rn(y[0], y[1]), b = __floats2half2_rn(y[2], y[3]);
  const float2 fa = __half22float2(a), fb = __half22float2(b);
  const __half2 la = __floats2half2_rn((y[0] - fa.x) * 2048.0f, (y[1] - fa.y) * 2048.0f);
  const __half2 lb = __floats2half2_rn((y[2] - fb.x) * 2048.0f, (y[3] - fb.y) * 2048.0f);
  out[0] = make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
  out[1] = make_uint2(*reinterpret_cast<const uint32_t *>(&la), *reinterpret_cast<const uint32_t *>(&lb));
}

// Two fp16 parts (HALF, of x times mul) or PARTS bf16 parts of x as it is.
template <int PARTS, bool HALF>
__device__ __forceinline__ void split_any(float4 x, float mul, uint2 (&out)[PARTS]) {
  if constexpr (HALF) split4_half(x, mul, out);
  else split4<PARTS, false>(x, 0, out);
}

// min over four values of |x|'s bit pattern less one: a zero becomes the
// largest word, so it never is the smallest.
__device__ __forceinline__ uint32_t min4_bits(float4 x) {
  const uint32_t a = min(abs_bits(x.x) - 1u, abs_bits(x.y) - 1u);
  return min(a, min(abs_bits(x.z) - 1u, abs_bits(x.w) - 1u));
}

// An operand with an entry outside the fp16 window [low, 61440]
// times 2^-e, as bit patterns (both ends are normal numbers for |e| <= 100).
__device__ __forceinline__ bool outside_window(uint32_t mx, uint32_t mn, int e, uint32_t low) {
  const uint32_t shift = (uint32_t)e << 23;
  return mx > kHalfHighBits - shift || mn < low - shift - 1u;
}

// max |x| over four values as a float bit pattern
__device__ __forceinline__ uint32_t max4_bits(float4 x) {
  return umax(umax(abs_bits(x.x), abs_bits(x.y)), umax(abs_bits(x.z), abs_bits(x.w)));
}

// Eight maxima over the 16 lanes of a half warp at once (v[t], t = 0..7, in
// every lane): each exchange round sends the half of the slots that the
// partner keeps, so 8 shuffles replace 4 per slot.  Returns, in every lane,
// the half-warp maximum of slot t = (lane >> 1) & 7 (lanes 2t and 2t + 1 of
// the half warp hold slot t).  Every lane of the warp must call it.
__device__ __forceinline__ uint32_t half_warp_max8(const uint32_t (&v)[8]) {
  const int lane = threadIdx.x & 31;
  const bool b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
  uint32_t w[4], u[2];
#pragma unroll
  for (int j = 0; j < 4; j++) {  // lanes with bit 3 clear keep slots 0-3
    const uint32_t send = b3 ? v[j] : v[j + 4], keep = b3 ? v[j + 4] : v[j];
    w[j] = umax(keep, __shfl_xor_sync(0xffffffffu, send, 8));
  }
#pragma unroll
  for (int j = 0; j < 2; j++) {  // w[j] holds slot j + 4 b3
    const uint32_t send = b2 ? w[j] : w[j + 2], keep = b2 ? w[j + 2] : w[j];
    u[j] = umax(keep, __shfl_xor_sync(0xffffffffu, send, 4));
  }
  const uint32_t send = b1 ? u[0] : u[1], keep = b1 ? u[1] : u[0];  // u[j]: slot j + 2 b2 + 4 b3
  const uint32_t t = umax(keep, __shfl_xor_sync(0xffffffffu, send, 2));
  return umax(t, __shfl_xor_sync(0xffffffffu, t, 1));
}

// Barrier of the 256 threads that pack (a block may hold one more warp).
__device__ __forceinline__ void pack_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// One B pack tile (nt, kb) of split_pack_kernel: bn columns x 64 k,
// transposed through shared memory CW columns at a time.  `scaled` (kPackFix):
// the columns are scaled.
template <int PARTS, int MODE, int CW>
__device__ __forceinline__ void pack_b_tile(const SplitProb &pr, int b, uint2 *__restrict__ pack,
                                            float (&tile)[kPackK][128 + 1], int tid, bool scaled) {
  constexpr int kQuads = kPackK / 4;                 // groups of four bf16 per pack row
  constexpr int kIter = kPackK * (CW / 4) / 256;     // 16-byte loads per thread and chunk
  const int nt = b / pr.kt, kb = b % pr.kt;
  const int bn = pr.bn;
  const int64_t base = pr.b_row0 + (int64_t)b * PARTS * bn;
  const bool vec = aligned16(pr.B) && (pr.p & 3) == 0;
  for (int c0 = 0; c0 < bn; c0 += CW) {
    float4 vs[kIter];
#pragma unroll
    for (int it = 0; it < kIter; it++) {
      const int q = tid + it * 256;
      const int kk = q / (CW / 4), c4 = q % (CW / 4);
      const int64_t k = (int64_t)kb * kPackK + kk;
      const int64_t j = (int64_t)nt * bn + c0 + 4 * c4;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k < pr.m) {
        const float *src = pr.B + k * pr.p + j;
        if (vec && j + 4 <= pr.p) {
          v = __ldcs(reinterpret_cast<const float4 *>(src));
        } else {
          if (j < pr.p) v.x = src[0];
          if (j + 1 < pr.p) v.y = src[1];
          if (j + 2 < pr.p) v.z = src[2];
          if (j + 3 < pr.p) v.w = src[3];
        }
      }
      vs[it] = v;
    }
#pragma unroll
    for (int it = 0; it < kIter; it++) {
      const int q = tid + it * 256;
      const int kk = q / (CW / 4), c4 = q % (CW / 4);
      tile[kk][4 * c4 + 0] = vs[it].x;
      tile[kk][4 * c4 + 1] = vs[it].y;
      tile[kk][4 * c4 + 2] = vs[it].z;
      tile[kk][4 * c4 + 3] = vs[it].w;
    }
    __syncthreads();
    // column c = tid / 16 + 16 t of this chunk in round t: the 16 threads of
    // a half warp hold one column's 64 values
    constexpr int kCols = CW * kQuads / 256;
    uint32_t mxv[8];
#pragma unroll
    for (int t = 0; t < kCols; t++) {
      const int q = tid + t * 256;
      const int c = q / kQuads, kq = q % kQuads;
      const int64_t j = (int64_t)nt * bn + c0 + c;
      const int s = (MODE != kPackUnscaled && scaled && j < pr.p) ? scale_exponent(pr.tB[j]) : 0;
      const float4 x = make_float4(tile[4 * kq][c], tile[4 * kq + 1][c], tile[4 * kq + 2][c],
                                   tile[4 * kq + 3][c]);
      if (MODE == kPackUnscaled) mxv[t] = max4_bits(x);
      uint2 part[PARTS];
      split4<PARTS, MODE != kPackUnscaled>(x, s, part);
#pragma unroll
      for (int h = 0; h < PARTS; h++) pack[(base + h * bn + c0 + c) * kQuads + kq] = part[h];
    }
    if (MODE == kPackUnscaled) {
#pragma unroll
      for (int t = kCols; t < 8; t++) mxv[t] = 0;
      const uint32_t mx = half_warp_max8(mxv);
      const int t = (tid >> 1) & 7;
      const int64_t j = (int64_t)nt * bn + c0 + tid / kQuads + 16 * t;
      if ((tid & 1) == 0 && t < kCols && j < pr.p) pr.pB[(int64_t)kb * pr.p + j] = mx;
    }
    __syncthreads();
  }
}

// One A pack tile (mt, kb) of split_pack_kernel: rows mt*128.., k kb*64..; a
// warp covers two rows.
template <int PARTS, int MODE>
__device__ __forceinline__ void pack_a_tile(const SplitProb &pr, int local, uint2 *__restrict__ pack,
                                            int tid, bool scaled) {
  constexpr int kQuads = kPackK / 4;  // groups of four bf16 (8 bytes) per pack row
  constexpr int kAIter = kTcBM * kQuads / 256;
  static_assert(kAIter == 8, "eight A vectors per thread (one reduction slot each)");
  const int mt = local / pr.kt, kb = local % pr.kt;
  const int64_t base = pr.a_row0 + (int64_t)local * PARTS * kTcBM;
  const bool vec = aligned16(pr.A) && (pr.m & 3) == 0;
  float4 xs[kAIter];
#pragma unroll
  for (int it = 0; it < kAIter; it++) {
    const int q = tid + it * 256;
    const int r = q / kQuads, kq = q % kQuads;
    const int64_t i = (int64_t)mt * kTcBM + r;
    const int64_t k = (int64_t)kb * kPackK + 4 * kq;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < pr.n) {
      const float *row = pr.A + i * pr.m;
      if (vec && k + 4 <= pr.m) {
        x = __ldcs(reinterpret_cast<const float4 *>(row + k));
      } else {
        if (k < pr.m) x.x = row[k];
        if (k + 1 < pr.m) x.y = row[k + 1];
        if (k + 2 < pr.m) x.z = row[k + 2];
        if (k + 3 < pr.m) x.w = row[k + 3];
      }
    }
    xs[it] = x;
  }
  if (MODE == kPackUnscaled) {
    // row r = tid / 16 + 16 it: the 16 threads of a half warp hold one
    // row's 64 values
    uint32_t mxv[8];
#pragma unroll
    for (int it = 0; it < 8; it++) mxv[it] = max4_bits(xs[it]);
    const uint32_t mx = half_warp_max8(mxv);
    const int t = (tid >> 1) & 7;
    const int64_t i = (int64_t)mt * kTcBM + tid / kQuads + 16 * t;
    if ((tid & 1) == 0 && i < pr.n) pr.pA[(int64_t)kb * pr.n + i] = mx;
  }
#pragma unroll
  for (int it = 0; it < kAIter; it++) {
    const int q = tid + it * 256;
    const int r = q / kQuads, kq = q % kQuads;
    const int64_t i = (int64_t)mt * kTcBM + r;
    const int s = (MODE != kPackUnscaled && scaled && i < pr.n) ? scale_exponent(pr.sA[i]) : 0;
    uint2 part[PARTS];
    split4<PARTS, MODE != kPackUnscaled>(xs[it], s, part);
#pragma unroll
    for (int h = 0; h < PARTS; h++) pack[(base + h * kTcBM + r) * kQuads + kq] = part[h];
  }
}

// MODE: kPackUnscaled - no scaling; write the tile's row (A) / column (B)
//                       maxima to pA / pB; one block per pack tile;
//       kPackFix      - scale by 2^-s from the maxima in sA / tB; only the
//                       operands flagged by split_verify_kernel; a persistent
//                       grid over the pack tiles that returns at once when
//                       no operand of the table is flagged (*any == 0).
// Every thread first loads all its 16-byte vectors of a tile (eight of A, or
// four of a 64-column slice of B), then splits and stores them, so that each
// thread keeps several loads in flight.
template <int PARTS, int MODE>
__global__ void __launch_bounds__(256, 4)
split_pack_kernel(const __grid_constant__ ProbTable tab, const int *__restrict__ map,
                  const int *__restrict__ flags, const int *__restrict__ any, int total_tiles,
                  uint2 *__restrict__ pack) {
  __shared__ float tile[kPackK][128 + 1];
  const SplitProb *probs = tab.dev ? tab.dev : &tab.one;
  const int nprobs = tab.n;
  pdl_wait();
  if (MODE == kPackFix && *any == 0) return;
  const int tid = threadIdx.x;
  for (int item = blockIdx.x; item < total_tiles; item += gridDim.x) {
    const int g =
        find_problem(probs, nprobs, map, item, [](const SplitProb &q) { return q.pack_start; });
    const SplitProb &pr = probs[g];
    const int local = item - pr.pack_start;
    const bool a_tile = local < pr.mt * pr.kt;
    if (MODE == kPackFix && !(flags[g] & (a_tile ? kFlagScaleA : kFlagScaleB))) continue;
    if (a_tile) {
      pack_a_tile<PARTS, MODE>(pr, local, pack, tid, true);
    } else {
      // B tile (nt, kb): columns nt*bn.., k kb*64..; transposed through shared
      // memory 128 columns at a time (64 for bn = 64) so both the read and the
      // write coalesce, with eight 16-byte loads per thread in flight.
      const int b = local - pr.mt * pr.kt;
      if (pr.bn % 128 == 0)
        pack_b_tile<PARTS, MODE, 128>(pr, b, pack, tile, tid, true);
      else
        pack_b_tile<PARTS, MODE, 64>(pr, b, pack, tile, tid, true);
    }
  }
}

// Largest magnitude and smallest non-zero one (its bit pattern less one; the
// largest word if there is none) among kHalfSamples entries of an operand, at
// positions that depend on its size only, so the choice made from them is the
// same alone and in any table.  In every thread; all 256 must call it.
__device__ __forceinline__ uint2 sample_range(const float *__restrict__ X, int64_t count,
                                              uint32_t (&mx_s)[8], uint32_t (&mn_s)[8]) {
  uint32_t mx = 0, mn = 0xffffffffu;
#pragma unroll
  for (int t = 0; t < kHalfSamples / 256; t++) {
    // multiplicative hashing of the sample's index (Knuth, TAOCP 3, 6.4)
    const uint64_t h = (uint64_t)(threadIdx.x + 256 * t + 1) * 0x9E3779B97F4A7C15ull;
    const uint32_t b = abs_bits(X[__umul64hi(h, (uint64_t)count)]);
    mx = umax(mx, b);
    mn = min(mn, b - 1u);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  mn = __reduce_min_sync(0xffffffffu, mn);
  const int warp = threadIdx.x >> 5;
  pack_sync();
  if ((threadIdx.x & 31) == 0) {
    mx_s[warp] = mx;
    mn_s[warp] = mn;
  }
  pack_sync();
#pragma unroll
  for (int w = 0; w < 8; w++) {
    mx = umax(mx, mx_s[w]);
    mn = min(mn, mn_s[w]);
  }
  return make_uint2(mx, mn);
}

// The fp16 window's exponent e for an operand of that range: its largest
// sampled magnitude to [2^13, 2^14).  False where the sample does not fit.
__device__ __forceinline__ bool half_exponent(uint2 range, uint32_t low, int &e) {
  e = 0;
  if (range.x == 0) return true;  // nothing but zeros sampled
  if (range.x >= 0x7f800000u) return false;
  e = kHalfTopExp - ilogbf(__uint_as_float(range.x));
  return abs(e) <= kHalfExpMax && !outside_window(range.x, range.y, e, low);
}

// The form of a product from its operands' samples: 1 for three bf16 parts, 0
// for two fp16 parts with the exponents ea and eb.
__device__ __forceinline__ int half_form(uint2 ra, uint2 rb, int m, int &ea, int &eb) {
  const uint32_t low = half_low_bits(m);
  const bool fits = half_exponent(ra, low, ea) & half_exponent(rb, low, eb);
  return fits && m >= kHalfMinK ? 0 : 1;
}

// The same for kTcSplitF16x3 tables (bn = 128): a product's tiles as two fp16
// parts, or as three bf16 parts where its state says so (hx[kHalfX6]).
// It writes the state words of a table of one product, and sets hx[kHalfBad]
// (zeroed by the caller) and *any where an entry lies outside the fp16 window;
// split_fix_half_kernel packs such a product again, both operands, as three
// bf16 parts (scaled where verify flagged the operand), and otherwise the
// flagged operands as split_pack_kernel does.
//
// Memory-bound (4 bytes read and 4 written per entry).  A block per tile spent
// most of its time on the chain item -> map -> table -> state -> data, four
// dependent loads before the first entry arrives, which four blocks an SM do
// not cover on tables of small products.  Here a persistent grid's ninth warp
// runs that chain for 32 tiles at a time, a lane each, and leaves in shared
// memory all that a tile needs; eight warps copy the tile after next into
// shared memory (cp.async) before they split the current one, so that an SM's
// two blocks keep two to four tiles of 32 KB in flight; a table of one product
// draws its sample once a block instead of once a tile.  (1024 products of
// 32..1024: 941 us as a block per tile, 838 us so, 4.7 GB with the tiles'
// padding, 5.6 TB/s; a register double buffer instead of cp.async 995 us.)
struct __align__(16) PackItem {
  const float *src;   // the tile's first entry (null: no more tiles)
  uint32_t *maxima;   // of its rows (columns) in this K block
  uint2 *dst;         // its first pack row
  int32_t *bad;       // the product's kHalfBad word
  int32_t ld;         // entries between its rows (A) / K rows (B)
  int32_t outer, k;   // rows (columns) and K values from its first entry to the edge
  int32_t e;          // exponent of the fp16 parts
  uint32_t low;       // lower end of their window
  uint8_t is_a, x6, vec, pad;
};
constexpr int kPkStages = 3, kPkItems = 64;
constexpr int kPkSmem = kPkStages * kPackK * 128 * 4;

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Four consecutive floats into a 16-byte slot, those past `left` as zeros.
template <bool VEC>
__device__ __forceinline__ void copy_quad(uint32_t dst, const float *src, int left, const float *safe) {
  if (VEC) {  // wholly inside or outside
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(left >= 4 ? src : safe),
                 "r"(left >= 4 ? 16 : 0)
                 : "memory");
  } else {
#pragma unroll
    for (int t = 0; t < 4; t++)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * t),
                   "l"(left > t ? src + t : safe), "r"(left > t ? 4 : 0)
                   : "memory");
  }
}

// Slot of the 16-byte chunk c4 of K row kk of a B tile: the chunks of a row are
// permuted by the row's group of four, so that the sixteen threads that read
// a column's 64 values meet two on a bank instead of sixteen.
__device__ __forceinline__ int b_slot(int kk, int c4) { return kk * 32 + (c4 ^ ((kk >> 2) & 15)); }

// The eight 16-byte vectors of a tile that this thread copies: A's rows tid / 16
// + 16 it at K 4 (tid % 16); B's K rows tid / 32 + 8 it at columns 4 (tid % 32).
template <bool VEC>
__device__ __forceinline__ void copy_tile(const PackItem &d, int tid, uint32_t dst) {
  if (d.is_a) {
    const int k = 4 * (tid % 16), r0 = tid / 16;
    const float *src = d.src + (int64_t)r0 * d.ld + k;
#pragma unroll
    for (int it = 0; it < 8; it++)
      copy_quad<VEC>(dst + 16u * (uint32_t)(tid + 256 * it), src + (int64_t)it * 16 * d.ld,
                     r0 + 16 * it < d.outer ? d.k - k : 0, d.src);
  } else {
    const int c = 4 * (tid % 32), k0 = tid / 32;
    const float *src = d.src + (int64_t)k0 * d.ld + c;
#pragma unroll
    for (int it = 0; it < 8; it++)
      copy_quad<VEC>(dst + 16u * (uint32_t)b_slot(k0 + 8 * it, tid % 32), src + (int64_t)it * 8 * d.ld,
                     k0 + 8 * it < d.k ? d.outer - c : 0, d.src);
  }
}

// Splits a copied tile: in round t this thread holds four K values 4 (tid % 16)
// of row (column) tid / 16 + 16 t, so a half warp holds a row's 64 values and
// writes its 128-byte pack row of each part.  Returns whether an entry lies
// outside the fp16 window (HALF).
template <int PARTS, bool HALF>
__device__ __forceinline__ bool emit_tile(const PackItem &d, const float4 *t4, int tid) {
  const int kq = tid % 16, r0 = tid / 16;
  const float mul = HALF ? __int_as_float((d.e + 127) << 23) : 1.0f;
  const float *t = reinterpret_cast<const float *>(t4);
  uint2 *dst = d.dst + r0 * 16 + kq;
  uint32_t mxv[8], mn = 0xffffffffu;
#pragma unroll
  for (int it = 0; it < 8; it++) {
    float4 x;
    if (d.is_a) {
      x = t4[tid + 256 * it];
    } else {
      const int c = r0 + 16 * it;
      const int s0 = 4 * b_slot(4 * kq, c >> 2) + (c & 3);  // the group's rows lie 128 apart
      x = make_float4(t[s0], t[s0 + 128], t[s0 + 256], t[s0 + 384]);
    }
    mxv[it] = max4_bits(x);
    if (HALF) mn = min(mn, min4_bits(x));
    uint2 part[PARTS];
    split_any<PARTS, HALF>(x, mul, part);
#pragma unroll
    for (int h = 0; h < PARTS; h++) dst[(h * 128 + 16 * it) * 16] = part[h];
  }
  const uint32_t mx = half_warp_max8(mxv);
  const int r = r0 + 16 * ((tid >> 1) & 7);
  if ((tid & 1) == 0 && r < d.outer) d.maxima[r] = mx;
  return HALF && outside_window(mx, mn, d.e, d.low);
}

__global__ void __launch_bounds__(288, 2)
split_pack_half_kernel(const __grid_constant__ ProbTable tab, const int *__restrict__ map,
                       int *any, int total_tiles, uint2 *__restrict__ pack) {
  extern __shared__ __align__(16) float4 tiles[];  // kPkStages of 128 x 64 entries
  __shared__ PackItem items[kPkItems];
  __shared__ uint32_t mx_s[8], mn_s[8];
  __shared__ int one[3];  // the state words of a table of one product
  const SplitProb *probs = tab.dev ? tab.dev : &tab.one;
  const int nprobs = tab.n;
  const int tid = threadIdx.x;
  pdl_wait();
  if (map == nullptr && tid < 256) {
    int ea, eb;
    const uint2 ra = sample_range(probs->A, (int64_t)probs->n * probs->m, mx_s, mn_s);
    const uint2 rb = sample_range(probs->B, (int64_t)probs->m * probs->p, mx_s, mn_s);
    const int x6 = half_form(ra, rb, probs->m, ea, eb);
    if (tid == 0) {
      one[kHalfX6] = x6;
      one[kHalfExpA] = ea;
      one[kHalfExpB] = eb;
      if (blockIdx.x == 0) {
        probs->hx[kHalfX6] = x6;
        probs->hx[kHalfExpA] = ea;
        probs->hx[kHalfExpB] = eb;
      }
    }
  }
  __syncthreads();
  auto decode = [&](int it) {  // this block's tile `it` into its slot
    const int64_t item = (int64_t)blockIdx.x + (int64_t)it * gridDim.x;
    PackItem d;
    d.src = nullptr;
    if (item < total_tiles) {
      const int g =
          find_problem(probs, nprobs, map, (int)item, [](const SplitProb &q) { return q.pack_start; });
      const SplitProb &pr = probs[g];
      const int local = (int)item - pr.pack_start, b = local - pr.mt * pr.kt;
      const int *hx = map != nullptr ? pr.hx : one;
      d.is_a = b < 0;
      d.x6 = hx[kHalfX6] != 0;
      d.e = hx[b < 0 ? kHalfExpA : kHalfExpB];
      d.low = half_low_bits(pr.m);
      d.bad = &pr.hx[kHalfBad];
      const int t = b < 0 ? local : b;
      const int o0 = (t / pr.kt) * 128, kb = t % pr.kt;  // first row or column, K block
      const float *X = b < 0 ? pr.A : pr.B;
      d.ld = b < 0 ? pr.m : pr.p;
      d.src = b < 0 ? X + (int64_t)o0 * pr.m + kb * kPackK : X + (int64_t)kb * kPackK * pr.p + o0;
      d.outer = (b < 0 ? pr.n : pr.p) - o0;
      d.k = pr.m - kb * kPackK;
      d.maxima = b < 0 ? pr.pA + (int64_t)kb * pr.n + o0 : pr.pB + (int64_t)kb * pr.p + o0;
      d.dst = pack + ((b < 0 ? pr.a_row0 : pr.b_row0) + (int64_t)t * (d.x6 ? 3 : 2) * 128) * 16;
      d.vec = aligned16(X) && (d.ld & 3) == 0;
    }
    items[it % kPkItems] = d;
  };
  auto copy = [&](int it) {  // tile `it` into its stage, one group (empty past the end)
    const PackItem &d = items[it % kPkItems];
    if (d.src != nullptr) {
      const uint32_t dst = smem_addr(tiles + (it % kPkStages) * (kPackK * 32));
      if (d.vec) copy_tile<true>(d, tid, dst);
      else copy_tile<false>(d, tid, dst);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (tid >= 256) decode(tid - 256);
  __syncthreads();
  if (tid < 256) {
    copy(0);
    copy(1);
  }
  for (int it = 0;; it++) {
    const PackItem &d = items[it % kPkItems];
    if (d.src == nullptr) break;
    if (tid >= 256) {
      // the next 32 tiles at once, a lane each: the chain's latency once in 32
      if (it % 32 == 0) decode(it + 32 + tid - 256);
    } else {
      copy(it + 2);
      asm volatile("cp.async.wait_group 2;" ::: "memory");  // this thread's part of tile `it`
      if (!d.is_a) pack_sync();  // B: every thread's part (of A a thread reads what it copied)
      const float4 *t4 = tiles + (it % kPkStages) * (kPackK * 32);
      bool bad = false;
      if (d.x6) emit_tile<3, false>(d, t4, tid);
      else bad = emit_tile<2, true>(d, t4, tid);
      if (__any_sync(0xffffffffu, bad) && (tid & 31) == 0) {
        atomicOr(d.bad, 1);
        atomicOr(any, 1);
      }
    }
    __syncthreads();
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// The fix pass of such a table (a persistent grid, as split_pack_kernel's).
__global__ void __launch_bounds__(256, 4)
split_fix_half_kernel(const __grid_constant__ ProbTable tab, const int *__restrict__ map,
                      const int *__restrict__ flags, const int *__restrict__ any, int total_tiles,
                      uint2 *__restrict__ pack) {
  __shared__ float tile[kPackK][128 + 1];
  const SplitProb *probs = tab.dev ? tab.dev : &tab.one;
  const int nprobs = tab.n;
  pdl_wait();
  if (*any == 0) return;
  for (int item = blockIdx.x; item < total_tiles; item += gridDim.x) {
    const int g =
        find_problem(probs, nprobs, map, item, [](const SplitProb &q) { return q.pack_start; });
    const SplitProb &pr = probs[g];
    const int local = item - pr.pack_start;
    const bool scaled = (flags[g] & (local < pr.mt * pr.kt ? kFlagScaleA : kFlagScaleB)) != 0;
    if (!scaled && pr.hx[kHalfBad] == 0) continue;
    const int b = local - pr.mt * pr.kt;
    if (b < 0) pack_a_tile<3, kPackFix>(pr, local, pack, threadIdx.x, scaled);
    else pack_b_tile<3, kPackFix, 128>(pr, b, pack, tile, threadIdx.x, scaled);
  }
}

// A row/column maximum outside [2^-40, 2^40] (or not finite) needs scaling;
// zero needs none.
__device__ __forceinline__ bool needs_scale(uint32_t max_bits) {
  return max_bits != 0 && (max_bits < 0x2B800000u /* 2^-40 */ || max_bits > 0x53800000u /* 2^40 */);
}

// Verify items of 32 rows/columns of one problem; WPI warps per item split
// its K blocks, 8 / WPI items per block (WPI from the table's longest K, so
// that short products do not pay for idle warps): the maximum of a row of A
// over its K blocks -> sA (columns of B -> tB), and flags[g] |= kFlagScaleA /
// kFlagScaleB (and *any) where a maximum is outside the range packed
// unscaled.
template <int WPI>
__global__ void __launch_bounds__(256)
split_verify_kernel(const __grid_constant__ ProbTable tab, const int *__restrict__ map,
                    int total_items, int *__restrict__ flags, int *__restrict__ any,
                    bool write_cols) {
  __shared__ uint32_t part[8][32];
  const SplitProb *probs = tab.dev ? tab.dev : &tab.one;
  const int nprobs = tab.n;
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int sub = warp % WPI;
  const int item = blockIdx.x * (8 / WPI) + warp / WPI;
  const bool live = item < total_items;
  const SplitProb *pp = nullptr;
  int g = 0;
  int64_t w = 0;
  bool valid = false;
  uint32_t mx = 0;
  if (live) {
    g = find_problem(probs, nprobs, map, item, [](const SplitProb &q) { return q.ver_start; });
    pp = probs + g;
    w = (int64_t)(item - pp->ver_start) * 32 + lane;
    valid = w < (int64_t)pp->n + pp->p;
    // a product held in fp16 parts has no per-row scales
    if (pp->hx != nullptr && (pp->hx[kHalfX6] | pp->hx[kHalfBad]) == 0) valid = false;
    if (valid) {
      const bool is_row = w < pp->n;
      const uint32_t *src = is_row ? pp->pA + w : pp->pB + (w - pp->n);
      const int64_t stride = is_row ? pp->n : pp->p;
#pragma unroll 4
      for (int kb = sub; kb < pp->kt; kb += WPI) mx = umax(mx, src[kb * stride]);
    }
  }
  if (WPI > 1) {
    part[warp][lane] = mx;
    __syncthreads();
    if (sub == 0)
#pragma unroll
      for (int q = 1; q < WPI; q++) mx = umax(mx, part[warp + q][lane]);
  }
  if (sub != 0 || !live) return;
  int bad = 0;
  if (valid) {
    const bool is_row = w < pp->n;
    if (is_row) pp->sA[w] = mx; else if (write_cols) pp->tB[w - pp->n] = mx;
    if (needs_scale(mx)) bad = is_row ? kFlagScaleA : kFlagScaleB;
  }
  const unsigned mask = __activemask();
  const unsigned a = __ballot_sync(mask, bad & kFlagScaleA);
  const unsigned b = __ballot_sync(mask, bad & kFlagScaleB);
  if (lane == 0 && (a || b)) {
    atomicOr(&flags[g], (a ? kFlagScaleA : 0) | (b ? kFlagScaleB : 0));
    atomicOr(any, 1);
  }
}

// One block per problem: writes the problem's index over its ranges of MMA
// tiles, pack tiles and scale-reduction items, and the state words of a
// kTcSplitF16x3 product.
__global__ void __launch_bounds__(256)
split_maps_kernel(const __grid_constant__ ProbTable tab, int *__restrict__ unit_map,
                  int *__restrict__ pack_map, int *__restrict__ ver_map) {
  __shared__ uint32_t mx_s[8], mn_s[8];
  const int g = blockIdx.x;
  pdl_wait();
  const SplitProb &pr = (tab.dev ? tab.dev : &tab.one)[g];
  const int units = (int)split_units(pr);
  const int packs = pr.mt * pr.kt + pr.nt * pr.kt;
  if (unit_map)
    for (int i = threadIdx.x; i < units; i += blockDim.x) unit_map[pr.unit_start + i] = g;
  if (pack_map)
    for (int i = threadIdx.x; i < packs; i += blockDim.x) pack_map[pr.pack_start + i] = g;
  if (ver_map) {  // only tables that run split_verify_kernel
    const int vers = (int)verify_items(pr.n, pr.p);
    for (int i = threadIdx.x; i < vers; i += blockDim.x) ver_map[pr.ver_start + i] = g;
  }
  if (pr.hx) {
    const uint2 ra = sample_range(pr.A, (int64_t)pr.n * pr.m, mx_s, mn_s);
    const uint2 rb = sample_range(pr.B, (int64_t)pr.m * pr.p, mx_s, mn_s);
    if (threadIdx.x == 0) {
      int ea = 0, eb = 0;
      pr.hx[kHalfX6] = half_form(ra, rb, pr.m, ea, eb);
      pr.hx[kHalfExpA] = ea;
      pr.hx[kHalfExpB] = eb;
    }
  }
}

}  // namespace

cudaError_t launch_split_maps(const ProbTable &tab, int *unit_map, int *pack_map, int *ver_map,
                              cudaStream_t s) {
  if (tab.n <= 0) return cudaSuccess;
  TraceScope ts("split_maps", s);
  return launch_pdl(split_maps_kernel, (unsigned)tab.n, 256, 0, s, tab, unit_map, pack_map, ver_map);
}

cudaError_t launch_split_pack(TcKind kind, int mode, const ProbTable &tab, int total_tiles,
                              const int *map, const int *flags, int *any,
                              void *pack_base, cudaStream_t s) {
  if (total_tiles <= 0) return cudaSuccess;
  TraceScope ts(mode == kPackFix ? "split_fix" : "split_pack", s);
  auto *pk = static_cast<uint2 *>(pack_base);
  const bool x6 = kind == kTcSplitBf16x6;
  // the fix pass: a persistent grid of one wave (4 blocks per SM, the launch
  // bound) over the tiles, so that its early return when nothing is flagged
  // costs a single wave of blocks
  const int grid = mode == kPackFix ? std::min(total_tiles, sm_count() * 4) : total_tiles;
  if (kind == kTcSplitF16x3) {
    if (mode == kPackFix)
      return launch_pdl(split_fix_half_kernel, (unsigned)grid, 256, 0, s, tab, map, flags,
                        static_cast<const int *>(any), total_tiles, pk);
    static std::once_flag once;
    static cudaError_t attr_err = cudaSuccess;
    std::call_once(once, [] {
      attr_err = cudaFuncSetAttribute(split_pack_half_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      kPkSmem);
    });
    if (attr_err != cudaSuccess) return attr_err;
    return launch_pdl(split_pack_half_kernel, (unsigned)std::min(total_tiles, sm_count() * 2), 288, kPkSmem,
                      s, tab, map, any, total_tiles, pk);
  }
  auto kernel = mode == kPackUnscaled ? (x6 ? split_pack_kernel<3, kPackUnscaled> : split_pack_kernel<2, kPackUnscaled>)
                                      : (x6 ? split_pack_kernel<3, kPackFix> : split_pack_kernel<2, kPackFix>);
  return launch_pdl_if(grid <= sm_count() * 4, kernel, (unsigned)grid, 256, 0, s, tab, map, flags,
                       static_cast<const int *>(any), total_tiles, pk);
}

cudaError_t launch_split_verify(const ProbTable &tab, int64_t total_items,
                                const int *map, int *flags, int *any, int max_kt, cudaStream_t s,
                                bool write_cols) {
  if (tab.n <= 0 || total_items <= 0) return cudaSuccess;
  if (total_items > 0x7fffffffLL) return cudaErrorInvalidValue;
  TraceScope ts("split_verify", s);
  const int wpi = max_kt >= 64 ? 8 : (max_kt >= 32 ? 4 : (max_kt >= 16 ? 2 : 1));
  const int ti = (int)total_items;
  const unsigned blocks = (unsigned)((total_items * wpi + 7) / 8);
  auto kernel = wpi == 8 ? split_verify_kernel<8>
                         : (wpi == 4 ? split_verify_kernel<4>
                                     : (wpi == 2 ? split_verify_kernel<2> : split_verify_kernel<1>));
  return launch_pdl(kernel, blocks, 256, 0, s, tab, map, ti, flags, any, write_cols);
}

}  // namespace mm
