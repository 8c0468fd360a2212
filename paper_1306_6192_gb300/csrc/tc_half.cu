// Tensor-core kernel of the kTcSplitF16x3 kind (FP32 in/out, short inner
// dimensions): C = A.B from two fp16 parts per operand (split_prep.cu)
//     C_ij = 2^-(ea + eb) (sum_r (Ah Bh)_irj + 2^-11 sum_r (Ah Bl + Al Bh)_irj)
// with Bl, Al the parts scaled by 2^11; the products of the two low parts,
// below 2^-22 of a term (2^-18 at the window's low end, split_prep.cu), are dropped.
// A product whose magnitudes do not fit fp16, or with m <= 16, was packed as three bf16 parts and runs here as the six products of
// tc_gemm.cu's three-part kind (hx, SplitProb): one launch serves both.
//
// Why this form.  Six bf16 products were the bound of every product with a
// short inner dimension (m < 2237): 128 x 128 x 64 took 24 MMAs of N = 128.
// Three fp16 products halve them, and the two that share Ah run as ONE MMA of
// N = 256 against [Bh | Bl], which lie next to each other in the pack, into
// [main | low] accumulators that lie next to each other in tensor memory; the
// low accumulator keeps its own scale until the epilogue adds the two.  A
// 128 x 128 tile then holds 256 columns, so two tiles fit tensor memory and a
// tile's epilogue runs beside the next one's MMAs.  The main accumulator
// takes a sixth of the additions of the bf16 form.  The tensor cores' FP32 sums
// are not rounded to nearest, so a long sum of one sign drifts; every 512 K (256
// for products that the fused kernel's shorter sums served before; chunk, K
// blocks) the accumulator is therefore handed to the epilogue warps, which add the
// chunks in registers with round-to-nearest additions beside the next chunk's
// MMAs (2048^3, max error over |A||B|: signed entries 1.2e-7 against 2.0e-6 for the
// six bf16 products, entries in [0, 1) 3.0e-6 against 1.2e-5).
//
// Structure (persistent, one CTA per SM, 384 threads; the epilogue's two
// warpgroups take the registers that the first one gives back, 224 a thread
// against 56: at the launch's 168 its sums spilled, and beside 226 KB of shared
// memory the spills miss L1):
//   warp 0     TMEM allocation; lane 0 issues the TMA loads of each K block
//              (64 K: A's two parts, 256 pack rows of 128 bytes, and B's;
//              three-part products 32 K: six boxes of 128 x 64 bytes) into a
//              3-stage ring
//   warp 1     lane 0 issues the MMAs
//   warp 2     decodes the CTA's work units, 32 at a time, into a ring of
//              descriptors in shared memory, so that no role waits for the
//              chain unit list -> map -> table -> state words between tiles
//   warp 3     of the first CTA clears the words of the call before (ctx.h)
//   warps 4-11 epilogue: warp w reads lane quarter w & 3 and 64 of the 128
//              columns: both accumulators, their sum, the exact unscaling; the
//              accumulators go back to the MMAs before anything is stored.
//              C 32-byte aligned with p % 8 == 0: a lane stores its row in
//              whole 32-byte sectors, straight from registers; else 32 x 32
//              blocks turned in shared memory and stored a row at a time.  For
//              C = alpha (A.B) + beta D, D's blocks come by TMA, the next one
//              while this one is combined and stored (read by the lanes in
//              sectors, D took the 8192 x 512 x 8192 update from 176 to 261 us:
//              a warp's load touches 32 rows).
//
// Measured on GB300 (kernel times from the library's tracer): 8192 x 512 x 8192
// 153 us (six bf16 products: 305 for the call), with D 176 (395 before);
// 2048^3 43 us; 1024 uneven products of 32..1024 (0.29 TFLOP) 806 us (1916).  At
// 8192 x 2048 x 8192 the tensor cores set the time: 528 useful TFLOP/s, 86% of
// the measured bf16 rate over three products, at the power-capped clock.  A
// variant on CTA pairs (256 x 128 tiles, cta_group::2) read a quarter less from
// L2 but was no faster there (538 against 536 us) and slower on small products
// (2048^3 50 us), whose tiles it doubles.
// Tail-split units as in tc_gemm.cu.  Every wait is bounded; on expiry the
// error flag is set, the other roles stop at their next wait, and copies and
// MMAs in flight are drained before TMEM is freed.
#include <cuda.h>

#include <algorithm>

#include "ctx.h"
#include "tc_ptx.cuh"
#include "tc_units.cuh"

namespace mm {
namespace {

using namespace tcx;

constexpr int kBN = 128;                 // N tile
constexpr int kStages = 3;
constexpr int kPart = 128 * 128;         // a part of an operand: 128 rows x 128 bytes
constexpr int kStageBytes = 4 * kPart;   // A hi, A lo, B hi, B lo
constexpr int kPart6 = 128 * 64;         // three-part form: 64 bytes of K
constexpr int kStageBytes6 = 6 * kPart6;
static_assert(kStageBytes6 <= kStageBytes, "the three-part form fits the stage");
constexpr int kAccs = 2, kAccCols = 256;
constexpr int kUnits = 4;                // descriptor ring
constexpr int kEpiWarps = kHalfSplitCnt, kEpiThreads = 32 * kEpiWarps;
constexpr int kFirstEpi = 4;             // whole warpgroups share registers
constexpr int kThreads = 32 * kFirstEpi + kEpiThreads;
constexpr int kEpiRegs = 224, kRoleRegs = 56;
static_assert(kEpiThreads * kEpiRegs + 128 * kRoleRegs <= kThreads * 168, "registers of the launch");
constexpr uint64_t kWaitNs = 4000000000ull;
constexpr uint64_t kDrainNs = 200000000ull;

// What the roles need of one work unit.
struct __align__(16) Unit {
  float *C;
  const float *D;
  const uint32_t *sA, *tB;
  float *part;        // split tiles: the tile's first partial slot, else null
  int *cnt;
  int32_t arow, brow;  // first pack rows
  int32_t k0, k1;      // stages; k1 < 0: no more units
  int32_t x6, ex;      // three-part form; fp16 form: exponent of the result
  int32_t n, p, row0, col0;
  int32_t flags, vec8, split_s, h, epi_on, chunk;
  float alpha, beta;
};
static_assert(sizeof(Unit) <= 128, "descriptor slot");

struct Lay {
  static constexpr int kStgOff = kStages * kStageBytes;       // 32 x 32 FP32 per epilogue warp
  static constexpr int kUnitOff = kStgOff + kEpiWarps * 4096;
  static constexpr int kColOff = kUnitOff + kUnits * 128;     // column exponents, per epilogue warp
  static constexpr int kBarOff = kColOff + kEpiWarps * 64 * 2;
  // full[S], empty[S], acc full[A], acc empty[A], unit full[U], unit empty[U],
  // D full[epilogue warps], drain
  static constexpr int kNumBars = 2 * kStages + 2 * kAccs + 2 * kUnits + kEpiWarps + 1;
  static constexpr int kMiscOff = kBarOff + kNumBars * 8;
  static constexpr int kSmem = kMiscOff + 32 + 1024;          // + alignment slack
};
static_assert(Lay::kSmem + sizeof(SplitProb) <= 232448, "shared memory budget");

// mbar_wait with its slow path in line: a call would spill the epilogue's sums
// around it.
__device__ __forceinline__ bool epi_wait(uint32_t bar, uint32_t parity, int *err, int code,
                                         bool watch_err = true, uint64_t limit_ns = kWaitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 63u) == 0) {
      if (watch_err && *(volatile int *)err != 0) return false;
      if (globaltimer_ns() - t0 > limit_ns) {
        atomicCAS(err, 0, code);
        return false;
      }
    }
  }
}

// Instruction descriptor: FP32 accumulators, K-major fp16 (fmt 0) or bf16
// (fmt 1) operands, M = 128.
__device__ __forceinline__ uint32_t idesc_f16(uint32_t fmt, int bn) {
  return (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(kTcBM >> 4) << 24);
}

__global__ void __launch_bounds__(kThreads, 1)
tc_half_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap map6,
               const __grid_constant__ CUtensorMap map_d,
               const __grid_constant__ ProbTable tab, const int *__restrict__ unit_map,
               const int *__restrict__ flags, int total_units, const int *__restrict__ order, ClearWords clear,
               int *err) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t sbase = (raw + 1023u) & ~1023u;
  uint8_t *smem = smem_raw + (sbase - raw);
  const uint32_t bars = sbase + Lay::kBarOff;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (kStages + s); };
  auto accf_bar = [&](int a) { return bars + 8u * (2 * kStages + a); };
  auto acce_bar = [&](int a) { return bars + 8u * (2 * kStages + kAccs + a); };
  auto unitf_bar = [&](int u) { return bars + 8u * (2 * kStages + 2 * kAccs + u); };
  auto unite_bar = [&](int u) { return bars + 8u * (2 * kStages + 2 * kAccs + kUnits + u); };
  auto dfull_bar = [&](int w) { return bars + 8u * (2 * kStages + 2 * kAccs + 2 * kUnits + w); };
  const uint32_t drain_bar = bars + 8u * (2 * kStages + 2 * kAccs + 2 * kUnits + kEpiWarps);
  uint32_t *tmem_holder = reinterpret_cast<uint32_t *>(smem + Lay::kMiscOff);
  Unit *units = reinterpret_cast<Unit *>(smem + Lay::kUnitOff);
  auto unit_at = [&](int u) { return reinterpret_cast<Unit *>(reinterpret_cast<uint8_t *>(units) + 128 * u); };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ SplitProb shared_one;
  const SplitProb *probs = table_products(tab, &shared_one);
  const int nprobs = tab.n;

  if (warp == 0) {
    tmem_alloc(smem_u32(tmem_holder), kAccs * kAccCols);
    tmem_relinquish();
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < kStages; s++) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    for (int a = 0; a < kAccs; a++) {
      mbar_init(accf_bar(a), 1);
      mbar_init(acce_bar(a), kEpiWarps);
    }
    for (int u = 0; u < kUnits; u++) {
      mbar_init(unitf_bar(u), 1);
      mbar_init(unite_bar(u), 2 + kEpiWarps);  // producer, MMA issuer, epilogue warps
    }

    for (int w = 0; w < kEpiWarps; w++) mbar_init(dfull_bar(w), 1);
    mbar_init(drain_bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *reinterpret_cast<volatile uint32_t *>(tmem_holder);
  // the set-up above may run beside the end of the stream's previous kernel
  pdl_wait();

  if (warp < kFirstEpi) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRoleRegs));
    if (warp == 0) {
      if (lane == 0) {
        // ------------------------------------------------------ TMA producer
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map)) : "memory");
        int stage = 0, us = 0;
        uint32_t phase = 0, uphase = 0, issued = 0;
        bool ok = true;
        while (ok) {
          if (!mbar_wait(unitf_bar(us), uphase, err, 31, true, kWaitNs)) break;
          const Unit *d = unit_at(us);
          const int k0 = d->k0, k1 = d->k1, x6 = d->x6, arow = d->arow, brow = d->brow;
          mbar_arrive(unite_bar(us));
          if (++us == kUnits) us = 0, uphase ^= 1u;
          if (k1 < 0) break;
          for (int ki = k0; ki < k1; ki++) {
            if (!mbar_wait(empty_bar(stage), phase ^ 1u, err, 31, true, kWaitNs)) {
              ok = false;
              break;
            }
            ++issued;
            const uint32_t st = sbase + (uint32_t)(stage * kStageBytes);
            if (!x6) {
              // a tile's two parts of a K block are 256 consecutive pack rows
              mbar_arrive_expect_tx(full_bar(stage), kStageBytes);
              tma_load_2d(st, &map, 0, arow + ki * 256, full_bar(stage));
              tma_load_2d(st + 2 * kPart, &map, 0, brow + ki * 256, full_bar(stage));
            } else {
              mbar_arrive_expect_tx(full_bar(stage), kStageBytes6);
              const int x = (ki & 1) * 64, a = arow + (ki >> 1) * 384, b = brow + (ki >> 1) * 384;
#pragma unroll
              for (int q = 0; q < 3; q++) {
                tma_load_2d(st + q * kPart6, &map6, x, a + 128 * q, full_bar(stage));
                tma_load_2d(st + (3 + q) * kPart6, &map6, x, b + 128 * q, full_bar(stage));
              }
            }
            if (++stage == kStages) stage = 0, phase ^= 1u;
          }
        }
        if (*reinterpret_cast<volatile int *>(err) != 0) {
          // copies in flight must land before the shared memory goes away
          for (uint32_t j = issued > kStages ? issued - kStages : 0; j < issued; j++)
            mbar_wait(full_bar((int)(j % kStages)), (j / kStages) & 1u, err, 31, false, kDrainNs);
        }
      }
    } else if (warp == 1) {
      if (lane == 0) {
        // ------------------------------------------------------ MMA issuer
        int stage = 0, us = 0, acc = 0;
        uint32_t phase = 0, uphase = 0, aphase = 0;
        bool ok = true, issued = false;
        while (ok) {
          if (!mbar_wait(unitf_bar(us), uphase, err, 32, true, kWaitNs)) {
            ok = false;
            break;
          }
          const Unit *d = unit_at(us);
          const int k0 = d->k0, k1 = d->k1, x6 = d->x6, in_chunk = d->chunk - 1;
          mbar_arrive(unite_bar(us));
          if (++us == kUnits) us = 0, uphase ^= 1u;
          if (k1 < 0) break;
          uint32_t t0 = 0;
          for (int ki = k0; ki < k1; ki++) {
            const bool first = ((ki - k0) & in_chunk) == 0;
            if (first) {
              // the accumulator of the last chunk goes to the epilogue
              if (ki != k0) {
                tc_commit(accf_bar(acc));
                if (++acc == kAccs) acc = 0, aphase ^= 1u;
              }
              if (!mbar_wait(acce_bar(acc), aphase ^ 1u, err, 32, true, kWaitNs)) {
                ok = false;
                break;
              }
              t0 = tmem_base + (uint32_t)(acc * kAccCols);
            }
            if (!mbar_wait(full_bar(stage), phase, err, 33, true, kWaitNs)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t st = sbase + (uint32_t)(stage * kStageBytes);
            if (!x6) {
              const uint64_t ah = kmajor_desc<128>(st), al = kmajor_desc<128>(st + kPart);
              const uint64_t b = kmajor_desc<128>(st + 2 * kPart);  // hi rows, then lo rows
#pragma unroll
              for (int kk = 0; kk < 4; kk++) {  // 16 fp16 = 32 bytes of K per MMA
                const uint64_t adv = (uint64_t)(kk * 32) >> 4;
                tc_mma(t0, ah + adv, b + adv, idesc_f16(0, 256), (!first || kk != 0) ? 1u : 0u);
                tc_mma(t0 + kBN, al + adv, b + adv, idesc_f16(0, 128), 1u);
              }
            } else {
              const uint32_t id = idesc_f16(1, 128);
#pragma unroll
              for (int kk = 0; kk < 2; kk++) {
                const uint64_t adv = (uint64_t)(kk * 32) >> 4;
                const uint64_t a0 = kmajor_desc<64>(st) + adv, a1 = kmajor_desc<64>(st + kPart6) + adv;
                const uint64_t a2 = kmajor_desc<64>(st + 2 * kPart6) + adv;
                const uint64_t b0 = kmajor_desc<64>(st + 3 * kPart6) + adv;
                const uint64_t b1 = kmajor_desc<64>(st + 4 * kPart6) + adv;
                const uint64_t b2 = kmajor_desc<64>(st + 5 * kPart6) + adv;
                // hi, mid, lo: the products of relative size >= 2^-16, smallest first
                tc_mma(t0, a1, b1, id, (!first || kk != 0) ? 1u : 0u);
                tc_mma(t0, a0, b2, id, 1u);
                tc_mma(t0, a2, b0, id, 1u);
                tc_mma(t0, a0, b1, id, 1u);
                tc_mma(t0, a1, b0, id, 1u);
                tc_mma(t0, a0, b0, id, 1u);
              }
            }
            issued = true;
            tc_commit(empty_bar(stage));
            if (++stage == kStages) stage = 0, phase ^= 1u;
          }
          if (!ok) break;
          tc_commit(accf_bar(acc));
          if (++acc == kAccs) acc = 0, aphase ^= 1u;
        }
        if (!ok && issued) {
          // wait for MMAs in flight before TMEM is released
          tc_commit(drain_bar);
          mbar_wait(drain_bar, 0, err, 33, false, kDrainNs);
        }
      }
    } else if (warp == 2) {
      // -------------------------------------------------------- unit decoder
      // this CTA's units: the host's list (grid + 1 offsets, then the units), or
      // units c, c + grid, ...
      const int *ulist = order ? order + gridDim.x + 1 : nullptr;
      const int i_first = order ? order[blockIdx.x] : (int)blockIdx.x;
      const int i_end = order ? order[blockIdx.x + 1] : total_units;
      const int i_step = order ? 1 : (int)gridDim.x;
      const int count = i_first < i_end ? (i_end - i_first + i_step - 1) / i_step : 0;
      bool ok = true;
      for (int j0 = 0; j0 <= count && ok; j0 += 32) {
        const int j = j0 + lane;  // the entry after the last one ends the roles
        Unit d;
        d.k0 = 0;
        d.k1 = -1;
        if (j < count) {
          const int ui = i_first + j * i_step;
          const UnitCoord tc = decode_unit(probs, nprobs, unit_map, ulist ? ulist[ui] : ui);
          const SplitProb &pr = probs[tc.g];

          const int x6 = pr.hx[kHalfX6] | pr.hx[kHalfBad];
          const int rows = x6 ? 384 : 256;  // pack rows of a tile and K block
          d.x6 = x6;
          d.ex = -(pr.hx[kHalfExpA] + pr.hx[kHalfExpB]);
          d.arow = (int)(pr.a_row0 + (int64_t)tc.mt * pr.kt * rows);
          d.brow = (int)(pr.b_row0 + (int64_t)tc.nt * pr.kt * rows);
          if (x6) unit_krange<64>(pr, tc.h, (int)(((int64_t)pr.m * 2 + 63) / 64), d.k0, d.k1);
          else unit_krange<128>(pr, tc.h, pr.kt, d.k0, d.k1);
          d.C = pr.C;
          d.D = pr.epi.D;
          d.sA = pr.sA;
          d.tB = pr.tB;
          d.split_s = pr.split_s;
          // three parts, in stages of 32 K: one sum over K, as tc_gemm.cu's, or every
          // 64 K for products that the fused kernel served (magnitudes over many
          // binades, 1024^3: error 3.7e-6 in one sum, 2.6e-7 in the fused kernel's)
          d.chunk = !x6 ? pr.chunk : (pr.chunk < kHalfChunk ? 2 : 1 << 30);
          d.h = tc.h;
          const int st = tc.t - pr.split_from;
          d.part = tc.h >= 0 ? pr.part + (size_t)st * pr.split_s * (kTcBM * kBN) : nullptr;
          d.cnt = tc.h >= 0 ? pr.cnt + st * kHalfSplitCnt : nullptr;
          d.n = pr.n;
          d.p = pr.p;
          d.row0 = tc.mt * kTcBM;
          d.col0 = tc.nt * kBN;
          d.flags = x6 ? (flags ? flags[tc.g] : (kFlagScaleA | kFlagScaleB)) : 0;
          d.vec8 = (reinterpret_cast<uintptr_t>(pr.C) & 31u) == 0 && (pr.p & 7) == 0 &&
                   (pr.epi.on != 2 || (reinterpret_cast<uintptr_t>(pr.epi.D) & 15u) == 0);
          d.epi_on = pr.epi.on;
          d.alpha = pr.epi.alpha;
          d.beta = pr.epi.beta;
        }
        for (int t = 0; t < 32 && j0 + t <= count && ok; t++) {
          const int us = (j0 + t) % kUnits;
          const uint32_t par = (uint32_t)((j0 + t) / kUnits) & 1u;
          // the whole warp waits, so that it leaves together
          ok = __all_sync(0xffffffffu, mbar_wait(unite_bar(us), par ^ 1u, err, 34, true, kWaitNs));
          if (ok && lane == t) {
            *unit_at(us) = d;
            mbar_arrive(unitf_bar(us));
          }
          __syncwarp();
        }
      }
    } else if (blockIdx.x == 0) {
      clear_words(clear, lane, 32);
    }
  } else {
    // -------------------------------------------------------- epilogue
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kEpiRegs));
    const int q = warp & 3;                   // TMEM lane quarter this warp may access
    const int ch = (warp - kFirstEpi) >> 2;   // column half of the tile
    const int row = q * 32 + lane;
    float *buf = reinterpret_cast<float *>(smem + Lay::kStgOff + (warp - kFirstEpi) * 4096);
    int us = 0, acc = 0;
    uint32_t uphase = 0, aphase = 0;
    uint32_t dphase = 0;
    bool d_asked = false;  // D's first block of the coming unit is on its way
    bool d_out = false;    // a block of D is on its way
    // D's 32 columns cc of this warp's rows of a unit into its staging area (the
    // one block of it that was there has been read by every lane)
    auto ask_d = [&](const Unit *u, int cc) {
      const int i = u->row0 + q * 32, j = u->col0 + ch * 64 + cc * 32;
      d_out = i < u->n && j < u->p;
      if (lane == 0 && d_out) {
        mbar_arrive_expect_tx(dfull_bar(warp - kFirstEpi), 4096u);
        tma_load_2d(smem_u32(buf), &map_d, j, i, dfull_bar(warp - kFirstEpi));
      }
    };
    for (;;) {
      if (!__all_sync(0xffffffffu, epi_wait(unitf_bar(us), uphase, err, 35))) break;
      const Unit *d = unit_at(us);
      if (d->k1 < 0) break;
      const int n = d->n, p = d->p, x6 = d->x6, h = d->h, split_s = d->split_s, epi_on = d->epi_on;
      const int row0 = d->row0 + q * 32, col0 = d->col0;
      const int chunks = (d->k1 - d->k0 + d->chunk - 1) / d->chunk;
      // whole 32-byte sectors: C (and D) 32-byte aligned, p % 8 == 0
      const bool vec8 = d->vec8 != 0;
      const bool vec_d = vec8 && epi_on == 2;
      const int64_t at0 = (int64_t)(row0 + lane) * p + col0 + ch * 64;  // this row's 64 entries
      const int left = row0 + lane < n ? p - (col0 + ch * 64) : 0;     // of them inside the matrix
      float pre[64];  // sum of this thread's 64 columns over the chunks before the last
      if (vec_d && h < 0 && !d_asked) ask_d(d, 0);
      d_asked = false;
      int16_t *cexp = reinterpret_cast<int16_t *>(smem + Lay::kColOff) + 64 * (warp - kFirstEpi);
      if (x6) {
        __syncwarp();
        for (int c = lane; c < 64; c += 32) {
          const int j = col0 + ch * 64 + c;
          cexp[c] = (int16_t)((j < p && (d->flags & kFlagScaleB)) ? scale_exponent(d->tB[j]) : 0);
        }
        __syncwarp();
      }
      // 32 columns of the accumulator pair at column c of the tile
      auto load_acc = [&](int c, uint32_t (&v)[32]) {
        const uint32_t tacc = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * kAccCols);
        __syncwarp();  // tcgen05.ld is warp-collective: reconverge first
        tmem_ld_32x32b_x32(tacc + (uint32_t)c, v);
        if (!x6) {
          uint32_t w[32];
          tmem_ld_32x32b_x32(tacc + (uint32_t)(kBN + c), w);
          tmem_ld_wait();
#pragma unroll
          for (int e = 0; e < 32; e++)
            v[e] = __float_as_uint(fmaf(__uint_as_float(w[e]), 0x1p-11f, __uint_as_float(v[e])));
        } else {
          tmem_ld_wait();
        }
      };
      auto release_acc = [&] {  // this warp has read the accumulators
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce_bar(acc));
      };
      bool ok = true;
      for (int t = 0; t + 1 < chunks; t++) {
        ok = __all_sync(0xffffffffu, epi_wait(accf_bar(acc), aphase, err, 36));
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < 64; c += 32) {
          uint32_t v[32];
          load_acc(ch * 64 + c, v);
#pragma unroll
          for (int e = 0; e < 32; e++)
            pre[c + e] = t == 0 ? __uint_as_float(v[e]) : pre[c + e] + __uint_as_float(v[e]);
        }
        release_acc();
        if (++acc == kAccs) acc = 0, aphase ^= 1u;
      }
      ok = __all_sync(0xffffffffu, ok && epi_wait(accf_bar(acc), aphase, err, 36));
      if (!ok) break;
      tc_fence_after();
      const int si = !x6 ? d->ex
                         : ((row0 + lane < n && (d->flags & kFlagScaleA)) ? scale_exponent(d->sA[row0 + lane])
                                                                         : 0);
      // all 64 columns out of tensor memory first: the accumulator is free for
      // the MMAs while this tile is combined and stored
      float x[64];
#pragma unroll
      for (int c = 0; c < 64; c += 32) {
        uint32_t v[32];
        load_acc(ch * 64 + c, v);
#pragma unroll
        for (int e = 0; e < 32; e++)
          x[c + e] = chunks > 1 ? pre[c + e] + __uint_as_float(v[e]) : __uint_as_float(v[e]);
      }
      release_acc();

      // a split tile's parts: slots of 32 groups of 4 columns, each group 128
      // rows x 4 floats, so that a warp's 16-byte accesses to one group are
      // 512 consecutive bytes; the part that counts last adds all of them
      bool store = true;
      if (h >= 0) {
        constexpr size_t kSlot = (size_t)kTcBM * kBN;
        float4 *slots = reinterpret_cast<float4 *>(d->part) + (size_t)(ch * 16) * kTcBM + row;
#pragma unroll
        for (int k = 0; k < 16; k++)
          __stcg(slots + (size_t)h * (kSlot / 4) + (size_t)k * kTcBM,
                 make_float4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3]));
        __threadfence();
        __syncwarp();  // this warp's block of the part written and fenced
        int last = 0;
        int *cnt = d->cnt + (warp - kFirstEpi);
        if (lane == 0) last = atomicAdd(cnt, 1) == split_s - 1;
        store = __shfl_sync(0xffffffffu, last, 0) != 0;
        if (store) {
          __threadfence();
          // the parts in order 0..split_s-1 (this part's from its registers)
#pragma unroll
          for (int k = 0; k < 16; k++) {
            float4 y[kMaxSplit];
#pragma unroll
            for (int hh = 0; hh < kMaxSplit; hh++)
              if (hh < split_s)
                y[hh] = hh == h ? make_float4(x[4 * k], x[4 * k + 1], x[4 * k + 2], x[4 * k + 3])
                                : __ldcg(slots + (size_t)hh * (kSlot / 4) + (size_t)k * kTcBM);
            float4 sum = y[0];
#pragma unroll
            for (int hh = 1; hh < kMaxSplit; hh++)
              if (hh < split_s) {
                sum.x += y[hh].x;
                sum.y += y[hh].y;
                sum.z += y[hh].z;
                sum.w += y[hh].w;
              }
            x[4 * k] = sum.x;
            x[4 * k + 1] = sum.y;
            x[4 * k + 2] = sum.z;
            x[4 * k + 3] = sum.w;
          }
        }
      }
#pragma unroll
      for (int e0 = 0; e0 < 64; e0 += 32) {
        if (x6) {
#pragma unroll
          for (int e = e0; e < e0 + 32; e++) x[e] = scale_pow2(x[e], si + cexp[e]);
        } else if (si >= -126 && si <= 127) {
          const float f = __int_as_float((si + 127) << 23);
#pragma unroll
          for (int e = e0; e < e0 + 32; e++) x[e] *= f;
        } else {
          // 2^si beyond the normal range: two exact steps, the second of which
          // rounds once (|si| <= 200)
          const int s1 = si < 0 ? -126 : 127;
          const float f = __int_as_float((s1 + 127) << 23), g = __int_as_float((si - s1 + 127) << 23);
#pragma unroll
          for (int e = e0; e < e0 + 32; e++) x[e] = (x[e] * g) * f;
        }
      }
      if (vec8 && store) {
        const float al = d->alpha, be = d->beta;
        if (vec_d && h >= 0) ask_d(d, 0);
        bool d_ok = true;
#pragma unroll
        for (int cc = 0; cc < 2; cc++) {
          if (epi_on == 2) {
            if (row0 < n && col0 + ch * 64 + cc * 32 < p) {
              d_ok = __all_sync(0xffffffffu, epi_wait(dfull_bar(warp - kFirstEpi), dphase, err, 36));
              if (!d_ok) break;
              dphase ^= 1u;
              d_out = false;
            }
            // 16-byte chunk k of row `lane` at chunk k ^ (lane & 7) (the map's
            // 128-byte swizzle)
            const float4 *rowp = reinterpret_cast<const float4 *>(buf + lane * 32);
#pragma unroll
            for (int k = 0; k < 8; k++) {
              const float4 y = rowp[k ^ (lane & 7)];
              float *z = &x[cc * 32 + 4 * k];
              z[0] = fmaf(al, z[0], be * y.x);
              z[1] = fmaf(al, z[1], be * y.y);
              z[2] = fmaf(al, z[2], be * y.z);
              z[3] = fmaf(al, z[3], be * y.w);
            }
            __syncwarp();
            if (cc == 0) {
              ask_d(d, 1);
            } else if (h < 0) {
              // the next unit's first block, while this one is stored
              const int un = us + 1 == kUnits ? 0 : us + 1;
              d_ok = __all_sync(0xffffffffu, epi_wait(unitf_bar(un), un ? uphase : uphase ^ 1u, err, 35));
              if (!d_ok) break;
              const Unit *u = unit_at(un);
              d_asked = u->k1 >= 0 && u->h < 0;
              if (d_asked) ask_d(u, 0);
            }
          } else if (epi_on == 1) {
#pragma unroll
            for (int e = cc * 32; e < cc * 32 + 32; e++) x[e] = al * x[e];
          }
#pragma unroll
          for (int k = cc * 4; k < cc * 4 + 4; k++)
            if (8 * k < left) store8(d->C + at0 + 8 * k, &x[8 * k]);
        }
        if (!d_ok) break;
      }
#pragma unroll
      for (int cc = 0; cc < 2; cc++) {
        const int j0 = col0 + ch * 64 + cc * 32;
        if (vec8 || !store || j0 >= p) continue;  // the same for the whole warp
        // entry e of row `lane` at e ^ lane, conflict-free both ways; then the
        // block row by row, each store 32 consecutive columns of one row
#pragma unroll
        for (int e = 0; e < 32; e++) buf[lane * 32 + (e ^ lane)] = x[cc * 32 + e];
        __syncwarp();
        const int j = j0 + lane;
        if (j < p) {
          float *dst = d->C + (int64_t)row0 * p + j;
          const int left = n - row0, rows = left < 32 ? left : 32;
          if (epi_on == 0) {
#pragma unroll 8
            for (int r = 0; r < rows; r++, dst += p) __stcs(dst, buf[r * 32 + (lane ^ r)]);
          } else {
            // sixteen rows at a time: their values of D are loaded before any
            // of them is stored (D may be C)
            const float al = d->alpha, be = d->beta;
            const float *dcol = d->D + (int64_t)row0 * p + j;
#pragma unroll
            for (int hh = 0; hh < 32; hh += 16) {
              float dv[16];
#pragma unroll
              for (int r = 0; r < 16; r++)
                dv[r] = (epi_on == 2 && hh + r < rows) ? dcol[(int64_t)(hh + r) * p] : 0.f;
#pragma unroll
              for (int r = 0; r < 16; r++)
                if (hh + r < rows) {
                  const float x = buf[(hh + r) * 32 + (lane ^ (hh + r))];
                  __stcs(dst + (int64_t)(hh + r) * p, epi_on == 2 ? fmaf(al, x, be * dv[r]) : al * x);
                }
            }
          }
        }
        __syncwarp();
      }

      __syncwarp();
      if (lane == 0) mbar_arrive(unite_bar(us));
      if (++us == kUnits) us = 0, uphase ^= 1u;
      if (++acc == kAccs) acc = 0, aphase ^= 1u;
    }
    // left early: a copy in flight must land before the shared memory goes away
    if (d_out) epi_wait(dfull_bar(warp - kFirstEpi), dphase, err, 36, false, kDrainNs);
    __syncwarp();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kAccs * kAccCols);
  }
}

}  // namespace

cudaError_t launch_tc_half(const ProbTable &tab, int total_units,
                           const int *unit_map, const int *flags, void *pack_base,
                           int64_t pack_rows, int grid, int *d_err, cudaStream_t s,
                           const int *order, ClearWords clear) {
  // one CTA per SM: the kernel allocates all 512 TMEM columns
  static_assert(2 * Lay::kSmem > 232448, "must not fit twice on one SM");
  static std::once_flag once;
  static cudaError_t attr_err = cudaSuccess;
  std::call_once(once, [] {
    attr_err = cudaFuncSetAttribute(tc_half_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Lay::kSmem);
  });
  if (attr_err != cudaSuccess) return attr_err;
  CUtensorMap map, map6, map_d = {};
  cudaError_t e = encode_pack_map(&map, pack_base, pack_rows, 128, 256);
  if (e == cudaSuccess) e = encode_pack_map(&map6, pack_base, pack_rows, 64, 128);
  // (only a product of its own has an epilogue)
  const SplitProb &one = tab.one;
  if (e == cudaSuccess && tab.dev == nullptr && one.epi.on == 2 && tc_c_map_ok(one.epi.D, one.n, one.p))
    e = encode_c_map(&map_d, const_cast<float *>(one.epi.D), one.n, one.p);
  if (e != cudaSuccess) return e;
  TraceScope ts("split_tc", s);
  return launch_pdl(tc_half_kernel, (unsigned)grid, kThreads, Lay::kSmem, s, map, map6, map_d, tab, unit_map,
                    flags, total_units, order, clear, d_err);
}

}  // namespace mm
