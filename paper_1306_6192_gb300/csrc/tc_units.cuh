// Work units of the persistent tensor-core kernels (tc_gemm.cu, tc_half.cu).
#pragma once

#include "split_common.cuh"

namespace mm {

constexpr int kMaxSplit = 4;  // most K parts of a tail-split tile

// Work unit u of a table: problem g, output tile (mt, nt) = local tile t of
// the problem in raster order (bands of group_m row tiles), and part h of a
// tile split along K (h = -1: the whole tile).
struct UnitCoord {
  int g, mt, nt, t, h;
};

__device__ __forceinline__ UnitCoord decode_unit(const SplitProb *__restrict__ probs, int nprobs,
                                                 const int *__restrict__ map, int u) {
  const int g =
      find_problem(probs, nprobs, map, u, [](const SplitProb &q) { return q.unit_start; });
  const SplitProb &pr = probs[g];
  int t = u - pr.unit_start, h = -1;
  if (pr.split_s > 1 && t >= pr.split_from) {
    const int v = t - pr.split_from;
    t = pr.split_from + v / pr.split_s;
    h = v % pr.split_s;
  }
  const int gm = pr.group_m;
  const int band = gm * pr.nt;
  const int first = (t / band) * gm;
  const int rows = min(pr.mt - first, gm);
  const int in = t % band;
  return UnitCoord{g, first + in % rows, in / rows, t, h};
}

// Pipeline stages [k0, k1) of a unit: all kiters of a whole tile; for part h
// the stages of pack rows [h*kt/S, (h+1)*kt/S), so the split points do not
// depend on the stage depth BKB.
template <int BKB>
__device__ __forceinline__ void unit_krange(const SplitProb &pr, int h, int kiters, int &k0,
                                            int &k1) {
  if (h < 0) {
    k0 = 0;
    k1 = kiters;
    return;
  }
  constexpr int kStagesPerRow = kPackRowBytes / BKB;
  k0 = (int)((int64_t)h * pr.kt / pr.split_s) * kStagesPerRow;
  k1 = min((int)((int64_t)(h + 1) * pr.kt / pr.split_s) * kStagesPerRow, kiters);
}

}  // namespace mm
