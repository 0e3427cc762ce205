// The plateau schedule's question, "is the loss below best (1 - threshold)?",
// on FP32 loss sums: an FP64 comparison takes 16 cycles of an SM on GB300.
// Answers only where rounding cannot decide it; the caller asks FP64 there.
#pragma once

namespace dpf {

#ifdef __CUDACC__
#define DPF_HD __host__ __device__ __forceinline__
#else
#define DPF_HD inline
#endif

// Half width of the band left to FP64, relative to the bar.  keep (1 - threshold
// rounded once from FP64) and the product with the best sum are each off by
// 2^-24 of the bar, the band's edges by as much again: below 3e-7.
constexpr float PLATEAU_BAND = 1e-6f;

// The sum that the next improvement has to stay below; < 0: not usable
// (subnormal, overflowing or a threshold of 1 and above).
DPF_HD float plateau_bar(float best_sum, float keep) {
  const float bar = best_sum * keep;
  return bar > 1e-30f && bar < 1e37f ? bar : -1.f;
}
// 1: below the bar, -1: above it, 0: too near to tell (or no bar).
DPF_HD int plateau_side(float sum, float bar) {
  if (!(bar > 0.f)) return 0;
  return sum < bar * (1.f - PLATEAU_BAND) ? 1 : sum > bar * (1.f + PLATEAU_BAND) ? -1 : 0;
}

}  // namespace dpf
