// Sum of a thread's values in three FP32 words, by Knuth's two-sum from word to
// word, for totals whose FP64 adds would otherwise bound a kernel: GB300's FP64
// rate is a small fraction of its FP32 rate. What the third word rounds off is
// below 2^-70 of the summands' magnitudes, so that the sum is as good as rounded
// once to FP64 (a running FP64 sum rounds at every value). Two words keep 48
// bits, fewer than that; the third costs the position loss of 2M particles 15.6 ->
// 17.1 us and the gas sums, bound by memory, nothing. Values and sums have to stay
// finite.
#pragma once

#include <cuda_runtime.h>

struct Sum3 {
  float hi = 0.0f, mid = 0.0f, lo = 0.0f;
  // a + b = s + (what the FP32 sum s drops)
  __device__ static __forceinline__ float two_sum(float& a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    a = s;
    return e;
  }
  __device__ __forceinline__ void add_mid(float v) { lo = __fadd_rn(lo, two_sum(mid, v)); }
  __device__ __forceinline__ void add(float v) { add_mid(two_sum(hi, v)); }
  // v^2 with the part that its FP32 product drops (exact, by a fused multiply-add,
  // while that part is above FP32's smallest number)
  __device__ __forceinline__ void add_square(float v) {
    const float q = __fmul_rn(v, v);
    add(q);
    add_mid(__fmaf_rn(v, v, -q));
  }
  __device__ __forceinline__ double value() const { return double(hi) + (double(mid) + double(lo)); }
};
