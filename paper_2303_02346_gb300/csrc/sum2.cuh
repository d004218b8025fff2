// Sum of a thread's values to about 48 bits in two FP32 words (Knuth's
// two-sum), for totals whose FP64 adds would otherwise bound a kernel: GB300's
// FP64 rate is a small fraction of its FP32 rate.
#pragma once

#include <cuda_runtime.h>

struct Sum2 {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float v) {
    const float s = __fadd_rn(hi, v), bb = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(v, bb)));
    hi = s;
  }
  // v^2 with the part that its FP32 product drops (exact, by a fused multiply-add)
  __device__ __forceinline__ void add_square(float v) {
    const float q = __fmul_rn(v, v);
    lo = __fadd_rn(lo, __fmaf_rn(v, v, -q));
    add(q);
  }
  __device__ __forceinline__ double value() const { return double(hi) + double(lo); }
};
