// FP32 sums that keep what each addition rounds off (sm_103a).
#pragma once

#include <cuda_runtime.h>

namespace epic {
namespace {

// hi + lo += v without a rounding in hi's place (Knuth's TwoSum: about 48 bits).
__device__ __forceinline__ void add_kept(float& hi, float& lo, float v) {
  const float s = hi + v, t = s - hi;
  lo += (hi - (s - t)) + (v - t);
  hi = s;
}

}  // namespace
}  // namespace epic
