// Double-FP32 numbers hi + lo (48 significant bits): sums on the FP32 units,
// which GB300 runs at 64 times its FP64 rate.
#pragma once

namespace sg {

struct Df {
  float h, l;
};

// exact sum of two floats as hi + lo (TwoSum, Knuth)
__device__ __forceinline__ Df two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
// a + b with the rounding error gathered in the low word; symmetric in its
// arguments, so a butterfly gives every lane the same bits
__device__ __forceinline__ Df df_add(Df a, Df b) {
  const Df s = two_sum(a.h, b.h);
  return {s.h, __fadd_rn(__fadd_rn(a.l, b.l), s.l)};
}
// a running sum: a += b
__device__ __forceinline__ void df_accumulate(Df& a, float b) {
  const Df s = two_sum(a.h, b);
  a = {s.h, __fadd_rn(a.l, s.l)};
}
__device__ __forceinline__ float df_value(Df a) { return __fadd_rn(a.h, a.l); }

}  // namespace sg
