// two_float.cuh -- running sums held as two fp32 numbers (h + l, about 48
// bits): fp64 runs at about 1/64 of the fp32 rate on this part.
#pragma once

namespace tp {

// h + l += t
__device__ __forceinline__ void two_add(float& h, float& l, float t) {
  const float s = __fadd_rn(h, t);
  const float b = __fsub_rn(s, h);
  l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, b)), __fsub_rn(t, b)));
  h = s;
}
// h + l += h2 + l2; symmetric in the two sums
__device__ __forceinline__ void two_merge(float& h, float& l, float h2, float l2) {
  const float s = __fadd_rn(h, h2);
  const float b = __fsub_rn(s, h);
  l = __fadd_rn(__fadd_rn(l, l2), __fadd_rn(__fsub_rn(h, __fsub_rn(s, b)), __fsub_rn(h2, b)));
  h = s;
}

}  // namespace tp
