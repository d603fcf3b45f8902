// loss.cuh -- the per-row losses of the head kernels.
#pragma once

#include <stdint.h>

namespace tp {

// The 32-bit word of row r's label (an int32 class or an fp32 target); idx: the
// batch's row numbers, or null.  Two dependent loads: the head kernels ask
// for it beside the activations, not once the logits are there.
__device__ __forceinline__ uint32_t row_label(const void* y, const int32_t* idx, int64_t r) {
  return ((const uint32_t*)y)[idx ? (int64_t)idx[r] : r];
}

// Per-row loss and d(mean loss)/d(logits) of one row (fp32); y: row_label.
template <int DO>
__device__ __forceinline__ float row_loss(int task, int d_out, const float (&z)[DO], uint32_t y, float invB,
                                          float (&dl)[DO]) {
  float loss;
  if (task == 1) {  // multiclass: softmax cross-entropy
    const int yv = (int32_t)y;
    float mx = z[0];
#pragma unroll
    for (int c = 1; c < DO; ++c) if (c < d_out) mx = fmaxf(mx, z[c]);
    float s = 0.f;
#pragma unroll
    for (int c = 0; c < DO; ++c) if (c < d_out) s += expf(z[c] - mx);
    const float lse = mx + logf(s);
    float zy = 0.f;
#pragma unroll
    for (int c = 0; c < DO; ++c) {
      if (c == yv) zy = z[c];
      dl[c] = c < d_out ? (expf(z[c] - lse) - (c == yv ? 1.f : 0.f)) * invB : 0.f;
    }
    loss = lse - zy;
  } else if (task == 0) {  // binary: logistic loss on one logit
    const float yv = (float)(int32_t)y;
    const float x = z[0];
    loss = fmaxf(x, 0.f) - x * yv + log1pf(expf(-fabsf(x)));
#pragma unroll
    for (int c = 0; c < DO; ++c) dl[c] = 0.f;
    dl[0] = (1.f / (1.f + expf(-x)) - yv) * invB;
  } else {  // regression: squared error
    const float d = z[0] - __uint_as_float(y);
    loss = d * d;
#pragma unroll
    for (int c = 0; c < DO; ++c) dl[c] = 0.f;
    dl[0] = 2.f * d * invB;
  }
  return loss;
}

}  // namespace tp
