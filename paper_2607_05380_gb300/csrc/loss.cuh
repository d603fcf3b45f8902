// loss.cuh -- the per-row losses of the head kernels.
#pragma once

#include <stdint.h>

namespace tp {

// Per-row loss and d(mean loss)/d(logits) of one row (fp32).
template <int DO>
__device__ __forceinline__ float row_loss(int task, int d_out, const float (&z)[DO], const void* y, int64_t row,
                                          float invB, float (&dl)[DO]) {
  float loss;
  if (task == 1) {  // multiclass: softmax cross-entropy
    const int yv = ((const int32_t*)y)[row];
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
    const float yv = (float)((const int32_t*)y)[row];
    const float x = z[0];
    loss = fmaxf(x, 0.f) - x * yv + log1pf(expf(-fabsf(x)));
#pragma unroll
    for (int c = 0; c < DO; ++c) dl[c] = 0.f;
    dl[0] = (1.f / (1.f + expf(-x)) - yv) * invB;
  } else {  // regression: squared error
    const float d = z[0] - ((const float*)y)[row];
    loss = d * d;
#pragma unroll
    for (int c = 0; c < DO; ++c) dl[c] = 0.f;
    dl[0] = 2.f * d * invB;
  }
  return loss;
}

}  // namespace tp
