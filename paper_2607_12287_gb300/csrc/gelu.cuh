// GELU of the MLP's up-projection.
#pragma once

#include "internal.h"

namespace ivit {

// Hardware tanh (one MUFU instruction, relative error about 2^-11: below the bf16
// rounding the GELU output gets).
__device__ __forceinline__ float tanh_hw(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// kEpiGelu: gelu_mode 0 tanh form on the hardware's tanh, 1 erf form; kEpiGeluTanhf: the tanh form
// on tanhf.  (An epilogue of its own: a third form behind kEpiGelu's branch made a four-layer
// 224 px full encode 177.8 -> 181.8 us.)
template <int KIND>
__device__ __forceinline__ float gelu_f(float x, int mode) {
  if (KIND == kEpiGelu && mode == 1) return 0.5f * x * (1.f + erff(x * 0.70710678118654752f));
  const float c = 0.79788456080286536f;  // sqrt(2/pi)
  const float u = c * (x + 0.044715f * x * x * x);
  return 0.5f * x * (1.f + (KIND == kEpiGelu ? tanh_hw(u) : tanhf(u)));
}

}  // namespace ivit
