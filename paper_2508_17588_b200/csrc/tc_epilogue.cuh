// What the epilogues of the tensor-core kernels share: the activation and where a row goes.
#pragma once

#include "hero_internal.h"

namespace hero {
namespace tc {

__device__ __forceinline__ float gelu_tanh_f(float t) {
  // 0.5 t (1 + tanh(sqrt(2/pi) (t + 0.044715 t^3))) with the hardware tanh (one special-function
  // instruction, relative error 2^-11: below the bf16 rounding of the result).  The epilogue shares the
  // SM's power budget with the tensor core, so every instruction saved here is tensor clock gained.
  const float t2 = t * t;
  const float u = t * fmaf(0.0356774081f, t2, 0.7978845608f);
  float th;
  asm("tanh.approx.f32 %0, %1;" : "=f"(th) : "f"(u));
  const float h = 0.5f * t;
  return fmaf(h, th, h);
}

// Where one accumulator row goes.
struct RowOut {
  bool ok;                 // the row exists
  int m, b;                // row of the compact operand, its batch item
  long long scat;          // its row in a [B, n_rows] destination
};
__device__ __forceinline__ RowOut row_out(const GemmOut& out, int m, int M) {
  RowOut r;
  r.ok = m < M;
  r.m = m; r.b = 0; r.scat = 0;
  if (r.ok) {
    r.b = m / out.n_sel;
    const int li = m - r.b * out.n_sel;
    r.scat = (long long)r.b * out.n_rows + (out.idx ? __ldg(out.idx + li) : li);
  }
  return r;
}

}  // namespace tc
}  // namespace hero
