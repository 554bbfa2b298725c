// Activation functions shared by the GEMM epilogues and the one-launch
// forward, so that both compute bit-identical values.
#pragma once
#include "ptx.cuh"

namespace elasto {

// Coefficients of v below, lowest power first.
constexpr float kGeluB[3] = {-2.3011213394560093f, -0.10677572400312792f, 0.0010142630552981257f};

// GELU, phi in Eq. 5 (the exact x * Phi(x) of the base ViT), in the logistic
// form of the Hendrycks & Gimpel (2016) tanh approximation with one more odd
// term: GELU(x) ~= x / (1 + 2^v), v = -2 log2(e) u(x),
//   u(x) = x (a0 + a1 s + a2 s^2),  s = min(x^2, 36),
// a0..a2 refitted by minimax on [0, 8] (paper_2609_10018_gb300/gelu_fit.py).
// |error| <= 2.52e-5 for every x (the error is even in x, and the clamp keeps
// u increasing past |x| = 6, where the logistic has saturated), against the
// 2^-9 relative rounding of the bf16 output. Two MUFU operations (ex2, rcp)
// and six FMA-pipe operations: the FC1 epilogue is issue-bound, and an
// Abramowitz & Stegun 7.1.26 erf costs about twice as many.
__device__ __forceinline__ float gelu(float x) {
  constexpr float kB0 = -2.3011213394560093f;  // -2 log2(e) a0
  constexpr float kB1 = -0.10677572400312792f;  // -2 log2(e) a1
  constexpr float kB2 = 0.0010142630552981257f;  // -2 log2(e) a2
  static_assert(kB0 == kGeluB[0] && kB1 == kGeluB[1] && kB2 == kGeluB[2], "one set of coefficients");
  const float s = fminf(x * x, 36.0f);
  const float v = x * fmaf(fmaf(kB2, s, kB1), s, kB0);
  return x * rcp_approx(1.0f + ex2_approx(v));
}

// Two values with packed fp32 instructions, bit-identical to two gelu calls:
// 6 packed, 2 min and 4 MUFU instructions instead of 2 x 9.
__device__ __forceinline__ float2 gelu2(float2 x) {
  float2 s = mul2(x, x);
  s = make_float2(fminf(s.x, 36.0f), fminf(s.y, 36.0f));
  const float2 p = fma2(make_float2(kGeluB[2], kGeluB[2]), s, make_float2(kGeluB[1], kGeluB[1]));
  const float2 v = mul2(x, fma2(p, s, make_float2(kGeluB[0], kGeluB[0])));
  const float2 d = add2(make_float2(1.0f, 1.0f), make_float2(ex2_approx(v.x), ex2_approx(v.y)));
  return mul2(x, make_float2(rcp_approx(d.x), rcp_approx(d.y)));
}

}  // namespace elasto
