// Generated by paper_2609_09020_gb300/gen_gelu.py -- do not edit.
// Phi(-a) ~= 2^q(-a) on 0 <= a <= 5.8; max |GELU error| in fp32 ~ 5.2e-07.
#pragma once

namespace pic {

constexpr float kGeluZ = 5.800000190734863f;
constexpr float kGeluEps = 3.301103168595887e-09f;  // just above 2^q(-Z)
constexpr int kGeluDeg = 6;

// Coefficients of q, highest degree first (Horner order).
__host__ __device__ constexpr float gelu_c(int i) {
  constexpr float c[] = {
      3.3092816011048853e-05f,
      0.0007692197104915977f,
      0.008080716244876385f,
      0.05341210216283798f,
      -0.4587709605693817f,
      1.1512017250061035f,
      -0.999993085861206f,
  };
  return c[i];
}

}  // namespace pic
