// Logistic sigmoids of the GEMM epilogues, s(z) = 1 / (1 + e^-z).  Error bounds against 64 bits
// below, with u = 2^-24; tests/test_gpu_arithmetic.py holds all three to them over every float.
#pragma once

// From the hardware exponential and fast division.  The error budget of the BF16 path is set by
// its bf16 operands (unit roundoff 2^-8).  e^-z = inf for z < -88 gives 0, the correct limit.
// Relative error up to z = -87: (2.35 |z| + 4) u from the exponential, u from the sum, 4 u from
// the division.
__device__ __forceinline__ float sigm_fast(float z) { return __fdividef(1.f, 1.f + __expf(-z)); }

// s(z) = 1 / (1 + 2^(-z log2 e)) on the flush-to-zero units: two thirds of the instructions of
// sigm_fast, which it replaced in the residual gradient's epilogue (4.16 -> 4.13 ms of GEMMs at
// 1.06 million edges).  Relative error: 2 |z| u from rounding the exponent twice, 4 u from the
// power, u from the sum, 2 u from the reciprocal; a sigmoid below the normal range (z < -87.3)
// is 0.
__device__ __forceinline__ float sigm_ftz(float z) {
  float e, r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(z * -1.4426950408889634f));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.f + e));
  return r;
}

// FP32 path: expf and the hardware reciprocal with one Newton step, r' = r + r (1 - d r), without
// the branch of the IEEE division, which took a fifth of the SiLU epilogues' time.  Relative
// error: 4 u from expf, u from the sum, u from the step's last rounding.  The clamp keeps d
// finite: below z = -80 the result stays at s(-80) = 2e-35, an absolute error of no more than
// that.
__device__ __forceinline__ float sigm_nr(float z) {
  const float d = 1.f + expf(fminf(-z, 80.f));
  float r;   // d in [1, 6e34]: no denormals either side
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return fmaf(r, fmaf(-d, r, 1.f), r);
}
