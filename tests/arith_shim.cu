// Kernels and wrappers that the arithmetic tests call: built by the test into a library of its
// own, linked against libff.so.
#include <math.h>

#include "ff_internal.cuh"
#include "sigmoid.cuh"

namespace {

template <int WHICH>
__device__ __forceinline__ float sigmoid(float z) {
  return WHICH == 0 ? sigm_fast(z) : WHICH == 1 ? sigm_ftz(z) : sigm_nr(z);
}

// The bound on |s(z) - exact| of sigmoid.cuh, for finite z (1 % for the terms of second order).
template <int WHICH>
__device__ __forceinline__ double bound(double z, double exact) {
  const double u = 0x1p-24;
  if (WHICH == 2) return z >= -80.0 ? 1.01 * 6.0 * u * exact : 2e-35;
  if (z < -87.0) return 0x1p-125;
  return 1.01 * (WHICH == 0 ? 2.35 * fabs(z) + 9.0 : 2.0 * fabs(z) + 7.0) * u * exact;
}

// Every float: worst[0] = the largest |error| / bound (float bits, non-negative), worst[1] = inputs
// that break the limits (infinities; z s(z) must be NaN for a NaN).
template <int WHICH>
__global__ void k_check_sigmoid(unsigned* worst) {
  float top = 0.f;
  unsigned bad = 0;
  for (unsigned long long i = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
       i < (1ull << 32); i += (unsigned long long)gridDim.x * blockDim.x) {
    const float z = __uint_as_float((unsigned)i);
    const float s = sigmoid<WHICH>(z);
    if (isnan(z)) bad += !isnan(z * s);
    else if (isinf(z)) bad += z > 0.f ? s != 1.f : !(s >= 0.f && s <= 2e-35f);
    else {
      const double exact = 1.0 / (1.0 + exp(-(double)z));
      const float q = (float)(fabs((double)s - exact) / bound<WHICH>(z, exact));
      if (!(q <= top)) top = q;   // (a NaN stays)
    }
  }
  atomicMax(worst, isnan(top) ? 0x7f800000u : __float_as_uint(top));
  atomicAdd(worst + 1, bad);
}

}  // namespace

// which: 0 sigm_fast, 1 sigm_ftz, 2 sigm_nr; worst: two device words, zero.
extern "C" int shim_check_sigmoid(int which, unsigned* worst) {
  if (which == 0) k_check_sigmoid<0><<<1216, 256>>>(worst);
  else if (which == 1) k_check_sigmoid<1><<<1216, 256>>>(worst);
  else k_check_sigmoid<2><<<1216, 256>>>(worst);
  return (int)cudaDeviceSynchronize();
}

// out [M][N] = [A | A2] B by the FP32 GEMM, B^T = [W1 | W2] given as FP32 rows (K2 = 0: A, W1
// alone).  slices: 3 N split_ld(K1, K2) bf16 of device memory; err: the device error word.
extern "C" int shim_gemm_f32(const float* A, const float* A2, const float* W1, const float* W2,
                             int M, int N, int K1, int K2, __nv_bfloat16* slices, float* out,
                             int* err) {
  launch_split_weights(W1, N, K1, W2, K2, 1.0, slices, nullptr);
  EpiParams ep{};
  ep.alpha = 1.f;
  ep.out = out;
  ep.ldo = N;
  if (!launch_gemm_f32(EPI_STORE, M, N, K1, A, K1, slices, split_ld(K1, K2), ep, err, nullptr,
                       K2 > 0 ? A2 : nullptr, K2, K2))
    return -1;
  return (int)cudaDeviceSynchronize();
}

extern "C" int shim_split_ld(int K1, int K2) { return split_ld(K1, K2); }
