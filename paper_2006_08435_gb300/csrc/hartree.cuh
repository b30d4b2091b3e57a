// The weight of a plane wave in the Hartree energy's gradient, shared by the
// seed kernel (hartree.cu) and the inverse real transforms that apply it to the
// spectrum as they read it.
#pragma once

#include <cuda_runtime.h>

namespace fft3d {

// 1 / x by the hardware's approximate reciprocal (within 1 ulp by the PTX
// ISA's bound; the callers' x = |m|^2 is a positive integer below 2^24,
// exact in FP32).
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// v scale / |m|^2, 0 at m = 0 whatever v.  (Products rounded by themselves, as
// the seed kernel stores them: not fused into the sums that follow.)
__device__ __forceinline__ float2 weighted(float2 v, float scale, float m2) {
  const float w = scale * rcp_approx(m2);
  return m2 == 0.0f ? make_float2(0.0f, 0.0f) : make_float2(__fmul_rn(v.x, w), __fmul_rn(v.y, w));
}
// Index k of an axis of n points as a signed frequency.
__host__ __device__ __forceinline__ int signed_index(int k, int n) {
  return k < (n + 1) / 2 ? k : k - n;
}

// What the weighted inverse needs: scale = (float)(s grad[grid]).
struct HartreeWeight {
  const double* grad = nullptr;  // device, one per grid
  double s = 0.0;
};

// s = Omega 4 pi / (n^6 (2 pi / L)^2) (hartree.cu)
double hartree_s(int n, double L);
bool hartree_valid(int n, int batch, double L);

}  // namespace fft3d
