// The FP32 face fluxes' constants on arrays of FP64 values (tests/test_face_constants_gpu.py).
#include <cstdint>

#include "kernels.cuh"

namespace {
__global__ void constants(int64_t n, const double* a, const double* b, float* product, float* eps) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  product[i] = afe::f32_product(a[i], b[i]);
  eps[i] = afe::f32_face_eps<1>(a[i], b[i]);
  eps[n + i] = afe::f32_face_eps<2>(a[i], b[i]);
  eps[2 * n + i] = afe::f32_face_eps<3>(a[i], b[i]);
}
}  // namespace

// Device pointers; 0 on success.
extern "C" int face_constants(int64_t n, const double* a, const double* b, float* product, float* eps) {
  constants<<<(unsigned)((n + 255) / 256), 256>>>(n, a, b, product, eps);
  return cudaDeviceSynchronize() == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : 1;
}
