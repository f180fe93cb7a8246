// Elementwise device functions of the kernels, on arrays, for the tests.
#include "attn_core.cuh"

namespace {
__global__ void silu_kernel(const float* x, float* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = pard::silu(x[i]);
}
}  // namespace

// y[i] = silu(x[i]) for i < n, device pointers
extern "C" int device_silu(const float* x, float* y, int n) {
  silu_kernel<<<(n + 255) / 256, 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
