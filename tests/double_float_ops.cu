// Double-float operations on arrays, for test_gpu_double_float.py: host arrays in and out, one value per thread.
#include "common.cuh"

namespace {

using namespace hom;

__global__ void divide_kernel(const df64* a, const df64* b, df64* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = a[i] / b[i];
}

}  // namespace

extern "C" __attribute__((visibility("default"))) int df_divide(const df64* a, const df64* b, df64* out, int n) {
  df64 *d = nullptr;
  const size_t bytes = sizeof(df64) * n;
  if (cudaMalloc(&d, 3 * bytes) != cudaSuccess) return 1;
  cudaMemcpy(d, a, bytes, cudaMemcpyHostToDevice);
  cudaMemcpy(d + n, b, bytes, cudaMemcpyHostToDevice);
  divide_kernel<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, n);
  const cudaError_t e = cudaMemcpy(out, d + 2 * n, bytes, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e != cudaSuccess;
}
