// Double-float operations and wave vectors on arrays, for test_gpu_double_float.py: host arrays in and out, one value
// per thread.
#include "spectral.cuh"

namespace {

using namespace hom;

__global__ void divide_kernel(const df64* a, const df64* b, df64* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = a[i] / b[i];
}

__global__ void wave_kernel(const Geo g, int axis, int k0, int n, df64* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = wave_scaled<df64>(g, axis, k0 + i);
}

// FP32 wave vectors of CG's vectors with the rotated operator, [n3][n2][h + 1][3]
__global__ void rotated_kernel(const Geo g, const double* gtab, float* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int nh = g.h + 1;
  if (i >= (long long)g.n3 * g.n2 * nh) return;
  const int kx = (int)(i % nh), ky = (int)(i / nh % g.n2), n = (int)(i / nh / g.n2);
  cg_wave_vector<float>(g, 1, gtab, kx, ky, n, out[3 * i], out[3 * i + 1], out[3 * i + 2]);
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

// wave numbers k0 .. k0 + n - 1 of an axis of the grid; *scale: the axis' frequency per wave number in FP64
extern "C" __attribute__((visibility("default"))) int df_waves(const int* grid, int axis, int k0, int n, df64* out, double* scale) {
  Geo g{};
  g.n1 = grid[0];
  g.n2 = grid[1];
  g.n3 = grid[2];
  geo_wave_scale(g);
  *scale = axis == 0 ? g.xs1 : axis == 1 ? g.xs2 : g.xs3;
  df64* d = nullptr;
  if (cudaMalloc(&d, sizeof(df64) * n) != cudaSuccess) return 1;
  wave_kernel<<<(n + 255) / 256, 256>>>(g, axis, k0, n, d);
  const cudaError_t e = cudaMemcpy(out, d, sizeof(df64) * n, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e != cudaSuccess;
}

// gtab: ntab doubles as hom_create lays them out
extern "C" __attribute__((visibility("default"))) int rotated_vectors(const int* grid, const double* gtab, int ntab, float* out) {
  Geo g{};
  g.n1 = grid[0];
  g.n2 = grid[1];
  g.n3 = grid[2];
  g.h = g.n1 / 2;
  geo_wave_scale(g);
  const long long n = (long long)g.n3 * g.n2 * (g.h + 1);
  double* t = nullptr;
  float* d = nullptr;
  if (cudaMalloc(&t, sizeof(double) * ntab) != cudaSuccess || cudaMalloc(&d, sizeof(float) * 3 * n) != cudaSuccess) return 1;
  cudaMemcpy(t, gtab, sizeof(double) * ntab, cudaMemcpyHostToDevice);
  rotated_kernel<<<(unsigned)((n + 255) / 256), 256>>>(g, t, d);
  const cudaError_t e = cudaMemcpy(out, d, sizeof(float) * 3 * n, cudaMemcpyDeviceToHost);
  cudaFree(t);
  cudaFree(d);
  return e != cudaSuccess;
}
