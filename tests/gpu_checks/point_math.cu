// The point-wise functions of jf_math.cuh as the device evaluates them, one
// argument (or pair of face states) per thread, for tests/test_gpu_point_math.py.
#include <cuda_runtime.h>

#include "jf_math.cuh"

using namespace jf;

__global__ void unary_kernel(int f, const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = f == 0 ? trcp(x[i]) : tsqrt(x[i]);
}

static int finish() {
  const cudaError_t e = cudaGetLastError();
  return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}

extern "C" int pm_unary(int f, const double* x, double* y, int n) {
  unary_kernel<<<(n + 255) / 256, 256>>>(f, x, y, n);
  return finish();
}
