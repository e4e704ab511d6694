// The point-wise functions of jf_math.cuh and vjp_gen.cuh as the device evaluates them, one
// argument (or pair of face states) per thread, for tests/test_gpu_point_math.py.
#include <cuda_runtime.h>

#include "jf_math.cuh"
#include "vjp_gen.cuh"

using namespace jf;

__global__ void unary_kernel(int f, const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = f == 0 ? trcp(x[i]) : tsqrt(x[i]);
}

// W: [2][5][n] left and right states, F: [5][n]
__host__ __device__ void hllc_at(int i, const double* W, double* F, int n, const Gas<double>& g, int speeds) {
  double WL[5], WR[5], f[5];
  for (int c = 0; c < 5; ++c) {
    WL[c] = W[c * n + i];
    WR[c] = W[(5 + c) * n + i];
  }
  hllc<double, 0>(WL, WR, g, f, speeds);
  for (int c = 0; c < 5; ++c) F[c * n + i] = f[c];
}

__global__ void hllc_kernel(const double* W, double* F, int n, Gas<double> g, int speeds) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) hllc_at(i, W, F, n, g, speeds);
}

// the cotangent of the x momentum under a unit cotangent of the x velocity: 1 / rho
__global__ void prim_vjp_kernel(const float* rho, float* out, int n, Gas<float> g) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float W[5] = {rho[i], 0.3f, -0.2f, 0.1f, 1.0f}, Wb[5] = {0.0f, 1.0f, 0.0f, 0.0f, 0.0f};
  float Ub[5];
  prim_vjp(W, g, Wb, Ub);
  out[i] = Ub[1];
}

static int finish() {
  const cudaError_t e = cudaGetLastError();
  return (int)(e == cudaSuccess ? cudaDeviceSynchronize() : e);
}

extern "C" int pm_unary(int f, const double* x, double* y, int n) {
  unary_kernel<<<(n + 255) / 256, 256>>>(f, x, y, n);
  return finish();
}

// on the device, or (host arrays) in the host's branch of the same functions
extern "C" int pm_hllc(int host, const double* W, double* F, int n, double gamma, int speeds) {
  Gas<double> g{};
  g.gamma = gamma;
  g.gm1 = gamma - 1.0;
  g.inv_gm1 = 1.0 / (gamma - 1.0);
  if (host) {
    for (int i = 0; i < n; ++i) hllc_at(i, W, F, n, g, speeds);
    return 0;
  }
  hllc_kernel<<<(n + 255) / 256, 256>>>(W, F, n, g, speeds);
  return finish();
}

extern "C" int pm_prim_vjp(const float* rho, float* out, int n) {
  Gas<float> g{};
  g.gm1 = 0.4f;
  prim_vjp_kernel<<<(n + 255) / 256, 256>>>(rho, out, n, g);
  return finish();
}
