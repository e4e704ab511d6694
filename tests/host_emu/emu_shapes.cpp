// Host emulation (see emu.cpp) of the stage kernels' remaining families and
// tile shapes, with slip walls: the component-split 1D tiles of FP64, the FP64
// 2D and 3D shapes, the extended forms (walls, WENO3-JS) per cell and per
// face, and the Rusanov-NN kernels with the parameters, their transposed copy
// and the threads' hidden rows.  Shared memory is exactly launch_smem bytes and
// 16-byte aligned.  Test infrastructure only (tests/test_host_emulation_shapes.py).
#include <cstring>
#include <memory>
#include <thread>
#include <vector>

#include <cuda_runtime.h>
struct alignas(16) float4 { float x, y, z, w; };
inline float4 make_float4(float a, float b, float c, float d) { return float4{a, b, c, d}; }
#define JF_HOST_FLOAT4
#include "stage.cuh"

thread_local uint3 threadIdx;
thread_local uint3 blockIdx;
dim3 blockDim, gridDim;
static std::barrier<>* g_bar = nullptr;
static unsigned char* g_smem = nullptr;
void emu_syncthreads() { g_bar->arrive_and_wait(); }
unsigned char* emu_smem() { return g_smem; }

using namespace jf;

template <typename T, int DIM, bool VISC, int BX, int BY, int SCH>
static void run(const StageArgs<T>& A, const Gas<T>& g) {
  constexpr int NT = Geo<BX, BY, DIM, VISC>::NT;
  constexpr size_t smem = launch_smem<T, DIM, VISC, BX, BY, SCH>();
  gridDim.x = (A.nx + BX - 1) / BX;
  gridDim.y = plane_dims(DIM) == 2 ? (A.ny + BY - 1) / BY : 1;
  gridDim.z = marches(DIM) ? (A.nz + A.zchunk - 1) / A.zchunk : 1;
  blockDim.x = NT;
  for (unsigned bz = 0; bz < gridDim.z; ++bz)
    for (unsigned by = 0; by < gridDim.y; ++by)
      for (unsigned bx = 0; bx < gridDim.x; ++bx) {
        std::unique_ptr<unsigned char[]> sm(new unsigned char[smem]);
        std::memset(sm.get(), 0xFF, smem);
        g_smem = sm.get();
        std::barrier<> bar(NT);
        g_bar = &bar;
        std::vector<std::thread> th;
        for (int t = 0; t < NT; ++t)
          th.emplace_back([&, t] {
            threadIdx = uint3{(unsigned)t, 0, 0};
            blockIdx = uint3{bx, by, bz};
            stage_kernel<T, DIM, VISC, BX, BY, 1, SCH>(A, nullptr, nullptr, 0, 0, g);
          });
        for (auto& x : th) x.join();
      }
}

// Kernels of one precision by number, as the tables of stage_f32_*.cu and
// stage_f64*.cu compile them.
static int emulate(int kernel, bool visc, const StageArgs<double>& A, const Gas<double>& g) {
  using T = double;
#define KERNEL(k, DIM, V, BX, BY, SCH) \
  if (kernel == k && visc == V) return run<T, DIM, V, BX, BY, SCH>(A, g), 0
  KERNEL(0, 1, true, 30, 1, SCH_DEFAULT);
  KERNEL(0, 1, false, 30, 1, SCH_DEFAULT);
  KERNEL(1, 1, false, 30, 1, SCH_GENERAL_EXT);
  KERNEL(2, 1, true, 30, 1, SCH_ROE_EXT);
  KERNEL(3, 1, false, 30, 1, SCH_NN);
  KERNEL(4, 2, true, 32, 3, SCH_DEFAULT);
  KERNEL(5, 2, false, 32, 4, SCH_GENERAL);
  KERNEL(6, 2, true, 32, 3, SCH_GENERAL_EXT);
  KERNEL(6, 2, false, 32, 3, SCH_GENERAL_EXT);
  KERNEL(7, 2, false, 32, 8, SCH_GENERAL_EXT);
  KERNEL(8, 3, true, 32, 7, SCH_DEFAULT);
  KERNEL(9, 3, true, 32, 4, SCH_GENERAL_EXT);
  KERNEL(9, 3, false, 32, 4, SCH_GENERAL_EXT);
  KERNEL(10, 2, false, 32, 7, SCH_NN);
#undef KERNEL
  return -1;
}
static int emulate(int kernel, bool visc, const StageArgs<float>& A, const Gas<float>& g) {
  using T = float;
#define KERNEL(k, DIM, V, BX, BY, SCH) \
  if (kernel == k && visc == V) return run<T, DIM, V, BX, BY, SCH>(A, g), 0
  KERNEL(0, 1, false, 128, 1, SCH_GENERAL_EXT);
  KERNEL(1, 2, false, 32, 7, SCH_GENERAL_EXT);
  KERNEL(2, 2, true, 32, 8, SCH_GENERAL_EXT);
  KERNEL(2, 2, false, 32, 8, SCH_GENERAL_EXT);
  KERNEL(3, 3, true, 32, 7, SCH_GENERAL_EXT);
  KERNEL(3, 3, false, 32, 7, SCH_GENERAL_EXT);
  KERNEL(4, 3, true, 32, 8, SCH_GENERAL_EXT);
  KERNEL(4, 3, false, 32, 8, SCH_GENERAL_EXT);
  KERNEL(5, 2, false, 32, 3, SCH_NN);
  KERNEL(6, 2, true, 32, 8, SCH_NN);
  KERNEL(7, 3, false, 32, 7, SCH_NN);
#undef KERNEL
  return -1;
}

// out = L(Us).  gas = {gamma, R, mu, lambda, eps, flux, recon, speeds} (the last
// three as the jf_scheme codes), wall: bit 0 the low side, bit 1 the high one;
// theta: the network's parameters or null.  Returns the device flag, or -1.
template <typename T>
static int rhs(int kernel, const int* n, const int* periodic, const int* wall, const double* inv_h, const double* gas,
               int zchunk, const T* theta, const T* Us, T* out) {
  const long long N = (long long)n[0] * n[1] * n[2];
  std::unique_ptr<T[]> us(new T[5 * N]), o(new T[5 * N]), th(theta ? new T[NN_PARAMS] : nullptr);
  std::memcpy(us.get(), Us, sizeof(T) * 5 * N);
  if (theta) std::memcpy(th.get(), theta, sizeof(T) * NN_PARAMS);
  int flag = 0;
  StageArgs<T> A;
  std::memset(&A, 0, sizeof A);
  A.Us = us.get();
  A.out = o.get();
  A.nx = n[0];
  A.ny = n[1];
  A.nz = n[2];
  A.N = N;
  for (int d = 0; d < 3; ++d) {
    A.periodic[d] = periodic[d];
    A.wall[d] = wall[d];
    A.inv_h[d] = (T)inv_h[d];
  }
  A.rhs_only = 1;
  A.b = T(1);
  A.zchunk = zchunk;
  A.flag = &flag;
  Gas<T> g;
  std::memset(&g, 0, sizeof g);
  g.gamma = (T)gas[0];
  g.gm1 = (T)(gas[0] - 1.0);
  g.inv_gm1 = (T)(1.0 / (gas[0] - 1.0));
  g.inv_R = (T)(1.0 / gas[1]);
  g.mu = (T)gas[2];
  g.lambda = (T)gas[3];
  g.eps = (T)gas[4];
  g.flux = (int)gas[5];
  g.recon = (int)gas[6];
  g.speeds = (int)gas[7];
  g.nn = th.get();
  if (emulate(kernel, gas[2] > 0.0, A, g) != 0) return -1;
  std::memcpy(out, o.get(), sizeof(T) * 5 * N);
  return flag;
}

extern "C" int emu_rhs_f64(int kernel, const int* n, const int* periodic, const int* wall, const double* inv_h,
                           const double* gas, int zchunk, const double* theta, const double* Us, double* out) {
  return rhs<double>(kernel, n, periodic, wall, inv_h, gas, zchunk, theta, Us, out);
}
extern "C" int emu_rhs_f32(int kernel, const int* n, const int* periodic, const int* wall, const double* inv_h,
                           const double* gas, int zchunk, const float* theta, const float* Us, float* out) {
  return rhs<float>(kernel, n, periodic, wall, inv_h, gas, zchunk, theta, Us, out);
}
