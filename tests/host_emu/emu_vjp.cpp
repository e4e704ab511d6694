// Host emulation of the tiled adjoint kernels (vjp.cuh, vjp3.cuh), as emu.cpp
// for the stage kernel: their source compiled for the CPU, one std::thread per
// CUDA thread, a std::barrier per CTA, every buffer a heap array of exactly
// its size filled with NaN.  A program: reads one stage's inputs from the
// file argv[1] and writes its result, out = lam + dt J(Us)^T lam, to argv[2].
// Test infrastructure only (tests/test_host_emulation_vjp.py).
#include <cstring>
#include <fstream>
#include <memory>
#include <mutex>
#include <thread>
#include <type_traits>
#include <vector>

#include <cuda_runtime.h>

static std::mutex g_mu;  // additions to one accumulator from many threads
inline void atomicAdd(float* p, float v) { std::lock_guard<std::mutex> l(g_mu); *p += v; }
inline void atomicAdd(double* p, double v) { std::lock_guard<std::mutex> l(g_mu); *p += v; }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }

#include "vjp.cuh"
#include "vjp3.cuh"

thread_local uint3 threadIdx;
thread_local uint3 blockIdx;
dim3 blockDim, gridDim;
static std::barrier<>* g_bar = nullptr;
static unsigned char* g_smem = nullptr;
void emu_syncthreads() { g_bar->arrive_and_wait(); }
unsigned char* emu_smem() { return g_smem; }

using namespace jf;

template <typename F>
static void launch(dim3 grid, int threads, size_t smem, F body) {
  gridDim = grid;
  blockDim.x = threads;
  for (unsigned z = 0; z < grid.z; ++z)
    for (unsigned y = 0; y < grid.y; ++y)
      for (unsigned x = 0; x < grid.x; ++x) {
        std::unique_ptr<unsigned char[]> sm(new unsigned char[smem + 1]);
        std::memset(sm.get(), 0xFF, smem);
        g_smem = sm.get();
        std::barrier<> bar(threads);
        g_bar = &bar;
        std::vector<std::thread> th;
        for (int t = 0; t < threads; ++t)
          th.emplace_back([&, t] {
            threadIdx = uint3{(unsigned)t, 0, 0};
            blockIdx = uint3{x, y, z};
            body();
          });
        for (auto& q : th) q.join();
      }
}

template <typename T, int DIM, bool VISC, int BX, int BY, int NT>
static void box(const VjpArgs<T>& A, const Gas<T>& g) {
  dim3 grid;
  grid.x = (A.n[0] + BX - 1) / BX;
  grid.y = (A.n[1] + BY - 1) / BY;
  launch(grid, NT, vjp_smem_bytes<T, DIM, VISC, BX, BY>(),
         [&] { vjp_stage_kernel<T, DIM, VISC, BX, BY, 1, NT>(A, g); });
}

template <typename T, bool VISC, int BX, int BY, int NT>
static void march(const VjpArgs<T>& A, const Gas<T>& g, int zchunk) {
  std::unique_ptr<T[]> G(new T[(VISC ? 6 : 5) * A.N]());
  dim3 grid;
  grid.x = (A.n[0] + BX - 1) / BX;
  grid.y = (A.n[1] + BY - 1) / BY;
  grid.z = (A.n[2] + zchunk - 1) / zchunk;
  launch(grid, NT, vjp3_smem_bytes<T, VISC, BX, BY>(),
         [&] { vjp3_kernel<T, VISC, BX, BY, NT, 1>(A, g, G.get(), zchunk); });
  dim3 one;
  launch(one, 1, 0, [&] { vjp3_finish_kernel<T, VISC>(A, g, G.get()); });
}

// header: n[3], periodic[3], zchunk, visc, safe (ints), then inv_h[3], gamma, R,
// mu, lambda, eps, dt (doubles), then U and lam (5 N values of T each)
template <typename T>
static int run(std::ifstream& in, const char* path) {
  int h[9];
  double d[9];
  in.read((char*)h, sizeof h);
  in.read((char*)d, sizeof d);
  const long long N = (long long)h[0] * h[1] * h[2];
  std::unique_ptr<T[]> U(new T[5 * N]), lam(new T[5 * N]), out(new T[5 * N]);
  in.read((char*)U.get(), sizeof(T) * 5 * N);
  in.read((char*)lam.get(), sizeof(T) * 5 * N);
  if (!in) return 2;
  int flag = 0;
  Gas<T> g;
  std::memset(&g, 0, sizeof g);
  g.gamma = (T)d[3];
  g.gm1 = (T)(d[3] - 1.0);
  g.inv_gm1 = (T)(1.0 / (d[3] - 1.0));
  g.inv_R = (T)(1.0 / d[4]);
  g.mu = (T)d[5];
  g.lambda = (T)d[6];
  g.eps = (T)d[7];
  g.safe = h[8];
  VjpArgs<T> A;
  std::memset(&A, 0, sizeof A);
  A.Us = U.get();
  A.lam = lam.get();
  A.out = out.get();
  A.dt = &d[8];
  A.s_in = T(1);
  A.N = N;
  A.flag = &flag;
  for (int a = 0; a < 3; ++a) {
    A.n[a] = h[a];
    A.periodic[a] = h[3 + a];
    A.inv_h[a] = (T)d[a];
  }
  constexpr bool f32 = sizeof(T) == 4;
  const bool visc = h[7];
  if (h[2] > 1) {
    if (visc) march<T, true, f32 ? 32 : 16, f32 ? 8 : 4, f32 ? 576 : 224>(A, g, h[6]);
    else march<T, false, f32 ? 32 : 16, 8, f32 ? 576 : 320>(A, g, h[6]);
  } else if (h[1] > 1) {
    if (visc) box<T, 2, true, 16, 16, 384>(A, g); else box<T, 2, false, 16, 16, 384>(A, g);
  } else {
    if (visc) box<T, 1, true, 128, 1, 160>(A, g); else box<T, 1, false, 128, 1, 160>(A, g);
  }
  std::ofstream(path, std::ios::binary).write((char*)out.get(), sizeof(T) * 5 * N);
  return flag;
}

int main(int argc, char** argv) {
  std::ifstream in(argv[1], std::ios::binary);
  int f64 = 0;
  in.read((char*)&f64, sizeof f64);
  return f64 ? run<double>(in, argv[2]) : run<float>(in, argv[2]);
}
