// Point-wise numerics of the finite-volume stage, shared by the forward,
// batched and adjoint kernels of libjf.
//
// References (arXiv 2203.13760):
//   primitives        Section 2, Eq. (StiffenedGas) with B = 0
//   weno5             Section 3.3 (High-order Godunov approach, step 1),
//                     WENO5-JS of Jiang & Shu (1996) or WENO5-Z of Borges et
//                     al. (2008) (Table 2)
//   hllc              Section 3.3 steps 2-3, Eq. (ApproxRiemannSolver): HLLC
//                     (Toro 1994) with Einfeldt (1988), Davis (1988) or Toro
//                     (1994) signal speeds (Table 2)
//   hll, rusanov      Table 2: HLL (Harten, Lax, van Leer 1983) and local
//                     Lax-Friedrichs
//   rusanov_nn        Section 7.4: Rusanov flux with a learned dissipation
//   weno3             Table 2 WENO3-JS
//   df4 / dc4 / rc4   Section 3.4 fourth-order face derivative, cell-centre
//                     derivative and central interpolation to the face
#pragma once
#include <cuda_runtime.h>

// point-wise numerics compile for the host too (used by host-side checks)
#define JF_HD __host__ __device__ __forceinline__

namespace jf {

// Programmatic dependent launch of the kernels that follow one another on a
// stream (stages, CFL passes, adjoints): a launch may be made ready while its
// predecessor still runs, and its CTAs take the SMs that the predecessor's
// leave.  Every kernel launched this way starts with follow_predecessor(),
// which waits until the predecessor has finished and its writes are visible,
// and only then lets its own successor start, so that at most one kernel waits
// ahead.  These kernels read what their predecessor may have written with plain
// loads: no __ldg and no const __restrict__ pointers, whose loads are taken for
// read-only during the whole kernel and may move above the wait.  A launch after a
// copy, a memset or another library's kernel waits for that as usual.
//
// Before and after: FP64 step of a 200-cell tube 39 -> 32 us (four dependent
// launches of a few us each), 107 x 61 x 45 step 139 -> 132 us, gradient of 24
// 256^2 steps 2.78 -> 2.50 ms, a training step on a 32^2 batch 2.53 -> 2.31 ms;
// steps of a millisecond and more within 1 %.  Where it costs time the launch is
// plain (overlapped_launch, spreads_evenly and launch_batch).

// LET: let the successor's CTAs in now (else as this kernel ends).  FP64 kernels
// other than the stages do not: a stage that fills one slot of most SMs comes to
// rest two to an SM where its predecessor's CTAs leave fewer SMs empty than it
// has CTAs (FP64 128^2 step, after the CFL pass: 224 us with the early release,
// 147 without).
template <bool LET = true>
__device__ __forceinline__ void follow_predecessor() {
#ifdef __CUDA_ARCH__
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (LET) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
#endif
}

// A load of the stage input, which the kernel does not write: free to move past
// its stores like a read-only load, but (volatile) not above the wait.  A plain
// load costs the 128-register kernels a percent (256^3 step 4.21 -> 4.23 ms).
__device__ __forceinline__ float ld_state(const float* p) {
#ifdef __CUDA_ARCH__
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
#else
  return *p;
#endif
}
__device__ __forceinline__ double ld_state(const double* p) {
#ifdef __CUDA_ARCH__
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
#else
  return *p;
#endif
}

#ifdef __CUDACC__
template <typename... P, typename... A>
cudaError_t launch_next(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
  if (e != cudaSuccess) cudaGetLastError();  // returned here: not left for the next caller's check
  return e;
}
#endif

template <typename T>
struct Gas {
  T gamma;     // ratio of specific heats
  T gm1;       // gamma - 1
  T inv_gm1;   // 1 / (gamma - 1)
  T inv_R;     // 1 / R
  T mu;        // dynamic viscosity (0 if inviscid)
  T lambda;    // heat conductivity
  T eps;       // WENO5 epsilon
  int safe;    // first-order fallback for non-positive reconstructed rho / p
  int flux;    // 0 HLLC, 1 HLL, 2 Rusanov (local Lax-Friedrichs), 4 Rusanov-NN
  int recon;   // 0 WENO5-JS, 1 WENO5-Z, 2 WENO3-JS
  int speeds;  // 0 Einfeldt, 1 Davis, 2 Toro (PVRS)
  const T* nn; // Rusanov-NN parameters (NN_PARAMS values; shared memory in the kernels)
};

// The Rusanov-NN dissipation network (Section 7.4): inputs
// x = (|du_n|, mean u_n, mean c, |ds|), three hidden layers of NN_HIDDEN ReLU
// units, alpha = exp(output); parameters W1 [32][4], b1, W2 [32][32], b2,
// W3 [32][32], b3, W4 [32], b4 (row-major, outputs by inputs).
constexpr int NN_HIDDEN = 32;
constexpr int NN_PARAMS = 32 * 4 + 32 + 2 * (32 * 32 + 32) + 32 + 1;

// Reciprocal and square roots of the point-wise numerics.  FP32 device code
// takes the hardware approximations (rcp.approx.ftz: one MUFU operation,
// within 1 ulp for |x| < 2^126; host code divides exactly).  FP64 device code
// starts from the PTX approximations rcp / rsqrt.approx.ftz.f64 (about 20
// bits, not on the FP64 pipe) and refines them: the reciprocal with one
// third-order step (Chebyshev), y + y (e + e^2) with e = 1 - x y; the root
// r = x y with two Newton steps r + (x - r^2) y / 2, whose residuals a fused
// multiply-add forms exactly.  3 and 5 FP64 operations, where an IEEE division
// or square root takes about ten and the FP64 pipe (2 FMA per clock and SM) is
// what bounds the FP64 kernels.  The last operation rounds a correction of some
// 2^-20 (2^-40) of the result, so the error stays within 0.51 ulp; a form that
// rounds x y and takes one third-order step from it reaches 0.75.  Zero, infinity and NaN give
// what IEEE division and square root give; arguments and results below 2^-1022
// count as zero.  FP32: against __fdividef, whose
// multiplication it saves, the same bits, and the ROE step at 128^3 takes 903
// instead of 941 us, the default one at 256^3 4.205 instead of 4.264 ms.
template <typename T> JF_HD T trcp(T x);
template <> JF_HD float trcp<float>(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / x;
#endif
}
template <> JF_HD double trcp<double>(double x) {
#ifdef __CUDA_ARCH__
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0), r = fma(y, fma(e, e, e), y);
  // 1/0, 1/inf, 1/NaN: the approximation is the result, and e would be NaN
  // (its exponent field is 0 or 0x7ff; 32-bit operations)
  return ((__double2hiint(y) + 0x00100000) & 0x7fe00000) == 0 ? y : r;
#else
  return 1.0 / x;
#endif
}

// 1 / sqrt(x) in FP64, x > 0, one third-order step (Halley): 0.8 ulp, for the
// weights of a Roe average, which scale differences only.
JF_HD double trsqrt(double x) {
#ifdef __CUDA_ARCH__
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
#else
  return 1.0 / sqrt(x);
#endif
}

template <typename T> JF_HD T tsqrt(T x);
template <> JF_HD float tsqrt<float>(float x) { return sqrtf(x); }
template <> JF_HD double tsqrt<double>(double x) {
#ifdef __CUDA_ARCH__
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));  // y / 2
  const double r = x * y, r1 = fma(fma(-r, r, x), h, r), s = fma(fma(-r1, r1, x), h, r1);
  // sqrt(+-0) and sqrt(inf) are x itself (32-bit operations)
  const int hi = __double2hiint(x);
  return (hi & 0x7ff00000) == 0 || hi == 0x7ff00000 ? x : s;
#else
  return sqrt(x);
#endif
}

template <typename T> JF_HD T tmin(T a, T b) { return b < a ? b : a; }
template <typename T> JF_HD T tmax(T a, T b) { return a < b ? b : a; }

// WENO5-JS (Jiang & Shu 1996): value at x_{i+1/2} biased to the left, from
// v[i-2..i+2]: candidate stencils q_k, smoothness indicators beta_k, weights
// alpha_k = d_k / (eps + beta_k)^2 with d = (1/10, 6/10, 3/10),
// omega_k = alpha_k / sum(alpha).  With z != 0 the WENO5-Z weights of Borges
// et al. (2008) replace the JS ones: tau5 = |beta_0 - beta_2|,
// alpha_k = d_k (1 + tau5 / (eps + beta_k)).
//
// Evaluated in differences, which takes the fewest operations (the kernels
// are bound by the arithmetic pipes).  With D2 = v0 - v[-1], D3 = v[1] - v0
// and the second differences d0, d1, d2 of the three sub-stencils,
//   beta_0 = 4/3 d0^2 + d0 D2 + D2^2, beta_1 = 4/3 d1^2 + d1 D2 + D2^2,
//   beta_2 = 4/3 d2^2 + d2 D3 + D3^2
// (positive definite forms, no cancellation beyond a factor of 2), so that
// D2^2 + eps serves two of them, and with the weights (1, 6, 3) r_k
//   v^ = v0 + [a0 (d0/3 + D2/2) + a1 (d1/3 + D2/2) + a2 (d2/6 + D3/2)] / (a0 + a1 + a2).
template <typename T>
struct WenoTerms {
  T d0, d1, d2;  // second differences of the sub-stencils
  T h2, h3;      // D2 / 2, D3 / 2
  T t0, t1, t2;  // eps + beta_k
};

template <typename T>
JF_HD WenoTerms<T> weno5_terms(T vm2, T vm1, T v0, T vp1, T vp2, T eps) {
  WenoTerms<T> w;
  const T D2 = v0 - vm1, D3 = vp1 - v0;
  w.d0 = D2 + (vm2 - vm1);
  w.d1 = D3 - D2;
  w.d2 = D3 + (vp1 - vp2);
  const T q2 = D2 * D2 + eps, q3 = D3 * D3 + eps, k = T(4) / T(3);
  w.t0 = w.d0 * (k * w.d0 + D2) + q2;
  w.t1 = w.d1 * (k * w.d1 + D2) + q2;
  w.t2 = w.d2 * (k * w.d2 + D3) + q3;
  w.h2 = T(0.5) * D2;
  w.h3 = T(0.5) * D3;
  return w;
}

// The factors r_k of the weights, up to a common factor.  FP64: scaled by
// (t0 t1 t2)^2 (JS; WENO5-Z: t0 t1 t2), so that no reciprocal is taken here
// (the factors are >= eps, far inside the FP64 range).
template <typename T>
JF_HD void weno5_factors(const WenoTerms<T>& w, int z, T& r0, T& r1, T& r2) {
  if constexpr (sizeof(T) == 8) {
    if (z) {
      const T tau = fabs(w.t0 - w.t2);
      r0 = (w.t0 + tau) * (w.t1 * w.t2);
      r1 = (w.t1 + tau) * (w.t0 * w.t2);
      r2 = (w.t2 + tau) * (w.t0 * w.t1);
    } else {
      const T s0 = w.t0 * w.t0, s1 = w.t1 * w.t1, s2 = w.t2 * w.t2;
      r0 = s1 * s2;
      r1 = s0 * s2;
      r2 = s0 * s1;
    }
  } else {
    if (z) {
      const T tau = fabs(w.t0 - w.t2);
      r0 = (w.t0 + tau) * trcp(w.t0);
      r1 = (w.t1 + tau) * trcp(w.t1);
      r2 = (w.t2 + tau) * trcp(w.t2);
    } else {
      r0 = trcp(w.t0 * w.t0);
      r1 = trcp(w.t1 * w.t1);
      r2 = trcp(w.t2 * w.t2);
    }
  }
}

template <typename T>
JF_HD T weno5(T vm2, T vm1, T v0, T vp1, T vp2, T eps, int z = 0) {
  const WenoTerms<T> w = weno5_terms(vm2, vm1, v0, vp1, vp2, eps);
  T a0, a1, a2;
  weno5_factors(w, z, a0, a1, a2);
  a1 = T(6) * a1;
  a2 = T(3) * a2;
  const T third = T(1) / T(3), sixth = T(1) / T(6);
  const T num = a0 * (third * w.d0 + w.h2) + a1 * (third * w.d1 + w.h2) + a2 * (sixth * w.d2 + w.h3);
  return v0 + num * trcp(a0 + a1 + a2);
}

// WENO5 per cell: both face values one cell j contributes, from the same
// five values v[j-2..j+2]:
//   right = v^-_{j+1/2} (left-biased, the weno5 formula above),
//   left  = v^+_{j-1/2} (right-biased: the same formula on the mirrored
//           stencil v[j+2..j-2]).
// The mirrored stencil has the smoothness indicators in reverse order (the
// three 3-cell sub-stencils are the same) and the differences reversed and
// negated, so both values share the indicators and the factors r_k:
//   left = v0 - [r2 (d2/3 + D3/2) + 6 r1 (d1/6 + D2/2) + 3 r0 (d0/6 + D2/2)] / (r2 + 6 r1 + 3 r0).
template <typename T>
JF_HD void weno5_cell_lean(T vm2, T vm1, T v0, T vp1, T vp2, T eps, T& right, T& left, int z = 0) {
  const WenoTerms<T> w = weno5_terms(vm2, vm1, v0, vp1, vp2, eps);
  T r0, r1, r2;
  weno5_factors(w, z, r0, r1, r2);
  if constexpr (sizeof(T) == 8) {
    // the sums of products r_k d_k and r_2 D3 serve both numerators (46 FP64
    // operations with the reciprocal; 50 value by value):
    //   2 n_r = D2 (r0 + 6 r1) + 3 r2 D3 + 2/3 r0 d0 + 4 r1 d1 + r2 d2
    //   2 n_l = D2 (3 r0 + 6 r1) + r2 D3 + r0 d0 + 2 r1 d1 + 2/3 r2 d2
    const T D2 = v0 - vm1, D3 = vp1 - v0, k = T(2) / T(3);
    const T A = fma(T(6), r1, r0), C = fma(T(2), r0, A);
    const T Sr = fma(T(3), r2, A), Sl = C + r2;
    const T x0 = r0 * w.d0, x1 = r1 * w.d1, x2 = r2 * w.d2, y = r2 * D3;
    const T nr = fma(D2, A, fma(T(3), y, fma(k, x0, fma(T(4), x1, x2))));
    const T nl = fma(D2, C, y + fma(k, x2, fma(T(2), x1, x0)));
    // one reciprocal for both values: 1/S_r = S_l / (S_r S_l) and the converse
    // (S >= 1e-23 as every s_k >= eps^2; the product stays far inside the
    // FP64 range)
    const T inv = trcp((Sr + Sr) * Sl);
    right = fma(nr, Sl * inv, v0);
    left = fma(-nl, Sr * inv, v0);
  } else {
    const T a1 = T(6) * r1, a2 = T(3) * r2, c0 = T(3) * r0;
    const T third = T(1) / T(3), sixth = T(1) / T(6);
    const T nr = r0 * (third * w.d0 + w.h2) + a1 * (third * w.d1 + w.h2) + a2 * (sixth * w.d2 + w.h3);
    const T nl = c0 * (sixth * w.d0 + w.h2) + a1 * (sixth * w.d1 + w.h2) + r2 * (third * w.d2 + w.h3);
    right = v0 + nr * trcp(r0 + a1 + a2);
    left = v0 - nl * trcp(c0 + a1 + r2);
  }
}

// The FP32 tile kernels (1D, 2D, 3D) have an earlier grouping of the same
// formulas, with three independent indicators, of the same accuracy.  The lean
// form above, which serves the row tiles and FP64 (see cell_recon), would take
// 4 to 6 % off them; its other rounding moves a loss that is formed in FP64 from
// FP32 states by 1e-9 to 1e-7.
template <typename T>
JF_HD void weno5_cell(T vm2, T vm1, T v0, T vp1, T vp2, T eps, T& right, T& left, int z = 0) {
  if constexpr (sizeof(T) == 8) {
    weno5_cell_lean(vm2, vm1, v0, vp1, vp2, eps, right, left, z);
  } else {
    const T D1 = vm2 - vm1, D2 = v0 - vm1, D3 = vp1 - v0, D4 = vp1 - vp2;
    const T c13 = T(13) / T(12);
    const T d0 = D2 + D1, e0 = T(3) * D2 + D1;
    const T d1 = D3 - D2, e1 = D2 + D3;
    const T d2 = D3 + D4, e2 = T(3) * D3 + D4;
    const T t0 = eps + (c13 * d0 * d0 + T(0.25) * e0 * e0);
    const T t1 = eps + (c13 * d1 * d1 + T(0.25) * e1 * e1);
    const T t2 = eps + (c13 * d2 * d2 + T(0.25) * e2 * e2);
    // candidate offsets q_k - v0 (times 6) of both reconstructions
    const T g0 = T(5) * D2 + T(2) * D1, g1 = D2 + T(2) * D3, g2 = T(4) * D3 + D4;
    const T h0 = -(T(5) * D3 + T(2) * D4), h1 = -(D3 + T(2) * D2), h2 = -(T(4) * D2 + D1);
    T r0, r1, r2;
    if (z) {
      const T tau = fabs(t0 - t2);
      r0 = (t0 + tau) * trcp(t0);
      r1 = (t1 + tau) * trcp(t1);
      r2 = (t2 + tau) * trcp(t2);
    } else {
      r0 = trcp(t0 * t0);
      r1 = trcp(t1 * t1);
      r2 = trcp(t2 * t2);
    }
    const T a0 = T(0.1) * r0, a1 = T(0.6) * r1, a2 = T(0.3) * r2;
    const T b0 = T(0.1) * r2, b2 = T(0.3) * r0;
    right = v0 + (a0 * g0 + a1 * g1 + a2 * g2) * trcp(T(6) * (a0 + a1 + a2));
    left = v0 + (b0 * h0 + a1 * h1 + b2 * h2) * trcp(T(6) * (b0 + a1 + b2));
  }
}

__device__ __forceinline__ float2 splat2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 rcp2(float2 x) { return make_float2(trcp(x.x), trcp(x.y)); }

// The left and right WENO5-JS states of one face component in packed FP32x2
// arithmetic (sm_100+ FFMA2 / FADD2 / FMUL2): lane x reconstructs
// (v[i-2], .., v[i+2]) -> v^-, lane y the mirrored stencil
// (v[i+3], .., v[i-1]) -> v^+.  The formula of weno5, rearranged to fewer
// operations (equal up to rounding):
//  * with the differences D1 = vm2 - vm1, D2 = v0 - vm1, D3 = vp1 - v0,
//    D4 = vp1 - vp2 the candidates are q_k = v0 + delta_k / 6 with
//    delta = (5 D2 + 2 D1, D2 + 2 D3, 4 D3 + D4), and the smoothness terms
//    are d0 = D2 + D1, d1 = D3 - D2, |d2| = |D3 + D4|, e0 = 3 D2 + D1,
//    |e1| = |D2 + D3|, |e2| = |3 D3 + D4| (only their squares enter);
//  * every eps + beta_k is scaled by 12/13 (a common factor of the three
//    alpha_k, which cancels in omega_k), so t_k = d_k^2 + 3/13 e_k^2 + 12/13 eps;
//  * with r_k = 1 / t_k^2 and alpha_k scaled by 10/3 (weights 1/3, 2, 1),
//    v^ = v0 + (r0 delta0/18 + r1 delta1/3 + r2 delta2/6) / (r0/3 + 2 r1 + r2);
//  * WENO5-Z (z != 0): r_k = (t_k + tau) / t_k with tau = |t_0 - t_2| (the
//    same 12/13 scaling of tau5 = |beta_0 - beta_2|).
__device__ __forceinline__ float2 weno5_pair(float2 vm2, float2 vm1, float2 v0, float2 vp1, float2 vp2, float eps,
                                             int z = 0) {
  auto c = [](float x) { return make_float2(x, x); };
  const float2 m1 = c(-1.0f);
  const float2 D1 = __ffma2_rn(m1, vm1, vm2);
  const float2 D2 = __ffma2_rn(m1, vm1, v0);
  const float2 D3 = __ffma2_rn(m1, v0, vp1);
  const float2 D4 = __ffma2_rn(m1, vp2, vp1);
  const float2 d0 = __fadd2_rn(D2, D1), e0 = __ffma2_rn(c(3.0f), D2, D1);
  const float2 d1 = __ffma2_rn(m1, D2, D3), e1 = __fadd2_rn(D2, D3);
  const float2 d2 = __fadd2_rn(D3, D4), e2 = __ffma2_rn(c(3.0f), D3, D4);
  const float2 k3 = c(3.0f / 13.0f), ke = c(12.0f / 13.0f * eps);
  const float2 t0 = __ffma2_rn(d0, d0, __ffma2_rn(__fmul2_rn(k3, e0), e0, ke));
  const float2 t1 = __ffma2_rn(d1, d1, __ffma2_rn(__fmul2_rn(k3, e1), e1, ke));
  const float2 t2 = __ffma2_rn(d2, d2, __ffma2_rn(__fmul2_rn(k3, e2), e2, ke));
  // approximate reciprocals (t_k^2 >= (12/13 eps)^2 > 0, so the sum is > 0)
  float2 r0, r1, r2;
  if (z) {
    const float2 d02 = __ffma2_rn(m1, t2, t0);
    const float2 tau = make_float2(fabsf(d02.x), fabsf(d02.y));
    r0 = __fmul2_rn(__fadd2_rn(t0, tau), rcp2(t0));
    r1 = __fmul2_rn(__fadd2_rn(t1, tau), rcp2(t1));
    r2 = __fmul2_rn(__fadd2_rn(t2, tau), rcp2(t2));
  } else {
    r0 = rcp2(__fmul2_rn(t0, t0));
    r1 = rcp2(__fmul2_rn(t1, t1));
    r2 = rcp2(__fmul2_rn(t2, t2));
  }
  const float2 g0 = __ffma2_rn(c(5.0f / 18.0f), D2, __fmul2_rn(c(1.0f / 9.0f), D1));
  const float2 g1 = __ffma2_rn(c(2.0f / 3.0f), D3, __fmul2_rn(c(1.0f / 3.0f), D2));
  const float2 g2 = __ffma2_rn(c(2.0f / 3.0f), D3, __fmul2_rn(c(1.0f / 6.0f), D4));
  const float2 num = __ffma2_rn(r2, g2, __ffma2_rn(r1, g1, __fmul2_rn(r0, g0)));
  const float2 den = __ffma2_rn(c(1.0f / 3.0f), r0, __ffma2_rn(c(2.0f), r1, r2));
  return __ffma2_rn(num, rcp2(den), v0);
}

// weno5_cell for two components of one cell in the lanes of packed FP32x2
// operations (the arithmetic of weno5_pair: indicators scaled by 12/13,
// linear weights scaled by 10/3; z = 1: WENO5-Z as in weno5_cell).
__device__ __forceinline__ void weno5_cell_pair(float2 vm2, float2 vm1, float2 v0, float2 vp1, float2 vp2, float eps,
                                                float2& right, float2& left, int z = 0) {
  auto c = [](float x) { return make_float2(x, x); };
  const float2 m1 = c(-1.0f);
  const float2 D1 = __ffma2_rn(m1, vm1, vm2);
  const float2 D2 = __ffma2_rn(m1, vm1, v0);
  const float2 D3 = __ffma2_rn(m1, v0, vp1);
  const float2 D4 = __ffma2_rn(m1, vp2, vp1);
  const float2 d0 = __fadd2_rn(D2, D1), e0 = __ffma2_rn(c(3.0f), D2, D1);
  const float2 d1 = __ffma2_rn(m1, D2, D3), e1 = __fadd2_rn(D2, D3);
  const float2 d2 = __fadd2_rn(D3, D4), e2 = __ffma2_rn(c(3.0f), D3, D4);
  const float2 k3 = c(3.0f / 13.0f), ke = c(12.0f / 13.0f * eps);
  const float2 t0 = __ffma2_rn(d0, d0, __ffma2_rn(__fmul2_rn(k3, e0), e0, ke));
  const float2 t1 = __ffma2_rn(d1, d1, __ffma2_rn(__fmul2_rn(k3, e1), e1, ke));
  const float2 t2 = __ffma2_rn(d2, d2, __ffma2_rn(__fmul2_rn(k3, e2), e2, ke));
  float2 r0, r1, r2;
  if (z) {
    const float2 d02 = __ffma2_rn(m1, t2, t0);
    const float2 tau = make_float2(fabsf(d02.x), fabsf(d02.y));
    r0 = __fmul2_rn(__fadd2_rn(t0, tau), rcp2(t0));
    r1 = __fmul2_rn(__fadd2_rn(t1, tau), rcp2(t1));
    r2 = __fmul2_rn(__fadd2_rn(t2, tau), rcp2(t2));
  } else {
    r0 = rcp2(__fmul2_rn(t0, t0));
    r1 = rcp2(__fmul2_rn(t1, t1));
    r2 = rcp2(__fmul2_rn(t2, t2));
  }
  // right: v0 + (r0 g0 + r1 g1 + r2 g2) / (r0/3 + 2 r1 + r2)
  const float2 g0 = __ffma2_rn(c(5.0f / 18.0f), D2, __fmul2_rn(c(1.0f / 9.0f), D1));
  const float2 g1 = __ffma2_rn(c(2.0f / 3.0f), D3, __fmul2_rn(c(1.0f / 3.0f), D2));
  const float2 g2 = __ffma2_rn(c(2.0f / 3.0f), D3, __fmul2_rn(c(1.0f / 6.0f), D4));
  const float2 num = __ffma2_rn(r2, g2, __ffma2_rn(r1, g1, __fmul2_rn(r0, g0)));
  const float2 den = __ffma2_rn(c(1.0f / 3.0f), r0, __ffma2_rn(c(2.0f), r1, r2));
  right = __ffma2_rn(num, rcp2(den), v0);
  // left: the mirrored stencil (r and D reversed and negated)
  const float2 h0 = __ffma2_rn(c(-5.0f / 18.0f), D3, __fmul2_rn(c(-1.0f / 9.0f), D4));
  const float2 h1 = __ffma2_rn(c(-2.0f / 3.0f), D2, __fmul2_rn(c(-1.0f / 3.0f), D3));
  const float2 h2 = __ffma2_rn(c(-2.0f / 3.0f), D2, __fmul2_rn(c(-1.0f / 6.0f), D1));
  const float2 numl = __ffma2_rn(r0, h2, __ffma2_rn(r1, h1, __fmul2_rn(r2, h0)));
  const float2 denl = __ffma2_rn(c(1.0f / 3.0f), r2, __ffma2_rn(c(2.0f), r1, r0));
  left = __ffma2_rn(numl, rcp2(denl), v0);
}

// weno5_cell_lean for two components of one cell in the lanes: 41 packed
// operations and 10 reciprocals where weno5_cell_pair takes 46 and 10.
__device__ __forceinline__ void weno5_cell_pair_lean(float2 vm2, float2 vm1, float2 v0, float2 vp1, float2 vp2,
                                                     float eps, float2& right, float2& left, int z = 0) {
  const float2 m1 = splat2(-1.0f), k = splat2(4.0f / 3.0f), ke = splat2(eps);
  const float2 D2 = __ffma2_rn(m1, vm1, v0), D3 = __ffma2_rn(m1, v0, vp1);
  const float2 d0 = __fadd2_rn(D2, __ffma2_rn(m1, vm1, vm2));
  const float2 d1 = __ffma2_rn(m1, D2, D3);
  const float2 d2 = __fadd2_rn(D3, __ffma2_rn(m1, vp2, vp1));
  const float2 q2 = __ffma2_rn(D2, D2, ke), q3 = __ffma2_rn(D3, D3, ke);
  const float2 t0 = __ffma2_rn(d0, __ffma2_rn(k, d0, D2), q2);
  const float2 t1 = __ffma2_rn(d1, __ffma2_rn(k, d1, D2), q2);
  const float2 t2 = __ffma2_rn(d2, __ffma2_rn(k, d2, D3), q3);
  float2 r0, r1, r2;
  // approximate reciprocals (t_k^2 >= eps^2 > 0, so the sums are > 0)
  if (z) {
    const float2 d02 = __ffma2_rn(m1, t2, t0);
    const float2 tau = make_float2(fabsf(d02.x), fabsf(d02.y));
    r0 = __fmul2_rn(__fadd2_rn(t0, tau), rcp2(t0));
    r1 = __fmul2_rn(__fadd2_rn(t1, tau), rcp2(t1));
    r2 = __fmul2_rn(__fadd2_rn(t2, tau), rcp2(t2));
  } else {
    r0 = rcp2(__fmul2_rn(t0, t0));
    r1 = rcp2(__fmul2_rn(t1, t1));
    r2 = rcp2(__fmul2_rn(t2, t2));
  }
  const float2 a1 = __fmul2_rn(splat2(6.0f), r1), a2 = __fmul2_rn(splat2(3.0f), r2), c0 = __fmul2_rn(splat2(3.0f), r0);
  const float2 h2 = __fmul2_rn(splat2(0.5f), D2), h3 = __fmul2_rn(splat2(0.5f), D3);
  const float2 third = splat2(1.0f / 3.0f), sixth = splat2(1.0f / 6.0f);
  const float2 nr = __ffma2_rn(a2, __ffma2_rn(sixth, d2, h3),
                               __ffma2_rn(a1, __ffma2_rn(third, d1, h2), __fmul2_rn(r0, __ffma2_rn(third, d0, h2))));
  const float2 nl = __ffma2_rn(r2, __ffma2_rn(third, d2, h3),
                               __ffma2_rn(a1, __ffma2_rn(sixth, d1, h2), __fmul2_rn(c0, __ffma2_rn(sixth, d0, h2))));
  const float2 Sr = __fadd2_rn(__fadd2_rn(r0, a1), a2), Sl = __fadd2_rn(__fadd2_rn(c0, a1), r2);
  right = __ffma2_rn(nr, rcp2(Sr), v0);
  left = __ffma2_rn(nl, make_float2(trcp(-Sl.x), trcp(-Sl.y)), v0);
}

// WENO3-JS (Table 2): value at x_{i+1/2} biased to the left from
// v[i-1], v[i], v[i+1]: q0 = (3 v[i] - v[i-1]) / 2, q1 = (v[i] + v[i+1]) / 2,
// beta0 = (v[i] - v[i-1])^2, beta1 = (v[i+1] - v[i])^2,
// alpha_k = d_k / (eps + beta_k)^2, d = (1/3, 2/3), omega_k = alpha_k / sum.
// FP64: in differences, v0 + (r0 e0 + 2 r1 e1) / (2 (r0 + 2 r1)) with e0, e1 and
// r_k as below: one reciprocal, and its rounding only scales the correction.
template <typename T>
JF_HD T weno3(T vm1, T v0, T vp1, T eps) {
  if constexpr (sizeof(T) == 8) {
    const T e0 = v0 - vm1, e1 = vp1 - v0, t0 = eps + e0 * e0, t1 = eps + e1 * e1;
    const T r0 = t1 * t1, r1 = t0 * t0;
    return fma(fma(T(0.5), r0 * e0, r1 * e1), trcp(fma(T(2), r1, r0)), v0);
  } else {
    const T q0 = T(0.5) * (T(3) * v0 - vm1), q1 = T(0.5) * (v0 + vp1);
    const T t0 = eps + (v0 - vm1) * (v0 - vm1), t1 = eps + (vp1 - v0) * (vp1 - v0);
    const T a0 = T(1.0 / 3.0) * trcp(t0 * t0), a1 = T(2.0 / 3.0) * trcp(t1 * t1);
    return (a0 * q0 + a1 * q1) * trcp(a0 + a1);
  }
}
// Both WENO3-JS face values of one cell from v[j-1..j+1] (as weno5_cell):
// with e0 = v0 - v[-1], e1 = v[1] - v0 and r_k = 1 / (eps + e_k^2)^2,
//   right = v0 + (r0 e0 + 2 r1 e1) / (2 (r0 + 2 r1)),
//   left  = v0 - (r1 e1 + 2 r0 e0) / (2 (r1 + 2 r0)).
// FP64: r0, r1 scaled by (eps + e0^2)^2 (eps + e1^2)^2.  A reciprocal for each
// value: one for both, of the product of the sums, takes an operation more and
// ends the range of eps and of the jumps at the fourth root of FP64's.
template <typename T>
JF_HD void weno3_cell(T vm1, T v0, T vp1, T eps, T& right, T& left) {
  const T e0 = v0 - vm1, e1 = vp1 - v0;
  const T t0 = eps + e0 * e0, t1 = eps + e1 * e1;
  T r0, r1;
  if constexpr (sizeof(T) == 8) {
    r0 = t1 * t1;
    r1 = t0 * t0;
  } else {
    r0 = trcp(t0 * t0);
    r1 = trcp(t1 * t1);
  }
  const T Sr = r0 + T(2) * r1, Sl = r1 + T(2) * r0;
  const T p0 = r0 * e0, p1 = r1 * e1;
  if constexpr (sizeof(T) == 8) {  // halves taken in the numerators
    right = fma(fma(T(0.5), p0, p1), trcp(Sr), v0);
    left = fma(-fma(T(0.5), p1, p0), trcp(Sl), v0);
  } else {
    const T nr = p0 + T(2) * p1, nl = p1 + T(2) * p0;
    right = v0 + nr * trcp(T(2) * Sr);
    left = v0 - nl * trcp(T(2) * Sl);
  }
}
__device__ __forceinline__ float2 weno3_pair(float2 vm1, float2 v0, float2 vp1, float eps) {
  return make_float2(weno3(vm1.x, v0.x, vp1.x, eps), weno3(vm1.y, v0.y, vp1.y, eps));
}

// Signal speeds S_L <= S_R at a face along axis D (Table 2 estimates), from
// the side states W = [rho, u, v, w, p] and their total energies E, 1/rho
// and sound speeds c:
//   Einfeldt (1988): Roe averages (weights sqrt(rho)) u~, H~ (H = (E + p)/rho),
//     c~ = sqrt((gamma - 1)(H~ - |u~|^2/2)); S_L = min(u_L - c_L, u~ - c~),
//     S_R = max(u_R + c_R, u~ + c~);
//   Davis (1988): S_L = min(u_L - c_L, u_R - c_R), S_R = max(u_L + c_L, u_R + c_R);
//   Toro (1994): PVRS pressure p* = max(0, (p_L + p_R)/2 - (u_R - u_L)(rho_L + rho_R)(c_L + c_R)/8);
//     q_K = 1 if p* <= p_K else sqrt(1 + (gamma + 1)/(2 gamma)(p*/p_K - 1));
//     S_L = u_L - c_L q_L, S_R = u_R + c_R q_R.
// q = sqrt(rho_R / rho_L), read by Einfeldt's estimate.
template <typename T, int D>
JF_HD void signal_speeds(const T WL[5], const T WR[5], const Gas<T>& g, int speeds, T EL, T ER, T irL, T irR, T q,
                         T cL, T cR, T& SL, T& SR) {
  const T rL = WL[0], rR = WR[0], pL = WL[4], pR = WR[4];
  const T unL = WL[1 + D], unR = WR[1 + D];
  if (speeds == 1) {
    SL = tmin(unL - cL, unR - cR);
    SR = tmax(unL + cL, unR + cR);
  } else if (speeds == 2) {
    const T ps = tmax(T(0), T(0.5) * (pL + pR) - T(0.125) * (unR - unL) * (rL + rR) * (cL + cR));
    const T k = (g.gamma + T(1)) * trcp(T(2) * g.gamma);
    const T qL = ps > pL ? tsqrt(T(1) + k * (ps * trcp(pL) - T(1))) : T(1);
    const T qR = ps > pR ? tsqrt(T(1) + k * (ps * trcp(pR) - T(1))) : T(1);
    SL = unL - cL * qL;
    SR = unR + cR * qR;
  } else {
    // Roe weights sqrt(rho_K) / (sqrt(rho_L) + sqrt(rho_R)):
    // w_L = 1 / (1 + q), w_R = q w_L
    const T wL = trcp(T(1) + q), wR = q * wL;
    const T HL = (EL + pL) * irL, HR = (ER + pR) * irR;
    const T u0 = wL * WL[1] + wR * WR[1];
    const T u1 = wL * WL[2] + wR * WR[2];
    const T u2 = wL * WL[3] + wR * WR[3];
    const T Ht = wL * HL + wR * HR;
    const T ct = tsqrt(g.gm1 * (Ht - T(0.5) * (u0 * u0 + u1 * u1 + u2 * u2)));
    const T un_t = D == 0 ? u0 : (D == 1 ? u1 : u2);
    SL = tmin(unL - cL, un_t - ct);
    SR = tmax(unR + cR, un_t + ct);
  }
}

template <typename T>
JF_HD T total_energy(const T W[5], const Gas<T>& g) {
  return W[4] * g.inv_gm1 + T(0.5) * W[0] * (W[1] * W[1] + W[2] * W[2] + W[3] * W[3]);
}

// Total energy, 1/rho and sound speed of one side.
template <typename T>
JF_HD void side_state(const T W[5], const Gas<T>& g, T& E, T& ir, T& c) {
  E = W[4] * g.inv_gm1 + T(0.5) * W[0] * (W[1] * W[1] + W[2] * W[2] + W[3] * W[3]);
  ir = trcp(W[0]);
  c = tsqrt(g.gamma * W[4] * ir);
}

// Both sides' E, 1/rho and c, and q = sqrt(rho_R / rho_L); FP64 forms the two
// reciprocals from one, 1/rho_L = rho_R / (rho_L rho_R) and the converse.
template <typename T>
JF_HD void side_states(const T WL[5], const T WR[5], const Gas<T>& g, T& EL, T& ER, T& irL, T& irR, T& q, T& cL,
                       T& cR) {
  if constexpr (sizeof(T) == 8) {
    const T inv = trcp(WL[0] * WR[0]);
    irL = WR[0] * inv;
    irR = WL[0] * inv;
    EL = WL[4] * g.inv_gm1 + T(0.5) * WL[0] * (WL[1] * WL[1] + WL[2] * WL[2] + WL[3] * WL[3]);
    ER = WR[4] * g.inv_gm1 + T(0.5) * WR[0] * (WR[1] * WR[1] + WR[2] * WR[2] + WR[3] * WR[3]);
    cL = tsqrt(g.gamma * WL[4] * irL);
    cR = tsqrt(g.gamma * WR[4] * irR);
  } else {
    side_state(WL, g, EL, irL, cL);
    side_state(WR, g, ER, irR, cR);
  }
  q = tsqrt(WR[0] * irL);
}

// Physical flux along D and conservative state of one side.
template <typename T, int D>
JF_HD void side_flux(const T W[5], T E, T F[5], T U[5]) {
  const T un = W[1 + D], mass = W[0] * un;
  F[0] = mass;
  F[1] = mass * W[1];
  F[2] = mass * W[2];
  F[3] = mass * W[3];
  F[1 + D] += W[4];
  F[4] = un * (E + W[4]);
  U[0] = W[0];
  U[1] = W[0] * W[1];
  U[2] = W[0] * W[2];
  U[3] = W[0] * W[3];
  U[4] = E;
}

// The flux of hllc<double, D> with Einfeldt's speeds in about 100 FP64
// operations (116 by the general path): the Roe sound speed from
//   c~^2 = w_L c_L^2 + w_R c_R^2 + (gamma - 1)/2 w_L w_R |u_R - u_L|^2
// (the identity behind H~ - |u~|^2/2, without its cancellation), the energy of
// the chosen side only, and signs read from the high words.
// x >= 0 by 32-bit compares: +0 to +inf, or -0; false for the NaN of an invalid
// side, whose face must not pass as the regular flux of the other one.
JF_HD bool not_negative(double x) {
#ifdef __CUDA_ARCH__
  const unsigned hi = (unsigned)__double2hiint(x);
  return hi <= 0x7ff00000u || hi == 0x80000000u;
#else
  return x >= 0.0;
#endif
}
// S_K (U*_K - U_K) added to the mass, normal momentum and energy flux of a star
// side (FP64), from theta = (S* - u_n) / (S - S*): with fac = rho (1 + theta)
//   fac - rho = rho theta,  fac S* - rho u_n = rho (S* - u_n + theta S*),
//   fac (E/rho + (S* - u_n)(S* + p/m)) - E = E theta + fac (S* - u_n)(S* + p/m),
// without the cancellation of the left-hand sides and without 1/rho (a
// contact at rest keeps its fluxes 0, p, 0 exactly).  1 / (S - S*) and p / m from
// one reciprocal.
JF_HD void hllc_star(double r, double p, double un, double E, double mass, double S, double m, double Ss, double& F0,
                     double& Fn, double& F4) {
  const double d = S - Ss, x = trcp(m * d), k = Ss - un, theta = k * (m * x), rt = r * theta;
  F0 = fma(S, rt, mass);
  Fn = fma(S * r, fma(theta, Ss, k), Fn);
  F4 = fma(S, fma(E, theta, (r + rt) * k * fma(p * d, x, Ss)), F4);
}
template <int D>
JF_HD void hllc_einfeldt(const double WL[5], const double WR[5], const Gas<double>& g, double F[5]) {
  const double rL = WL[0], rR = WR[0], pL = WL[4], pR = WR[4], unL = WL[1 + D], unR = WR[1 + D];
  const double rr = rL * rR, gi = g.gamma * trcp(rr), q = rR * trsqrt(rr);  // q = sqrt(rho_R / rho_L)
  const double aL = pL * rR * gi, aR = pR * rL * gi;                       // c_K^2
  const double wL = trcp(1.0 + q), wR = q * wL;
  const double du = WR[1] - WL[1], dv = WR[2] - WL[2], dw = WR[3] - WL[3];
  const double jump = fma(dw, dw, fma(dv, dv, du * du));
  const double ct = tsqrt(fma(0.5 * g.gm1 * (wL * wR), jump, fma(wR, aR, wL * aL)));
  const double ut = fma(wR, unR, wL * unL);
  const double SL = tmin(unL - tsqrt(aL), ut - ct), SR = tmax(unR + tsqrt(aR), ut + ct);
  const double mL = rL * (SL - unL), mR = rR * (SR - unR);
  const double Ss = fma(-mR, unR, fma(mL, unL, pR - pL)) * trcp(mL - mR);
  const bool sup = not_negative(SL), left = sup || not_negative(Ss);
  const bool star = left ? !sup : SR > 0.0;
  const double r = left ? rL : rR, p = left ? pL : pR, un = left ? unL : unR;
  const double w0 = left ? WL[1] : WR[1], w1 = left ? WL[2] : WR[2], w2 = left ? WL[3] : WR[3];
  const double S = left ? SL : SR, m = left ? mL : mR;
  const double E = fma(0.5 * r, fma(w2, w2, fma(w1, w1, w0 * w0)), p * g.inv_gm1);
  const double mass = r * un;
  double F0 = mass, Fn = fma(mass, un, p), F4 = un * (E + p);
  if (star) hllc_star(r, p, un, E, mass, S, m, Ss, F0, Fn, F4);
  F[0] = F0;
  F[1] = F0 * w0;
  F[2] = F0 * w1;
  F[3] = F0 * w2;
  F[1 + D] = Fn;
  F[4] = F4;
}

// HLLC flux along axis D from the reconstructed primitive states
// W = [rho, u, v, w, p] left (WL) and right (WR) of the face; `speeds` picks
// the signal speed estimate (0 Einfeldt, 1 Davis, 2 Toro).
//   U_K, F_K                conservative state and physical flux of side K
//   S_L, S_R                signal speeds of the selected estimate
//   S*  = (p_R - p_L + rho_L u_L (S_L - u_L) - rho_R u_R (S_R - u_R))
//         / (rho_L (S_L - u_L) - rho_R (S_R - u_R))
//   F*_K = F_K + S_K (U*_K - U_K),
//   U*_K = rho_K (S_K - u_K)/(S_K - S*) [1, S*, u_t, E_K/rho_K + (S* - u_K)(S* + p_K/(rho_K (S_K - u_K)))]
template <typename T, int D>
JF_HD void hllc(const T WL[5], const T WR[5], const Gas<T>& g, T F[5], int speeds = 0) {
  if constexpr (sizeof(T) == 8) {
    if (speeds == 0) return hllc_einfeldt<D>(WL, WR, g, F);
  }
  const T rL = WL[0], rR = WR[0], pL = WL[4], pR = WR[4];
  const T unL = WL[1 + D], unR = WR[1 + D];
  // every division goes through a reciprocal (1/rho of each side shared)
  T EL, ER, irL, irR, q, cL, cR;
  side_states(WL, WR, g, EL, ER, irL, irR, q, cL, cR);
  T SL, SR;
  signal_speeds<T, D>(WL, WR, g, speeds, EL, ER, irL, irR, q, cL, cR, SL, SR);
  const T mL = rL * (SL - unL), mR = rR * (SR - unR);
  const T Ss = (pR - pL + mL * unL - mR * unR) * trcp(mL - mR);
  // side selection: F_L if 0 <= S_L; F*_L if S_L < 0 <= S*; F*_R if S* < 0 < S_R; F_R if S_R <= 0
  const bool left = (SL >= T(0)) || (Ss >= T(0));
  const bool star = left ? !(SL >= T(0)) : (SR > T(0));
  const T r = left ? rL : rR, p = left ? pL : pR, un = left ? unL : unR, E = left ? EL : ER;
  const T w0 = left ? WL[1] : WR[1], w1 = left ? WL[2] : WR[2], w2 = left ? WL[3] : WR[3];
  const T S = left ? SL : SR, m = left ? mL : mR;
  // physical flux F_K of the chosen side, plus S_K (U*_K - U_K) on a star
  // side.  Mass: r u_n + S (fac - r); a tangential momentum component is
  // (r u_n + S (fac - r)) u_t on either branch (its U* - U is (fac - r) u_t),
  // so it is the mass flux times u_t; normal momentum: r u_n^2 + p +
  // S (fac S* - r u_n); energy: u_n (E + p) + S (fac e* - E).
  const T mass = r * un;
  T F0 = mass, Fn = mass * un + p, F4 = un * (E + p);
  if (star) {
    // (m and S - S* are non-zero on a star side: S_L < u_L - c_L, S_L < 0 <= S*,
    // and the mirror image)
    if constexpr (sizeof(T) == 8) {
      hllc_star(r, p, un, E, mass, S, m, Ss, F0, Fn, F4);
    } else {
      const T ir = left ? irL : irR, fac = m * trcp(S - Ss), p_m = p * trcp(m);
      F0 = mass + S * (fac - r);
      Fn = Fn + S * (fac * Ss - mass);
      F4 = F4 + S * (fac * (E * ir + (Ss - un) * (Ss + p_m)) - E);
    }
  }
  F[0] = F0;
  F[1] = F0 * w0;
  F[2] = F0 * w1;
  F[3] = F0 * w2;
  F[1 + D] = Fn;
  F[4] = F4;
}

// HLL flux (Harten, Lax, van Leer 1983): F_L if 0 <= S_L, F_R if S_R <= 0,
// else (S_R F_L - S_L F_R + S_L S_R (U_R - U_L)) / (S_R - S_L).
template <typename T, int D>
JF_HD void hll(const T WL[5], const T WR[5], const Gas<T>& g, T F[5], int speeds = 0) {
  T EL, ER, irL, irR, q, cL, cR;
  side_states(WL, WR, g, EL, ER, irL, irR, q, cL, cR);
  T SL, SR;
  signal_speeds<T, D>(WL, WR, g, speeds, EL, ER, irL, irR, q, cL, cR, SL, SR);
  T FL[5], FR[5], UL[5], UR[5];
  side_flux<T, D>(WL, EL, FL, UL);
  side_flux<T, D>(WR, ER, FR, UR);
  if (SL >= T(0)) {
#pragma unroll
    for (int q = 0; q < 5; ++q) F[q] = FL[q];
  } else if (SR <= T(0)) {
#pragma unroll
    for (int q = 0; q < 5; ++q) F[q] = FR[q];
  } else {
    const T inv = trcp(SR - SL);
#pragma unroll
    for (int q = 0; q < 5; ++q) F[q] = (SR * FL[q] - SL * FR[q] + SL * SR * (UR[q] - UL[q])) * inv;
  }
}

// Local Lax-Friedrichs (Rusanov): a = max(|u_L| + c_L, |u_R| + c_R),
// F = (F_L + F_R)/2 - a (U_R - U_L)/2.
template <typename T, int D>
JF_HD void rusanov(const T WL[5], const T WR[5], const Gas<T>& g, T F[5]) {
  T EL, ER, irL, irR, q, cL, cR;
  side_states(WL, WR, g, EL, ER, irL, irR, q, cL, cR);
  const T a = tmax(fabs(WL[1 + D]) + cL, fabs(WR[1 + D]) + cR);
  T FL[5], FR[5], UL[5], UR[5];
  side_flux<T, D>(WL, EL, FL, UL);
  side_flux<T, D>(WR, ER, FR, UR);
#pragma unroll
  for (int q = 0; q < 5; ++q) F[q] = T(0.5) * (FL[q] + FR[q]) - T(0.5) * a * (UR[q] - UL[q]);
}

template <typename T> JF_HD T texp(T x);
template <> JF_HD float texp<float>(float x) { return expf(x); }
template <> JF_HD double texp<double>(double x) { return exp(x); }
template <typename T> JF_HD T tlog(T x);
template <> JF_HD float tlog<float>(float x) { return logf(x); }
template <> JF_HD double tlog<double>(double x) { return log(x); }

// alpha = exp(NN(x)) of the Rusanov-NN flux; th: the network parameters.
// Not inlined: one copy of the ~2200 multiply-adds serves every face
// direction, and its 64 hidden values do not add to the register pressure
// of the tile code around the call.
#if defined(__CUDACC__) || defined(JF_HOST_FLOAT4)  // (a host build that has float4)
// Four consecutive network parameters (or hidden-row values) from a 16-byte
// aligned address: every weight row of the parameter layout starts at a
// multiple of 4 elements, and the kernels place the parameters at a 16-byte
// aligned offset of their shared memory.
__device__ __forceinline__ void ld4(const float* p, float o[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  o[0] = q.x; o[1] = q.y; o[2] = q.z; o[3] = q.w;
}
__device__ __forceinline__ void ld4(const double* p, double o[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
  o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
#endif

template <typename T>
__host__ __device__ __noinline__ T nn_alpha(const T* th, const T x[4]) {
  const T* W1 = th;
  const T* b1 = W1 + NN_HIDDEN * 4;
  const T* W2 = b1 + NN_HIDDEN;
  const T* b2 = W2 + NN_HIDDEN * NN_HIDDEN;
  const T* W3 = b2 + NN_HIDDEN;
  const T* b3 = W3 + NN_HIDDEN * NN_HIDDEN;
  const T* W4 = b3 + NN_HIDDEN;
  const T b4 = W4[NN_HIDDEN];
  T h1[NN_HIDDEN], h2[NN_HIDDEN];
#ifdef __CUDA_ARCH__
  // device: th is 16-byte aligned shared memory; weight rows read four at a time
#pragma unroll
  for (int i = 0; i < NN_HIDDEN; ++i) {
    T w[4];
    ld4(W1 + 4 * i, w);
    h1[i] = tmax(T(0), b1[i] + w[0] * x[0] + w[1] * x[1] + w[2] * x[2] + w[3] * x[3]);
  }
#pragma unroll
  for (int i = 0; i < NN_HIDDEN; ++i) {
    T z = b2[i];
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4) {
      T w[4];
      ld4(W2 + NN_HIDDEN * i + j, w);
      z += w[0] * h1[j] + w[1] * h1[j + 1] + w[2] * h1[j + 2] + w[3] * h1[j + 3];
    }
    h2[i] = tmax(T(0), z);
  }
  T out = b4;
#pragma unroll 4
  for (int i = 0; i < NN_HIDDEN; ++i) {
    T z = b3[i];
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; j += 4) {
      T w[4];
      ld4(W3 + NN_HIDDEN * i + j, w);
      z += w[0] * h2[j] + w[1] * h2[j + 1] + w[2] * h2[j + 2] + w[3] * h2[j + 3];
    }
    out += W4[i] * tmax(T(0), z);
  }
#else
#pragma unroll
  for (int i = 0; i < NN_HIDDEN; ++i) {
    const T z = b1[i] + W1[4 * i] * x[0] + W1[4 * i + 1] * x[1] + W1[4 * i + 2] * x[2] + W1[4 * i + 3] * x[3];
    h1[i] = tmax(T(0), z);
  }
#pragma unroll
  for (int i = 0; i < NN_HIDDEN; ++i) {
    T z = b2[i];
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; ++j) z += W2[NN_HIDDEN * i + j] * h1[j];
    h2[i] = tmax(T(0), z);
  }
  T out = b4;
#pragma unroll 4
  for (int i = 0; i < NN_HIDDEN; ++i) {
    T z = b3[i];
#pragma unroll
    for (int j = 0; j < NN_HIDDEN; ++j) z += W3[NN_HIDDEN * i + j] * h2[j];
    out += W4[i] * tmax(T(0), z);
  }
#endif
  return texp(out);
}

// The transposed weights for nn_alpha_pair: W1 [4][NN_HIDDEN], then W2 and W3
// [NN_HIDDEN][NN_TPITCH], a row per input.
constexpr int NN_TPITCH = NN_HIDDEN + 4, NN_T2 = 4 * NN_HIDDEN, NN_T3 = NN_T2 + NN_HIDDEN * NN_TPITCH,
              NN_TELEMS = NN_T3 + NN_HIDDEN * NN_TPITCH;
// Where parameter i goes in them (-1: a bias or W4, not there).
JF_HD int nn_transposed(int i) {
  constexpr int W2 = 5 * NN_HIDDEN, W3 = W2 + (NN_HIDDEN + 1) * NN_HIDDEN;
  if (i < 4 * NN_HIDDEN) return i % 4 * NN_HIDDEN + i / 4;
  if (i >= W2 && i < W2 + NN_HIDDEN * NN_HIDDEN) return NN_T2 + (i - W2) % NN_HIDDEN * NN_TPITCH + (i - W2) / NN_HIDDEN;
  if (i >= W3 && i < W3 + NN_HIDDEN * NN_HIDDEN) return NN_T3 + (i - W3) % NN_HIDDEN * NN_TPITCH + (i - W3) / NN_HIDDEN;
  return -1;
}

#if defined(__CUDACC__) || defined(JF_HOST_FLOAT4)
// nn_alpha of two faces (the lanes of x), from the parameters th and the
// transposed weights tt (16-byte aligned): per face the operations of nn_alpha
// in its order, so the same bits.  Two outputs of a layer share a packed FP32x2
// operation, so that four weights of one load serve both faces: with every
// weight stored twice and the faces in the lanes a pass took twice the loads, and
// the stage of 20 boxes of 32^2 18.6 us in the place of 16.4.
// A layer runs over its inputs four at a time (from `row`, this thread's
// NN_PAIR_ROW values of shared memory) with all its outputs in registers:
// independent sums, and a loop whose code stays in the instruction cache.
constexpr int NN_PAIR_ROW = 2 * NN_HIDDEN + 4;  // 17 x 16 bytes: conflict-free 16-byte accesses
static __device__ __noinline__ float2 nn_alpha_pair(const float* th, const float* tt, const float2 x[4], float* row) {
  const float* b1 = th + NN_HIDDEN * 4;
  const float* b2 = b1 + NN_HIDDEN + NN_HIDDEN * NN_HIDDEN;
  const float* b3 = b2 + NN_HIDDEN + NN_HIDDEN * NN_HIDDEN;
  const float* W4 = b3 + NN_HIDDEN;
  auto ld2 = [](const float* p, float2& a, float2& b) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    a = make_float2(q.x, q.y);
    b = make_float2(q.z, q.w);
  };
  auto splat = [](float v) { return make_float2(v, v); };
  float2 zx[NN_HIDDEN / 2], zy[NN_HIDDEN / 2];
  auto bias = [&](const float* b) {
#pragma unroll
    for (int i = 0; i < NN_HIDDEN / 2; i += 2) {
      ld2(b + 2 * i, zx[i], zx[i + 1]);
      zy[i] = zx[i];
      zy[i + 1] = zx[i + 1];
    }
  };
  auto keep = [&]() {  // the layer's values to this thread's row
#pragma unroll
    for (int i = 0; i < NN_HIDDEN / 2; i += 2) {
      *reinterpret_cast<float4*>(row + 2 * i) = make_float4(tmax(0.0f, zx[i].x), tmax(0.0f, zx[i].y),
                                                            tmax(0.0f, zx[i + 1].x), tmax(0.0f, zx[i + 1].y));
      *reinterpret_cast<float4*>(row + NN_HIDDEN + 2 * i) = make_float4(tmax(0.0f, zy[i].x), tmax(0.0f, zy[i].y),
                                                                        tmax(0.0f, zy[i + 1].x), tmax(0.0f, zy[i + 1].y));
    }
  };
  auto layer = [&](const float* W, const float* b) {
    bias(b);
#pragma unroll 1
    for (int j = 0; j < NN_HIDDEN; j += 4) {
      float hx[4], hy[4];
      ld4(row + j, hx);
      ld4(row + NN_HIDDEN + j, hy);
#pragma unroll
      for (int i = 0; i < NN_HIDDEN / 2; i += 2) {
        float2 w[4][2];
#pragma unroll
        for (int m = 0; m < 4; ++m) ld2(W + (j + m) * NN_TPITCH + 2 * i, w[m][0], w[m][1]);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          auto sum = [&](const float h[4]) {
            return __ffma2_rn(w[3][q], splat(h[3]), __ffma2_rn(w[2][q], splat(h[2]),
                                                               __ffma2_rn(w[0][q], splat(h[0]), __fmul2_rn(w[1][q], splat(h[1])))));
          };
          zx[i + q] = __fadd2_rn(zx[i + q], sum(hx));
          zy[i + q] = __fadd2_rn(zy[i + q], sum(hy));
        }
      }
    }
  };
  bias(b1);
#pragma unroll
  for (int i = 0; i < NN_HIDDEN / 2; i += 2)
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      float2 w[2];
      ld2(tt + NN_HIDDEN * m + 2 * i, w[0], w[1]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        zx[i + q] = __ffma2_rn(w[q], splat(x[m].x), zx[i + q]);
        zy[i + q] = __ffma2_rn(w[q], splat(x[m].y), zy[i + q]);
      }
    }
  keep();
  layer(tt + NN_T2, b2);
  keep();
  layer(tt + NN_T3, b3);
  float ox = W4[NN_HIDDEN], oy = ox;
#pragma unroll
  for (int i = 0; i < NN_HIDDEN; ++i) {
    const float w = W4[i];
    ox = fmaf(w, tmax(0.0f, i & 1 ? zx[i / 2].y : zx[i / 2].x), ox);
    oy = fmaf(w, tmax(0.0f, i & 1 ? zy[i / 2].y : zy[i / 2].x), oy);
  }
  return make_float2(texp(ox), texp(oy));
}
#else
constexpr int NN_PAIR_ROW = 0;  // host: face by face, no hidden rows
inline float2 nn_alpha_pair(const float* th, const float*, const float2 x[4], float*) {
  float a[4], b[4];
  for (int m = 0; m < 4; ++m) { a[m] = x[m].x; b[m] = x[m].y; }
  return make_float2(nn_alpha(th, a), nn_alpha(th, b));
}
#endif

// Network inputs of the Rusanov-NN flux at a face along D (Section 7.4):
// |u_R - u_L|, (u_L + u_R)/2, (c_L + c_R)/2, |s_R - s_L| with u the normal
// velocity and s = ln(p / rho^gamma) / (gamma - 1).
template <typename T, int D>
JF_HD void nn_inputs(const T WL[5], const T WR[5], const Gas<T>& g, T cL, T cR, T x[4]) {
  const T sL = (tlog(WL[4]) - g.gamma * tlog(WL[0])) * g.inv_gm1;
  const T sR = (tlog(WR[4]) - g.gamma * tlog(WR[0])) * g.inv_gm1;
  x[0] = fabs(WR[1 + D] - WL[1 + D]);
  x[1] = T(0.5) * (WL[1 + D] + WR[1 + D]);
  x[2] = T(0.5) * (cL + cR);
  x[3] = fabs(sR - sL);
}

// Rusanov-NN (Section 7.4, Eq. (Rusanov)): F = (F_L + F_R)/2 - alpha (U_R - U_L)/2
// with alpha = exp(NN(x)).
template <typename T, int D>
JF_HD void rusanov_nn(const T WL[5], const T WR[5], const Gas<T>& g, T F[5], T a) {
  const T EL = total_energy(WL, g), ER = total_energy(WR, g);
  T FL[5], FR[5], UL[5], UR[5];
  side_flux<T, D>(WL, EL, FL, UL);
  side_flux<T, D>(WR, ER, FR, UR);
#pragma unroll
  for (int q = 0; q < 5; ++q) F[q] = T(0.5) * (FL[q] + FR[q]) - T(0.5) * a * (UR[q] - UL[q]);
}

// The network's inputs of a face from its states.
template <typename T, int D>
JF_HD void nn_face_inputs(const T WL[5], const T WR[5], const Gas<T>& g, T x[4]) {
  T EL, ER, irL, irR, q, cL, cR;
  side_states(WL, WR, g, EL, ER, irL, irR, q, cL, cR);
  nn_inputs<T, D>(WL, WR, g, cL, cR, x);
}
template <typename T, int D>
JF_HD void rusanov_nn(const T WL[5], const T WR[5], const Gas<T>& g, T F[5]) {
  T x[4];
  nn_face_inputs<T, D>(WL, WR, g, x);
  rusanov_nn<T, D>(WL, WR, g, F, nn_alpha(g.nn, x));
}

// The Riemann solver and signal speeds of the configuration (uniform branch;
// the default kernels call hllc with Einfeldt speeds directly).
template <typename T, int D>
JF_HD void riemann_flux(const T WL[5], const T WR[5], const Gas<T>& g, T F[5]) {
  if (g.flux == 1) hll<T, D>(WL, WR, g, F, g.speeds);
  else if (g.flux == 2) rusanov<T, D>(WL, WR, g, F);
  else hllc<T, D>(WL, WR, g, F, g.speeds);
}

// Section 3.4 stencils (without the 1/h factor).
template <typename T>
JF_HD T df4(T a, T b, T c, T d) {  // face derivative * h
  return (a - T(27) * b + T(27) * c - d) * (T(1) / T(24));
}
template <typename T>
JF_HD T dc4(T m2, T m1, T p1, T p2) {  // cell-centre derivative * h
  return (m2 - T(8) * m1 + T(8) * p1 - p2) * (T(1) / T(12));
}
template <typename T>
JF_HD T rc4(T a, T b, T c, T d) {  // face interpolation
  return (-a + T(9) * b + T(9) * c - d) * (T(1) / T(16));
}

}  // namespace jf
